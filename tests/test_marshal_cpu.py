"""The packed arguments of a call hold what the C structures hold: every field against a ctypes structure built on its
own, for each head format and grid length, and the values the packed form leaves to ctypes."""

import ctypes
import math

import pytest
import torch

import paper_2609_33887_gb300.bdcommit as B


def fields(s):
    return [getattr(s, n) for n, *_ in s._fields_ if n not in ("tau", "eps")]


def heads():
    w = torch.zeros(6, 32)
    yield w, None
    yield w.bfloat16()[:, :24], None
    yield w.to(torch.float8_e4m3fn), torch.ones(6)
    yield B.Nvfp4Head(torch.zeros(6, 16, dtype=torch.uint8), torch.zeros(6, 4, dtype=torch.uint8)[:, :2], 31), None


@pytest.mark.parametrize("T", [1, 4, 31, 32])
@pytest.mark.parametrize("head", range(4))
def test_step_arguments(head, T):
    weight, scale = list(heads())[head]
    hidden = torch.zeros(10, 48, dtype=torch.bfloat16)[:, :32]
    mask, flags = torch.ones(10, dtype=torch.uint8), torch.ones(5, dtype=torch.uint8)
    tau = [k / 7 for k in range(T)]
    hf, wf = B._hidden_fields(hidden), B._weight_fields(weight, scale)
    mf = B._mask_state_fields(mask, flags, 5, 1, 2, 3)
    ef = (11, 12, 13, 14, 15, 16, 3, 1)
    buf, base = B._pack(B._STEP, B._StepArgs, tau, (*hf, *wf[:5], wf[5] or 0, wf[6] or 0, wf[7], *mf), ef)
    a = B._StepArgs.from_buffer(buf)
    assert ctypes.addressof(a) == base
    assert fields(a.h) == fields(B.make_hidden(hidden))
    assert fields(a.w) == fields(B.make_weight(weight, scale))
    assert fields(a.ms) == fields(B.make_mask_state(mask, flags, 5, 1, 2, 3))
    assert fields(a.ex) == list(ef)
    grid, _ = B.make_tau_grid(tau)
    assert a.grid.T == grid.T == T
    assert [a.grid.tau[k] for k in range(T)] == [grid.tau[k] for k in range(T)]


def test_verify_arguments():
    hidden, (weight, scale) = torch.zeros(10, 32, dtype=torch.bfloat16), list(heads())[2]
    hf, wf = B._hidden_fields(hidden), B._weight_fields(weight, scale)
    buf, _ = B._pack(B._VERIFY, B._VerifyArgs, [0.5, 0.25], (*hf, *wf[:5], wf[5], 0, wf[7], 2, 4, 77), (1, 2, 3, 4, 5, 6, 0, 0))
    a = B._VerifyArgs.from_buffer(buf)
    assert fields(a.h) == fields(B.make_hidden(hidden)) and fields(a.w) == fields(B.make_weight(weight, scale))
    assert (a.dr.n_req, a.dr.n_draft, a.dr.draft) == (2, 4, 77)
    assert a.grid.E == 2 and [a.grid.eps[0], a.grid.eps[1]] == [0.5, 0.25] and fields(a.ex) == [1, 2, 3, 4, 5, 6, 0, 0]


@pytest.mark.parametrize("tau,last", [([0.5] * 33, 0), (["x"], 0), ([0.5], 2 ** 40)])
def test_left_to_ctypes(tau, last):
    before = (*[0] * 13, 1, 1, 1, -1, 0, 0)
    assert B._pack(B._STEP, B._StepArgs, tau, before, (0, 0, 0, 0, 0, 0, 0, last)) is None


def test_nan_and_infinite_thresholds_are_packed():
    before = (*[0] * 13, 1, 1, 1, -1, 0, 0)
    tau = [math.nan, math.inf, 1e300]  # a value beyond float32 becomes infinite, as in a ctypes array
    buf, _ = B._pack(B._STEP, B._StepArgs, tau, before, (0,) * 8)
    v = B._StepArgs.from_buffer(buf).values
    assert math.isnan(v[0]) and v[1] == math.inf and v[2] == (ctypes.c_float * 1)(1e300)[0] == math.inf
