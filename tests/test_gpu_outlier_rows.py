"""Rows whose largest element dwarfs the rest, as large models' activations have them. The outlier meets a head column
of zeros, so it adds nothing to a logit or to the rounding of its sum: what moves is what the row's other elements lost
when the row was encoded. Compared with float64, for every head format: verification multiplies the rows as they are,
so its error stays that of a float32 sum; the commit step on an E4M3 head holds two E4M3 terms per element, whose
bound is stated; on an NVFP4 head float16 scaled by a power of two, exact here.
"""

import pytest
import torch

pytestmark = pytest.mark.gpu

bdc = pytest.importorskip("paper_2609_33887_gb300")

E2M1 = (0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


def make(head, R, V, d, top, seed):
    """(hidden, weight, scale, the logits in float64, the head in float64) with element 7 of every row at `top`."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.randn(V, d, generator=g, device="cuda") / d ** 0.5
    scale = None
    if head == "nvfp4":
        code = torch.randint(0, 16, (V, d), generator=g, device="cuda")
        code[:, 7] = 0
        nb = (d // 16 + 15) // 16 * 16
        bs = torch.randint(40, 60, (V, nb), generator=g, device="cuda", dtype=torch.int32).to(torch.uint8)
        scale = (torch.rand(V, generator=g, device="cuda") + 0.5) / d ** 0.5
        val = torch.tensor(E2M1, device="cuda", dtype=torch.float64)[code & 7] * (1 - 2 * (code >> 3).double())
        block = bs[:, :d // 16].view(torch.float8_e4m3fn).double().repeat_interleave(16, 1)
        w64 = val * block * scale[:, None].double()
        w = bdc.Nvfp4Head((code[:, 0::2] | (code[:, 1::2] << 4)).to(torch.uint8), bs, d)
    else:
        w[:, 7] = 0
        if head == "e4m3":
            scale = w.abs().amax(1) / 448
            w = (w / scale[:, None]).to(torch.float8_e4m3fn)
            w64 = w.double() * scale[:, None].double()
        else:
            w = w.bfloat16()
            w64 = w.double()
    h = torch.randn(R, d, generator=g, device="cuda")
    # half of the rows point at a head row: probabilities of every size, where they move most
    tok = torch.randint(0, V, (R,), generator=g, device="cuda")
    push = torch.linspace(0, 12, R, device="cuda")[torch.randperm(R, generator=g, device="cuda")]
    wr = w64[tok].float()
    h += push[:, None] * wr / (wr * wr).sum(1, keepdim=True)
    h[:, 7] = top
    h = h.bfloat16()
    return h, w, scale, h.double() @ w64.t(), w64


# Verification: float32 sums of at most 1024 products with logits of at most ~20, as in the tests of token groups
P_TOL, H_TOL, GAP = 4e-4, 4e-3, 1e-3


@pytest.mark.parametrize("top", [1.0, 100.0, 1000.0, 10000.0])
@pytest.mark.parametrize("head", ["bf16", "e4m3", "nvfp4"])
def test_verify_step(head, top):
    n_req, D, V, d, eps = 60, 4, 4096, 1024, [0.3, 0.05]
    R = n_req * (D + 1)
    h, w, scale, logit, _ = make(head, R, V, d, top, 11)
    best = logit.argmax(1)
    rows = torch.arange(R, device="cuda").view(n_req, D + 1)[:, :D].reshape(-1)
    draft = best[rows].int()
    draft[1::3] = (draft[1::3] + 1) % V
    out = bdc.verify_step(h, w, draft, n_req, D, eps, weight_scale=scale)
    assert bdc.bd_get_device_status() == 0
    logp = logit.log_softmax(1)
    p = logp[rows].gather(1, draft.long()[:, None])[:, 0].exp()
    assert float((out["p_draft"][rows].double() - p).abs().max()) < P_TOL
    assert float((out["entropy"].double() + (logp.exp() * logp).sum(1)).abs().max()) < H_TOL
    two = logit.topk(2, dim=1).values
    sure = two[:, 0] - two[:, 1] > GAP
    assert torch.equal(out["tokens"][sure].long(), best[sure])
    lossless = (out["accept"][rows] < 0)  # bit 31
    assert torch.equal(lossless[sure[rows]], (draft.long() == best[rows])[sure[rows]])


@pytest.mark.parametrize("head", ["bf16", "e4m3", "nvfp4"])
def test_verify_step_with_a_broken_row(head):
    # an infinite activation leaves infinite logits (NaN where the head holds a
    # zero): no positive probability, nothing accepted at any eps, and only there
    n_req, D, V, d, eps = 8, 4, 1000, 256, [0.3, 0.05]
    R = n_req * (D + 1)
    h, w, scale, logit, w64 = make(head, R, V, d, 1.0, 12)
    h[12, 9] = float("inf")
    assert float(w64[:, 9].abs().max()) > 0
    draft = logit.argmax(1).view(n_req, D + 1)[:, :D].int().reshape(-1).contiguous()
    out = bdc.verify_step(h, w, draft, n_req, D, eps, weight_scale=scale)
    assert bdc.bd_get_device_status() == 0
    assert not float(out["p_draft"][12]) > 0 and int(out["accept"][12]) & 3 == 0
    others = torch.arange(R, device="cuda") != 12
    assert torch.isfinite(out["p_draft"][others]).all() and torch.isfinite(out["entropy"][others]).all()


@pytest.mark.parametrize("top", [1.0, 100.0, 1000.0, 10000.0])
@pytest.mark.parametrize("head", ["bf16", "e4m3", "nvfp4"])
def test_commit_step(head, top):
    P, V, d = 300, 4096, 1024
    h, w, scale, logit, w64 = make(head, P, V, d, top, 13)
    ones = torch.ones(P, dtype=torch.uint8, device="cuda")
    tok, conf, _, _ = bdc.commit_step(h, w, ones, ones, P, 1, 1, [0.5], weight_scale=scale)
    assert bdc.bd_get_device_status() == 0
    # E4M3: an element below 2^-10 of the row's largest is held to within 2^-17 of it, so a
    # logit moves by at most 2^-17 max|h| times the sum of its head row's |w| (column 7 is 0)
    moved = 2.0 ** -17 * float(h.abs().max()) * float(w64.abs().sum(1).max()) if head == "e4m3" and top > 10 else 0.0
    # a probability moves by at most twice the logits' shift
    p = (logit.amax(1) - logit.logsumexp(1)).exp()
    assert float((conf.double() - p).abs().max()) < P_TOL + 2 * moved
    two = logit.topk(2, dim=1).values
    sure = two[:, 0] - two[:, 1] > GAP + 2 * moved
    assert torch.equal(tok[sure].long(), logit.argmax(1)[sure])
