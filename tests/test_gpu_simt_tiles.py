"""The float32 LM head at the edges of its tiles: row counts around its groups of 8 R rows, vocabularies around its
tiles of 32, 64, 112 and 128 entries, widths around its 16-column stages, row strides and base addresses with no more than the
4-byte alignment the entry points ask for, and a workspace without room for every runner's partials. Compared with a
float64 evaluation of every position.
"""

import pytest
import torch

pytestmark = pytest.mark.gpu

bdc = pytest.importorskip("paper_2609_33887_gb300")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


def strided(rows, cols, pad, g):
    """[rows, cols] float32 N(0, 1), row stride cols + pad, one element off the allocation's start."""
    buf = torch.randn(rows * (cols + pad) + 1, generator=g, device="cuda")[1:]
    return buf.view(rows, cols + pad)[:, :cols]


def check_step(h, w, N, V, mid, out, tol):
    tok, conf = out
    logit = h.double() @ w.double().t()
    if mid >= 0:
        logit[:, mid] = -float("inf")
    ref = (logit.amax(1) - logit.logsumexp(1)).exp()
    assert float((conf.double() - ref).abs().max()) < tol
    top = logit.topk(min(2, V), dim=1).values
    sure = top[:, 0] - top[:, -1] > 2 * tol
    assert torch.equal(tok[sure].long(), logit.argmax(1)[sure])


# float32 sums of at most 100 products with partial sums of up to ~20, whose rounding errors add up like a random walk
# (four standard deviations: 4 * sqrt(100) * 2^-24 * 20 = 5e-5 on a logit, at most as much on a probability); the
# base-2 exponential's 2^-22 and the sums over the vocabulary add less than 1e-5
TOL = 6e-5


@pytest.mark.parametrize("N", [1, 7, 8, 9, 33, 40, 63, 64, 65, 77, 129, 200])
@pytest.mark.parametrize("V,d,pad", [(5, 1, 0), (31, 15, 2), (33, 16, 0), (257, 17, 3), (4096, 100, 1),
                                     (39000, 20, 0), (40001, 33, 5), (9001, 100, 1), (9024, 20, 0),
                                     (17024, 16, 0), (17026, 33, 3), (19001, 15, 0), (19456, 20, 0)])
def test_commit_step(N, V, d, pad):
    g = torch.Generator(device="cuda").manual_seed(N * V + d)
    h, w = strided(N, d, pad, g), strided(V, d, pad, g) / max(1, d) ** 0.5 * 2
    w = torch.as_strided(w.contiguous(), (V, d), (d, 1)) if pad == 0 else w
    mask = torch.ones(N, dtype=torch.uint8, device="cuda")
    flags = torch.ones(N, dtype=torch.uint8, device="cuda")
    mid = V // 2 if V > 5 else -1
    tok, conf, _, _ = bdc.commit_step(h, w, mask, flags, N, 1, 1, [0.5], mask_token_id=mid)
    assert bdc.bd_get_device_status() == 0
    check_step(h, w, N, V, mid, (tok, conf), TOL)


@pytest.mark.parametrize("n_req", [1, 9, 13, 40])  # 5, 45, 65 and 200 rows
@pytest.mark.parametrize("V,d", [(33, 16), (4096, 100), (39000, 20), (19001, 33), (17024, 20)])
def test_verify_step(n_req, V, d):
    D, g = 4, torch.Generator(device="cuda").manual_seed(n_req + V)
    h, w = strided(n_req * (D + 1), d, 1, g), strided(V, d, 0, g) / d ** 0.5 * 2
    logit = h.double() @ w.double().t()
    draft = logit.argmax(1).view(n_req, D + 1)[:, :D].int().reshape(-1).contiguous()
    draft[1::2] = torch.randint(0, V, draft[1::2].shape, generator=g, device="cuda", dtype=torch.int32)
    out = bdc.verify_step(h, w, draft, n_req, D, [0.3])
    assert bdc.bd_get_device_status() == 0
    logp = logit.log_softmax(1)
    rows = torch.arange(n_req * (D + 1), device="cuda").view(n_req, D + 1)[:, :D].reshape(-1)
    p = logp[rows].gather(1, draft.long()[:, None])[:, 0].exp()
    assert float((out["p_draft"][rows].double() - p).abs().max()) < TOL
    assert float((out["entropy"].double() + (logp.exp() * logp).sum(1)).abs().max()) < 10 * TOL  # sums of p (l - max)


@pytest.mark.parametrize("head", ["bf16", "e4m3", "nvfp4"])
def test_other_heads_forced_onto_it(head):
    N, V, d = 45, 4001, 48
    g = torch.Generator(device="cuda").manual_seed(V)
    h = torch.randn(N, d, generator=g, device="cuda").bfloat16()
    scale = None
    if head == "nvfp4":
        codes = torch.randint(0, 256, (V, 32), generator=g, device="cuda", dtype=torch.int32).to(torch.uint8)
        bs = torch.randint(40, 60, (V, 16), generator=g, device="cuda", dtype=torch.int32).to(torch.uint8)
        w = bdc.Nvfp4Head(codes, bs, d)
        nib = torch.stack([codes & 15, codes >> 4], 2).view(V, -1)[:, :d].long()
        val = torch.tensor([0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0], device="cuda")[nib & 7] * (1 - 2 * (nib >> 3))
        w64 = val.double() * bs.view(torch.float8_e4m3fn).double().repeat_interleave(16, 1)[:, :d]
    else:
        w = (torch.randn(V, d, generator=g, device="cuda") / 4).to(
            torch.bfloat16 if head == "bf16" else torch.float8_e4m3fn)
        w64 = w.double()
        if head == "e4m3":
            scale = torch.rand(V, generator=g, device="cuda") + 0.5
            w64 = w64 * scale[:, None].double()
    ones = torch.ones(N, dtype=torch.uint8, device="cuda")
    tok, conf, _, _ = bdc.commit_step(h, w, ones, ones, N, 1, 1, [0.5], weight_scale=scale, variant=1)
    check_step(h, w64, N, V, -1, (tok, conf), TOL)


def test_scratch_that_holds_fewer_partials():
    # 8000 rows: the full set of runners' partials exceeds the allocation-free
    # call's 32 MiB array, fewer runners' fit
    N, V, d = 8000, 100000, 8
    g = torch.Generator(device="cuda").manual_seed(1)
    h, w = torch.randn(N, d, generator=g, device="cuda"), torch.randn(V, d, generator=g, device="cuda")
    ones = torch.ones(N, dtype=torch.uint8, device="cuda")
    args = (h, w, None, ones, ones, N, 1, 1, -1, [0.5])
    assert bdc.bd_workspace_size(*args) > 32 << 20
    out = [torch.empty(N, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.int32)]
    assert bdc.bdcommit.bd_commit_step_static(*args, *out) == 0
    tok, conf, commit, _ = bdc.commit_step(h, w, ones, ones, N, 1, 1, [0.5])
    torch.cuda.synchronize()
    assert torch.equal(out[0], tok) and float((out[1] - conf).abs().max()) < 1e-5


@pytest.mark.parametrize("V", [300, 5000, 9000, 40000])  # tiles of 32, 64, 112 and 128 entries
@pytest.mark.parametrize("N", [1, 40, 77])
def test_infinite_and_missing_logits(N, V):
    # a head row that overflows to one infinite logit takes all the probability
    # (two such rows half each, the lower id), one of -inf takes none, and a NaN
    # logit leaves no confidence: nothing commits without the fallback
    d = 16
    g = torch.Generator(device="cuda").manual_seed(V + N)
    h, w = torch.randn(N, d, generator=g, device="cuda"), torch.randn(V, d, generator=g, device="cuda")
    ones = torch.ones(N, dtype=torch.uint8, device="cuda")
    step = lambda h, w: bdc.commit_step(h, w, ones, ones, N, 1, 1, [0.25])  # noqa: E731
    h[:, 0], w[:, 0] = 1e30, 0.0
    top = (V * 2 // 3, V - 1)
    for n in (1, 2):
        w[top[-n:], 0] = 1e30  # 1e60: infinite in float32
        tok, conf, commit, _ = step(h, w)
        assert torch.equal(tok, torch.full_like(tok, top[-n])) and torch.equal(conf, torch.full_like(conf, 1 / n))
        assert torch.equal(commit, torch.ones_like(commit))
    w[top[0], 0] = w[top[1], 0] = -1e30
    tok, conf, _, _ = step(h, w)
    live = torch.ones(V, dtype=torch.bool, device="cuda")
    live[list(top)] = False
    assert live[tok.long()].all()
    logit = h[:, 1:].double() @ w[:, 1:].double().t()
    p = (logit[:, live].amax(1) - logit[:, live].logsumexp(1)).exp()
    assert float((conf.double() - p).abs().max()) < TOL
    w[V // 4, 3] = float("nan")
    _, conf, commit, _ = step(h, w)
    assert torch.isnan(conf).all() and not commit.any()
    assert bdc.bd_get_device_status() == 0


@pytest.mark.parametrize("V", [2500, 4096, 4800])
def test_units_of_narrow_tiles_run_at_once(V):
    # two CTAs with tiles of 32 entries fit an SM: the plan of a window that one
    # round could hold does not count on more (which staged the head once more
    # per group and left a second, partial round)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for P in (48, 77, 96, 150, 192):
        h, w = torch.zeros(P, 64, device="cuda"), torch.zeros(V, 64, device="cuda")
        ones = torch.ones(P, dtype=torch.uint8, device="cuda")
        hdr = bdc.bdcommit.bd_plan_header(h, w, None, ones, ones, P, 1, 1, -1, [0.5], P)
        band, parts = hdr[2], hdr[3]
        assert band * parts <= 2 * sms
