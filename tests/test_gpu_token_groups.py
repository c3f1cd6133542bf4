"""Windows around one token group (256 compacted rows), where the clusters' layout is chosen on the device: the two
pairs share token rows for a single group and head tiles for two; and around the group sizes of heads decoded in the
kernel (at most 192 rows, with four, three or two operand stages in flight). Every position is compared with a float64
evaluation, over vocabularies of one, three (an odd last pair of v-tiles) and many v-tiles, and with workspaces that
hold the partial slots of both layouts or only of the second.
"""

import pytest
import torch

pytestmark = pytest.mark.gpu

bdc = pytest.importorskip("paper_2609_33887_gb300")
B = bdc.bdcommit


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


def make(head, P, V, d, seed):
    """(hidden, weight, scale, the float64 logits the step computes)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    h = (3 * torch.randn(P, d, generator=g, device="cuda")).bfloat16()
    w = torch.randn(V, d, generator=g, device="cuda") / d ** 0.5
    h64 = h.double()
    if head == "w8a8":
        amax = h.float().abs().amax(1, keepdim=True)
        top = torch.full_like(amax, 448.0)
        h64 = (h.float() * (top / amax)).to(torch.float8_e4m3fn).double() * (amax / top).double()
    if head == "bf16":
        w = w.bfloat16()
        return h, w, None, h64 @ w.double().t()
    if head == "nvfp4":
        pad = (-((d + 15) // 16)) % 16  # 16-byte aligned rows of codes and block scales
        codes = torch.randint(0, 256, (V, (d + 31) // 32 * 16), generator=g, device="cuda", dtype=torch.int32)
        bs = torch.randint(40, 60, (V, (d + 15) // 16 + pad), generator=g, device="cuda", dtype=torch.int32)
        scale = (torch.rand(V, generator=g, device="cuda") + 0.5) / d ** 0.5
        nib = torch.stack([codes & 15, codes >> 4], 2).view(V, -1)[:, :d]
        val = torch.tensor([0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0], device="cuda")[(nib & 7).long()] * (1 - 2 * (nib >> 3))
        bs = bs.to(torch.uint8)
        block = bs.view(torch.float8_e4m3fn).double().repeat_interleave(16, 1)[:, :d]
        w64 = val.double() * block * scale[:, None].double()
        return h, bdc.Nvfp4Head(codes.to(torch.uint8), bs, d), scale, h64 @ w64.t()
    scale = w.abs().amax(1) / 448
    w = (w / scale[:, None]).to(torch.float8_e4m3fn)
    return h, w, scale, h64 @ (w.double() * scale[:, None].double()).t()


@pytest.mark.parametrize("N", [1, 33, 255, 256, 257, 300])
@pytest.mark.parametrize("V", [200, 700, 19001])
@pytest.mark.parametrize("head", ["bf16", "e4m3", "w8a8"])
def test_commit_step(head, V, N, monkeypatch):
    n_seq, L, d, mid = 8, 64, 336, 5
    P = n_seq * L
    h, w, scale, logit = make(head, P, V, d, N)
    logit[:, mid] = -float("inf")
    mask = torch.zeros(P, dtype=torch.uint8, device="cuda")
    mask[torch.randperm(P, generator=torch.Generator(device="cuda").manual_seed(V), device="cuda")[:N]] = 1
    flags = torch.full((n_seq,), 3, dtype=torch.uint8, device="cuda")
    args = (h, w, scale, mask, flags, n_seq, 1, L, mid, [0.5])
    fp8 = B.BD_EXEC_FP8_ACTIVATIONS if head == "w8a8" else 0
    full = bdc.bd_workspace_size(*args)
    monkeypatch.setenv("BD_PAIR_SHARE", "0")
    least = bdc.bd_workspace_size(*args)  # partial slots for shared head tiles only
    monkeypatch.delenv("BD_PAIR_SHARE")
    assert least <= full
    for size in (full, least):
        ws = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
        ws = ws[(-ws.data_ptr()) % 256:][:size]
        tok, conf, commit = (torch.empty(P, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.int32))
        assert bdc.bd_commit_step_ex(*args, tok, conf, commit, workspace=ws, flags=fp8) == 0
        assert bdc.bd_get_device_status() == 0
        live = mask != 0
        assert torch.equal(tok >= 0, live)
        top = logit[live].topk(2, dim=1).values
        ref = (top[:, 0] - logit[live].logsumexp(1)).exp()
        # logits of at most ~20: float32 accumulation of 336 products errs by well under 336 * 2^-24 * 20 = 4e-4
        assert float((conf[live].double() - ref).abs().max()) < 4e-4
        sure = top[:, 0] - top[:, 1] > 8e-4
        assert torch.equal(tok[live][sure].long(), logit[live].argmax(1)[sure])


@pytest.mark.parametrize("N", [1, 32, 33, 96, 97, 128, 129, 160, 161, 192, 193, 300, 385, 9001])
@pytest.mark.parametrize("V,d", [(200, 336), (5001, 64), (19001, 640), (700, 1056)])
@pytest.mark.parametrize("head", ["nvfp4", "e4m3"])
def test_head_decoded_in_the_kernel(head, V, d, N, monkeypatch):
    monkeypatch.setenv("BD_E4M3_SPLIT", "0")
    h, w, scale, logit = make(head, N, V, d, N)
    ones = torch.ones(N, dtype=torch.uint8, device="cuda")
    tok, conf, _, _ = bdc.commit_step(h, w, ones, ones, N, 1, 1, [0.5], weight_scale=scale)
    assert bdc.bd_get_device_status() == 0
    top = logit.topk(2, dim=1).values
    # as above, with logits of at most ~40 and 1056 products
    assert float((conf.double() - (top[:, 0] - logit.logsumexp(1)).exp()).abs().max()) < 2e-3
    sure = top[:, 0] - top[:, 1] > 4e-3
    assert torch.equal(tok[sure].long(), logit.argmax(1)[sure])


@pytest.mark.parametrize("n_req", [1, 38, 51, 52, 60])  # 5, 190, 255, 260 and 300 rows
@pytest.mark.parametrize("V", [200, 700, 19001])
@pytest.mark.parametrize("head", ["bf16", "e4m3", "nvfp4"])
def test_verify_step(head, V, n_req):
    D, d, eps = 4, 336, [0.3, 0.05]
    R = n_req * (D + 1)
    h, w, scale, logit = make(head, R, V, d, V)
    g = torch.Generator(device="cuda").manual_seed(n_req)
    best = logit.argmax(1).view(n_req, D + 1)[:, :D]
    other = torch.randint(0, V, best.shape, generator=g, device="cuda")
    draft = torch.where(torch.rand(best.shape, generator=g, device="cuda") < 0.5, best, other).int().reshape(-1)
    draft[0] = V  # outside the vocabulary: probability 0
    out = bdc.verify_step(h, w, draft, n_req, D, eps, weight_scale=scale)
    assert bdc.bd_get_device_status() == 0
    logp = logit.log_softmax(1)
    ent = -(logp.exp() * logp).sum(1)
    rows = torch.arange(R, device="cuda").view(n_req, D + 1)[:, :D].reshape(-1)
    p = logp[rows].gather(1, draft.clamp(max=V - 1).long()[:, None])[:, 0].exp()
    p[0] = 0
    # as above; the entropy sums p (l - max) over the vocabulary: twice the logits' error
    assert float((out["p_draft"][rows].double() - p).abs().max()) < 4e-4
    assert float((out["entropy"].double() - ent).abs().max()) < 2e-3
    bar = torch.stack([torch.minimum(torch.full_like(ent, e), e ** 0.5 * (-ent).exp()) for e in eps], 1)[rows]
    bits = torch.stack([(out["accept"][rows] >> k) & 1 for k in range(2)], 1) != 0
    clear = (p[:, None] - bar).abs() > 4e-3
    assert torch.equal(bits[clear], (p[:, None] > bar)[clear])


def test_verify_with_the_workspace_of_rows_read_in_place(monkeypatch):
    # verification on an E4M3 head reads its rows in place (the head is decoded
    # in the kernel), whatever room there is beyond the partial slots
    n_req, D, d, V = 6, 4, 336, 700
    h, w, scale, logit = make("e4m3", n_req * (D + 1), V, d, 3)
    draft = logit.argmax(1).view(n_req, D + 1)[:, :D].int().reshape(-1).contiguous()
    monkeypatch.setenv("BD_E4M3_SPLIT", "0")
    least = bdc.bd_verify_workspace_size(h, w, scale, draft, n_req, D, [0.3])
    monkeypatch.delenv("BD_E4M3_SPLIT")
    want = bdc.verify_step(h, w, draft, n_req, D, [0.3], weight_scale=scale)
    for size in (least, least + 64 * 1024):
        ws = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
        ws = ws[(-ws.data_ptr()) % 256:][:size]
        got = bdc.verify_step(h, w, draft, n_req, D, [0.3], weight_scale=scale, workspace=ws)
        assert torch.equal(got["tokens"], want["tokens"]) and torch.equal(got["accepted"], want["accepted"])
        assert float((got["p_draft"] - want["p_draft"]).abs().max()) < 4e-4


def test_verify_with_the_workspace_of_a_decoded_copy(monkeypatch):
    # the head decoded to a bf16 copy, with room beside it for the slots of
    # shared head tiles only
    n_req, D, d, V = 60, 4, 336, 200
    h, w, scale, logit = make("e4m3", n_req * (D + 1), V, d, 5)
    draft = logit.argmax(1).view(n_req, D + 1)[:, :D].int().reshape(-1).contiguous()
    want = bdc.verify_step(h, w, draft, n_req, D, [0.3], weight_scale=scale)
    monkeypatch.setenv("BD_FUSED_DECODE", "0")
    monkeypatch.setenv("BD_E4M3_SPLIT", "0")
    monkeypatch.setenv("BD_PAIR_MC", "2")
    least = bdc.bd_verify_workspace_size(h, w, scale, draft, n_req, D, [0.3])
    monkeypatch.delenv("BD_E4M3_SPLIT")
    monkeypatch.delenv("BD_PAIR_MC")
    ws = torch.empty(least + 256, dtype=torch.uint8, device="cuda")
    ws = ws[(-ws.data_ptr()) % 256:][:least]
    got = bdc.verify_step(h, w, draft, n_req, D, [0.3], weight_scale=scale, workspace=ws)
    assert torch.equal(got["tokens"], want["tokens"]) and torch.equal(got["accepted"], want["accepted"])
    assert float((got["p_draft"] - want["p_draft"]).abs().max()) < 4e-4
