"""Quantised heads in windows above 8192 positions, where two kernels may serve them: whatever room the caller or the
allocation-free call's 32 MiB array leaves for one of them is enough, and the results are those of the step. Compared
with a float64 evaluation of every position.
"""

import pytest
import torch

pytestmark = pytest.mark.gpu

bdc = pytest.importorskip("paper_2609_33887_gb300")
B = bdc.bdcommit

E2M1 = (0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


def nvfp4(V, d, g):
    """(head the kernels can read as stored, row scale, the head in float64)."""
    codes = torch.randint(0, 256, (V, d // 2), generator=g, device="cuda", dtype=torch.int32).to(torch.uint8)
    nb = d // 16
    bs = torch.randint(40, 60, (V, (nb + 15) // 16 * 16), generator=g, device="cuda", dtype=torch.int32).to(torch.uint8)
    scale = (torch.rand(V, generator=g, device="cuda") + 0.5) / d ** 0.5
    nib = torch.stack([codes & 15, codes >> 4], 2).view(V, -1)
    val = torch.tensor(E2M1, device="cuda", dtype=torch.float64)[(nib & 7).long()] * (1 - 2 * (nib >> 3).double())
    block = bs[:, :nb].view(torch.float8_e4m3fn).double().repeat_interleave(16, 1)
    return bdc.Nvfp4Head(codes, bs, d), scale, val * block * scale[:, None].double()


def aligned(nbytes):
    ws = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    return ws[(-ws.data_ptr()) % 256:][:nbytes]


def top(h, w64):
    """Per row: the largest probability, the argmax, the gap to the next logit."""
    out = []
    for r in range(0, len(h), 2048):
        l = h[r:r + 2048].double() @ w64.t()
        t = l.topk(2, dim=1)
        out.append(((t.values[:, 0] - l.logsumexp(1)).exp(), t.indices[:, 0], t.values[:, 0] - t.values[:, 1]))
    return [torch.cat(x) for x in zip(*out)]


def check(tok, conf, want):
    p, a, gap = want
    # logits of at most ~40, sums of 128 products in float32: errors under 128 * 2^-24 * 40 = 3e-4
    assert float((conf.double() - p).abs().max()) < 6e-4
    assert torch.equal(tok[gap > 1e-3].long(), a[gap > 1e-3])


def test_commit_step(monkeypatch):
    V, d = 19456, 128
    g = torch.Generator(device="cuda").manual_seed(0)
    w, scale, w64 = nvfp4(V, d, g)
    for P in (9000, 16384, 16400):
        h = torch.randn(P, d, generator=g, device="cuda").bfloat16()
        ones = torch.ones(P, dtype=torch.uint8, device="cuda")
        args = (h, w, scale, ones, ones, P, 1, 1, -1, [0.5])
        want = top(h, w64)
        out = [torch.empty(P, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.int32)]
        assert B.bd_commit_step_static(*args, *out) == 0
        assert B.bd_static_device_status() == 0
        check(*out[:2], want)
        for line in ("8192", "1000000"):  # the room of the one-CTA kernel, and of the pair kernel
            monkeypatch.setenv("BD_PAIR_MAX_P", line)
            size = bdc.bd_workspace_size(*args)
            monkeypatch.delenv("BD_PAIR_MAX_P")
            assert B.bd_commit_step_ex(*args, *out, workspace=aligned(size)) == 0
            assert bdc.bd_get_device_status() == 0
            check(*out[:2], want)
            short = min(size, bdc.bd_workspace_size(*args)) // 2
            assert B.bd_commit_step_ex(*args, *out, workspace=aligned(short)) == B.BD_ERR_WORKSPACE


@pytest.mark.parametrize("V", [256, 5000])
def test_verify_step(V, monkeypatch):
    d, D, n_req = 128, 1, 4400
    R = n_req * (D + 1)
    g = torch.Generator(device="cuda").manual_seed(V)
    w, scale, w64 = nvfp4(V, d, g)
    h = torch.randn(R, d, generator=g, device="cuda").bfloat16()
    p, a, gap = top(h, w64)
    draft = a.view(n_req, D + 1)[:, :D].int().reshape(-1).contiguous()
    for line in ("8192", "1000000"):
        monkeypatch.setenv("BD_PAIR_MAX_P", line)
        size = bdc.bd_verify_workspace_size(h, w, scale, draft, n_req, D, [0.3])
        monkeypatch.delenv("BD_PAIR_MAX_P")
        out = bdc.verify_step(h, w, draft, n_req, D, [0.3], weight_scale=scale, workspace=aligned(size))
        assert bdc.bd_get_device_status() == 0
        rows = torch.arange(0, R, D + 1, device="cuda")
        check(out["tokens"][rows], out["p_draft"][rows], (p[rows], a[rows], gap[rows]))


def test_w8a8_in_the_documented_workspace():
    # bd_workspace_size covers W8A8 too: above 256 MiB of two-term rows the plain
    # step takes clusters, W8A8 rows of half the bytes single pairs with more partials
    P, V, d, N = 131100, 40000, 1024, 300
    g = torch.Generator(device="cuda").manual_seed(3)
    h = torch.randn(P, d, generator=g, device="cuda", dtype=torch.bfloat16)
    w = torch.randn(V, d, generator=g, device="cuda") / d ** 0.5
    scale = w.abs().amax(1) / 448
    w = (w / scale[:, None]).to(torch.float8_e4m3fn)
    mask = torch.zeros(P, dtype=torch.uint8, device="cuda")
    mask[torch.randperm(P, generator=g, device="cuda")[:N]] = 1
    flags = torch.ones(P, dtype=torch.uint8, device="cuda")
    args = (h, w, scale, mask, flags, P, 1, 1, -1, [0.5])
    outs = []
    for ws in (None, aligned(bdc.bd_workspace_size(*args))):
        out = [torch.empty(P, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.int32)]
        assert B.bd_commit_step_ex(*args, *out, workspace=ws, flags=B.BD_EXEC_FP8_ACTIVATIONS) == 0
        assert bdc.bd_get_device_status() == 0
        outs.append(out)
    assert torch.equal(outs[0][0], outs[1][0]) and int((outs[0][0] >= 0).sum()) == N
    assert float((outs[0][1] - outs[1][1]).abs().max()) < 1e-5  # the same float32 sums, grouped by fewer parts
