"""The compaction kernel at the sizes where its counting can go wrong: block lengths that a 16-byte or 4-byte mask
load straddles, mask arrays that do not start on a 16-byte boundary, window sizes around a chunk and a whole
256-position scan, and windows whose chunks take several scans. Small heads, so that a wrong row shows in the outputs:
every position is compared with a float64 evaluation of the same step.
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


# (n_seq, n_slots, block_len, offset of the mask array, masked share)
WINDOWS = [(1, 1, 1, 0, 1.0), (3, 5, 1, 0, 0.5), (5, 3, 3, 1, 0.5), (7, 2, 5, 0, 0.7), (2, 2, 7, 3, 1.0),
           (8, 1, 8, 0, 0.3), (4, 3, 18, 8, 0.4), (9, 3, 20, 0, 0.5), (13, 2, 63, 0, 0.6), (16, 4, 64, 16, 0.5),
           (16384, 2, 5, 0, 0.02), (4096, 1, 64, 1, 0.01)]


@pytest.mark.parametrize("head", ["f32", "bf16", "e4m3"])
@pytest.mark.parametrize("window", WINDOWS)
def test_every_position_is_the_right_row(window, head):
    n_seq, n_slots, L, off, share = window
    d, V, tau = 32, 320, [0.02, 0.2]
    g = torch.Generator(device="cuda").manual_seed(n_seq * 64 + L)
    P = n_seq * n_slots * L
    dt = torch.float32 if head == "f32" else torch.bfloat16
    hidden = (4 * torch.randn(P, d, generator=g, device="cuda")).to(dt)
    w = torch.randn(V, d, generator=g, device="cuda") / d ** 0.5
    scale = None
    if head == "e4m3":
        scale = torch.full((V,), 1 / 64, device="cuda")
        w = (64 * w).to(torch.float8_e4m3fn)
        w64 = w.double() / 64
    else:
        w = w.to(dt)
        w64 = w.double()
    mask = torch.zeros(P + off, dtype=torch.uint8, device="cuda")[off:]
    mask[torch.rand(P, generator=g, device="cuda") < share] = 255  # any nonzero value means masked
    flags = torch.randint(0, 4, (n_seq * n_slots,), generator=g, device="cuda", dtype=torch.uint8)
    tok, conf, commit, counts = bdc.commit_step(hidden, w, mask, flags, n_seq, n_slots, L, tau, weight_scale=scale,
                                                counts=True)
    assert bdc.bd_get_device_status() == 0
    live = (mask != 0) & ((flags & 1) != 0).repeat_interleave(L)
    assert torch.equal(tok >= 0, live) and torch.equal(conf > 0, live)
    pos = torch.nonzero(live).view(-1)
    if pos.numel():
        logit = hidden[pos].double() @ w64.t()
        top = logit.topk(2, dim=1).values
        ref = (top[:, 0] - logit.logsumexp(1)).exp()
        # logits of at most ~40 in float32: 32 products, errors under 32 * 2^-24 * 40 < 1e-4
        assert float((conf[pos].double() - ref).abs().max()) < 2e-4
        sure = top[:, 0] - top[:, 1] > 2e-4
        assert torch.equal(tok[pos][sure].long(), logit.argmax(1)[sure])
    bits = torch.stack([(commit >> k) & 1 for k in range(2)], 1).view(n_seq, -1, 2).sum(1).int()
    assert torch.equal(counts, bits)
