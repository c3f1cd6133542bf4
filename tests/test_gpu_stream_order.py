"""Calls queued one behind another on a stream, with no host wait and no other kernel between them. The first kernel of
a call is let in while the last kernel of the call before it still runs, and that kernel may write what the first one
reads: the commit sweep moves the window on in place, and calls that share a workspace write the same arrays. Each
queued run is compared, word for word, with the same calls made one at a time.
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


def head(kind, V, d, g):
    """(weight, its row scale, the hidden rows' type) of a random head of that format."""
    w = torch.randn(V, d, generator=g, device="cuda") / d ** 0.5
    if kind == "e4m3":
        scale = w.abs().amax(1) / 448
        return (w / scale[:, None]).to(torch.float8_e4m3fn), scale, torch.bfloat16
    dt = torch.float32 if kind == "f32" else torch.bfloat16
    return w.to(dt), None, dt


def aligned(nbytes):
    ws = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    return ws[(-ws.data_ptr()) % 256:][:nbytes]


# from one CTA of each kernel to windows whose compaction takes many CTAs while the sweep still writes its last ones
@pytest.mark.parametrize("n_seq,n_slots,L", [(1, 2, 8), (16, 4, 32), (256, 8, 32)])
@pytest.mark.parametrize("kind", ["f32", "bf16", "e4m3"])
def test_step_then_sweep_in_place(kind, n_seq, n_slots, L):
    P, V, d, steps, tau = n_seq * n_slots * L, 500, 64, 24, [0.1, 0.3]
    g = torch.Generator(device="cuda").manual_seed(P)
    w, scale, dt = head(kind, V, d, g)
    hidden = [(4 * torch.randn(P, d, generator=g, device="cuda")).to(dt) for _ in range(3)]
    mask0 = (torch.rand(P, generator=g, device="cuda") < 0.7).to(torch.uint8)
    flags0 = torch.full((n_seq * n_slots,), bdc.BD_BLOCK_ACTIVE, dtype=torch.uint8, device="cuda")
    flags0[::n_slots] |= bdc.BD_BLOCK_FALLBACK_ELIGIBLE
    args = (hidden[0], w, scale, mask0, flags0, n_seq, n_slots, L, -1, tau)
    ws = aligned(bdc.bd_workspace_size(*args))
    options = bdc.BD_SWEEP_ADMIT | bdc.BD_SWEEP_ELIGIBLE_OLDEST

    def loop(wait):
        window = torch.full((P,), 7, dtype=torch.int32, device="cuda")
        mask, flags = mask0.clone(), flags0.clone()
        out = [tuple(torch.empty(P, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.int32))
               + tuple(torch.zeros(n, dtype=torch.int32, device="cuda") for n in (P, n_seq, n_seq))
               for _ in range(steps)]
        torch.cuda.synchronize()
        for i, (tok, conf, commit, cache, ncom, nres) in enumerate(out):
            assert B.bd_commit_step_ex(hidden[i % 3], w, scale, mask, flags, n_seq, n_slots, L, -1, tau, tok, conf,
                                       commit, workspace=ws) == 0
            if wait:
                torch.cuda.synchronize()
            assert B.bd_commit_sweep(window, mask, flags, n_seq, n_slots, L, -1, tok, commit, i % 2, options, cache,
                                     ncom, nres) == 0
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert bdc.bd_get_device_status() == 0
        return [window, mask, flags] + [t for o in out for t in o]

    want = loop(True)
    assert sum(int(o.sum()) for o in want[7::6]) > 0  # blocks were committed on the way
    for _ in range(3):
        for a, b in zip(loop(False), want):
            assert torch.equal(a, b)


@pytest.mark.parametrize("kind", ["bf16", "e4m3"])
def test_verifications_that_share_a_workspace(kind):
    V, d, D, eps = 700, 336, 4, [0.3, 0.05]
    g = torch.Generator(device="cuda").manual_seed(1)
    w, scale, dt = head(kind, V, d, g)
    calls = []
    for i in range(24):
        n_req = (1, 60, 13)[i % 3]
        hidden = (3 * torch.randn(n_req * (D + 1), d, generator=g, device="cuda")).to(dt)
        draft = torch.randint(0, V, (n_req * D,), generator=g, device="cuda", dtype=torch.int32)
        calls.append((hidden, w, scale, draft, n_req, D, eps))
    ws = aligned(max(bdc.bd_verify_workspace_size(*c) for c in calls))

    def run(wait):
        out = []
        for hidden, _, _, draft, n_req, _, _ in calls:
            R = n_req * (D + 1)
            out.append([torch.empty(R, dtype=t, device="cuda")
                        for t in (torch.int32, torch.float32, torch.float32, torch.int32)]
                       + [torch.empty(n_req, len(eps) + 1, dtype=torch.int32, device="cuda")])
        torch.cuda.synchronize()
        for c, o in zip(calls, out):
            assert B.bd_verify_step(*c, *o, workspace=ws) == 0
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert bdc.bd_get_device_status() == 0
        return [t for o in out for t in o]

    want = run(True)
    for _ in range(3):
        for a, b in zip(run(False), want):
            assert torch.equal(a, b)
