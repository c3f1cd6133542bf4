"""Which calls take clusters of two CTA pairs, whose loads are multicast: commit steps and verifications of a run on one
GPU. A rank's shard of a vocabulary-parallel head (lmhead_partials) runs single pairs whatever the environment asks
for, and BD_PAIR_MC=1 keeps every call on them. The kernel's last template argument tells the two apart.
"""

import ctypes
import re

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


def multicast(call, path):
    """Whether the LM-head launches of `call` may multicast, from the kernels' names in a captured graph."""
    call()  # the workspace and the module's first load stay outside the capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        call()
    with open("/proc/self/maps") as f:
        runtime = next(line.split()[-1] for line in f if "libcudart.so" in line)
    print_dot = ctypes.CDLL(runtime).cudaGraphDebugDotPrint
    assert print_dot(ctypes.c_void_p(g.raw_cuda_graph()), str(path).encode(), ctypes.c_uint(1)) == 0  # 1: verbose
    with open(path, errors="replace") as f:
        text = f.read()
    found = {m.group(1) for m in re.finditer(r"lmhead_pair_kernelILi\d+ELb[01]ELb([01])EE", text)}
    assert len(found) == 1, text[:4000]
    return found == {"1"}


def window(kind, P, V, d):
    g = torch.Generator(device="cuda").manual_seed(P)
    h = torch.randn(P, d, generator=g, device="cuda").bfloat16()
    w = torch.randn(V, d, generator=g, device="cuda") / d ** 0.5
    scale = None
    if kind == "e4m3":
        scale = w.abs().amax(1) / 448
        w = (w / scale[:, None]).to(torch.float8_e4m3fn)
    else:
        w = w.bfloat16()
    ones = torch.ones(P, dtype=torch.uint8, device="cuda")
    return h, w, scale, ones


@pytest.mark.parametrize("P", [64, 512])
@pytest.mark.parametrize("kind", ["bf16", "e4m3"])
def test_clusters_per_call(kind, P, monkeypatch, tmp_path):
    V, d = 3000, 64
    h, w, scale, ones = window(kind, P, V, d)
    step = lambda: bdc.commit_step(h, w, ones, ones, P, 1, 1, [0.5], weight_scale=scale)  # noqa: E731
    shard = lambda: bdc.lmhead_partials(h, w, 0, ones, ones, P, 1, 1, shard_scale=scale)  # noqa: E731
    monkeypatch.delenv("BD_PAIR_MC", raising=False)
    assert multicast(step, tmp_path / "graph.dot")
    assert not multicast(shard, tmp_path / "graph.dot")
    monkeypatch.setenv("BD_PAIR_MC", "2")
    monkeypatch.setenv("BD_PAIR_SPILL", "1")
    assert not multicast(shard, tmp_path / "graph.dot")
    monkeypatch.setenv("BD_PAIR_MC", "1")
    assert not multicast(step, tmp_path / "graph.dot")
    assert not multicast(shard, tmp_path / "graph.dot")
    assert bdc.bd_get_device_status() == 0


@pytest.mark.parametrize("P", [64, 512])
@pytest.mark.parametrize("kind", ["bf16", "e4m3"])
def test_shard_in_the_workspace_of_the_documented_size(kind, P, monkeypatch):
    # bd_workspace_size counts the partial slots of the step's own layout, and
    # of head tiles shared by clusters (what it counted before token rows were)
    V, d = 40000, 64
    h, w, scale, ones = window(kind, P, V, d)
    args = (h, w, scale, ones, ones, P, 1, 1, -1, [0.5])
    sizes = [bdc.bd_workspace_size(*args)]
    monkeypatch.setenv("BD_PAIR_SHARE", "0")
    sizes.append(bdc.bd_workspace_size(*args))
    monkeypatch.delenv("BD_PAIR_SHARE")
    want = bdc.lmhead_partials(h, w, 7, ones, ones, P, 1, 1, shard_scale=scale)
    for size in sizes:
        ws = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
        ws = ws[(-ws.data_ptr()) % 256:][:size]
        got = bdc.lmhead_partials(h, w, 7, ones, ones, P, 1, 1, shard_scale=scale, workspace=ws)
        assert bdc.bd_get_device_status() == 0
        assert torch.equal(got[0], want[0]) and torch.equal(got[2], want[2])
        assert float((got[1] / want[1] - 1).abs().max()) < 1e-5  # the same float32 sums, grouped by fewer parts
