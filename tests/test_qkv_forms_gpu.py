"""nystra_qkv's two forms: the fused kernel (the C entry point) and the
projection and attention by turns over a workspace, in one chunk and in several
(a ragged last one, per-window score biases, streams), and the calls at the
edges of the rule that picks between them."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2506_08520_gb300 import binding, workloads
from tests.parity import ROUND, fused_qkv, per_unit_rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2506_08520_gb300 import build
    build.build()


CASES = [  # windows, heads, N, d, m, pooling, bias (None, "heads", "windows"), dtype
    (5, 2, 1024, 16, 8, "segments", None, "bf16"), (3, 1, 1024, 32, 32, "segments", None, "f16"),
    (4, 2, 1024, 30, 16, "patches", "heads", "bf16"), (7, 4, 256, 32, 16, "segments", "windows", "bf16"),
    (5, 6, 256, 30, 16, "patches", "windows", "f16"), (1027, 3, 64, 30, 16, "segments", "heads", "bf16"),
    (1025, 4, 64, 20, 8, "segments", "windows", "f16"),
]


@pytest.mark.parametrize("nw,heads,N,d,m,lm,kind,dtype", CASES)
def test_both_forms_match_the_oracle(nw, heads, N, d, m, lm, kind, dtype, monkeypatch):
    x, w, b = workloads.random_x_wqkv(nw, N, heads, d, dtype, seed=N + m + d)
    rng = np.random.default_rng(N)
    bias = None if kind is None else torch.from_numpy(
        0.3 * rng.standard_normal(((nw, heads) if kind == "windows" else (heads,)) + (N, N))).float()
    xd, wd, bd = x.cuda(), w.cuda(), b.cuda()
    pooled = None if bias is None else binding.pool_bias(bias.cuda(), m, lm)
    assert binding._two_pass(nw, N, heads, d, m, 5, lm, xd, wd, bd, pooled, nw if kind == "windows" else 1,
                             torch.empty_like(xd), None)
    one = binding.nystra_qkv(xd, wd, heads, m, 5, b_qkv=bd, pooled=pooled, landmarks=lm)
    fused = fused_qkv(xd, wd, heads, m, 5, bd, pooled, lm)
    monkeypatch.setattr(binding, "QKV_WORKSPACE", 3 * (nw // 2) * heads * N * d * 2)  # two or three chunks
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    some = binding.nystra_qkv(xd, wd, heads, m, 5, b_qkv=bd, pooled=pooled, landmarks=lm, stream=s)
    s.synchronize()
    torch.cuda.synchronize()
    assert binding.status() == binding.NYSTRA_OK
    assert torch.equal(one, some)  # every window on its own, whatever the chunks
    idx = np.unique(np.linspace(0, nw - 1, 6).astype(int))
    q, k, v = oracle.project_qkv(x[idx], w, b, heads)
    bb = None if bias is None else bias.double().numpy()[idx] if kind == "windows" else bias.double().numpy()[None]
    ref = oracle.nystra_attention(q, k, v, m, 5, lm, bb).reshape(-1, N, d)
    for out in (one, fused):
        err = per_unit_rel(out.cpu()[idx].double().numpy(), ref)
        assert err.max() <= 3 * ROUND[dtype], err.max()  # Q and K, V and the output are rounded


def test_what_was_refused_stays_refused():
    x, w, b = (t.cuda() for t in workloads.random_x_wqkv(4, 256, 4, 32, "bf16", seed=1))
    for kw in ({"m": 32}, {"m": 64}, {"m": 16, "iters": 13}, {"m": 8, "landmarks": "patches"}):
        with pytest.raises(binding.NystraError):
            binding.nystra_qkv(x, w, 4, **kw)
    with pytest.raises(binding.NystraError):  # out over the tokens
        binding.nystra_qkv(x, w, 4, 16, 6, out=x.view(4, 4, 256, 32))
    big = torch.zeros(4 * 256 * 128 + 8, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(binding.NystraError):  # tokens not 16-byte aligned
        binding.nystra_qkv(big[4:4 + 4 * 256 * 128].view(4, 256, 128), w, 4, 16, 6)
    with pytest.raises(binding.NystraError):
        binding.nystra_qkv(x.float(), w.float(), 4, 16, 6)
    torch.cuda.synchronize()
    assert binding.status() == binding.NYSTRA_OK


@pytest.mark.parametrize("N,heads,d", [(64, 6, 30), (256, 1, 32), (256, 6, 30), (1024, 1, 16), (1024, 6, 30)])
@pytest.mark.parametrize("kind", [None, "heads", "windows"])
def test_no_windows_is_a_no_op(N, heads, d, kind):
    x, w, b = (t.cuda() for t in workloads.random_x_wqkv(1, N, heads, d, "bf16", seed=N))
    pooled = None
    if kind is not None:
        lead = (heads,) if kind == "heads" else (0, heads)
        pooled = tuple(torch.zeros(lead + s, device="cuda") for s in ((N, 16), (16, N), (16, 16)))
    out = binding.nystra_qkv(x[:0], w, heads, 16, 6, b_qkv=b, pooled=pooled)
    torch.cuda.synchronize()
    assert out.shape == (0, heads, N, d) and binding.status() == binding.NYSTRA_OK


def test_without_memory_and_under_capture(monkeypatch):
    x, w, b = (t.cuda() for t in workloads.random_x_wqkv(6, 1024, 2, 32, "bf16", seed=2))
    ref = binding.nystra_qkv(x, w, 2, 16, 6, b_qkv=b)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = binding.nystra_qkv(x, w, 2, 16, 6, b_qkv=b)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)
    monkeypatch.setattr(binding, "_qkv_two_pass", lambda *a: None)  # no memory: the fused kernel
    out = binding.nystra_qkv(x, w, 2, 16, 6, b_qkv=b)
    assert torch.equal(out, fused_qkv(x, w, 2, 16, 6, b))


@pytest.mark.parametrize("given", [False, True])
def test_a_capture_begun_outside_torch(given):
    # the runtime captures, and torch's allocator knows nothing of it: what the
    # graph writes at a replay is the result's own storage, not what came after it
    x, w, b = (t.cuda() for t in workloads.random_x_wqkv(6, 1024, 2, 32, "bf16", seed=3))
    rt = ctypes.CDLL("libcudart.so.13")
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph, run = ctypes.c_void_p(), ctypes.c_void_p()
    with torch.cuda.stream(s):
        ref = binding.nystra_qkv(x, w, 2, 16, 6, b_qkv=b)
        fused = fused_qkv(x, w, 2, 16, 6, b)
        mine = torch.zeros_like(ref) if given else None
        s.synchronize()
        assert rt.cudaStreamBeginCapture(ctypes.c_void_p(s.cuda_stream), 2) == 0  # relaxed
        out = binding.nystra_qkv(x, w, 2, 16, 6, b_qkv=b, out=mine)
        assert rt.cudaStreamEndCapture(ctypes.c_void_p(s.cuda_stream), ctypes.byref(graph)) == 0
        assert rt.cudaGraphInstantiate(ctypes.byref(run), graph, ctypes.c_ulonglong(0)) == 0
        later = [torch.full((n,), 7, dtype=torch.uint8, device="cuda") for n in [6 * 2 * 1024 * 32 * 2 * 3] * 4]
        out.zero_()
        for _ in range(2):
            assert rt.cudaGraphLaunch(run, ctypes.c_void_p(s.cuda_stream)) == 0
        s.synchronize()
    assert torch.equal(out, fused if given else ref)
    assert all(bool((t == 7).all()) for t in later)
    assert rt.cudaGraphExecDestroy(run) == 0 and rt.cudaGraphDestroy(graph) == 0
    assert binding.status() == binding.NYSTRA_OK


@pytest.mark.parametrize("explicit", [False, True])
def test_a_failing_workspace_allocation(explicit, monkeypatch):
    x, w, b = (t.cuda() for t in workloads.random_x_wqkv(6, 1024, 2, 32, "bf16", seed=4))
    fused, real = fused_qkv(x, w, 2, 16, 6, b), torch.empty
    torch.cuda.synchronize()

    def empty(*a, **k):
        if k.get("dtype") is torch.uint8:
            raise torch.OutOfMemoryError("no memory for the workspace")
        return real(*a, **k)
    monkeypatch.setattr(torch, "empty", empty)
    s = torch.cuda.Stream() if explicit else None
    out = binding.nystra_qkv(x, w, 2, 16, 6, b_qkv=b, stream=s)
    torch.cuda.synchronize()
    assert torch.equal(out, fused)
