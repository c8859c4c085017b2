"""Kernels that begin while the one before them on the stream still runs: chains of calls without anything in between."""
import ctypes
import gc

import pytest
import torch

from test_gpu_parity import S  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

# dtype, heads, T, d, block_q, block_k: a form of every attention kernel
FORMS = [
    (torch.bfloat16, 16, 3000, 128, 64, 64), (torch.bfloat16, 8, 1500, 64, 64, 64),   # tcgen05
    (torch.bfloat16, 8, 1500, 128, 32, 32), (torch.bfloat16, 8, 1500, 64, 32, 32),    # tcgen05, blocks of 32
    (torch.bfloat16, 4, 1100, 128, 1, 64),                                            # tcgen05, per-token masks
    (torch.bfloat16, 8, 1100, 256, 64, 64), (torch.bfloat16, 4, 700, 64, 1, 16),      # mma.sync, and its merged walk
    (torch.float32, 8, 1500, 64, 32, 32), (torch.float32, 8, 1000, 64, 32, 32),       # fp32, P over the key tile or not
    (torch.float32, 8, 1500, 32, 32, 32), (torch.float32, 4, 1100, 128, 32, 32),
    (torch.float32, 2, 700, 64, 32, 32),                                              # a row over a cluster
]


@pytest.fixture(scope="module", autouse=True)
def leave_no_garbage():  # (what follows counts the allocator's bytes around a call: no collection may fall there)
    yield
    gc.collect()


@pytest.mark.parametrize("dtype,heads,T,d,block_q,block_k", FORMS)
def test_attentions_that_feed_each_other(S, dtype, heads, T, d, block_q, block_k):
    """Every output is the queries or the values of the next call, and its buffer is written again two or three calls later: a
    kernel has to see the results of the one before, and of those before that, and may not write what they still read."""
    torch.manual_seed(d + block_q)
    q, k, v = (torch.randn(1, heads, T, d, device="cuda").to(dtype) for _ in range(3))
    kw = dict(block_q=block_q, block_k=block_k)
    mask = S.build_mask(q, k, k_top=5, **kw).mask
    calls = [("q", "v", "a"), ("a", "v", "b"), ("b", "a", "c"), ("c", "b", "a"), ("a", "c", "b"), ("q", "b", "c"), ("c", "a", "a2"), ("a2", "c", "a")]

    def chain(wait):
        x = dict(q=q, v=v, **{n: torch.full_like(q, float("nan")) for n in ("a", "b", "c", "a2")})
        torch.cuda.synchronize()
        for at_q, at_v, to in calls * 3:
            S.sparse_attention(x[at_q], k, x[at_v], mask, out=x[to], **kw)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return x

    want = chain(True)
    for _ in range(3):
        got = chain(False)
        for n in ("a", "b", "c", "a2"):
            assert torch.isfinite(want[n]).all() and torch.equal(got[n], want[n]), n


def test_a_call_that_failed_does_not_fail_the_next(S):
    """A synchronisation on a stream that is being captured is refused on the host. The refusal is that call's alone: the
    calls after it report their own errors, none here."""
    torch.manual_seed(0)
    q, k, v = (torch.randn(1, 2, 300, 64, device="cuda") for _ in range(3))
    kw = dict(block_q=32, block_k=32)
    mask = S.build_mask(q, k, k_top=4, **kw).mask
    want = S.sparse_attention(q, k, v, mask, **kw)
    torch.cuda.synchronize()
    rt = ctypes.CDLL("libcudart.so.12")  # the one that torch has loaded
    side, graph = torch.cuda.Stream(), ctypes.c_void_p()
    for call in (lambda: S.sparse_attention(q, k, v, mask, **kw), lambda: S.build_mask(q, k, k_top=4, **kw).mask,
                 lambda: S.mask_difference(mask, mask)[0]):
        assert rt.cudaStreamBeginCapture(ctypes.c_void_p(side.cuda_stream), 2) == 0  # (relaxed: other streams go on as ever)
        with pytest.raises(S.StreamError):
            S.stream_check_device_status(side)
        assert rt.cudaStreamEndCapture(ctypes.c_void_p(side.cuda_stream), ctypes.byref(graph)) != 0  # the capture is lost
        rt.cudaGetLastError()  # (that error is this test's own)
        call()
        torch.cuda.synchronize()
    assert torch.equal(S.sparse_attention(q, k, v, mask, **kw), want)


@pytest.mark.parametrize("dtype,heads,T,d,block_q,block_k", FORMS)
def test_capture_in_a_graph(S, dtype, heads, T, d, block_q, block_k):
    """Two passes of mask and attention and a second attention behind them, captured once, replayed on changed inputs."""
    torch.manual_seed(d)
    kw = dict(block_q=block_q, block_k=block_k)
    inputs = [tuple(torch.randn(1, heads, T, d, device="cuda").to(dtype) for _ in range(3)) for _ in range(2)]
    want = []
    for q, k, v in inputs:
        mask = S.build_mask(q, k, k_top=5, **kw).mask
        out = S.sparse_attention(q, k, v, mask, **kw)
        torch.cuda.synchronize()
        want.append((mask, out, S.sparse_attention(out, k, v, mask, **kw)))
        torch.cuda.synchronize()
    q, k, v = (x.clone() for x in inputs[0])
    mask, out, out2 = (torch.empty_like(x) for x in want[0])
    ws = torch.empty(256, dtype=torch.uint8, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(2):
            S.build_mask(q, k, k_top=5, mask_out=mask, workspace=ws, **kw)
            S.sparse_attention(q, k, v, mask, out=out, **kw)
            S.sparse_attention(out, k, v, mask, out=out2, **kw)
    for i in (0, 1, 1, 0):
        for dst, src in zip((q, k, v), inputs[i]):
            dst.copy_(src)
        mask.fill_(-7)
        out.zero_()
        out2.zero_()
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(mask, want[i][0]) and torch.equal(out, want[i][1]) and torch.equal(out2, want[i][2])


def test_capture_of_several_k_one_k_a_row_and_the_library_s_scratch(S):
    torch.manual_seed(3)
    kw = dict(block_q=64, block_k=64)
    inputs = [tuple(torch.randn(1, h, 3000, 128, device="cuda").bfloat16() for h in (8, 2)) for _ in range(2)]
    q, k = (x.clone() for x in inputs[0])
    p = S.make_problem(q, k, k_top=12, **kw)
    k_row = S.k_schedule(p, 1 / 4).cuda()
    static = torch.empty(1, 8, S.n_query_blocks(p), 12, dtype=torch.int32, device="cuda")

    def calls():
        S.stream_build_mask_static(p, q, k, static, None)
        return [static, S.build_masks(q, k, [12, 3, 7], **kw).mask, S.build_masks(q, k, [12, 3, 7], share=False, **kw).mask,
                S.build_mask(q, k, k_top=12, k_row=k_row, **kw).mask]

    want = []
    for i in (0, 1):  # (the first call on the library's scratch asks for its address, which no capture allows)
        q.copy_(inputs[i][0])
        k.copy_(inputs[i][1])
        want.append([x.clone() for x in calls()])
        torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = calls()
    for i in (1, 0, 1):
        q.copy_(inputs[i][0])
        k.copy_(inputs[i][1])
        for x in got:
            x.fill_(-7)
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, want[i]))
