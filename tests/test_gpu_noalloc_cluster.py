"""spinq_w4a4_gemm_noalloc where the clustered kernel serves the call: it uses
none of the library's array, so nothing but the kernel goes on the stream (a
captured call is one graph node) and calls on two streams at once do not share
anything; where split-K serves it, the array is cleared first as before."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    from paper_2405_16406_gb300 import spinq
    return spinq


def _case(S, M, N, K, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    codes = lambda r: torch.randint(0, 256, (r, K // 2), dtype=torch.uint8, device="cuda", generator=g)
    a = S.ActCodes(codes(M), torch.rand(M, device="cuda", generator=g) + 0.1, None)
    wc = codes(N)
    u = torch.stack([wc & 15, wc >> 4], -1).reshape(N, -1).int()
    w = S.WeightCodes(wc, torch.rand(N, device="cuda", generator=g) * 0.01, torch.where(u > 7, u - 16, u).sum(1).int())
    return a, w, torch.full((M, N), float("nan"), dtype=torch.float16, device="cuda")


def _call(S, case, stream):
    a, w, y = case
    p = lambda t: t.data_ptr()
    return S.spinq_w4a4_gemm_noalloc(p(a.codes), p(a.scale), None, p(w.codes), p(w.scale), p(w.rowsum), y.shape[0],
                                     y.shape[1], a.codes.shape[1] * 2, p(y), None, stream.cuda_stream)


def _nodes(graph):
    n = ctypes.c_size_t(0)
    assert ctypes.CDLL("libcuda.so.1").cuGraphGetNodes(ctypes.c_void_p(graph.raw_cuda_graph()), None, ctypes.byref(n)) == 0
    return n.value


@pytest.mark.parametrize("M,N,K,cluster", [(77, 4096, 4096, True), (32, 3072, 8192, True), (77, 4096, 4096, False)])
def test_only_the_kernel_is_enqueued(S, M, N, K, cluster):
    case = _case(S, M, N, K, 1)
    assert S.spinq_w4a4_gemm_workspace_bytes(M, N, K) > 0
    prev = S.spinq_gemm_select_kernel(S.SPINQ_GEMM_AUTO if cluster else S.SPINQ_GEMM_SPLITK)
    try:
        assert (S.spinq_w4a4_gemm_cluster_plan(M, N, K) > 0) == cluster
        side = torch.cuda.Stream()
        assert _call(S, case, side) == S.SPINQ_OK   # first use: address and attributes
        torch.cuda.synchronize()
        case[2].fill_(float("nan"))
        graph = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(graph, stream=side):
            assert _call(S, case, torch.cuda.current_stream()) == S.SPINQ_OK
        assert _nodes(graph) == (1 if cluster else 2)
        graph.replay()
    finally:
        S.spinq_gemm_select_kernel(prev)
    assert torch.equal(case[2], S.w4a4_gemm_splitk(case[0], case[1]))


def test_clustered_calls_on_two_streams(S):
    cases = [_case(S, 77, 4096, 4096, s) for s in (1, 2)]
    want = [S.w4a4_gemm_splitk(a, w) for a, w, _ in cases]
    assert S.spinq_w4a4_gemm_cluster_plan(77, 4096, 4096) > 0
    streams = [torch.cuda.Stream() for _ in cases]
    torch.cuda.synchronize()
    for _ in range(50):
        for case, s in zip(cases, streams):
            assert _call(S, case, s) == S.SPINQ_OK
    torch.cuda.synchronize()
    for case, y in zip(cases, want):
        assert torch.equal(case[2], y)
    assert S.spinq_device_status()[0] == S.SPINQ_OK
