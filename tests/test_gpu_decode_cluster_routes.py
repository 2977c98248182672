"""The clustered decode GEMM by name: every cluster size forced, with the query
that says which kernel serves a call, so that what is compared is known to be
the clustered kernel.  Token counts and channels at the edges of its tiles, K
steps that divide unevenly, one K step, and the longest K with the codes that
make the largest sums.  The accumulator is exact and the outputs are those of
the split-K kernel bit for bit (one epilogue formula)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    from paper_2405_16406_gb300 import spinq
    return spinq


@pytest.fixture
def cluster(S):
    yield S.spinq_gemm_cluster
    S.spinq_gemm_cluster(0)


def _signed(codes):
    u = torch.stack([codes & 15, codes >> 4], -1).reshape(codes.shape[0], -1).double()
    return torch.where(u > 7, u - 16, u)


def _case(S, M, N, K, symmetric, extreme=False):
    g = torch.Generator(device="cuda").manual_seed(M * 7 + N + K)

    def codes(rows, byte):
        if extreme:
            return torch.full((rows, K // 2), byte, dtype=torch.uint8, device="cuda")
        return torch.randint(0, 256, (rows, K // 2), dtype=torch.uint8, device="cuda", generator=g)

    # scales small enough for fp16 outputs at any K
    a = S.ActCodes(codes(M, 0x88 if symmetric else 0xFF), (torch.rand(M, device="cuda", generator=g) + 0.1) / K,
                   None if symmetric else -torch.rand(M, device="cuda", generator=g) / K)
    wc = codes(N, 0x88)
    wi = _signed(wc)
    w = S.WeightCodes(wc, torch.rand(N, device="cuda", generator=g) + 0.1, wi.sum(1).to(torch.int32))
    ai = _signed(a.codes) if symmetric else torch.stack([a.codes & 15, a.codes >> 4], -1).reshape(M, -1).double() - 8
    return a, w, ai @ wi.T   # |sums| <= 64 K < 2^53: exact in double


def _splitk(S, a, w):
    prev = S.spinq_gemm_select_kernel(S.SPINQ_GEMM_SPLITK)
    try:
        return S.w4a4_gemm_splitk(a, w)
    finally:
        S.spinq_gemm_select_kernel(prev)


@pytest.mark.parametrize("size", range(1, 9))
@pytest.mark.parametrize("M,N,K", [(1, 16, 1024), (16, 272, 1152), (17, 144, 4224), (77, 1040, 1664), (128, 400, 2048),
                                   (97, 3072, 128)])
@pytest.mark.parametrize("symmetric", [True, False])
def test_every_cluster_size(S, cluster, size, M, N, K, symmetric):
    a, w, ref = _case(S, M, N, K, symmetric)
    assert cluster(size) == 0
    assert S.spinq_w4a4_gemm_cluster_plan(M, N, K) == min(size, K // 128)
    y, acc = S.w4a4_gemm_splitk(a, w, want_acc=True)
    again = S.w4a4_gemm_splitk(a, w)
    cluster(0)
    assert torch.equal(acc.double(), ref)
    assert torch.equal(y, again) and torch.equal(y, _splitk(S, a, w))
    assert S.spinq_device_status()[0] == S.SPINQ_OK


@pytest.mark.parametrize("size", [1, 3, 8])
@pytest.mark.parametrize("M", [16, 80, 128])
@pytest.mark.parametrize("symmetric", [True, False])
def test_largest_sums(S, cluster, size, M, symmetric):
    K = 65536
    a, w, ref = _case(S, M, 256, K, symmetric, extreme=True)
    cluster(size)
    assert S.spinq_w4a4_gemm_cluster_plan(M, 256, K) == size
    y, acc = S.w4a4_gemm_splitk(a, w, want_acc=True)
    cluster(0)
    assert torch.equal(acc.double(), ref)
    assert torch.isfinite(y).all() and torch.equal(y, _splitk(S, a, w))


def test_who_serves_a_call(S, cluster):
    """The automatic choice, and what takes the clustered kernel out of it."""
    plan = S.spinq_w4a4_gemm_cluster_plan
    for M, N, K in ((77, 4096, 4096), (77, 4096, 14336), (24, 4096, 4096), (128, 3072, 8192), (40, 8192, 3072)):
        assert 1 <= plan(M, N, K) <= 8
        assert S.spinq_w4a4_gemm_workspace_bytes(M, N, K) > 0 or S.spinq_w4a4_gemm_splitk_plan(M, N, K)[1] <= 1
    assert plan(1, 4096, 4096) == plan(16, 4096, 4096) == plan(129, 4096, 4096) == 0
    assert plan(77, 28672, 4096) == 0        # the tiles need a second wave
    for choose, restore in ((lambda: S.spinq_gemm_select_kernel(S.SPINQ_GEMM_SPLITK), S.spinq_gemm_select_kernel),
                            (lambda: S.spinq_gemm_split_k(2), S.spinq_gemm_split_k)):
        prev = choose()
        try:
            cluster(4)
            assert plan(77, 4096, 4096) == 0
        finally:
            restore(prev)
            cluster(0)
    cluster(8)
    assert plan(1, 4096, 4096) == 8 and plan(128, 4096, 4096) == 8 and plan(129, 4096, 4096) == 0
    assert plan(77, 4096, 256) == 2
