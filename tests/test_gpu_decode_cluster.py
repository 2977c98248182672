"""The clustered decode GEMM (K split over a cluster of CTAs, partial sums over
distributed shared memory), which the split-K entry point takes for most shapes
of up to 128 tokens: token counts around its tiles, ragged channel counts, one
to eight CTAs, uneven slices, the longest K with extreme codes, and a wait that
runs out.  The accumulator is exact, so it has to equal the integer product, and
the outputs those of the split-K kernel bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    from paper_2405_16406_gb300 import spinq
    return spinq


def _signed(codes):
    u = torch.stack([codes & 15, codes >> 4], -1).reshape(codes.shape[0], -1).double()
    return torch.where(u > 7, u - 16, u)


def _case(S, M, N, K, symmetric, extreme=False):
    g = torch.Generator(device="cuda").manual_seed(M * 7 + N + K)

    def codes(rows, byte):
        if extreme:
            return torch.full((rows, K // 2), byte, dtype=torch.uint8, device="cuda")
        return torch.randint(0, 256, (rows, K // 2), dtype=torch.uint8, device="cuda", generator=g)

    a = S.ActCodes(codes(M, 0x88 if symmetric else 0xFF), torch.rand(M, device="cuda", generator=g) + 0.1,
                   None if symmetric else -torch.rand(M, device="cuda", generator=g))
    wc = codes(N, 0x88)
    wi = _signed(wc)
    w = S.WeightCodes(wc, torch.rand(N, device="cuda", generator=g) * 0.01 + 0.001, wi.sum(1).to(torch.int32))
    ai = _signed(a.codes) if symmetric else torch.stack([a.codes & 15, a.codes >> 4], -1).reshape(M, -1).double() - 8
    return a, w, ai @ wi.T   # |sums| <= 64 K < 2^53: exact in double


def _check(S, a, w, acc_ref, symmetric, entry):
    y, acc = entry(a, w, want_acc=True)
    assert torch.equal(acc.double(), acc_ref)
    al = a.scale.double()[:, None]
    beta = 0.0 if symmetric else a.zero.double()[:, None] + 8 * al
    ref = w.scale.double() * (al * acc_ref + beta * w.rowsum.double())
    # one fp32 epilogue of three roundings and one fp16 rounding
    tol = 2.0 ** -10 * ref.abs() + 2.0 ** -20 * (w.scale.double() * (al * acc_ref).abs()) + 2.0 ** -24
    if not symmetric:
        tol = tol + 2.0 ** -20 * (w.scale.double() * (beta * w.rowsum.double()).abs())
    over = (ref.abs() >= 65504) & torch.isinf(y) & (torch.sign(y) == torch.sign(ref))   # past fp16's range
    assert torch.all(((y.double() - ref).abs() <= tol) | over)
    return y


SHAPES = [(m, n, k) for m in (17, 32, 33, 64, 77, 96, 97, 113, 128)
          for n, k in ((400, 4096), (1040, 1152), (3072, 1664), (4096, 2048), (6160, 4096), (272, 8192), (16, 128))]
SHAPES += [(9, 2064, 4224), (16, 272, 4224), (24, 16384, 3072)]


@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("symmetric", [True, False])
def test_decode_cluster_exact(S, M, N, K, symmetric):
    a, w, ref = _case(S, M, N, K, symmetric)
    y, acc = S.w4a4_gemm_splitk(a, w, want_acc=True)
    assert torch.equal(acc.double(), ref)
    prev = S.spinq_gemm_select_kernel(S.SPINQ_GEMM_SPLITK)
    try:
        y2, acc2 = S.w4a4_gemm_splitk(a, w, want_acc=True)
    finally:
        S.spinq_gemm_select_kernel(prev)
    assert torch.equal(acc2.double(), ref)
    if S.spinq_w4a4_gemm_splitk_plan(M, N, K)[0] == S.SPINQ_GEMM_SPLITK:   # (the prefill kernels round otherwise)
        assert torch.equal(y, y2)
    assert torch.equal(S.w4a4_gemm_splitk(a, w), y)
    assert S.spinq_device_status()[0] == S.SPINQ_OK


@pytest.mark.parametrize("M", [16, 80, 128])
@pytest.mark.parametrize("symmetric", [True, False])
def test_decode_cluster_extreme_codes_long_k(S, M, symmetric):
    a, w, ref = _case(S, M, 256, 65536, symmetric, extreme=True)
    _check(S, a, w, ref, symmetric, S.w4a4_gemm_splitk)


def test_decode_cluster_is_repeatable(S):
    a, w, ref = _case(S, 77, 6144, 4096, False)
    first = _check(S, a, w, ref, False, S.w4a4_gemm_splitk)
    for _ in range(30):
        assert torch.equal(S.w4a4_gemm_splitk(a, w), first)


def test_decode_cluster_wait_gives_up_and_reports_timeout(S):
    a, w, ref = _case(S, 32, 4096, 4096, True)
    try:
        assert S.spinq_debug_set_wait_limit_ns(1_000_000) == S.SPINQ_OK
        assert S.spinq_debug_stall_launches(1) == 0
        S.w4a4_gemm_splitk(a, w)
        assert S.spinq_device_status()[0] == S.SPINQ_ETIMEOUT
        assert S.spinq_debug_stall_launches(0) == 0     # the stalled launch happened
    finally:
        S.spinq_debug_stall_launches(0)
        S.spinq_debug_set_wait_limit_ns(2_000_000_000)
    _check(S, a, w, ref, True, S.w4a4_gemm_splitk)
    assert S.spinq_device_status()[0] == S.SPINQ_OK
