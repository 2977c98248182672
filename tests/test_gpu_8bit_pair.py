"""The 8-bit GEMMs on SM pairs (more than 128 rows): every tile width, ragged
rows and columns, odd numbers of 128-deep K steps, several tiles per pair, and
a wait that runs out.  The W4A8 accumulator is exact.  FP8: products exact, the
fp32 accumulation of K / 32 partial sums, each within 2^-22 of the running sum
of magnitudes, so within 2^-13 of it for K <= 4224 with room; two fp32
roundings and one to fp16."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# (rows, columns, K): tiles 192 wide unless noted
SHAPES = [(129, 16, 128), (256, 192, 256), (257, 400, 384), (300, 1040, 4224), (1531, 2064, 1024),
          (2048, 4080, 384), (2041, 4096, 512),      # 224
          (1531, 14336, 256)]                        # 256


@pytest.fixture(scope="module")
def S():
    from paper_2405_16406_gb300 import spinq
    return spinq


def _fp8(S, M, N, K):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    a, w = ((torch.randn(r, K, generator=g, device="cuda") * 40).to(torch.float8_e4m3fn) for r in (M, N))
    al, sn = (torch.rand(r, generator=g, device="cuda") * 1e-3 + 1e-4 for r in (M, N))
    return a, w, al, sn, S.ActCodes(a.view(torch.uint8), al, None), S.WeightCodes(w.view(torch.uint8), sn, None)


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_fp8_pair(S, M, N, K):
    a, w, al, sn, qa, qw = _fp8(S, M, N, K)
    y = S.fp8_gemm(qa, qw).double()
    s = al.double()[:, None] * sn.double()
    ref = s * (a.double() @ w.double().T)
    mag = s * (a.double().abs() @ w.double().abs().T)
    assert torch.all((y - ref).abs() <= 2.0 ** -10 * ref.abs() + 2.0 ** -13 * mag + 2.0 ** -24)
    assert S.spinq_device_status()[0] == S.SPINQ_OK


@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("symmetric", [True, False])
def test_w4a8_pair_exact(S, M, N, K, symmetric):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    x = torch.randn(M, K, generator=g, device="cuda").half()
    qa = S.rotate_quant_act8(x, None, S.SPINQ_FMT_INT8_PLANES, symmetric=symmetric)
    qw = S.quant_weight8(torch.randn(N, K, generator=g, device="cuda").half(), None, S.SPINQ_FMT_INT4_BYTES)
    c = qa.codes.view(torch.float8_e4m3fn).double()
    ref = (c[:, :K] + c[:, K:]) @ qw.codes.view(torch.float8_e4m3fn).double().T
    y, acc = S.w4a8_gemm(qa, qw, want_acc=True)
    assert torch.equal(acc.double(), ref)
    assert torch.equal(S.w4a8_gemm(qa, qw), y)
    al = qa.scale.double()[:, None]
    bias = 0.0 if symmetric else (qa.zero.double()[:, None] + 128 * al) * qw.rowsum.double()
    out = qw.scale.double() * (al * ref + bias)
    mag = qw.scale.double() * ((al * ref).abs() + abs(bias))
    assert torch.all((y.double() - out).abs() <= 2.0 ** -10 * out.abs() + 2.0 ** -20 * mag + 2.0 ** -24)


def test_pair_wait_gives_up_and_reports_timeout(S):
    _, _, _, _, qa, qw = _fp8(S, 512, 512, 512)
    good = S.fp8_gemm(qa, qw)
    try:
        assert S.spinq_debug_set_wait_limit_ns(1_000_000) == S.SPINQ_OK
        assert S.spinq_debug_stall_launches(1) == 0
        S.fp8_gemm(qa, qw)
        assert S.spinq_device_status()[0] == S.SPINQ_ETIMEOUT
        assert S.spinq_debug_stall_launches(0) == 0     # the stalled launch happened
    finally:
        S.spinq_debug_stall_launches(0)
        S.spinq_debug_set_wait_limit_ns(2_000_000_000)
    assert torch.equal(S.fp8_gemm(qa, qw), good)
    assert S.spinq_device_status()[0] == S.SPINQ_OK
