"""256-row tiles of 192 columns, taken where they save work for whole waves:
ragged rows and columns, one and several tiles per CTA, odd and single K steps.
The accumulator is exact and the outputs are those of the 128-row tiles bit for
bit (one epilogue formula)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _signed(codes):
    u = torch.stack([codes & 15, codes >> 4], -1).reshape(codes.shape[0], -1).double()
    return torch.where(u > 7, u - 16, u)


@pytest.mark.parametrize("M,N,K", [(129, 16, 128), (256, 192, 256), (257, 208, 384), (300, 400, 4224),
                                   (513, 4112, 512), (1531, 14336, 256), (1000, 14352, 640)])
@pytest.mark.parametrize("symmetric", [True, False])
def test_slim_tiles_exact(M, N, K, symmetric):
    from paper_2405_16406_gb300 import spinq as S
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    codes = lambda r: torch.randint(0, 256, (r, K // 2), dtype=torch.uint8, device="cuda", generator=g)
    a = S.ActCodes(codes(M), torch.rand(M, device="cuda", generator=g) + 0.1,
                   None if symmetric else -torch.rand(M, device="cuda", generator=g))
    wc = codes(N)
    wi = _signed(wc)
    w = S.WeightCodes(wc, torch.rand(N, device="cuda", generator=g) * 0.01 + 0.001, wi.sum(1).to(torch.int32))
    ai = _signed(a.codes) if symmetric else torch.stack([a.codes & 15, a.codes >> 4], -1).reshape(M, -1).double() - 8
    prev = S.spinq_gemm_select_kernel(S.SPINQ_GEMM_TILE256)
    try:
        y, acc = S.w4a4_gemm(a, w, want_acc=True)
        again = S.w4a4_gemm(a, w)
        S.spinq_gemm_select_kernel(S.SPINQ_GEMM_TILE128)
        y128 = S.w4a4_gemm(a, w)
    finally:
        S.spinq_gemm_select_kernel(prev)
    assert torch.equal(acc.double(), ai @ wi.T)
    assert torch.equal(y, again) and torch.equal(y, y128)
    assert S.spinq_device_status()[0] == S.SPINQ_OK
