"""256-row tiles of 192 columns as the automatic choice reaches them: the cost
model weighs the width that the launch takes, so calls whose narrower tiles fit
in one wave go to them and not to the SM pair.  Accumulators are exact and the
outputs those of the 128-row tiles bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _signed(codes):
    u = torch.stack([codes & 15, codes >> 4], -1).reshape(codes.shape[0], -1).double()
    return torch.where(u > 7, u - 16, u)


# one wave of 192-column tiles (77 to 152 of them; SM pairs would take two waves)
@pytest.mark.parametrize("M,N,K", [(300, 14336, 4096), (640, 8192, 3072), (1500, 4096, 3072), (200, 28160, 3072),
                                   (1300, 4096, 4096)])
@pytest.mark.parametrize("symmetric", [True, False])
def test_automatic_choice_reaches_the_slim_tiles(M, N, K, symmetric):
    from paper_2405_16406_gb300 import spinq as S
    assert S.spinq_w4a4_gemm_plan(M, N, K) == S.SPINQ_GEMM_TILE256
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    codes = lambda r: torch.randint(0, 256, (r, K // 2), dtype=torch.uint8, device="cuda", generator=g)
    a = S.ActCodes(codes(M), torch.rand(M, device="cuda", generator=g) + 0.1,
                   None if symmetric else -torch.rand(M, device="cuda", generator=g))
    wc = codes(N)
    wi = _signed(wc)
    w = S.WeightCodes(wc, torch.rand(N, device="cuda", generator=g) * 0.01 + 0.001, wi.sum(1).to(torch.int32))
    ai = _signed(a.codes) if symmetric else torch.stack([a.codes & 15, a.codes >> 4], -1).reshape(M, -1).double() - 8
    y, acc = S.w4a4_gemm(a, w, want_acc=True)
    assert torch.equal(acc.double(), ai @ wi.T)
    prev = S.spinq_gemm_select_kernel(S.SPINQ_GEMM_TILE128)
    try:
        y128 = S.w4a4_gemm(a, w)
    finally:
        S.spinq_gemm_select_kernel(prev)
    assert torch.equal(y, y128)
    assert S.spinq_device_status()[0] == S.SPINQ_OK
