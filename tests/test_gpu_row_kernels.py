"""GPU parity of the row kernels (weights, and the 8-bit and small activation
shapes) at the edges of their stages: the smallest and largest power-of-two
blocks, one and two shared-memory passes and the third one at 16384, every
small factor, and plain rows of one chunk up to the largest K.

Bars as in the other quantizer tests: codes within +-1 on at most 1e-4 of the
elements, scales within 1e-5 relative (fp32 butterflies against double), the
row sum equal to the sum of the codes produced."""
import numpy as np
import pytest
import torch

import oracle
from paper_2405_16406_gb300 import synth
from tests import parity_util as pu

pytestmark = pytest.mark.gpu

HADS = [(1, 32), (1, 64), (1, 512), (1, 1024), (1, 8192), (1, 16384), (12, 8), (28, 16), (20, 32), (12, 128),
        (28, 256), (12, 2048), (28, 1024)]


@pytest.fixture(scope="module")
def S():
    from paper_2405_16406_gb300 import spinq
    return spinq


@pytest.mark.parametrize("had,K", [(h, h[0] * h[1]) for h in HADS] + [(None, k) for k in (32, 2080, 4096, 16384, 32768)])
@pytest.mark.parametrize("clip", [1.0, 0.9])
def test_weight_rows(S, had, K, clip):
    rng = np.random.default_rng(K)
    w = synth.weights(rng, 21, K)
    w[3] = 0
    out = S.quant_weight(torch.from_numpy(w).cuda(), had, clip)
    ref = oracle.quant_weight(w, had, 4, clip)
    got = pu.gpu_codes(out.codes.cpu().numpy(), True)
    pu.assert_codes_close(got, ref.codes, f"had={had} K={K}")
    pu.assert_scale_close(out.scale.cpu().numpy(), ref.scale, f"had={had} K={K} scale")
    assert np.array_equal(out.rowsum.cpu().numpy(), got.sum(1))


def test_weight_rows_more_than_one_wave(S):
    """More rows than resident CTAs, an odd number of them: every CTA walks
    several rows and prefetches the next."""
    rng = np.random.default_rng(3)
    w = synth.weights(rng, 2501, 768)
    out = S.quant_weight(torch.from_numpy(w).cuda(), (12, 64), 1.0)
    ref = oracle.quant_weight(w, (12, 64))
    pu.assert_codes_close(pu.gpu_codes(out.codes.cpu().numpy(), True), ref.codes, "rows")
    pu.assert_scale_close(out.scale.cpu().numpy(), ref.scale, "rows scale")


@pytest.mark.parametrize("had", [None, (1, 256), (1, 8192), (12, 2048)])
def test_fp8_rows(S, had):
    K = 2176 if had is None else had[0] * had[1]
    rng = np.random.default_rng(K + 1)
    w = synth.weights(rng, 19, K)
    out = S.quant_weight8(torch.from_numpy(w).cuda(), had, S.SPINQ_FMT_E4M3)
    ref = oracle.quant_weight_fp8(w, had)
    pu.assert_scale_close(out.scale.cpu().numpy(), ref.alpha, "fp8 scale")
    got = out.codes.view(torch.float8_e4m3fn).float().cpu().numpy()
    want = torch.from_numpy(np.ascontiguousarray(ref.codes).astype(np.uint8)).view(torch.float8_e4m3fn).float().numpy()
    off = got != want
    assert off.mean() <= 1e-4
    # a tie goes to the neighbouring grid value: at most 2^-3 of it, or one subnormal step
    assert np.all(np.abs(got - want)[off] <= np.maximum(np.abs(want[off]) / 8, 2.0 ** -9))
