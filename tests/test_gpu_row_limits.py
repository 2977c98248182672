"""Rotated rows whose fp32 copy in shared memory is as large as a block's
default limit: K = 12288 = 12 x 1024 is 48 KB, to which the row kernels'
reduction arrays are added.  Every quantizer that has a row kernel, against
the oracle, and a plain row after each (no launch error may be left over)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2405_16406_gb300 import synth
from tests import parity_util as pu

pytestmark = pytest.mark.gpu

HAD, K = (12, 1024), 12288


@pytest.fixture(scope="module")
def S():
    from paper_2405_16406_gb300 import spinq
    return spinq


@pytest.fixture
def rows(S):
    w = synth.weights(np.random.default_rng(12288), 9, K)
    yield w, torch.from_numpy(w).cuda()
    plain = S.quant_weight(torch.from_numpy(w[:, :256].copy()).cuda(), None)
    assert np.array_equal(pu.gpu_codes(plain.codes.cpu().numpy(), True).sum(1), plain.rowsum.cpu().numpy())


def test_weights_of_48_kb_rows(S, rows):
    w, wt = rows
    out, ref = S.quant_weight(wt, HAD), oracle.quant_weight(w, HAD)
    got = pu.gpu_codes(out.codes.cpu().numpy(), True)
    pu.assert_codes_close(got, ref.codes, "weights")
    pu.assert_scale_close(out.scale.cpu().numpy(), ref.scale, "weights")
    assert np.array_equal(out.rowsum.cpu().numpy(), got.sum(1))


def test_byte_weights_of_48_kb_rows(S, rows):
    w, wt = rows
    out, ref = S.quant_weight8(wt, HAD, S.SPINQ_FMT_INT4_BYTES), oracle.quant_weight(w, HAD)
    got = out.codes.view(torch.float8_e4m3fn).float().cpu().numpy().astype(np.int64)
    pu.assert_codes_close(got, ref.codes, "byte weights")
    assert np.array_equal(out.rowsum.cpu().numpy(), got.sum(1))
    pu.assert_scale_close(S.quant_weight8(wt, HAD, S.SPINQ_FMT_E4M3).scale.cpu().numpy(),
                          oracle.quant_weight_fp8(w, HAD).alpha, "fp8 weights")


@pytest.mark.parametrize("symmetric", [True, False])
def test_clipped_activations_of_48_kb_rows(S, rows, symmetric):
    w, wt = rows
    out, ref = S.rotate_quant_act(wt, HAD, symmetric, clip=0.9), oracle.rotate_quant_act(w, HAD, 4, symmetric, 0.9)
    pu.assert_codes_close(pu.gpu_codes(out.codes.cpu().numpy(), symmetric), ref.codes, "act")
    pu.assert_scale_close(out.scale.cpu().numpy(), ref.alpha, "act")
    o8 = S.rotate_quant_act8(wt, HAD, S.SPINQ_FMT_INT8_PLANES, symmetric, clip=0.9)
    r8 = oracle.rotate_quant_act(w, HAD, 8, symmetric, 0.9)
    pu.assert_scale_close(o8.scale.cpu().numpy(), r8.alpha, "act8")
    p = o8.codes.view(torch.float8_e4m3fn).float().cpu().numpy().astype(np.int64)
    pu.assert_codes_close(p[:, :K] + p[:, K:] + (0 if symmetric else 128), r8.codes, "act8")
