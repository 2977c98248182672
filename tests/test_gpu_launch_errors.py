"""A call answers for its own launches only: an error that an earlier CUDA call
of the program left in the thread's last-error slot (here a cudaSetDevice that
the runtime refuses on the host) is neither reported nor taken by it."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu

INVALID_DEVICE = 101


def _calls(S):
    g = torch.Generator(device="cuda").manual_seed(1)
    f16 = lambda *s: torch.randn(*s, generator=g, device="cuda").half()
    x, big, paley = f16(8, 512), f16(2048, 8192), f16(160, 14336)
    w = S.quant_weight(f16(512, 512), (1, 512))
    a8 = S.rotate_quant_act8(f16(200, 512), None, S.SPINQ_FMT_E4M3)
    w8 = S.quant_weight8(f16(512, 512), None, S.SPINQ_FMT_E4M3)
    many = [S.rotate_quant_act(f16(m, 512), None) for m in (1, 8, 40, 300)]
    q, k = f16(2, 64, 8, 64), f16(2, 64, 4, 64)
    q1, kv = f16(2, 8, 64), S.rotate_quant_kv(q, k, k)
    pos = torch.arange(64, dtype=torch.int32, device="cuda").repeat(2, 1)
    table = torch.rand(64, 32, 2, generator=g, device="cuda")
    R = torch.eye(128, device="cuda").repeat(3, 1, 1)
    ws = S.gemm_workspace(40, 512, 512)
    return {"act": lambda: S.rotate_quant_act(x, (1, 512)), "act_tc": lambda: S.rotate_quant_act(big, (1, 8192)),
            "paley": lambda: S.rotate_quant_act(paley, (28, 512)), "weight": lambda: S.quant_weight(x, None),
            "act8": lambda: S.rotate_quant_act8(x, None, S.SPINQ_FMT_INT8_PLANES), "fp8": lambda: S.fp8_gemm(a8, w8),
            **{f"gemm{m.codes.shape[0]}": (lambda m=m: S.w4a4_gemm(m, w)) for m in many},
            "splitk": lambda: S.w4a4_gemm_splitk(many[2], w, workspace=ws), "kv": lambda: S.rotate_quant_kv(q, k, k),
            "rope": lambda: S.rope_rotate_quant_kv(q, k, k, pos, table),
            "attention": lambda: S.decode_attention_kv4(q1, kv), "cayley": lambda: S.cayley_step(R, R, 0.1)
            }


def test_a_pending_error_is_not_the_calls_own():
    from paper_2405_16406_gb300 import spinq as S
    rt = ctypes.CDLL("libcudart.so.13")   # the runtime that libspinq.so is linked with
    for name, call in _calls(S).items():
        call()                            # outputs of its size are in torch's cache now
        torch.cuda.synchronize()
        assert rt.cudaSetDevice(1 << 20) == INVALID_DEVICE
        try:
            call()
            assert rt.cudaPeekAtLastError() == INVALID_DEVICE, name
        finally:
            rt.cudaGetLastError()
        torch.cuda.synchronize()
    assert S.spinq_device_status()[0] == S.SPINQ_OK
