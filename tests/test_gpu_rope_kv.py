"""The RoPE form of the KV quantizer, where a warp takes 8 tokens and a range
of heads: token counts around 8, odd head counts, head ranges that cross from Q
to K to V, batches that take the wide CTAs, clamped positions, in place.

The reference is the plain form (checked against the oracle elsewhere) on
inputs rotated here: RoPE is two fp32 products, one fp32 sum and one rounding
to fp16 per element, so the two agree in every bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu

FIELDS = ("q_out", "k_codes", "k_scale", "k_zero", "v_codes", "v_scale", "v_zero")


def _rope(x, pos, cs):
    """x [B, S, H, D] fp16 at positions [B, S]: rotate-half, products rounded apart."""
    half = x.shape[-1] // 2
    t = cs[pos.long().clamp(0, cs.shape[0] - 1)][:, :, None]
    cos, sin = t[..., 0], t[..., 1]
    a, b = x[..., :half].float(), x[..., half:].float()
    return torch.cat([a * cos + (-b) * sin, b * cos + a * sin], -1).half()


@pytest.mark.parametrize("B,S,Hq,Hkv,D", [(1, 1, 1, 1, 128), (1, 7, 3, 1, 64), (3, 3, 5, 5, 128), (2, 8, 12, 2, 64),
                                          (77, 1, 32, 8, 128), (1, 203, 7, 7, 128), (16, 1, 48, 12, 64),
                                          (2, 1023, 32, 8, 128), (3, 1365, 6, 3, 64)])
@pytest.mark.parametrize("clip", [1.0, 0.9])
def test_rope_form_equals_plain_form_on_rotated_inputs(B, S, Hq, Hkv, D, clip):
    from paper_2405_16406_gb300 import spinq
    g = torch.Generator(device="cuda").manual_seed(B * S + Hq)
    q, k, v = (torch.randn(B, S, h, D, generator=g, device="cuda").half() for h in (Hq, Hkv, Hkv))
    k[..., 3] *= 16
    ang = torch.rand(S + 2, D // 2, generator=g, device="cuda") * 6.3
    cs = torch.stack([ang.cos(), ang.sin()], -1).contiguous()
    pos = torch.randint(-2, S + 5, (B, S), generator=g, device="cuda", dtype=torch.int32)   # some outside the table
    out = spinq.rope_rotate_quant_kv(q, k, v, pos, cs, clip=clip)
    ref = spinq.rotate_quant_kv(_rope(q, pos, cs), _rope(k, pos, cs), v, clip=clip)
    for f in FIELDS:
        assert torch.equal(getattr(out, f), getattr(ref, f)), f
    q2 = q.clone()
    spinq.rope_rotate_quant_kv(q2, k, v, pos, cs, clip=clip, in_place_q=True)
    assert torch.equal(q2, out.q_out)
