"""What the fp16 rounding of the value product's weights may cost in decode
attention.  The weights P' = p v_scale / r are rounded by 2^-11 relative (p the
softmax weight, r the largest v_scale a warp meets), and the kernel adds back
8 (p v_scale - P' r) in fp32, so an element moves by at most 2^-11 times the
weighted mean of |v_scale (u - 8)|, not of v_scale u.  With every code 8 and
v_zero close to -8 v_scale that term vanishes and the outputs are small.

Beside it: fp32 scores of magnitude below 2^6 and the base-2 exponential move p
by at most 2^-14 relative, fp32 sums of at most 2^9 terms a lane of size
8 v_scale and v_zero add 2^-18 of them, fp16 rounds the output by 2^-11."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _nib(c):
    return torch.stack([c & 15, c >> 4], -1).reshape(*c.shape[:-1], -1).double()


@pytest.mark.parametrize("B,S,Hq,Hkv,D", [(3, 200, 32, 8, 128), (1, 2048, 32, 8, 128), (2, 700, 8, 1, 64),
                                          (2, 1432, 8, 2, 128), (4, 951, 8, 4, 64), (77, 130, 8, 8, 64)])
@pytest.mark.parametrize("eights", [True, False])
def test_rounding_of_the_weights(B, S, Hq, Hkv, D, eights):
    from paper_2405_16406_gb300 import spinq
    g = torch.Generator(device="cuda").manual_seed(S + D)
    rnd = lambda *s: torch.rand(*s, generator=g, device="cuda")
    codes = lambda: torch.randint(0, 256, (B, S, Hkv, D // 2), dtype=torch.uint8, device="cuda", generator=g)
    vs = rnd(B, S, Hkv) * 0.2 + 0.1
    vz = -8 * vs + 0.02 * rnd(B, S, Hkv) if eights else -2 * rnd(B, S, Hkv)
    vc = torch.full((B, S, Hkv, D // 2), 0x88, dtype=torch.uint8, device="cuda") if eights else codes()
    cache = spinq.KVCodes(None, codes(), rnd(B, S, Hkv) * 0.04 + 0.02, -0.3 * rnd(B, S, Hkv), vc, vs, vz)
    q = torch.randn(B, Hq, D, generator=g, device="cuda").half()
    o = spinq.decode_attention_kv4(q, cache)
    for b in sorted({0, B // 2, B - 1}):
        k = _nib(cache.k_codes[b]) * cache.k_scale[b, ..., None].double() + cache.k_zero[b, ..., None].double()
        s = torch.einsum("hgd,thd->hgt", q[b].double().reshape(Hkv, -1, D), k) / D ** 0.5
        assert s.abs().max() < 64
        p = torch.softmax(s, -1)
        u, a, z = _nib(vc[b]), vs[b, ..., None].double(), vz[b, ..., None].double()
        mean = lambda t: torch.einsum("hgt,thd->hgd", p, t).reshape(Hq, D)
        ref = mean(a * u + z)
        tol = (2.0 ** -11 * mean(a * (u - 8).abs()) + 2.0 ** -14 * mean((a * u + z).abs())
               + 2.0 ** -18 * mean((8 * a + z.abs()).expand_as(u)) + 2.0 ** -11 * ref.abs() + 2.0 ** -25)
        assert torch.all((o[b].double() - ref).abs() <= tol)
