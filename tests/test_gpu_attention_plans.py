"""Decode attention over long caches: the chunks that the SMs take at once (the
workspace holds that many partial results) are all used, or nearly so, once the
cache is long enough for their merge to pay, and every cut gives the attention
of the reference.  A cut into several clusters shows in the workspace, which
then receives (max, sum, o[D]) of each cluster.

Bar as in the other split tests: the fp16 weights move an element by at most
2^-10 times 15 v_scale, the fp16 output by 2^-11 of itself."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _nib(c):
    return torch.stack([c & 15, c >> 4], -1).reshape(*c.shape[:-1], -1).double()


# sequences * kv heads: 72 -> 8 chunks, 67 -> 9, 56 -> 10, 48 -> 12, 43 -> 14, 40 -> 15, 38 -> 16, 32 -> 19, 24 -> 25,
# 21 -> 28, 16 -> 38 (152 SMs)
@pytest.mark.parametrize("B,Hq,Hkv,D,S,most_idle", [
    (67, 1, 1, 64, 16385, 0), (7, 16, 8, 64, 12289, 0), (6, 8, 8, 64, 7000, 0), (43, 2, 1, 64, 6145, 0),
    (5, 32, 8, 128, 8193, 1), (38, 1, 1, 128, 12289, 0), (4, 8, 8, 64, 20000, 0), (3, 8, 8, 64, 10300, 1),
    (3, 8, 8, 64, 25000, 0), (21, 4, 1, 128, 30000, 0), (2, 16, 8, 64, 40000, 2), (9, 8, 8, 64, 41000, 0)])
@pytest.mark.parametrize("ragged", [False, True])
def test_long_caches_use_the_chunks(B, Hq, Hkv, D, S, most_idle, ragged):
    from paper_2405_16406_gb300 import spinq
    g = torch.Generator(device="cuda").manual_seed(S + D + B)
    rnd = lambda *s: torch.rand(*s, generator=g, device="cuda")
    codes = lambda: torch.randint(0, 256, (B, S, Hkv, D // 2), dtype=torch.uint8, device="cuda", generator=g)
    cache = spinq.KVCodes(None, codes(), rnd(B, S, Hkv) * 0.2 + 0.1, -2 * rnd(B, S, Hkv),
                          codes(), rnd(B, S, Hkv) * 0.2 + 0.1, -2 * rnd(B, S, Hkv))
    q = torch.randn(B, Hq, D, generator=g, device="cuda").half()
    lens = torch.full((B,), S, dtype=torch.int32, device="cuda")
    if ragged:
        lens[0], lens[-1] = 0, S - 1
        lens[B // 2] = 17
    need = spinq.spinq_decode_attention_workspace_bytes(B, S, Hq, Hkv, D)
    n = need // (B * Hq * (D + 2) * 4)
    ws = torch.full((need // 4,), float("nan"), device="cuda")
    o = torch.full_like(q, float("nan"))
    spinq.decode_attention_kv4(q, cache, lens=lens, out=o, workspace=ws.view(torch.uint8))
    assert spinq.spinq_device_status()[0] == spinq.SPINQ_OK
    written = (~torch.isnan(ws)).sum().item()
    clusters = written // (B * Hq * (D + 2))
    assert written == clusters * B * Hq * (D + 2) and clusters > 1
    # a cluster has at most 8 CTAs, the same number in each
    assert n - clusters * min(8, n // clusters) <= most_idle
    for b in sorted({0, B // 2, B - 1}):
        m = int(lens[b])
        if m == 0:
            assert torch.all(o[b] == 0)
            continue
        k = _nib(cache.k_codes[b, :m]) * cache.k_scale[b, :m, :, None].double() + cache.k_zero[b, :m, :, None].double()
        v = _nib(cache.v_codes[b, :m]) * cache.v_scale[b, :m, :, None].double() + cache.v_zero[b, :m, :, None].double()
        s = torch.einsum("hgd,thd->hgt", q[b].double().reshape(Hkv, -1, D), k) / D ** 0.5
        assert s.abs().max() < 512
        ref = torch.einsum("hgt,thd->hgd", torch.softmax(s, -1), v).reshape(Hq, D)
        tol = 2.0 ** -10 * 15 * cache.v_scale[b, :m].max().item() + 2.0 ** -11 * ref.abs()
        assert torch.all((o[b].double() - ref).abs() <= tol)
