"""Decode attention over every split of the cache length that the launch
chooses: one to eight chunks in a cluster, several clusters with a merge,
chunks that are empty or a part of a step, lengths of zero and one.

Bar: the fp16 weights p v_scale / r round by 2^-11 relative, so a head's sum
moves by at most 2^-11 times its weighted mean of |v_scale u|, at most 15
v_scale; products and sums in fp32 and the base-2 exponential add 2^-11 of the
same at most for scores below 2^9 (fp32 scores, 2^-23 relative each); the fp16
output adds 2^-11 |o|."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _nib(c):
    return torch.stack([c & 15, c >> 4], -1).reshape(*c.shape[:-1], -1).double()


@pytest.mark.parametrize("B,S,Hq,Hkv,D,lens", [
    (77, 130, 8, 8, 64, None),               # one chunk
    (38, 200, 32, 8, 128, [1, 200, 65, 0]),  # two
    (25, 321, 8, 8, 128, [16, 17, 321]),     # three
    (16, 300, 64, 8, 64, [300, 33]),         # four
    (5, 513, 96, 24, 128, [513, 80, 81]),    # five
    (2, 383, 16, 8, 64, [383, 7]),           # six
    (3, 448, 12, 3, 128, [448, 449, 112]),   # seven
    (2, 1000, 2, 1, 128, [1000, 0]),         # eight
    (1, 8193, 8, 1, 64, None),               # two clusters
    (2, 20000, 4, 2, 128, [20000, 129]),     # three clusters, most chunks empty
])
def test_every_split(B, S, Hq, Hkv, D, lens):
    from paper_2405_16406_gb300 import spinq
    g = torch.Generator(device="cuda").manual_seed(S + D)
    rnd = lambda *s: torch.rand(*s, generator=g, device="cuda")
    codes = lambda: torch.randint(0, 256, (B, S, Hkv, D // 2), dtype=torch.uint8, device="cuda", generator=g)
    cache = spinq.KVCodes(None, codes(), rnd(B, S, Hkv) * 0.2 + 0.1, -2 * rnd(B, S, Hkv),
                          codes(), rnd(B, S, Hkv) * 0.2 + 0.1, -2 * rnd(B, S, Hkv))
    q = torch.randn(B, Hq, D, generator=g, device="cuda").half()
    L = [S] * B if lens is None else [lens[b % len(lens)] for b in range(B)]
    o = torch.full_like(q, float("nan"))
    spinq.decode_attention_kv4(q, cache, lens=torch.tensor(L, dtype=torch.int32, device="cuda"), out=o)
    assert spinq.spinq_device_status()[0] == spinq.SPINQ_OK
    for b in sorted({0, 1 % B, 2 % B, B - 1}):
        n = min(L[b], S)
        if n == 0:
            assert torch.all(o[b] == 0)
            continue
        k = _nib(cache.k_codes[b, :n]) * cache.k_scale[b, :n, :, None].double() + cache.k_zero[b, :n, :, None].double()
        v = _nib(cache.v_codes[b, :n]) * cache.v_scale[b, :n, :, None].double() + cache.v_zero[b, :n, :, None].double()
        s = torch.einsum("hgd,thd->hgt", q[b].double().reshape(Hkv, -1, D), k) / D ** 0.5
        assert s.abs().max() < 512
        ref = torch.einsum("hgt,thd->hgd", torch.softmax(s, -1), v).reshape(Hq, D)
        tol = 2.0 ** -10 * 15 * cache.v_scale[b, :n].max().item() + 2.0 ** -11 * ref.abs()
        assert torch.all((o[b].double() - ref).abs() <= tol)
