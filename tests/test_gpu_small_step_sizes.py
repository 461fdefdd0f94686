"""The one-kernel step against the general path over the cluster sizes and lengths that it is taken for, told apart by what the library
says it launches: both get the same descriptor, the general path from a build that takes it whatever the size.

Masks, block counts and status are the same bit for bit (the same bounds); outputs differ by the order of fp32 sums of at most 2^16
terms and exponentials to 2^-21: at most 2 * 2^-20 * max |v| <= 1.4e-5 for values up to 7."""
import pytest
import torch

from tests.test_gpu_small_step import _eb, _Side

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# batch, KV heads, G, d, b, most full blocks, tokens past them, parameters
@pytest.mark.parametrize("B,Hkv,G,d,b,NB,tail,kw", [
    (4, 1, 4, 128, 64, 511, 63, {}), (1, 4, 2, 64, 32, 512, 0, {}), (1, 1, 8, 128, 128, 64, 0, {}),       # clusters of 16
    (8, 1, 4, 128, 64, 263, 0, dict(lwb=3)), (13, 1, 2, 64, 64, 190, 5, dict(rescue_window=191)),       # of 8
    (2, 8, 4, 128, 64, 200, 0, {}), (5, 4, 1, 128, 32, 118, 3, dict(rescue_window=1)),               # of 6
    (23, 1, 4, 64, 64, 121, 0, dict(flags=2)), (8, 4, 8, 128, 64, 127, 64 - 1, {}),                   # of 5 and 4
    (11, 4, 2, 128, 64, 70, 1, {}), (8, 8, 4, 64, 32, 47, 31, {}), (16, 8, 4, 128, 64, 23, 1, {}),       # of 3, 2 and 1
])
def test_paths_agree(B, Hkv, G, d, b, NB, tail, kw):
    eb = _eb()
    from paper_2609_20888_b200 import build as ebuild
    general = eb.load(ebuild.build_general_variant())
    T = NB * b + tail
    gen = torch.Generator(device=DEV).manual_seed(NB + B)
    randn = lambda *s: torch.randn(s, generator=gen, device=DEV)  # noqa: E731
    K = (randn(B, Hkv, 1 + T // b, 1, d) + 0.6 * randn(B, Hkv, 1 + T // b, b, d)).reshape(B, Hkv, -1, d)[:, :, :T].bfloat16()
    V = randn(B, Hkv, T, d).bfloat16()
    q = (randn(B, Hkv, 1, d) + 0.3 * randn(B, Hkv, G, d)).reshape(B, Hkv * G, d).bfloat16()
    lens = torch.randint(0, T + 1, (B,), generator=gen, device=DEV, dtype=torch.int32)
    lens[0] = T
    if B > 2:
        lens[1], lens[2] = T // 2 // b * b, 0
    side = _Side(eb, K, V, lens, Hkv * G, b, NB + (1 if tail else 0), False, False)
    params = eb.DecodeParams(**kw)
    assert eb.eta_decode_launches(side.desc, params) == 1
    for level in (0.6, 1.4, float("inf"), float("-inf")):
        tau = level + 0.2 * randn(B, Hkv * G)
        got = side.decode(params, q, tau, None)
        product, eb._lib = eb._lib, general
        try:
            ref = side.decode(params, q, tau, None)
        finally:
            eb._lib = product
        assert torch.equal(got[1], ref[1]) and torch.equal(got[2], ref[2]) and got[3] == ref[3]
        assert float((got[0] - ref[0]).abs().max()) <= 1.4e-5
