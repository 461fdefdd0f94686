"""Summaries of keys beyond the L2 (128 MiB), which are read with a hint that they will not be needed again: the same bytes as
a build of a few rows of them.  All rows share one row of keys."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,b,T,packed", [(128, 64, 4096 + 37, False), (64, 32, 8192 + 31, True), (128, 128, 4096, True)])
def test_large_build_equals_a_small_one(d, b, T, packed):
    from paper_2609_20888_b200 import binding as eb
    dev, Hkv = "cuda:0", 8
    g = torch.Generator(device=dev).manual_seed(T)
    K1 = torch.randn((1, 1, T, d), generator=g, device=dev).bfloat16()

    def build(B):
        K = K1.expand(B, Hkv, T, d)
        desc = eb.CacheDesc(B, Hkv, Hkv, d, b, T, T // b, *K.stride()[:3], *K.stride()[:3])
        musig, mnorm = eb.alloc_summaries(desc, dev, packed=packed)
        musig.zero_(), mnorm.zero_()
        eb.eta_build_block_summaries(desc, K, torch.full((B,), T, dtype=torch.int32, device=dev), musig, mnorm,
                                     eb.ETA_BUILD_PACKED_SIGMA if packed else 0)
        torch.cuda.synchronize()
        return musig.view(torch.uint8), mnorm

    B = (160 << 20) // (Hkv * T * d * 2) + 1
    assert B * Hkv * (T // b * b) * d * 2 > 128 << 20
    small, large = build(1), build(B)
    for x, y in zip(small, large):
        assert bool((x != 0).any()) and torch.equal(x.expand_as(y), y)
