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


@pytest.mark.parametrize("paged", [False, True])
def test_records_do_not_depend_on_the_capacity(paged):
    """What decides how the keys are read is how long a sequence is, not the room it has: short and long sequences of one build,
    on either side of the line of 128 MiB (here 16384 tokens a sequence), give the bytes of a build of just their size."""
    from paper_2609_20888_b200 import binding as eb
    dev, B, Hkv, d, b, T = "cuda:0", 4, 8, 128, 64, 18432
    g = torch.Generator(device=dev).manual_seed(5)
    lens = torch.tensor([T, 16384, 16383, 700], dtype=torch.int32, device=dev)
    K = torch.empty((B, Hkv, T, d), dtype=torch.bfloat16, device=dev).normal_(generator=g)
    want = []
    for i in range(B):                       # one at a time: far below the line
        desc = eb.cache_desc(K[i:i + 1], K[i:i + 1], Hkv, b)
        mu, mn = eb.alloc_summaries(desc, dev)
        eb.eta_build_block_summaries(desc, K[i:i + 1], lens[i:i + 1], mu, mn)
        want.append((mu, mn))
    if paged:
        nb = T // b
        pool = K.view(B, Hkv, nb, b, d).transpose(1, 2).reshape(B * nb, Hkv, b, d).contiguous()
        table = torch.arange(B * nb, dtype=torch.int32, device=dev).view(B, nb)
        desc = eb.paged_cache_desc(pool, pool, B, Hkv, t_cap=T)
        mu, mn = eb.alloc_summaries(desc, dev)
        eb.eta_build_block_summaries_paged(desc, eb.page_table(table, B * nb), pool, lens, mu, mn)
    else:
        wide = torch.zeros((B, Hkv, 2 * T, d), dtype=torch.bfloat16, device=dev)
        wide[:, :, :T] = K
        desc = eb.cache_desc(wide, wide, Hkv, b)
        mu, mn = eb.alloc_summaries(desc, dev)
        eb.eta_build_block_summaries(desc, wide, lens, mu, mn)
    torch.cuda.synchronize()
    for i in range(B):
        assert torch.equal(mu[i, :, :T // b], want[i][0][0]) and torch.equal(mn[i, :, :T // b], want[i][1][0])
