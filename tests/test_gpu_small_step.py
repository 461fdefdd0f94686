"""The one-kernel step of small problems against the general path.

Which of the two eta_decode takes goes by the capacity of the cache, so the same tokens in a cache with room for more than 512
blocks a sequence go the general way.  Bounds are the same arithmetic on both: masks, block counts and status must be equal bit for
bit.  Outputs are averages of the values with weights that either path computes in fp32 (exponentials to 2^-21, sums of at most
2^16 terms in another order): |difference| <= 2 * 2^-20 * max |v| <= 1.4e-5 for values up to 7.  Against the oracle the small sizes
of the other tests run."""
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _eb():
    from paper_2609_20888_b200 import binding as eb
    from paper_2609_20888_b200 import build as ebuild
    ebuild.build()
    eb.load()
    return eb


class _Side:
    """A cache of `blocks` blocks a sequence, contiguous or in pages, with its index."""

    def __init__(self, eb, K, V, lens, Hq, b, blocks, packed, paged):
        B, Hkv, T, d = K.shape
        self.eb, self.lens, self.packed = eb, lens, packed
        shape = (B, Hkv, blocks * b, d)
        self.K, self.V = torch.full(shape, 7.0, dtype=torch.bfloat16, device=DEV), torch.full(shape, -7.0, dtype=torch.bfloat16, device=DEV)
        n = min(T, blocks * b)
        self.K[:, :, :n], self.V[:, :, :n] = K[:, :, :n], V[:, :, :n]
        self.pages = None
        if paged:
            perm = torch.randperm(B * blocks, generator=torch.Generator().manual_seed(1)).to(DEV)
            pool = lambda X: torch.empty(B * blocks, Hkv, b, d, dtype=X.dtype, device=DEV).index_copy_(  # noqa: E731
                0, perm, X.view(B, Hkv, blocks, b, d).transpose(1, 2).reshape(B * blocks, Hkv, b, d))
            self.K, self.V = pool(self.K), pool(self.V)
            self.table = perm.view(B, blocks).to(torch.int32)
            self.pages = eb.page_table(self.table, B * blocks)
            self.desc = eb.paged_cache_desc(self.K, self.V, B, Hq, t_cap=blocks * b)
        else:
            self.desc = eb.cache_desc(self.K, self.V, Hq, b)
        self.musig, self.mnorm = eb.alloc_summaries(self.desc, DEV, packed=packed)
        flags = eb.ETA_BUILD_PACKED_SIGMA if packed else 0
        if paged:
            eb.eta_build_block_summaries_paged(self.desc, self.pages, self.K, lens, self.musig, self.mnorm, flags)
        else:
            eb.eta_build_block_summaries(self.desc, self.K, lens, self.musig, self.mnorm, flags)
        raw = torch.zeros(eb.eta_workspace_bytes(self.desc) + 256, dtype=torch.uint8, device=DEV)
        self.ws = raw[-raw.data_ptr() % 256:]

    def decode(self, params, q, tau, const):
        B, Hq, d = q.shape
        Hkv = self.desc.n_kv_heads
        out = torch.full((B, Hq, d), float("nan"), device=DEV)
        sel = torch.full((B, Hkv, self.desc.nb_cap), 0x55, dtype=torch.uint8, device=DEV)
        stats = torch.full((B, Hkv), -1, dtype=torch.int32, device=DEV)
        status = torch.zeros(1, dtype=torch.int32, device=DEV)
        args = (params, q, self.K, self.V, self.lens, self.musig, self.mnorm, tau, const, out, sel, self.ws)
        if self.pages is None:
            self.eb.eta_decode(self.desc, *args, stats=stats, status=status)
        else:
            self.eb.eta_decode_paged(self.desc, self.pages, *args, stats=stats, status=status)
        torch.cuda.synchronize()
        return out.cpu(), sel.cpu(), stats.cpu(), int(status)


# batch, KV heads (rows: every cluster size), G, d, b, most blocks, tokens past the last full block, what else
CASES = [
    (1, 1, 1, 64, 32, 1, 0, {}), (1, 1, 8, 128, 64, 2, 1, {}), (1, 2, 4, 64, 32, 64, 0, {}), (2, 1, 2, 128, 128, 65, 127, {}),
    (2, 2, 4, 128, 64, 70, 63, dict(paged=True)), (1, 4, 4, 128, 64, 193, 0, dict(rescue_window=1000)),
    (1, 4, 8, 64, 64, 385, 5, dict(packed=True)), (4, 2, 4, 128, 64, 192, 0, dict(rescue_window=192)),
    (1, 8, 1, 128, 64, 512, 0, {}), (2, 4, 2, 128, 32, 511, 31, dict(lwb=3)), (3, 4, 4, 128, 64, 33, 0, dict(flags=2)),
    (2, 8, 4, 128, 64, 200, 1, dict(packed=True, paged=True)), (16, 1, 8, 64, 32, 130, 7, dict(frozen=True)),
    (3, 8, 2, 64, 128, 61, 0, dict(flags=2, lwb=1)), (8, 4, 4, 128, 64, 128, 0, {}), (5, 8, 4, 64, 64, 100, 63, {}),
    (32, 2, 1, 128, 32, 64, 0, dict(rescue_window=1)), (16, 8, 4, 64, 64, 31, 2, {}),
]


@pytest.mark.parametrize("B,Hkv,G,d,b,NB,tail,kw", CASES)
def test_small_step_equals_the_general_path(B, Hkv, G, d, b, NB, tail, kw):
    eb = _eb()
    kw = dict(kw)
    packed, paged, frozen = kw.pop("packed", False), kw.pop("paged", False), kw.pop("frozen", False)
    if packed:
        kw["flags"] = kw.get("flags", 0) | eb.ETA_FLAG_PACKED_SIGMA
    Hq, T = G * Hkv, NB * b + tail
    gen = torch.Generator().manual_seed(NB * 1000 + tail * 10 + B)
    K = (torch.randn((B, Hkv, 1 + T // b, 1, d), generator=gen) + 0.6 * torch.randn((B, Hkv, 1 + T // b, b, d), generator=gen))
    K = K.reshape(B, Hkv, -1, d)[:, :, :T].bfloat16().to(DEV)
    V = torch.randn((B, Hkv, T, d), generator=gen).bfloat16().to(DEV)
    q = (torch.randn((B, Hkv, 1, d), generator=gen) + 0.3 * torch.randn((B, Hkv, G, d), generator=gen)).reshape(B, Hq, d).bfloat16().to(DEV)
    lens = torch.full((B,), T, dtype=torch.int32)
    for i, n in enumerate([T, 0, max(1, T // 2 // b * b), 1, b, max(1, T - 1), T + 9][:B]):
        lens[i] = n
    lens = lens.to(DEV)
    cap = NB + (1 if tail else 0)
    assert cap <= 512
    small = _Side(eb, K, V, lens, Hq, b, cap, packed, paged)
    # (a length beyond this cache's capacity is not beyond the other's: that one gets the clamped length)
    large = _Side(eb, K, V, lens.clamp(max=cap * b), Hq, b, 513, packed, paged)
    for level in (0.6, 1.4, float("inf"), float("-inf")):
        tau = level + 0.2 * torch.randn((B, Hq), generator=gen)
        tau, const = (None, tau[0].contiguous().to(DEV)) if frozen else (tau.to(DEV), None)
        params = eb.DecodeParams(**kw)
        got, ref = small.decode(params, q, tau, const), large.decode(params, q, tau, const)
        assert torch.equal(got[1], ref[1][:, :, :cap]) and not ref[1][:, :, cap:].any()
        assert torch.equal(got[2], ref[2])
        clamped = eb.ETA_DEV_LEN_CLAMPED if int(lens.max()) > cap * b else 0
        assert got[3] == ref[3] | clamped
        assert float((got[0] - ref[0]).abs().max()) <= 1.4e-5
        again = small.decode(params, q, tau, const)
        assert all(torch.equal(x, y) for x, y in zip(got[:3], again[:3]))


@pytest.mark.parametrize("B,Hkv,b,NB", [(255, 1, 32, 20), (256, 1, 32, 17), (257, 1, 32, 16), (32, 8, 32, 19), (129, 2, 64, 17)])
def test_a_batch_equals_its_sequences_alone(B, Hkv, b, NB):
    """Batches that the general path splits over its CTAs by up to 256 or more granules of segments, in one or more warps, against each
    sequence by itself, which goes the other way."""
    eb = _eb()
    G, d, T = 2, 64, NB * b + 9
    gen = torch.Generator().manual_seed(B)
    K = (torch.randn((B, Hkv, NB + 1, 1, d), generator=gen) + 0.6 * torch.randn((B, Hkv, NB + 1, b, d), generator=gen))
    K = K.reshape(B, Hkv, -1, d)[:, :, :T].bfloat16().to(DEV)
    V = torch.randn((B, Hkv, T, d), generator=gen).bfloat16().to(DEV)
    q = torch.randn((B, G * Hkv, d), generator=gen).bfloat16().to(DEV)
    lens = torch.randint(0, T + 1, (B,), generator=gen, dtype=torch.int32)
    lens[:4 if B > 4 else 1] = torch.tensor([T, 0, b, b - 1][:4 if B > 4 else 1], dtype=torch.int32)
    tau = (0.8 + 0.3 * torch.randn((B, G * Hkv), generator=gen)).to(DEV)
    side = _Side(eb, K, V, lens.to(DEV), G * Hkv, b, NB + 1, False, False)
    out, sel, stats, _ = side.decode(eb.DecodeParams(), q, tau, None)
    for i in range(B):
        one = _Side(eb, K[i:i + 1], V[i:i + 1], lens[i:i + 1].to(DEV), G * Hkv, b, NB + 1, False, False)
        o, m, n, _ = one.decode(eb.DecodeParams(), q[i:i + 1], tau[i:i + 1], None)
        assert torch.equal(m[0], sel[i]) and torch.equal(n[0], stats[i])
        assert float((o[0] - out[i]).abs().max()) <= 1.4e-5
