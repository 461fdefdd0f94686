"""A capacity beyond twice the L2 makes the streaming kernel's copies leave the L2 first and the screening kernel start the first
survivors of every segment on their way; neither may change a result.  The same sequences are decoded through a cache of just
their size and through one whose capacity lies past the line (256 MiB of K and V)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hkv,G,d,b,nb,nb_large,paged", [
    (1, 8, 4, 128, 64, 130, 1025, False),      # a segment of 64 blocks and a remainder
    (2, 8, 2, 64, 32, 200, 2049, True),        # the pool is small, the page table's width is not
    (1, 4, 1, 128, 128, 65, 1025, False),      # two copies per block
    (1, 4, 8, 64, 32, 1, 8193, True),         # a single block
])
def test_results_do_not_depend_on_the_capacity(B, Hkv, G, d, b, nb, nb_large, paged):
    from paper_2609_20888_b200 import binding as eb
    dev = "cuda:0"
    g = torch.Generator(device=dev).manual_seed(nb + d)
    randn = lambda *s: torch.randn(s, generator=g, device=dev)
    T = nb * b + b // 2
    q, K, V = randn(B, Hkv * G, d).bfloat16(), randn(B, Hkv, T, d).bfloat16(), randn(B, Hkv, T, d).bfloat16()
    lens = torch.tensor([T] + [T - 2 * b] * (B - 1), device=dev, dtype=torch.int32)
    mu, sg = randn(B, Hkv, nb, d).half(), torch.rand((B, Hkv, nb, d), generator=g, device=dev).half()
    tau = randn(B, Hkv * G) * 0.5 + 1.0

    def decode(nb_cap, V):
        t_cap = nb_cap * b if nb_cap > nb else T
        musig = torch.zeros((B, Hkv, nb_cap, 2, d), dtype=torch.float16, device=dev)
        musig[:, :, :nb, 0], musig[:, :, :nb, 1] = mu, sg
        mn = torch.full((B, Hkv, nb_cap), 30.0, device=dev)
        pages = None
        if paged:
            per = nb + 1
            perm = torch.randperm(B * per, generator=torch.Generator().manual_seed(3)).to(dev).view(B, per)
            table = torch.full((B, max(nb_cap, per)), -1, dtype=torch.int32, device=dev)
            table[:, :per] = perm
            pool = [torch.zeros((B * per, Hkv, b, d), dtype=torch.bfloat16, device=dev) for _ in range(2)]
            for p, x in zip(pool, (K, V)):
                full = torch.zeros((B, Hkv, per * b, d), dtype=torch.bfloat16, device=dev)
                full[:, :, :T] = x
                p[perm.flatten()] = full.view(B, Hkv, per, b, d).transpose(1, 2).reshape(B * per, Hkv, b, d)
            Kc, Vc = pool
            pages = eb.PageTable(table.data_ptr(), table.shape[1], B * per)
        else:
            Kc = torch.zeros((B, Hkv, t_cap, d), dtype=torch.bfloat16, device=dev)
            Vc = torch.zeros_like(Kc)
            Kc[:, :, :T], Vc[:, :, :T] = K, V
        desc = eb.CacheDesc(B, Hkv * G, Hkv, d, b, t_cap, nb_cap, *Kc.stride()[:3], *Vc.stride()[:3])
        ws = torch.zeros(eb.eta_workspace_bytes(desc) + 256, dtype=torch.uint8, device=dev)
        ws = ws[-ws.data_ptr() % 256:]
        out = torch.empty((B, Hkv * G, d), device=dev)
        sel = torch.empty((B, Hkv, nb_cap), dtype=torch.uint8, device=dev)
        status = torch.zeros(1, dtype=torch.int32, device=dev)
        if paged:
            eb.eta_decode_paged(desc, pages, eb.DecodeParams(), q, Kc, Vc, lens, musig, mn, tau, None, out, sel, ws, status=status)
        else:
            eb.eta_decode(desc, eb.DecodeParams(), q, Kc, Vc, lens, musig, mn, tau, None, out, sel, ws, status=status)
        torch.cuda.synchronize()
        assert int(status) == 0
        return out, sel

    out, sel = decode(nb, V)
    out_l, sel_l = decode(nb_large, V)
    assert torch.equal(sel_l[..., :nb], sel) and not bool(sel_l[..., nb:].any())
    assert bool(sel.any())
    # another split of the same sums: each weight is off by 2^-17 at most (a bf16 value and its bf16 residual) and by a few
    # fp32 roundings of exponent, sum and scale, on either side
    scale = decode(nb, V.abs())[0]
    assert bool(((out_l - out).abs() <= 2 ** -15 * scale).all())
