"""Block selection at the edges of the screening kernel's tiles, passes and groups of passes.

The reference is the selection rule on bounds evaluated in double from the same records; thresholds sit in the middle of
gaps between bounds that are wider than the 1e-5 near-tie band on either side.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hkv,G,d,nb,packed", [
    (3, 2, 4, 128, 65, False),       # one record past a segment
    (2, 4, 1, 128, 15, True),        # less than a tile
    (2, 2, 8, 64, 129, False),       # one record past a pass of 128 records
    (64, 16, 1, 64, 700, False),     # more rows than CTA slots: six passes per CTA, a second group of passes
    (128, 8, 2, 128, 330, True),     # the same with 64-record passes
    (1, 1, 4, 128, 4096, False),     # one row over many CTAs
])
def test_selection_matches_the_rule(B, Hkv, G, d, nb, packed):
    from paper_2609_20888_b200 import binding as eb
    dev, b = "cuda:0", 32
    g = torch.Generator(device=dev).manual_seed(nb + d)
    lens = torch.randint(0, nb * b + 1, (B,), generator=g, device=dev, dtype=torch.int32)
    lens[0] = nb * b
    T = nb * b
    # K and V are never looked at by the rule: all heads of all sequences share one row
    K = torch.zeros((1, 1, T, d), dtype=torch.bfloat16, device=dev).expand(B, Hkv, T, d)
    desc = eb.CacheDesc(B, Hkv * G, Hkv, d, b, T, nb, 0, 0, d, 0, 0, d)
    q = torch.randn((B, Hkv * G, d), generator=g, device=dev).to(torch.bfloat16)
    mu = torch.randn((B, Hkv, nb, d), generator=g, device=dev).half()
    sg = torch.rand((B, Hkv, nb, d), generator=g, device=dev).half()
    if packed:
        code = sg.float().to(torch.float8_e4m3fn)
        musig = torch.cat([mu.view(torch.uint8).view(B, Hkv, nb, 2 * d), code.view(torch.uint8)], -1).contiguous()
        sgv = code.double()
    else:
        musig, sgv = torch.stack([mu, sg], 3).contiguous(), sg.double()
    mn = torch.full((B, Hkv, nb), 30.0, device=dev)
    qd = q.double().view(B, Hkv, G, d)
    bound = torch.empty((B, Hkv, G, nb), dtype=torch.float64, device=dev)
    for i in range(B):
        dot = torch.einsum("hgd,hnd->hgn", qd[i], mu[i].double())
        sq = torch.einsum("hgd,hnd->hgn", qd[i].square(), sgv[i].square()).sqrt()
        bound[i] = torch.minimum(dot + sq, qd[i].norm(dim=2, keepdim=True) * 30.0) * d ** -0.5
    full = torch.arange(nb, device=dev)[None, :] < (lens // b)[:, None]
    full = full[:, None, None, :].expand_as(bound)
    srt = bound.masked_fill(~full, -1e3).sort(dim=3).values
    gap = srt[..., 1:] - srt[..., :-1] if nb > 1 else torch.zeros_like(srt)
    at = gap[..., nb // 2:].argmax(3) + nb // 2               # a wide gap in the upper half
    tau = ((srt.gather(3, at[..., None]) + srt.gather(3, at[..., None] + 1)) / 2)[..., 0].float()
    tau = torch.where(gap.gather(3, at[..., None])[..., 0] > 4e-5, tau, -50.0)
    want = full & (bound >= tau.double()[..., None])
    near = full & ((bound - tau.double()[..., None]).abs() <= 1e-5)
    # top-1 rescue in the first 128 blocks for a head that admits none of them
    window = want[..., :128].any(3)
    best = bound.masked_fill(~full, -1e9)[..., :128].argmax(3, keepdim=True)
    resc = torch.zeros_like(want).scatter_(3, best, True) & full & ~window[..., None]
    want = want | resc
    ws = torch.zeros(eb.eta_workspace_bytes(desc) + 256, dtype=torch.uint8, device=dev)
    ws = ws[-ws.data_ptr() % 256:]
    out = torch.empty((B, Hkv * G, d), device=dev)
    sel = torch.zeros((B, Hkv, nb), dtype=torch.uint8, device=dev)
    stats = torch.zeros((B, Hkv), dtype=torch.int32, device=dev)
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    eb.eta_decode(desc, eb.DecodeParams(flags=eb.ETA_FLAG_PACKED_SIGMA if packed else 0), q, K, K, lens, musig, mn,
                  tau.reshape(B, Hkv * G).contiguous(), None, out, sel, ws, stats=stats, status=status)
    torch.cuda.synchronize()
    assert int(status) & ~4 == 0                                # only "some sequence is empty" may be reported
    got = torch.stack([(sel >> k) & 1 for k in range(G)], 2).bool()
    assert not bool(near.any())
    assert torch.equal(got, want), int((got != want).sum())
    assert torch.equal(stats.long(), want.any(2).sum(2))
    assert torch.equal(out, torch.zeros_like(out))
