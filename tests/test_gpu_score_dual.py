"""eta_score_dual at the edges of its tiles, against the definition evaluated in double on the same records.

Both sums are accumulated in fp32 over head_dim = d products that are exact (centroid term: fp16 x fp16 after an exact
scaling; variance term: the parts of q^2 and sigma^2), so each is within d 2^-24 of the sum of its absolute terms:
|<q, mu>| <= ||q|| ||mu||, and the square root halves the variance term's relative error.  Twice that, plus 4 ulp for the
norm and the final operations, bounds the difference.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _e4m3(x):
    return x.to(torch.float8_e4m3fn).view(torch.uint8), x.to(torch.float8_e4m3fn).float()


LENS = [(32 * 31, 32 * 33 + 5), (0, 32), (32 * 129, 32 * 640 + 31)]


@pytest.mark.parametrize("lens", LENS)
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("G", [1, 2, 4, 8])
@pytest.mark.parametrize("packed", [False, True])
@pytest.mark.parametrize("room", [3, 4097])          # blocks past the longest: few bounds in all, or more than 4096 (tiles)
def test_bounds_match_the_definition(lens, d, G, packed, room):
    _check(lens, d, G, packed, 0, room)


@pytest.mark.parametrize("lens", LENS)
@pytest.mark.parametrize("d", [64, 128])
def test_bounds_of_queries_off_a_16_byte_boundary(lens, d):
    _check(lens, d, 2, False, 1, 4097)


def _check(lens, d, G, packed, offset, room):
    from paper_2609_20888_b200 import binding as eb
    Hkv, b, B = 2, 32, 2
    T = max(max(lens), 1)
    nb = T // b + room
    g = torch.Generator().manual_seed(d + G + T)
    desc = eb.CacheDesc(B, Hkv * G, Hkv, d, b, T, nb, Hkv * T * d, T * d, d, Hkv * T * d, T * d, d)
    q = torch.randn((B, Hkv * G, d), generator=g).to(torch.bfloat16)
    q[1, 0] *= 2.0 ** 50                  # outside fp16's range
    q[1, 1] *= 2.0 ** -40
    mu = torch.randn((B, Hkv, nb, d), generator=g).half()
    sg = torch.rand((B, Hkv, nb, d), generator=g).half()
    mn = torch.rand((B, Hkv, nb), generator=g) * 30
    if lens[0] >= b:
        sg[0, 0, 0, 3] = 448 if packed else float("inf")     # inf: no split into parts
        mn[0, 0, 0] = 1e4
    if packed:
        code, val = _e4m3(sg.float())
        musig = torch.cat([mu.view(torch.uint8).view(B, Hkv, nb, 2 * d), code], -1).contiguous()
        sgv = val.double()
    else:
        musig, sgv = torch.stack([mu, sg], 3).contiguous(), sg.double()
    qd = q.double().view(B, Hkv, G, d)
    dot = torch.einsum("bhgd,bhnd->bhgn", qd, mu.double())
    sq = torch.einsum("bhgd,bhnd->bhgn", qd.square(), sgv.square()).sqrt()
    qn = qd.norm(dim=3, keepdim=True)
    z, scale = 1.25, d ** -0.5
    ref = scale * torch.minimum(dot + z * sq, qn * mn.double()[:, :, None])
    tol = scale * (2 * d * 2.0 ** -24 * (qn * mu.double().norm(dim=3)[:, :, None] + z * torch.where(sq.isinf(), 0, sq)))
    tol = (tol + 4 * 2.0 ** -23 * ref.abs()).view(B, Hkv * G, nb)
    dev = "cuda:0"
    raw = torch.zeros(q.numel() + 8, dtype=torch.bfloat16, device=dev)
    qg = raw[offset:offset + q.numel()].view(q.shape)
    qg.copy_(q)
    bound = torch.full((B, Hkv * G, nb), -7.0, device=dev)
    eb.eta_score_dual(desc, eb.DecodeParams(z=z, flags=eb.ETA_FLAG_PACKED_SIGMA if packed else 0), qg,
                      torch.tensor(lens, dtype=torch.int32, device=dev), musig.to(dev), mn.to(dev), bound)
    torch.cuda.synchronize()
    got = bound.double().cpu()
    for i, t in enumerate(lens):
        n = t // b
        err = (got[i, :, :n] - ref.view(B, Hkv * G, nb)[i, :, :n]).abs()
        assert bool((err <= tol[i, :, :n]).all()), (i, float((err - tol[i, :, :n]).max()))
        assert bool((got[i, :, n:] == -7.0).all())          # blocks that are not full are left alone
