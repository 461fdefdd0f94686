"""Top-1 rescue with windows longer than what the first CTA of a row screens (rescue_kernel settles those), against the oracle.

Heads 0 and 1 of every group ask the same query with a threshold nothing reaches, so both rescue the same block.  In the first
group another head with that query admits exactly that block (its bit joins an entry that exists), in the second nobody
does (the entry is new).  The block with the largest bound lies past the first CTA's passes.
"""
import numpy as np
import pytest
import torch

from oracle import eta_oracle as orc
from tests.helpers import bits, compare_masks, gpu_decode, heads_without_near_tie, output_errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,G,nb,window", [
    (128, 4, 700, 1 << 30), (128, 8, 300, 257), (128, 4, 330, 256), (128, 8, 200, 129), (128, 2, 129, 1 << 30),
    (64, 8, 1200, 1 << 30), (64, 4, 530, 513), (64, 8, 530, 512), (64, 1, 260, 257),
])
def test_long_windows_match_the_oracle(d, G, nb, window):
    B, Hkv, b = 3, 2, 32
    T = nb * b
    rng = np.random.default_rng(nb + d + G)
    K = torch.from_numpy(rng.standard_normal((B, Hkv, T, d))).to(torch.bfloat16)
    V = torch.from_numpy(rng.standard_normal((B, Hkv, T, d))).to(torch.bfloat16)
    lens = np.array([T, T - 7, 5 * b + 3], np.int32)                    # the last one shorter than any window
    q = torch.from_numpy(rng.standard_normal((B, Hkv * G, d))).to(torch.bfloat16).view(B, Hkv, G, d)
    twins = [h for h in (0, 1, 3) if h < G]
    q[:, :, twins] = q[:, :, :1].clone()
    best = min(window, nb) - 3                                          # late in the window, and a larger one past its end
    for j, strength in ((best, 0.5), (best + 4, 0.9)):
        K[:2, :, j * b:(j + 1) * b] += strength * q[:2, :, :1]
    q = q.reshape(B, Hkv * G, d)
    c = orc.Cache(bits(K), bits(V), lens, b)
    musig, mnorm = orc.block_summaries(c)
    bound = orc.score_dual(bits(q), musig, mnorm, lens, b, 1.0)
    tau = np.full((B, Hkv, G), np.inf, np.float32)
    for i in range(B):
        n = int(lens[i]) // b
        for h in range(4, G):                                           # ordinary heads beside them
            tau[i, :, h] = np.quantile(bound[i].reshape(Hkv, G, nb)[:, h, :n], 0.97, axis=1) + 2e-4
        if G > 3:                                                       # between the largest bound of the window and the next
            top = np.sort(bound[i, 3, :min(n, window)])[-2:]
            tau[i, 0, 3] = top.mean()
            assert top[1] - top[0] > 1e-4
    tau = tau.reshape(B, Hkv * G)
    ref = orc.decode_step(bits(q), c, musig, mnorm, tau=tau, rescue_window=window)
    assert (ref["rescued"].reshape(B, Hkv, G)[:2, :, 0] == best).all()
    out, sel, stats, status = gpu_decode(q, K, V, lens, b, musig, mnorm, tau=tau, rescue_window=window)
    assert status == 0
    near = compare_masks(sel, ref["sel"], ref["bound"], tau.astype(np.float64), lens, b, G, rescued=ref["rescued"])
    keep = heads_without_near_tie(near, B, Hkv * G)
    assert keep.mean() > 0.9
    mx, mean = output_errors(out[keep], ref["out"][keep])
    assert mx <= 1e-2 and mean <= 1e-3, (mx, mean)
    assert np.array_equal(stats, [[int((sel[i, hk, :int(lens[i]) // b] != 0).sum()) for hk in range(Hkv)] for i in range(B)])


def _step(rows, nb, G, tau, d=128, b=32):
    """A step on synthetic records (K and V are one row of zeros that all rows share); -> function of the window, mask, bounds"""
    from paper_2609_20888_b200 import binding as eb
    dev = "cuda:0"
    g = torch.Generator(device=dev).manual_seed(1)
    K = torch.zeros((1, 1, nb * b, d), dtype=torch.bfloat16, device=dev)
    desc = eb.CacheDesc(rows, G, 1, d, b, nb * b, nb, 0, 0, d, 0, 0, d)
    q = torch.randn((rows, G, d), generator=g, device=dev).to(torch.bfloat16)
    musig = torch.rand((rows, 1, nb, 2, d), generator=g, device=dev).half()
    mn = torch.full((rows, 1, nb), 30.0, device=dev)
    taus = torch.full((rows, G), tau, device=dev)
    lens = torch.full((rows,), nb * b, dtype=torch.int32, device=dev)
    ws = torch.zeros(eb.eta_workspace_bytes(desc) + 256, dtype=torch.uint8, device=dev)
    ws = ws[-ws.data_ptr() % 256:]
    out, sel = torch.empty((rows, G, d), device=dev), torch.zeros((rows, 1, nb), dtype=torch.uint8, device=dev)
    bound = torch.empty((rows, G, nb), device=dev)
    eb.eta_score_dual(desc, eb.DecodeParams(), q, lens, musig, mn, bound)
    run = lambda window: eb.eta_decode(desc, eb.DecodeParams(rescue_window=window), q, K, K, lens, musig, mn, taus, None, out, sel, ws)
    return run, sel, bound


def test_a_window_of_several_groups_of_passes_in_one_cta():
    """Rows that are one CTA's work each: it settles a window longer than the bounds it keeps at a time.  600 rows of counts are also
    more than the streaming kernel reads in one round trip."""
    G, nb = 2, 640                                     # ten passes of 64 blocks, four of them at a time
    run, sel, bound = _step(600, nb, G, 1e30)
    run(nb - 1)
    torch.cuda.synchronize()
    best = bound[..., :nb - 1].argmax(2)
    want = torch.zeros((600, nb), dtype=torch.uint8, device=sel.device)
    for h in range(G):
        want[torch.arange(600, device=sel.device), best[:, h]] |= 1 << h
    assert torch.equal(sel[:, 0], want)


def test_a_long_window_is_not_one_ctas_work():
    """One row of 16384 blocks: with the whole row as its window a step takes little more than with 128 blocks (screened one pass
    after another by a single CTA it would take ten times as long; the bound is far from both)."""
    run, _, _ = _step(1, 16384, 4, 1e30)

    def us(window):
        best = float("inf")
        for _ in range(6):
            a, z = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                run(window)
            z.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(z) * 50)
        return best

    short, whole = us(128), us(16384)
    assert whole < 2 * short, (short, whole)
