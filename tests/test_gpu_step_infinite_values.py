"""Infinite values in blocks that a head does not attend: the head's output is that of the blocks it attends.

A tile is read once for all heads of a group, and a probability of 0 times an infinite value is a NaN in the part of a warp
that had the tile.  The one-kernel step adds up parts of twelve warps in three groups, which take a CTA's tiles in turn: here
every third block, one group's share, holds the infinities, and all heads but one attend another group's blocks."""
import numpy as np
import pytest
import torch

from oracle import eta_oracle as orc
from tests.helpers import bits, compare_masks, gpu_decode, output_errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,G,b,value", [(128, 4, 64, float("inf")), (64, 2, 32, float("-inf")), (128, 8, 32, float("nan"))])
def test_a_head_does_not_see_the_values_of_blocks_it_does_not_attend(d, G, b, value):
    nb = 24                                    # three tiles for each of the eight CTAs of the row
    rng = np.random.default_rng(d + G)
    q = torch.from_numpy(rng.standard_normal((1, G, d))).bfloat16()
    K = torch.from_numpy(0.1 * rng.standard_normal((1, 1, nb * b, d)))
    V = torch.from_numpy(rng.standard_normal((1, 1, nb * b, d)))
    blocks = lambda X: X.view(nb, b, d)  # noqa: E731
    blocks(K)[1::3] += 0.5 * q[0].double().mean(0)
    K = K.bfloat16()
    Vi = V.clone()
    blocks(Vi)[0::3] = value
    V, Vi = V.bfloat16(), Vi.bfloat16()
    lens = np.array([nb * b], np.int32)
    c = orc.Cache(bits(K), bits(V), lens, b)
    musig, mnorm = orc.block_summaries(c)
    bound = orc.score_dual(bits(q), musig, mnorm, lens, b, 1.0)
    inside, outside = bound[0, :, 1::3].min(1), np.delete(bound[0], np.s_[1::3], axis=1).max(1)
    assert (inside > outside + 1e-3).all()
    tau = ((inside + outside) / 2).astype(np.float32)[None]
    tau[0, 0] = -100.0                         # head 0 attends every block
    ref = orc.decode_step(bits(q), c, musig, mnorm, tau=tau)
    out, sel, stats, status = gpu_decode(q, K, Vi, lens, b, musig, mnorm, tau=tau)
    assert status == 0 and (stats == nb).all()
    assert not compare_masks(sel, ref["sel"], ref["bound"], tau.astype(np.float64), lens, b, G, rescued=ref["rescued"])
    assert not np.isfinite(out[0, 0]).any()
    mx, mean = output_errors(out[0, 1:], ref["out"][0, 1:])
    assert mx <= 1e-2 and mean <= 1e-3, (mx, mean)
