"""The root search of the offline calibration on its own: the constant in double precision that the kernels leave in the
scratch against a bisection, in numpy, of the same equation on the histogram and the density they left there.

Bound: both sides evaluate g(c) = sum_b H[b] sigmoid(beta (s_b - c)) in double; with H >= 0 and sum H = 1 the sum of n_bins
terms is off by at most n_bins 2^-53 + a few 2^-52 for the exponentials, and a relative 2^-53 per partial sum of the density,
which moves the root by that over |g'|.  The last step of the search leaves beta d^2 / 2 for a step of beta d <= 2e-8."""
import numpy as np
import pytest
import torch

from tests.helpers import calibration_scratch

pytestmark = pytest.mark.gpu


def _g(H, s, beta, c):
    x = beta * (s - c)
    e = np.exp(-np.abs(x))
    return float((H * np.where(x >= 0, 1.0, e) / (1.0 + e)).sum()), float((H * beta * e / (1.0 + e) ** 2).sum())


# one bin per thread and its neighbours, the most bins, the fewest; thresholds below, within and far above the scores; gates
# that are nearly steps and nearly constant
@pytest.mark.parametrize("n_bins,beta,mean", [(511, 5.0, 0.3), (512, 5.0, -3.0), (513, 50.0, 0.3), (4096, 0.5, 1.0), (2, 5.0, 0.0),
                                              (1000, 5.0, 4.0), (2048, 5.0, 6.0), (2048, 20.0, 2.0), (4095, 5.0, 0.5)])
def test_root_of_the_density_equation(n_bins, beta, mean):
    from paper_2609_20888_b200 import binding as eb
    from paper_2609_20888_b200 import build as ebuild
    ebuild.build()
    dev = torch.device("cuda:0")
    n_seq, Hq, T, d, lim = 2, 8, 300, 64, 8.0
    gen = torch.Generator().manual_seed(n_bins)
    Q = torch.randn((n_seq, Hq, T, d), generator=gen).to(torch.bfloat16).to(dev)
    K = torch.randn((n_seq, 4, T, d), generator=gen).to(torch.bfloat16).to(dev)
    tau = (mean + 0.4 * torch.randn((n_seq, Hq, T), generator=gen)).to(dev)
    hc, dbar = torch.empty(Hq, device=dev), torch.empty(Hq, device=dev)
    ws = eb.eta_calibrate_head_const(Q, K, tau, hc, dbar, beta=beta, n_bins=n_bins, s_min=-lim, s_max=lim)
    torch.cuda.synchronize()
    H, parts, got = calibration_scratch(ws, n_seq, Hq, T, n_bins)
    H = H.astype(np.float64)
    s = -lim + (np.arange(n_bins) + 0.5) * (2 * lim / n_bins)
    for h in range(Hq):
        Hn, target = H[h] / H[h].sum(), parts[:, h].sum() / (n_seq * T)
        lo, hi = -lim - 40.0 / beta, lim + 40.0 / beta
        for _ in range(200):
            c = (lo + hi) / 2
            lo, hi = (c, hi) if _g(Hn, s, beta, c)[0] > target else (lo, c)
        slope = _g(Hn, s, beta, c)[1]
        bound = (n_bins * 2.0 ** -53 + 2.0 ** -48) / slope + 2e-16 / beta + 1e-14 * (lim + 40.0 / beta)
        assert abs(got[h] - c) <= bound, (h, got[h], c, bound)
        assert hc[h].item() == np.float32(got[h]) and abs(dbar[h].item() - target) <= 2.0 ** -24 * target
