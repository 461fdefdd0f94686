"""The calibration's histogram with two copies of its planes (up to 2048 bins) against the one with one: of bins half as wide, two
neighbours hold what one of the wide bins holds, exactly (a width that is halved scales a score's place by two, which rounds
nothing)."""
import pytest
import torch

from tests.helpers import calibration_scratch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bins,T,d,spread", [(2048, 700, 128, 1.0), (2047, 513, 64, 3.0), (1025, 1025, 128, 0.0), (2048, 129, 64, 0.02)])
def test_two_copies_hold_what_one_holds(n_bins, T, d, spread):
    from paper_2609_20888_b200 import binding as eb
    from paper_2609_20888_b200 import build as ebuild
    ebuild.build()
    n_seq, Hq, dev = 2, 4, "cuda:0"
    gen = torch.Generator().manual_seed(T)
    Q = (spread * torch.randn((n_seq, Hq, T, d), generator=gen)).bfloat16().to(dev)
    K = torch.randn((n_seq, 2, T, d), generator=gen).bfloat16().to(dev)
    tau = torch.randn((n_seq, Hq, T), generator=gen).to(dev)
    H = []
    for bins in (n_bins, 2 * n_bins):
        hc, dbar = torch.empty(Hq, device=dev), torch.empty(Hq, device=dev)
        ws = eb.eta_calibrate_head_const(Q, K, tau, hc, dbar, n_bins=bins)
        torch.cuda.synchronize()
        H.append((calibration_scratch(ws, n_seq, Hq, T, bins)[0], dbar))
    assert (H[1][0].reshape(Hq, n_bins, 2).sum(axis=2) == H[0][0]).all()
    assert torch.equal(H[0][1], H[1][1])
    total = n_seq * sum(t * ((2 ** 40 + t // 2) // t) for t in range(1, T + 1))
    assert [int(h.sum()) for h in H[0][0]] == [total] * Hq
