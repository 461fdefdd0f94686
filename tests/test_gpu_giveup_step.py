"""A bounded wait of the one-kernel step that runs out, on purpose, without faulting or hanging anything.

A build of the same sources (-DETA_TEST_SKIP_STAGE_ARRIVE -DETA_WAIT_LIMIT=65536) in which one consumer warp of the first CTA never
releases the stages that it has read, with waits of 2^16 polls (a few milliseconds: far longer than a copy takes).  The first CTA has
more tiles than stages: the warp that issues the copies finds no free stage, gives up and lets the copies under way land; the
warps that wait for its tiles give up; all of them go on to the barriers of the cluster, which have no limit of their own, so that
the other CTAs, which wait there, leave too.  Checked: the call returns and reports ETA_DEV_TIMEOUT, rows of other clusters are as
ever, and ordinary calls on the same buffers right afterwards are correct on either path."""
import numpy as np
import pytest
import torch

from oracle import eta_oracle as orc
from tests.helpers import bits, compare_masks, heads_without_near_tie, output_errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hkv,d,b,nb", [(1, 8, 128, 64, 263), (2, 2, 64, 32, 500), (64, 2, 128, 64, 23)])
def test_a_stage_that_is_never_released_ends_in_a_timeout(B, Hkv, d, b, nb):
    from paper_2609_20888_b200 import binding as eb
    from paper_2609_20888_b200 import build as ebuild
    ebuild.build()
    eb.load()
    variant = eb.load(ebuild.build_giveup_step_variant())
    dev, G, T = "cuda:0", 2, nb * b + 5
    rng = np.random.default_rng(nb)
    cap = (nb + 1) * b
    K = torch.from_numpy(rng.standard_normal((B, Hkv, cap, d), dtype=np.float32)).bfloat16()
    V = torch.from_numpy(rng.standard_normal((B, Hkv, cap, d), dtype=np.float32)).bfloat16()
    q = torch.from_numpy(rng.standard_normal((B, Hkv * G, d), dtype=np.float32)).bfloat16()
    lens = np.full(B, T, np.int32)
    c = orc.Cache(bits(K), bits(V), lens, b)
    musig, mnorm = orc.block_summaries(c)
    bound = orc.score_dual(bits(q), musig, mnorm, lens, b, 1.0)
    tau = (np.nanquantile(bound, 0.2, axis=2) + 3e-4).astype(np.float32)
    ref = orc.decode_step(bits(q), c, musig, mnorm, tau=tau)
    Kd, Vd, qd = K.to(dev), V.to(dev), q.to(dev)
    st = eb.DecodeState(Kd, Vd, Hkv * G, b)
    st.musig.copy_(torch.from_numpy(musig.view(np.int16)).view(torch.float16))
    st.mnorm.copy_(torch.from_numpy(mnorm))
    lens_d, tau_d = torch.from_numpy(lens).to(dev), torch.from_numpy(tau).to(dev)
    assert eb.eta_decode_launches(st.desc, eb.DecodeParams()) == 1

    def call(lib=None, desc=st.desc, sel=st.sel_mask, ws=st.workspace, musig=st.musig, mnorm=st.mnorm, K=Kd, V=Vd):
        st.status.zero_()
        st.out.fill_(float("nan"))
        eb.eta_decode(desc, eb.DecodeParams(), qd, K, V, lens_d, musig, mnorm, tau_d, None, st.out, sel, ws,
                      stats=st.stats, status=st.status, lib=lib)
        torch.cuda.synchronize()
        return int(st.status)

    def check(rows, sel):
        near = compare_masks(sel.cpu().numpy()[..., :ref["sel"].shape[2]], ref["sel"], ref["bound"], tau.astype(np.float64), lens, b, G, rescued=ref["rescued"])
        keep = heads_without_near_tie(near, B, Hkv * G) & rows
        assert keep.sum() > 0.9 * rows.sum()
        mx, mean = output_errors(st.out.cpu().numpy()[keep], ref["out"][keep])
        assert mx <= 1e-2 and mean <= 1e-3, (mx, mean)

    assert call(variant) == eb.ETA_DEV_TIMEOUT, "the wait did not run out, or did not report it"
    rows = np.ones((B, Hkv * G), bool)
    rows[0, :G] = False                        # the first row is the first cluster's
    check(rows, st.sel_mask)
    rows[:] = True
    assert call() == 0
    check(rows, st.sel_mask)
    # the general path (a descriptor of more than 512 blocks, the index laid out for it)
    desc = eb.cache_desc(Kd, Vd, Hkv * G, b, nb_cap=513)
    assert eb.eta_decode_launches(desc, eb.DecodeParams()) == 3
    m2, n2 = eb.alloc_summaries(desc, dev)
    m2[:, :, :st.desc.nb_cap], n2[:, :, :st.desc.nb_cap] = st.musig, st.mnorm
    sel = torch.zeros((B, Hkv, 513), dtype=torch.uint8, device=dev)
    ws = torch.full((eb.eta_workspace_bytes(desc) + 256,), 0x5a, dtype=torch.uint8, device=dev)
    assert call(desc=desc, sel=sel, ws=ws[-ws.data_ptr() % 256:], musig=m2, mnorm=n2) == 0
    check(rows, sel)
