"""What eta_decode_launches says of a call is what the call does: the one-kernel step leaves the workspace alone, the general path
writes it (a survivor count per segment at least)."""
import json
import os
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("B,Hkv,G,d,b,nb,kw,launches", [
    (1, 2, 4, 64, 32, 64, {}, 1), (8, 1, 4, 128, 64, 263, {}, 1), (4, 1, 1, 128, 128, 256, dict(rescue_window=1 << 20), 1),
    (16, 8, 2, 64, 64, 24, dict(flags=4), 1),                              # one CTA a row
    (1, 2, 4, 64, 32, 513, {}, 3), (6, 1, 4, 128, 64, 511, {}, 3), (96, 1, 4, 128, 64, 32, {}, 3), (1, 2, 4, 64, 32, 64, dict(flags=1), 3),
    (1, 1, 4, 128, 64, 700, dict(rescue_window=129), 4), (1, 1, 4, 128, 64, 700, dict(rescue_window=128), 3),
    (1, 1, 4, 64, 64, 700, dict(rescue_window=257), 4), (1, 1, 4, 128, 64, 700, dict(rescue_window=700, flags=1), 3),
])
def test_launches_are_what_the_call_does(B, Hkv, G, d, b, nb, kw, launches):
    from paper_2609_20888_b200 import binding as eb
    dev = "cuda:0"
    K = torch.zeros((1, 1, nb * b, d), dtype=torch.bfloat16, device=dev)
    desc = eb.CacheDesc(B, Hkv * G, Hkv, d, b, nb * b, nb, 0, 0, d, 0, 0, d)
    params = eb.DecodeParams(**kw)
    assert eb.eta_decode_launches(desc, params) == launches
    musig, mnorm = eb.alloc_summaries(desc, dev, packed=bool(params.flags & eb.ETA_FLAG_PACKED_SIGMA))
    ws = torch.full((eb.eta_workspace_bytes(desc) + 256,), 0x5a, dtype=torch.uint8, device=dev)
    ws = ws[-ws.data_ptr() % 256:]
    out = torch.full((B, Hkv * G, d), float("nan"), device=dev)
    sel = torch.empty((B, Hkv, nb), dtype=torch.uint8, device=dev)
    eb.eta_decode(desc, params, torch.zeros((B, Hkv * G, d), dtype=torch.bfloat16, device=dev), K, K,
                  torch.full((B,), nb * b, dtype=torch.int32, device=dev), musig, mnorm, torch.zeros((B, Hkv * G), device=dev), None, out, sel, ws)
    torch.cuda.synchronize()
    assert bool((ws == 0x5a).all()) == (launches == 1)
    assert not out.isnan().any() and bool((sel == (1 << G) - 1).all())       # a bound of 0 is not below a threshold of 0


def test_the_first_call_of_a_process_may_be_captured():
    """What the library asks of the device on a first call (attributes, clusters that fit) is allowed during a capture."""
    code = """if True:
        import torch
        from paper_2609_20888_b200 import binding as eb
        dev, B, Hkv, G, d, b, nb = "cuda:0", 2, 4, 4, 128, 64, 100
        K = torch.randn((B, Hkv, nb * b, d), device=dev).bfloat16()
        st = eb.DecodeState(K, K, Hkv * G, b)
        q, tau = torch.randn((B, Hkv * G, d), device=dev).bfloat16(), torch.zeros((B, Hkv * G), device=dev)
        lens = torch.full((B,), nb * b - 5, dtype=torch.int32, device=dev)
        run = lambda: eb.eta_decode(st.desc, eb.DecodeParams(), q, K, K, lens, st.musig, st.mnorm, tau, None, st.out, st.sel_mask, st.workspace)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            run()
        g.replay()
        got = st.out.clone()
        assert eb.eta_decode_launches(st.desc, eb.DecodeParams()) == 1
        run()
        assert torch.equal(got, st.out) and float(got.abs().max()) > 0
    """
    out = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]


def test_bench_counts_the_launches_of_a_small_workload():
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--workload", "c1_tiny", "--steps", "4", "--warmup", "3", "--no-cpu",
                          "--no-sweep"], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert out.returncode == 0, out.stderr[-2000:]
    line = json.loads(out.stdout.strip().splitlines()[-1])
    assert line["gpu_launches"] == 4 * 3 and line["roofline"]["kernel"] == "step_kernel"
