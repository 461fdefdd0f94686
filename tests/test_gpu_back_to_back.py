"""Decode steps queued one after the other: the first kernel of a step may be on the GPU before the step in front of it has
ended.  Every step has its own query and length, all share cache, index and workspace; the results are compared, bit for
bit, with the same steps run with a synchronisation after each."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,d,b,T,frozen", [
    (1, 8, 2, 64, 32, 600, False),         # launches and latency only
    (4, 16, 4, 128, 64, 4000, False),
    (8, 32, 8, 128, 32, 8190, True),       # no predictor between the append and the screening
])
def test_queued_steps_equal_separate_steps(B, Hq, Hkv, d, b, T, frozen):
    from paper_2609_20888_b200 import binding as eb
    dev, steps = "cuda:0", 40
    g = torch.Generator(device=dev).manual_seed(T)
    randn = lambda *s: torch.randn(s, generator=g, device=dev)
    cap = T + steps + b
    K, V = randn(B, Hkv, cap, d).bfloat16(), randn(B, Hkv, cap, d).bfloat16()
    q = randn(steps, B, Hq, d).bfloat16()
    W, bias = 0.1 * randn(Hq * d, Hq), torch.full((Hq,), 0.8, device=dev)
    # every step completes a block of some sequences
    lens = torch.stack([T + s + 7 * torch.arange(B, device=dev) % b for s in range(steps)]).clamp(max=cap).int()
    desc = eb.cache_desc(K, V, Hq, b)
    ws = torch.zeros(eb.eta_workspace_bytes(desc) + 256, dtype=torch.uint8, device=dev)
    ws = ws[-ws.data_ptr() % 256:]
    tau = torch.empty(B, Hq, device=dev)
    musig, mnorm = eb.alloc_summaries(desc, dev)

    def run(separately):
        musig.zero_(), mnorm.zero_()
        eb.eta_build_block_summaries(desc, K, lens[0] - 1, musig, mnorm)
        outs = torch.zeros(steps, B, Hq, d, device=dev)
        sels = torch.zeros(steps, B, Hkv, desc.nb_cap, dtype=torch.uint8, device=dev)
        status = torch.zeros(1, dtype=torch.int32, device=dev)
        torch.cuda.synchronize()
        for s in range(steps):
            eb.eta_append_summary(desc, K, lens[s], musig, mnorm)
            if not frozen:
                eb.eta_predict_threshold(q[s], W, bias, tau)
            eb.eta_decode(desc, eb.DecodeParams(), q[s], K, V, lens[s], musig, mnorm, None if frozen else tau,
                          bias if frozen else None, outs[s], sels[s], ws, status=status)
            if separately:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert int(status) == 0
        return outs, sels, musig.clone(), mnorm.clone()

    for a, c in zip(run(True), run(False)):
        assert torch.equal(a, c)


def _aligned(eb, desc, dev):
    ws = torch.zeros(eb.eta_workspace_bytes(desc) + 256, dtype=torch.uint8, device=dev)
    return ws[-ws.data_ptr() % 256:]


def _both_ways(run):
    """The results of run(after), bit for bit the same with a synchronisation after every call (after()) and without any."""
    torch.cuda.synchronize()
    want = [t.clone() for t in run(torch.cuda.synchronize)]
    torch.cuda.synchronize()
    for _ in range(3):
        got = run(lambda: None)
        torch.cuda.synchronize()
        for a, c in zip(want, got):
            assert torch.equal(a, c)


@pytest.mark.parametrize("B,Hq,Hkv,d", [(1, 8, 2, 64), (16, 32, 8, 128), (64, 16, 4, 64)])
def test_thresholds_written_where_the_step_before_left_its_output(B, Hq, Hkv, d):
    """A predictor queued right behind a step, with its thresholds in memory that the step's output has just been in (as an
    allocator hands it out): what the later call writes is what stays."""
    from paper_2609_20888_b200 import binding as eb
    dev, b, T = "cuda:0", 32, 900
    g = torch.Generator(device=dev).manual_seed(B)
    randn = lambda *s: torch.randn(s, generator=g, device=dev)
    K, V, q = randn(B, Hkv, T, d).bfloat16(), randn(B, Hkv, T, d).bfloat16(), randn(B, Hq, d).bfloat16()
    W, bias = 0.1 * randn(Hq * d, Hq), torch.full((Hq,), 0.8, device=dev)
    lens = torch.full((B,), T, dtype=torch.int32, device=dev)
    desc = eb.cache_desc(K, V, Hq, b)
    ws = _aligned(eb, desc, dev)
    musig, mnorm = eb.alloc_summaries(desc, dev)
    eb.eta_build_block_summaries(desc, K, lens, musig, mnorm)
    sel = torch.zeros(B, Hkv, desc.nb_cap, dtype=torch.uint8, device=dev)

    def run(after):
        tau = []
        for _ in range(20):
            out = torch.zeros(B, Hq, d, device=dev)
            eb.eta_decode(desc, eb.DecodeParams(), q, K, V, lens, musig, mnorm, None, bias, out, sel, ws)
            after()
            tau.append(out.view(-1)[:B * Hq].view(B, Hq))
            eb.eta_predict_threshold(q, W, bias, tau[-1])
            after()
        return [torch.stack(tau)]

    _both_ways(run)
