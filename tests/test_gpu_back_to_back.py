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
    """The results of run(after), bit for bit the same with a synchronisation after every call (after()) and without any: a
    kernel of some 5 ms goes in front then, so that the calls pile up behind it and run one right after the other."""
    torch.cuda.synchronize()
    want = [t.clone() for t in run(torch.cuda.synchronize)]
    torch.cuda.synchronize()
    for _ in range(3):
        pile_up = iter([10_000_000])
        got = run(lambda: [torch.cuda._sleep(n) for n in pile_up])
        torch.cuda.synchronize()
        for a, c in zip(want, got):
            assert torch.equal(a, c)


@pytest.mark.parametrize("d,refill", [(64, False), (128, False), (128, True)])
def test_queued_calibrations_share_a_scratch(d, refill):
    """Calibrations of different sizes and inputs on one scratch (each clears what the root search of the one before reads), two
    in three followed by a step that uses the constants; refill: the inputs are written by a kernel right before the call."""
    from paper_2609_20888_b200 import binding as eb
    dev, Hq, Hkv, n_bins, b, T = "cuda:0", 8, 2, 513, 32, 2048
    g = torch.Generator(device=dev).manual_seed(d)
    randn = lambda *s: torch.randn(s, generator=g, device=dev)
    sizes = [(1, 1), (2, 64), (3, 130), (1, 257), (4, 300), (2, 96)] * 3
    splits = [(randn(n, Hq, t, d).bfloat16(), randn(n, Hkv, t, d).bfloat16(), 0.3 + 0.5 * randn(n, Hq, t)) for n, t in sizes]
    bufs = {s: tuple(torch.empty_like(x) for x in splits[k]) for k, s in enumerate(sizes)}
    scratch = torch.zeros(1 << 20, dtype=torch.uint8, device=dev)
    scratch = scratch[-scratch.data_ptr() % 256:]
    K, V, q = randn(1, Hkv, T, d).bfloat16(), randn(1, Hkv, T, d).bfloat16(), randn(1, Hq, d).bfloat16()
    lens = torch.full((1,), T - 5, dtype=torch.int32, device=dev)
    desc = eb.cache_desc(K, V, Hq, b)
    ws = _aligned(eb, desc, dev)
    musig, mnorm = eb.alloc_summaries(desc, dev)
    eb.eta_build_block_summaries(desc, K, lens, musig, mnorm)

    def run(after):
        const, dbar = torch.zeros(len(sizes), Hq, device=dev), torch.zeros(len(sizes), Hq, device=dev)
        outs = torch.zeros(len(sizes), 1, Hq, d, device=dev)
        sel = torch.zeros(len(sizes), 1, Hkv, desc.nb_cap, dtype=torch.uint8, device=dev)
        for k, split in enumerate(splits):
            if refill:
                for x, y in zip(bufs[sizes[k]], split):
                    x.copy_(y)
                split = bufs[sizes[k]]
            after()
            eb.eta_calibrate_head_const(*split, const[k], dbar[k], n_bins=n_bins, workspace=scratch)
            after()
            if k % 3:
                eb.eta_decode(desc, eb.DecodeParams(), q, K, V, lens, musig, mnorm, None, const[k], outs[k], sel[k], ws)
                after()
        return const, dbar, outs, sel

    _both_ways(run)


@pytest.mark.parametrize("append", [True, False])
@pytest.mark.parametrize("B,Hq,Hkv,d,b,T", [(1, 8, 2, 64, 32, 600), (2, 32, 8, 128, 64, 9000), (16, 32, 4, 64, 32, 1500)])
def test_queued_steps_fetch_their_queries_into_one_buffer(B, Hq, Hkv, d, b, T, append):
    """Every step fetches its own query from the host into the buffer that the step before it may still be reading."""
    from paper_2609_20888_b200 import binding as eb
    dev, steps = "cuda:0", 40
    g = torch.Generator(device=dev).manual_seed(T)
    randn = lambda *s: torch.randn(s, generator=g, device=dev)
    cap = T + steps + b
    K, V = randn(B, Hkv, cap, d).bfloat16(), randn(B, Hkv, cap, d).bfloat16()
    q_host = randn(steps, B, Hq, d).bfloat16().cpu().pin_memory()
    W, bias = 0.1 * randn(Hq * d, Hq), torch.full((Hq,), 0.8, device=dev)
    lens = torch.stack([T + s + 7 * torch.arange(B, device=dev) % b for s in range(steps)]).clamp(max=cap).int()
    desc = eb.cache_desc(K, V, Hq, b)
    ws = _aligned(eb, desc, dev)
    tau, q = torch.empty(B, Hq, device=dev), torch.empty(B, Hq, d, dtype=torch.bfloat16, device=dev)
    musig, mnorm = eb.alloc_summaries(desc, dev)

    def run(after):
        eb.eta_build_block_summaries(desc, K, lens[0] - 1 if append else lens[-1], musig, mnorm)
        outs = torch.zeros(steps, B, Hq, d, device=dev)
        taus = torch.zeros(steps, B, Hq, device=dev)
        sels = torch.zeros(steps, B, Hkv, desc.nb_cap, dtype=torch.uint8, device=dev)
        torch.cuda.synchronize()
        for s in range(steps):
            eb.eta_stage_query(q_host[s], q)
            after()
            if append:
                eb.eta_append_summary(desc, K, lens[s], musig, mnorm)
                after()
            eb.eta_predict_threshold(q, W, bias, taus[s])
            after()
            eb.eta_decode(desc, eb.DecodeParams(), q, K, V, lens[s], musig, mnorm, taus[s], None, outs[s], sels[s], ws)
            after()
        return outs, taus, sels, q

    _both_ways(run)


@pytest.mark.parametrize("T", [600, 40000])          # 336 bounds, a warp each; 10192, in tiles
@pytest.mark.parametrize("packed", [False, True])
def test_queued_bounds_between_append_and_step(T, packed):
    """The bounds of records that the append in front of them has just written, with a step and the next append right behind,
    and of an index that a build in front of them has just written."""
    from paper_2609_20888_b200 import binding as eb
    dev, B, Hq, Hkv, d, b, steps = "cuda:0", 2, 4, 2, 64, 32, 24
    g = torch.Generator(device=dev).manual_seed(T)
    randn = lambda *s: torch.randn(s, generator=g, device=dev)
    cap = T // b * b + steps * b
    K, V = randn(B, Hkv, cap, d).bfloat16(), randn(B, Hkv, cap, d).bfloat16()
    q, const = randn(steps, B, Hq, d).bfloat16(), torch.full((Hq,), 0.8, device=dev)
    # every step completes a block of both sequences
    lens = torch.stack([torch.full((B,), T // b * b + (s + 1) * b, device=dev) for s in range(steps)]).int()
    desc = eb.cache_desc(K, V, Hq, b)
    ws = _aligned(eb, desc, dev)
    musig, mnorm = eb.alloc_summaries(desc, dev, packed=packed)
    flags = eb.ETA_BUILD_PACKED_SIGMA if packed else 0
    params = eb.DecodeParams(flags=eb.ETA_FLAG_PACKED_SIGMA if packed else 0)

    def run(after):
        musig.zero_(), mnorm.zero_()
        bound = torch.zeros(steps + 1, B, Hq, desc.nb_cap, device=dev)
        outs = torch.zeros(steps, B, Hq, d, device=dev)
        sel = torch.zeros(steps, B, Hkv, desc.nb_cap, dtype=torch.uint8, device=dev)
        after()
        eb.eta_build_block_summaries(desc, K, lens[0] - b, musig, mnorm, flags)
        after()
        eb.eta_score_dual(desc, params, q[0], lens[0] - b, musig, mnorm, bound[steps])
        after()
        for s in range(steps):
            eb.eta_append_summary(desc, K, lens[s], musig, mnorm, flags)
            after()
            eb.eta_score_dual(desc, params, q[s], lens[s], musig, mnorm, bound[s])
            after()
            eb.eta_decode(desc, params, q[s], K, V, lens[s], musig, mnorm, None, const, outs[s], sel[s], ws)
            after()
        return bound, outs, sel, musig, mnorm

    _both_ways(run)


@pytest.mark.parametrize("T", [600, 70000])
def test_captured_calibration_bounds_and_staged_query(T):
    """The same calls captured into a graph, behind a memset, a copy and a join of two streams, replayed with other inputs."""
    from paper_2609_20888_b200 import binding as eb
    dev, Hq, Hkv, d, b = "cuda:0", 4, 2, 64, 32
    g = torch.Generator(device=dev).manual_seed(T)
    randn = lambda *s: torch.randn(s, generator=g, device=dev)
    K = randn(1, Hkv, T, d).bfloat16()
    desc = eb.cache_desc(K, K, Hq, b)
    musig, mnorm = eb.alloc_summaries(desc, dev)
    lens = torch.full((1,), T, dtype=torch.int32, device=dev)
    Q, Kc, tau = randn(2, Hq, 200, d).bfloat16(), randn(2, Hkv, 200, d).bfloat16(), randn(2, Hq, 200)
    q_host = torch.zeros(1, Hq, d, dtype=torch.bfloat16).pin_memory()
    q = torch.empty(1, Hq, d, dtype=torch.bfloat16, device=dev)
    const, dbar, bound = torch.zeros(Hq, device=dev), torch.zeros(Hq, device=dev), torch.zeros(1, Hq, desc.nb_cap, device=dev)
    Q2 = torch.empty_like(Q)
    scratch = eb.eta_calibrate_head_const(Q, Kc, tau, const, dbar)
    side = torch.cuda.Stream()

    def calls():
        bound.zero_(), const.zero_()
        main = torch.cuda.current_stream()
        side.wait_stream(main)
        with torch.cuda.stream(side):
            eb.eta_build_block_summaries(desc, K, lens, musig, mnorm)
        Q2.copy_(Q)
        eb.eta_calibrate_head_const(Q2, Kc, tau, const, dbar, workspace=scratch)
        eb.eta_stage_query(q_host, q)
        main.wait_stream(side)
        eb.eta_score_dual(desc, eb.DecodeParams(), q, lens, musig, mnorm, bound)
        eb.eta_calibrate_head_const(Q2, Kc, tau, const, dbar, workspace=scratch)

    calls()                       # the kernels are loaded before the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls()
    for k in range(3):
        Q.copy_(randn(*Q.shape)), K.copy_(randn(*K.shape)), tau.copy_(randn(*tau.shape))
        q_host.copy_(randn(*q.shape).cpu())
        musig.zero_(), mnorm.zero_()
        for _ in range(2):
            graph.replay()
        torch.cuda.synchronize()
        got = [t.clone() for t in (const, dbar, bound, q, musig, mnorm)]
        for t in (const, dbar, bound, q, musig, mnorm):
            t.zero_()
        calls()
        torch.cuda.synchronize()
        for a, c in zip(got, (const, dbar, bound, q, musig, mnorm)):
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
