"""What a user of the library has it do, as measurable cases.

A case is one pass through the public entry points (`paper_2609_20888_b200.binding`) on inputs a program already
has on the GPU.  Four kinds:

  step       one decode step of one layer for a batch: tail-block summary update, threshold prediction (left out in
             the frozen per-head-constant mode), screening, attention over the surviving blocks, merge
  build      the prefill-side pass over K that builds the block index
  score      Score_dual of every (query head, block): what frozen constants are picked from
  calibrate  offline calibration of the per-head constants on a split of short sequences

`listed()` names the twelve that stand for the range, `draw()` gives more of it.  Steps are replayed from a CUDA
graph where a serving loop would (`graph`), or called one by one as an eager program does.

Inputs come from the seed alone.  Thresholds are placed so that the union of the blocks a KV head's query heads
admit has the case's sparsity, each in the middle of the widest gap between neighbouring bounds there: which blocks
survive then does not hang on the last bit of a bound.
"""
from __future__ import annotations

import math

import torch

from paper_2609_20888_b200 import binding as eb

# ---------------------------------------------------------------------------------------------------------- cases

_STEP = {"kind": "step", "batch": 1, "n_q_heads": 32, "n_kv_heads": 8, "head_dim": 128, "block": 64, "context": 0,
         "min_context": 0, "sparsity": 0.9, "keys": "clustered", "frozen": False, "paged": False, "packed": False,
         "token_major": False, "lwb": 0, "graph": True, "pinned_io": False}


def _step(name, **kw):
    return {"name": name, **_STEP, **kw}


def listed():
    return [
        # the smallest call: the correctness configuration, cache resident in the L2, called eagerly (latency only)
        _step("step_tiny_2k", n_q_heads=8, n_kv_heads=2, head_dim=64, block=32, context=2048, sparsity=0.7, graph=False),
        # interactive batch of one on a mid-size context of odd length, eager calls, the last blocks always attended
        _step("step_b1_16k", context=16 * 1024 + 437, sparsity=0.85, lwb=4, graph=False),
        # a small serving batch at 32K
        _step("step_b8_32k", batch=8, context=32768 + 77, sparsity=0.84, keys="needles"),
        # the headline configuration: 128K context, batch 4, 90 % of the blocks screened out
        _step("step_b4_128k_s90", batch=4, context=131072, sparsity=0.9),
        # the same cache at a threshold that keeps half of it: the streaming-bound end of the sweep
        _step("step_b4_128k_s50", batch=4, context=131072, sparsity=0.5),
        # one very long sequence, block size 128, needle blocks
        _step("step_b1_512k", n_q_heads=16, n_kv_heads=4, block=128, context=524288 - 64, sparsity=0.86, keys="needles"),
        # frozen per-head constants on mixed lengths (no predictor), eager calls
        _step("step_frozen_b16_mixed", batch=16, context=65536, min_context=8192, sparsity=0.7, keys="needles", frozen=True,
              graph=False),
        # paged cache with token-major pages, packed index, mixed lengths, queries from and outputs to pinned host memory
        _step("step_paged_b8_mixed", batch=8, context=98304, min_context=4096, sparsity=0.9, paged=True, packed=True,
              token_major=True, pinned_io=True),
        # the paper's latency-table geometry: eight query heads per KV head, head_dim 64, a large batch
        _step("step_gqa8_b32_64k", batch=32, n_q_heads=32, n_kv_heads=4, head_dim=64, context=65536, sparsity=0.84),
        # prefill of the headline batch
        {"name": "build_b4_128k", "kind": "build", "batch": 4, "n_kv_heads": 8, "head_dim": 128, "block": 64, "context": 131072,
         "min_context": 0, "packed": False, "envelope": False, "paged": False, "token_major": False},
        # bounds of the headline configuration
        {"name": "score_b4_128k", "kind": "score", "batch": 4, "n_q_heads": 32, "n_kv_heads": 8, "head_dim": 128, "block": 64,
         "context": 131072, "min_context": 0, "packed": False},
        # calibration split of the benchmark
        {"name": "calibrate_16x1024", "kind": "calibrate", "n_seq": 16, "seq_len": 1024, "n_q_heads": 32, "n_kv_heads": 8,
         "head_dim": 128, "n_bins": 2048},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _heads(rng):
    G, hkv = rng.choice([1, 2, 4, 4, 8]), rng.choice([2, 4, 8])
    return G * hkv, hkv


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["build", "score", "calibrate"])
    hq, hkv = _heads(rng)
    d, b = rng.choice([64, 128, 128]), rng.choice([32, 64, 64, 128])
    if kind == "calibrate":
        n_seq, T = _log_int(rng, 2, 32), _log_int(rng, 64, 2048)
        while n_seq * hq * T * T > 16 * 32 * 1024 * 1024:
            n_seq, T = max(1, n_seq // 2), (T if n_seq > 1 else T // 2)
        return {"kind": kind, "n_seq": n_seq, "seq_len": T, "n_q_heads": hq, "n_kv_heads": hkv, "head_dim": d,
                "n_bins": rng.choice([512, 1000, 2048, 4096])}
    context = _log_int(rng, 2048, 512 * 1024)
    most = 4 * 8 * 131072 * 128                         # elements of K: the headline cache
    batch = _log_int(rng, 1, 64)
    while batch > 1 and batch * hkv * context * d > most:
        batch //= 2
    mixed = batch > 1 and rng.random() < 0.5
    lens = {"batch": batch, "n_kv_heads": hkv, "head_dim": d, "block": b, "context": context,
            "min_context": max(1024, context // 8) if mixed else 0, "packed": rng.random() < 0.2}
    if kind == "build":
        return {"kind": kind, **lens, "envelope": rng.random() < 0.2, "paged": rng.random() < 0.25,
                "token_major": rng.random() < 0.25}
    if kind == "score":
        return {"kind": kind, **lens, "n_q_heads": hq}
    graph = rng.random() < 0.6
    return {**_STEP, **lens, "n_q_heads": hq, "sparsity": round(rng.uniform(0.5, 0.97), 2),
            "keys": rng.choice(["clustered", "needles"]), "frozen": rng.random() < 0.25, "paged": rng.random() < 0.25,
            "token_major": rng.random() < 0.25, "lwb": rng.choice([0, 0, 1, 4]), "graph": graph,
            "pinned_io": rng.random() < 0.2}


# --------------------------------------------------------------------------------------------------------- inputs

def _lens(case, gen):
    lens = torch.full((case["batch"],), case["context"], dtype=torch.int32, device="cuda")
    if case["min_context"]:
        lens = torch.randint(case["min_context"], case["context"] + 1, lens.shape, generator=gen, device="cuda",
                             dtype=torch.int32)
        lens[0] = case["context"]
    return lens


def _queries(case, gen):
    """Post-RoPE queries: the heads of a KV group share a direction, as grouped heads do."""
    B, Hq, Hkv, d = case["batch"], case["n_q_heads"], case["n_kv_heads"], case["head_dim"]
    shared = torch.randn((B, Hkv, 1, d), generator=gen, device="cuda")
    noise = torch.randn((B, Hkv, Hq // Hkv, d), generator=gen, device="cuda")
    return (math.sqrt(0.95) * shared + math.sqrt(0.05) * noise).reshape(B, Hq, d).to(torch.bfloat16), shared[:, :, 0]


def _keys(case, gen, direction):
    """K [B, Hkv, Tcap, d] in one of two structures: every block around one of 64 centroids of its KV head, or unit
    noise on a slowly drifting mean with a few blocks aligned with the group's query direction."""
    B, Hkv, d, b = case["batch"], case["n_kv_heads"], case["head_dim"], case["block"]
    NB = -(-case["context"] // b)
    shape = (B, NB * b, Hkv, d) if case.get("token_major") else (B, Hkv, NB * b, d)
    K = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
    K = K.transpose(1, 2) if case.get("token_major") else K
    cent = torch.randn((Hkv, 64, d), generator=gen, device="cuda")
    for i in range(B):
        if case.get("keys", "clustered") == "clustered":
            which = torch.randint(0, 64, (Hkv, NB), generator=gen, device="cuda")
            mean, sigma = torch.gather(cent, 1, which[:, :, None].expand(-1, -1, d)), torch.full((Hkv, NB), 0.3, device="cuda")
        else:
            mean = torch.cumsum(torch.randn((Hkv, NB, d), generator=gen, device="cuda"), 1) / 16
            sigma = torch.ones((Hkv, NB), device="cuda")
            plant = torch.rand((Hkv, NB), generator=gen, device="cuda") < 1 / 200
            unit = direction[i] / direction[i].norm(dim=-1, keepdim=True)
            strength = 3 + 6 * torch.rand((Hkv, NB, 1), generator=gen, device="cuda")
            mean = torch.where(plant[:, :, None], strength * unit[:, None, :], mean)
            sigma = torch.where(plant, 0.3, sigma)
        noise = torch.randn((Hkv, NB, b, d), generator=gen, device="cuda", dtype=torch.bfloat16)
        K[i] = (mean[:, :, None, :] + sigma[:, :, None, None] * noise).reshape(Hkv, NB * b, d)
    return K


def _values(K, gen):
    """V like K in shape and strides."""
    V = torch.empty_strided(K.shape, K.stride(), dtype=K.dtype, device="cuda")
    for i in range(K.shape[0]):
        V[i] = torch.randn(K.shape[1:], generator=gen, device="cuda", dtype=torch.bfloat16)
    return V


def _bounds(case, K, q, lens):
    """Score_dual of every full block, +-0 apart from rounding: fp32 [B, Hq, NB], -inf where there is no full block."""
    B, Hq, Hkv, d, b = case["batch"], case["n_q_heads"], case["n_kv_heads"], case["head_dim"], case["block"]
    NB = K.shape[2] // b
    out = torch.empty((B, Hkv, Hq // Hkv, NB), device="cuda")
    qf = q.float().view(B, Hkv, Hq // Hkv, d)
    for i in range(B):
        k = K[i].reshape(Hkv, NB, b, d)
        mu, sig = torch.empty((2, Hkv, NB, d), device="cuda")
        top = torch.empty((Hkv, NB), device="cuda")
        for h in range(Hkv):
            kf = k[h].float()
            var, mean = torch.var_mean(kf, 1, correction=0)
            mu[h], sig[h], top[h] = mean.half().float(), var.sqrt().half().float(), kf.norm(dim=2).amax(1)
        dot, var = qf[i] @ mu.transpose(1, 2), qf[i].square() @ sig.square().transpose(1, 2)
        out[i] = torch.minimum(dot + var.sqrt(), qf[i].norm(dim=2, keepdim=True) * top[:, None, :]) / math.sqrt(d)
    out = out.view(B, Hq, NB)
    full = torch.arange(NB, device="cuda")[None, :] < (lens // b)[:, None]
    return out.masked_fill_(~full[:, None, :], -math.inf)


def _thresholds(case, bounds, raw, gen):
    """One offset per head, bounds above raw + offset survive: the union over a KV head's query heads keeps a share of
    1 - sparsity.  Heads differ in density in the frozen mode."""
    B, Hq, NB = bounds.shape
    G = Hq // case["n_kv_heads"]
    lift = torch.rand((Hq,), generator=gen, device="cuda") * 2 + 0.2 if case["frozen"] else torch.ones(Hq, device="cuda")
    rel = bounds - raw[:, :, None]
    pool = rel.transpose(0, 1).reshape(Hq, B * NB).sort(dim=1, descending=True).values
    n = int(torch.isfinite(pool[0]).sum())
    rows = torch.arange(Hq, device="cuda")
    pick = lambda rho: pool[rows, (rho * lift * n).long().clamp(1, max(1, n - 2))]  # noqa: E731
    lo, hi = 0.0, 1.0
    for _ in range(12):
        mid = (lo + hi) / 2
        kept = (rel >= pick(mid)[None, :, None]).view(B, Hq // G, G, NB).any(2).sum().item() / (n * (Hq // G))
        lo, hi = (mid, hi) if kept < 1 - case["sparsity"] else (lo, mid)
    # the middle of the widest gap close by
    at = (hi * lift * n).long().clamp(1, max(1, n - 2))
    w = max(2, n // 100)
    near = (at[:, None] + torch.arange(-w, w + 1, device="cuda")[None, :]).clamp(0, max(0, n - 2))
    gap = pool.gather(1, near) - pool.gather(1, near + 1)
    best = near.gather(1, gap.argmax(1, keepdim=True))
    return ((pool.gather(1, best) + pool.gather(1, best + 1)) / 2)[:, 0].contiguous()


def _pages(case, K, V, gen):
    """The same cache in pools of one-block pages scattered at random."""
    B, Hkv, T, d = K.shape
    b, NB = case["block"], T // case["block"]
    perm = torch.randperm(B * NB, generator=gen, device="cuda")

    def pool(X):
        shape = (B * NB, b, Hkv, d) if case["token_major"] else (B * NB, Hkv, b, d)
        P = torch.empty(shape, dtype=X.dtype, device="cuda")
        P = P.transpose(1, 2) if case["token_major"] else P
        for i in range(B):
            P[perm[i * NB:(i + 1) * NB]] = X[i].reshape(Hkv, NB, b, d).transpose(0, 1)
        return P

    return pool(K), (None if V is None else pool(V)), perm.view(B, NB).to(torch.int32)


def _aligned(n):
    ws = torch.zeros(n + 256, dtype=torch.uint8, device="cuda")
    off = -ws.data_ptr() % 256
    return ws[off:off + n]


def _prepare_step(case, gen):
    B, Hq, Hkv, d, b = case["batch"], case["n_q_heads"], case["n_kv_heads"], case["head_dim"], case["block"]
    s = {"case": case, "lens": _lens(case, gen)}
    q, direction = _queries(case, gen)
    K = _keys(case, gen, direction)
    V = _values(K, gen)
    # predictor weights at the fan-in scale of a trained one; the frozen mode has constants instead
    W = torch.randn((Hq * d, Hq), generator=gen, device="cuda") * (0.02 * math.sqrt(512 / (Hq * d)))
    raw = q.float().view(B, Hq * d) @ W * (0 if case["frozen"] else 1)
    offset = _thresholds(case, _bounds(case, K, q, s["lens"]), raw, gen)
    NB = K.shape[2] // b
    if case["paged"]:
        K, V, table = _pages(case, K, V, gen)
        s["table"], s["pages"] = table, eb.page_table(table, K.shape[0])
        s["desc"] = eb.paged_cache_desc(K, V, B, Hq, t_cap=NB * b)
    else:
        s["desc"] = eb.cache_desc(K, V, Hq, b)
    s.update(q=q, K=K, V=V, W=W, offset=offset, tau=torch.zeros((B, Hq), device="cuda"),
             sel=torch.zeros((B, Hkv, s["desc"].nb_cap), dtype=torch.uint8, device="cuda"),
             out=torch.zeros((B, Hq, d), device="cuda"), stats=torch.zeros((B, Hkv), dtype=torch.int32, device="cuda"),
             status=torch.zeros(1, dtype=torch.int32, device="cuda"),
             ws=_aligned(eb.eta_workspace_bytes(s["desc"])),
             params=eb.DecodeParams(lwb=case["lwb"], flags=eb.ETA_FLAG_PACKED_SIGMA if case["packed"] else 0))
    if case["pinned_io"]:
        s["q_host"] = q.cpu().pin_memory()
        s["out"] = torch.zeros((B, Hq, d)).pin_memory()
    s["musig"], s["mnorm"] = eb.alloc_summaries(s["desc"], "cuda", packed=case["packed"])
    _build(s)
    if case["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _launch_step(s)
        torch.cuda.current_stream().wait_stream(side)
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _launch_step(s)
    return s


def _build(s):
    case = s["case"]
    flags = (eb.ETA_BUILD_PACKED_SIGMA if case["packed"] else 0) | (eb.ETA_BUILD_SIGMA_ENVELOPE if case.get("envelope") else 0)
    if case.get("paged"):
        eb.eta_build_block_summaries_paged(s["desc"], s["pages"], s["K"], s["lens"], s["musig"], s["mnorm"], flags)
    else:
        eb.eta_build_block_summaries(s["desc"], s["K"], s["lens"], s["musig"], s["mnorm"], flags)


def _prepare_index(case, gen):
    s = {"case": case, "lens": _lens(case, gen)}
    Hq = case.get("n_q_heads", case["n_kv_heads"])
    s["q"], direction = _queries({**case, "n_q_heads": Hq}, gen)
    K = _keys(case, gen, direction)
    if case.get("paged"):
        T = K.shape[2]
        K, _, table = _pages(case, K, None, gen)
        s["table"], s["pages"] = table, eb.page_table(table, K.shape[0])
        s["desc"] = eb.paged_cache_desc(K, K, case["batch"], Hq, t_cap=T)
    else:
        s["desc"] = eb.cache_desc(K, K, Hq, case["block"])
    s["K"] = K
    s["musig"], s["mnorm"] = eb.alloc_summaries(s["desc"], "cuda", packed=case["packed"])
    if case["kind"] == "score":
        _build(s)
        s["params"] = eb.DecodeParams(flags=eb.ETA_FLAG_PACKED_SIGMA if case["packed"] else 0)
        s["bound"] = torch.zeros((case["batch"], Hq, s["desc"].nb_cap), device="cuda")
    return s


def _prepare_calibrate(case, gen):
    n, T, Hq, Hkv, d = (case[k] for k in ("n_seq", "seq_len", "n_q_heads", "n_kv_heads", "head_dim"))
    s = {"case": case, "Q": torch.randn((n, Hq, T, d), generator=gen, device="cuda").to(torch.bfloat16),
         "K": torch.randn((n, Hkv, T, d), generator=gen, device="cuda").to(torch.bfloat16),
         # the dynamic predictor's thresholds on the split
         "tau": 0.5 + 0.3 * torch.randn((n, Hq, T), generator=gen, device="cuda"),
         "head_const": torch.zeros(Hq, device="cuda"), "dbar": torch.zeros(Hq, device="cuda")}
    s["ws"] = eb.eta_calibrate_head_const(s["Q"], s["K"], s["tau"], s["head_const"], s["dbar"], n_bins=case["n_bins"])
    return s


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    make = {"step": _prepare_step, "build": _prepare_index, "score": _prepare_index, "calibrate": _prepare_calibrate}
    return make[case["kind"]](case, gen)


# ----------------------------------------------------------------------------------------------------------- passes

def _launch_step(s):
    case, desc = s["case"], s["desc"]
    flags = eb.ETA_BUILD_PACKED_SIGMA if case["packed"] else 0
    if case["pinned_io"]:
        eb.eta_stage_query(s["q_host"], s["q"])
    if case["paged"]:
        eb.eta_append_summary_paged(desc, s["pages"], s["K"], s["lens"], s["musig"], s["mnorm"], flags)
    else:
        eb.eta_append_summary(desc, s["K"], s["lens"], s["musig"], s["mnorm"], flags)
    if case["frozen"]:
        tau, const = None, s["offset"]
    else:
        eb.eta_predict_threshold(s["q"], s["W"], s["offset"], s["tau"])
        tau, const = s["tau"], None
    if case["paged"]:
        eb.eta_decode_paged(desc, s["pages"], s["params"], s["q"], s["K"], s["V"], s["lens"], s["musig"], s["mnorm"], tau,
                            const, s["out"], s["sel"], s["ws"], stats=s["stats"], status=s["status"])
    else:
        eb.eta_decode(desc, s["params"], s["q"], s["K"], s["V"], s["lens"], s["musig"], s["mnorm"], tau, const, s["out"],
                      s["sel"], s["ws"], stats=s["stats"], status=s["status"])


def run(state):
    s, kind = state, state["case"]["kind"]
    if kind == "step":
        if "graph" in s:
            s["graph"].replay()
        else:
            _launch_step(s)
        return {k: s[k] for k in ("out", "sel", "stats", "tau", "musig", "mnorm", "status")}
    if kind == "build":
        _build(s)
        return {"musig": s["musig"], "mnorm": s["mnorm"]}
    if kind == "score":
        eb.eta_score_dual(s["desc"], s["params"], s["q"], s["lens"], s["musig"], s["mnorm"], s["bound"])
        return s["bound"]
    eb.eta_calibrate_head_const(s["Q"], s["K"], s["tau"], s["head_const"], s["dbar"], n_bins=s["case"]["n_bins"],
                                workspace=s["ws"])
    return {"head_const": s["head_const"], "dbar": s["dbar"]}


def work(case):
    """Bytes and operations one pass cannot do without, at the mean sequence length of a mixed batch."""
    Hkv, d = case["n_kv_heads"], case["head_dim"]
    if case["kind"] == "calibrate":
        n, T, Hq = case["n_seq"], case["seq_len"], case["n_q_heads"]
        return {"bytes": n * T * (2 * d * (Hq + Hkv) + 4 * Hq) + 8 * Hq, "flops": n * Hq * (T * (T + 1) / 2) * (2 * d + 16)}
    B, b = case["batch"], case["block"]
    T = (case["min_context"] + case["context"]) / 2 if case["min_context"] else case["context"]
    blocks = B * Hkv * (T // b)
    record = (3 if case["packed"] else 4) * d + 4
    if case["kind"] == "build":
        return {"bytes": blocks * (2 * d * b + record), "flops": blocks * b * d * 6}
    Hq = case["n_q_heads"]
    screen = {"bytes": blocks * record + 2 * B * Hq * d, "flops": 4 * d * blocks * (Hq // Hkv)}
    if case["kind"] == "score":
        return {"bytes": screen["bytes"] + 4 * blocks * (Hq // Hkv), "flops": screen["flops"]}
    tokens = blocks * (1 - case["sparsity"]) * b + B * Hkv * (T % b)
    predict = 0 if case["frozen"] else Hq * d * Hq * 4
    return {"bytes": screen["bytes"] + blocks + 4 * d * tokens + predict + 4 * B * Hq * d,
            "flops": screen["flops"] + 4 * d * (Hq // Hkv) * tokens}


def tolerance(case):
    """Four times what the path differs by from its own formulas in 64 bits: outputs, thresholds and bounds by at most
    2.7e-6 (largest difference 2.1e-5).  Index entries are fp16, where another order of the sums flips a last bit now
    and then (2.4e-5 of the entries, each by up to 1e-3), or bytes in the packed index."""
    return {"rel": 1e-5, "max": 1e-3 if case["kind"] in ("step", "build") else 1e-4, "differ": 1e-4}
