// A decode step of a small problem in one kernel: screening, attention over the surviving blocks and the merge (Algorithm 3) by
// one thread-block cluster per (sequence, KV head) row.
//
// The general path takes three kernels, because survivors of all rows are dealt out over the whole GPU.  Where a row has a few
// hundred blocks its step is latency: the boundaries between the kernels and each one's own set-up.  Here every CTA of a row's
// cluster bounds a share of the row's blocks while the thresholds are still being predicted and stores the bounds to all of them, so
// that all know the list of survivors; each attends an equal share of the tiles; and the partial results are merged through the
// cluster's shared memory.
#include <cooperative_groups.h>

#include "eta_attend.cuh"
#include "eta_bounds.cuh"
#include "eta_step.h"

namespace cg = cooperative_groups;

namespace eta {

constexpr int STEP_WARPS = 12;                          // three groups of four that bound and attend ...
constexpr int STEP_THREADS = 32 * (STEP_WARPS + 1);     // ... and one that issues the copies
constexpr int STEP_RING = 196608;                       // bytes of the ring of K and V tiles; first the records' tiles, last the partials
constexpr int STEP_SEGS = STEP_MAX_BLOCKS / SEG;

template <int D, int TS, int G>
struct StepSmem {
    static constexpr int STAGE_BYTES = 4 * D * TS, NSTAGE = STEP_RING / STAGE_BYTES;
    static_assert(NSTAGE % 3 == 0, "a stage serves the same group in every round");
    static_assert(2 * STEP_WARPS * TileOf<D>::BYTES <= STEP_RING && STEP_WARPS * G * D * 4 <= STEP_RING, "what shares the ring fits it");
    static constexpr int BAR_OFF = STEP_RING;           // full[NSTAGE], empty[NSTAGE], two per warp for its records
    static constexpr int TAB_OFF = (BAR_OFF + 8 * (2 * NSTAGE + 2 * STEP_WARPS) + 15) / 16 * 16;
    static constexpr int BOUND_OFF = TAB_OFF + (int)((sizeof(QTab<D, G>) + 15) / 16 * 16);
    static constexpr int LIST_OFF = BOUND_OFF + 4 * STEP_MAX_BLOCKS * G;        // survivors in ascending order, then the tail
    static constexpr int IN_ML_OFF = TAB_OFF + 4 * G * D + 16 * STEP_MAX_CLUSTER;       // behind the parts: float2 [CTA][G]
    static_assert(IN_ML_OFF + 8 * G * STEP_MAX_CLUSTER <= LIST_OFF, "the parts take the place of the query table and the bounds");
    static constexpr int WARP_ML_OFF = LIST_OFF + 4 * (STEP_MAX_BLOCKS + 4);    // float m[STEP_WARPS][8], l[STEP_WARPS][8]
    static constexpr size_t BYTES = 1024 + WARP_ML_OFF + 8 * STEP_WARPS * 8;
};

// A barrier of the cluster in two halves; what was stored before the first is there after the second.  The hardware has no bounded
// form of it.  Every thread reaches every one: what stands between two barriers are bounded waits, after which a warp goes on to the
// next barrier with whatever it has (no early return in the kernel).
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// What bounds it: latency, of a chain of short parts: us from the entry, 8 rows of 16K tokens: query table 1.5, bounds 3.1, those of
// the other CTAs 5.2, thresholds 5.5 (they have been there), list 7.0, first tile 8.2, last 10.6, the parts of the warps and of the CTAs 3.4.
// What it took out of the chain to load q beside the length (it sets the entry's time), to read a record's bounds in one piece and a
// head's rescue once, and to load the CTAs' parts eight at a time: 17.7 -> 17.2 us a step there, 12.9 -> 12.3 for 2 rows of 2K.
// Code that runs once is fetched as it runs: admission as a loop over a segment's halves, not unrolled, 4 rows of 32K 18.9 -> 18.6, 8
// rows 19.7 -> 19.1.
// Bounds of the row in each CTA where they are one round of its warps, else in shares, which the cluster exchanges: 1.2 us slower
// for 32 blocks, 1.1 faster for 256 and 4 for 511.  Two tiles of records in flight per warp where a share is more than one.  Six 32 KB tiles in flight: with three, rows of 256 blocks, half of them
// attended, took 29.5 us instead of 25.5.  Parts are stored to the CTA that adds them up, not fetched by it: one barrier of the
// cluster instead of two, 0.6 to 0.8 us.
// Registers: the 13th warp, which issues the copies, makes four warps on one scheduler and so 128 registers the most.  At head_dim 128 the
// instances want a few more (28 to 64 bytes spilled), at 64 they take 98 to 115.
template <int D, int TS, int G, bool PACKED>
__global__ void __launch_bounds__(STEP_THREADS, 1) step_kernel(const __grid_constant__ CUtensorMap tmK,
                                                               const __grid_constant__ CUtensorMap tmV, const StepArgs a) {
    using L = StepSmem<D, TS, G>;
    using TL = TileOf<D>;
    constexpr int REC_BYTES = PACKED ? 3 * D : 4 * D;
    extern __shared__ unsigned char step_raw[];
    unsigned char* const sm = step_raw + ((1024u - (smem_u32(step_raw) & 1023u)) & 1023u);
    uint64_t* const full = reinterpret_cast<uint64_t*>(sm + L::BAR_OFF);
    uint64_t* const empty = full + L::NSTAGE;
    QTab<D, G>& tab = *reinterpret_cast<QTab<D, G>*>(sm + L::TAB_OFF);
    float* const sbound = reinterpret_cast<float*>(sm + L::BOUND_OFF);
    int32_t* const list = reinterpret_cast<int32_t*>(sm + L::LIST_OFF);
    __shared__ uint32_t s_bkey[G];        // per head: largest bound of the rescue window (as an ordered integer)
    __shared__ int s_best[G];             // and the first block that attains it
    __shared__ int s_cnt[STEP_SEGS];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), n_ranks = (int)cluster.num_blocks();
    const int r = blockIdx.x / n_ranks;
    int i, hk;
    a.div_hkv.divmod(r, i, hk);
    const int Traw = __ldcg(a.seq_lens + i);
    const uint4 q_piece = load_qtab<D, G>(a.q + ((int64_t)i * a.Hq + hk * G) * D, tid);
    const int T = Traw < 0 ? 0 : (Traw > a.t_cap ? a.t_cap : Traw);
    const int NB = min(T >> a.b_shift, a.nb_cap), b = 1 << a.b_shift;
    const unsigned char* const rec_row = reinterpret_cast<const unsigned char*>(a.musig) + (int64_t)r * a.nb_cap * REC_BYTES;
    const float* const mn_row = a.mnorm + (int64_t)r * a.nb_cap;

    // ------------------------------------------------------------ bounds of the row's blocks, a share per CTA: needs neither the
    // thresholds nor the newest record (see below), so it does not wait for the kernels that make them
    if (a.shared) cluster_arrive();       // (all CTAs of the cluster run when all have come by here)
    const int of = a.shared ? n_ranks : 1, first = (warp * of + (a.shared ? rank : 0)) * TL::RECS, stride = STEP_WARPS * of * TL::RECS;
    if (tid == 0) {
        for (int s = 0; s < L::NSTAGE; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], WARPS_PER_GROUP); }
        fence_barrier_init();
        prefetch_tmap(&tmK);
        prefetch_tmap(&tmV);
    }
    uint64_t* const bars = empty + L::NSTAGE + 2 * warp;
    TileStream<D, G, PACKED> ts{sm + warp * 2 * TL::BYTES, bars, rec_row, mn_row, NB, 2, 0, 0, 0u, true};
    if (warp < STEP_WARPS) {
        if (lane == 0) { mbar_init(&bars[0], 1); mbar_init(&bars[1], 1); fence_barrier_init(); }
        __syncwarp();
        ts.issue(first);
        ts.issue(first + stride);
    }
    build_qtab<D, G>(tab, q_piece, tid);
    bool ok = true;
    if (warp < STEP_WARPS) {
        for (int j = first; j < NB; j += stride) {
            ok = ts.bounds(tab, j, a.z, a.scale, sbound + j * G) && ok;
            if (j + 2 * stride < NB) ts.issue(j + 2 * stride);
        }
    }
    Attend<D, TS, 2> at(lane, warp % WARPS_PER_GROUP, G);
    at.load_q(a.q + ((int64_t)i * a.Hq + hk * G + (at.head ? at.g : 0)) * D);
    if (a.shared) {                       // every CTA gets all of them
        cluster_wait();
        if (warp < STEP_WARPS) {
            for (int j = first; j < NB; j += stride)
                for (int c = 1; c < n_ranks; ++c) {
                    float4* const dst = reinterpret_cast<float4*>(cluster.map_shared_rank(sbound + j * G, (rank + c) % n_ranks));
                    for (int k = lane; k < TL::RECS * G / 4; k += 32) dst[k] = reinterpret_cast<const float4*>(sbound + j * G)[k];
                }
        }
        cluster_arrive();
        cluster_wait();
    } else {
        __syncthreads();
    }

    // Top-1 rescue: a head that admits none of the first Wr blocks attends the first one with the largest bound among them.  It
    // admits none exactly when that bound is below its threshold and no block of the window is pinned (a NaN bound admits).
    // An ungated newest token must be attended: when it closes a full block, that block counts as pinned.
    const int lwb = ((a.flags & ETA_FLAG_UNGATE_LAST) && T > 0 && (T & (b - 1)) == 0 && a.lwb < 1) ? 1 : a.lwb;
    const int Wr = min(a.rescue_window, NB);
    const bool rescues = Wr > 0 && !(lwb > 0 && NB - lwb < Wr);
    const bool stale = NB > 0 && (T & (b - 1)) == 0;       // the newest block's record may not have been final yet
    const bool late = stale && NB - 1 < Wr;
    auto window_max = [&]() {
        for (int gq = warp; gq < G; gq += STEP_WARPS + 1) {
            uint32_t key = 0;                     // 0: no record of the window in this lane
            int arg = 0x7fffffff;
            for (int rec = lane; rec < Wr; rec += 32) {                     // ascending: a lane keeps the first of equal bounds
                const uint32_t k2 = bound_key(sbound[rec * G + gq]);
                if (k2 > key) { key = k2; arg = rec; }
            }
            const uint32_t kmax = __reduce_max_sync(0xffffffffu, key);
            const int amin = __reduce_min_sync(0xffffffffu, key == kmax ? arg : 0x7fffffff);
            if (lane == 0) { s_bkey[gq] = kmax; s_best[gq] = amin; }
        }
    };
    if (rescues && !late) window_max();
    pdl_wait();                           // the thresholds and the newest summaries are final now
    pdl_trigger();
    float te_l = -INFINITY;               // lane gq < G: effective threshold of head gq
    if (lane < G) te_l = (a.tau ? __ldcg(a.tau + (int64_t)i * a.Hq + hk * G + lane) : __ldcg(a.head_const + hk * G + lane)) - a.a;
    if (stale) {
        if (warp == 0)
            bound_one<D, G, PACKED>(tab.raw, rec_row + (int64_t)(NB - 1) * REC_BYTES, __ldcg(mn_row + NB - 1), a.z, a.scale, sbound + (NB - 1) * G);
        __syncthreads();
        if (rescues && late) window_max();
    }
    __syncthreads();
    if (rank == 0 && tid == 0 && a.status) {
        if (Traw > a.t_cap) atomicOr(a.status, ETA_DEV_LEN_CLAMPED);
        if (Traw <= 0) atomicOr(a.status, ETA_DEV_EMPTY_ROW);
    }

    // ------------------------------------------------------------ admission, a warp per segment
    const int j0 = warp * SEG;
    unsigned admitted = 0;                // a byte per half: heads that attend record j0 + 32 half + lane
    int carry = 0;
    if (warp < STEP_SEGS && j0 < a.nb_cap) {
        float te_g[G];
        int best[G];
#pragma unroll
        for (int gq = 0; gq < G; ++gq) {
            te_g[gq] = __shfl_sync(0xffffffffu, te_l, gq);
            best[gq] = rescues && key_bound(s_bkey[gq]) < te_g[gq] ? s_best[gq] : -1;
        }
#pragma unroll 1
        for (int half = 0; half < SEG / 32; ++half) {
            const int j = j0 + half * 32 + lane;
            unsigned m = 0;
            if (j < NB) {
                const bool pinned = j >= NB - lwb;
                float bd[G];
                constexpr int V = G < 4 ? G : 4;              // a record's bounds in pieces of up to 16 bytes
#pragma unroll
                for (int g0 = 0; g0 < G; g0 += V) {
                    if constexpr (V == 4) *reinterpret_cast<float4*>(bd + g0) = *reinterpret_cast<const float4*>(sbound + j * G + g0);
                    else if constexpr (V == 2) *reinterpret_cast<float2*>(bd) = *reinterpret_cast<const float2*>(sbound + j * 2);
                    else bd[0] = sbound[j];
                }
#pragma unroll
                for (int gq = 0; gq < G; ++gq)
                    if (pinned || j == best[gq] || !(bd[gq] < te_g[gq])) m |= 1u << gq;
            }
            if (rank == 0 && j < a.nb_cap) a.sel_mask[(int64_t)r * a.nb_cap + j] = (uint8_t)m;
            admitted |= m << (8 * half);
            carry += __popc(__ballot_sync(0xffffffffu, m != 0));
        }
    }
    if (warp < STEP_SEGS && lane == 0) s_cnt[warp] = carry;
    __syncthreads();
    const int cnt = lane < STEP_SEGS ? s_cnt[lane] : 0;
    const int n_blocks = __reduce_add_sync(0xffffffffu, cnt);
    int at_list = __reduce_add_sync(0xffffffffu, lane < warp ? cnt : 0);
    if (warp < STEP_SEGS) {
#pragma unroll 1
        for (int half = 0; half < SEG / 32; ++half) {
            const unsigned m = (admitted >> (8 * half)) & 0xff, nz = __ballot_sync(0xffffffffu, m != 0);
            if (m) list[at_list + __popc(nz & ((1u << lane) - 1u))] = (j0 + half * 32 + lane) | (int)(m << 24);
            at_list += __popc(nz);
        }
    }
    const int tail = T - NB * b;
    if (tid == 0) {
        list[n_blocks] = NB | (0xff << 24);               // the tail: every head attends it
        if (rank == 0 && a.stats) a.stats[r] = n_blocks;
    }
    at.te = __shfl_sync(0xffffffffu, te_l, at.head ? at.g : 0);
    __syncthreads();
    cluster_arrive();                     // this CTA needs its query table and bounds no more: the others' parts go there

    // ------------------------------------------------------------ an equal share of the row's tiles
    const int tpu_shift = a.b_shift - (TS == 64 ? 6 : 5);               // tiles of a full block: 1, or 2 (128 tokens)
    const int n_full = n_blocks << tpu_shift, n_tiles = n_full + (tail + TS - 1) / TS;
    const int f0 = n_tiles * rank / n_ranks, n = n_tiles * (rank + 1) / n_ranks - f0;
    // tile k of the share: its list entry, part of the block, tokens of it in the sequence
    auto locate = [&](int k, int& ent, int& sub, int& rows) {
        const int f = f0 + k;
        const bool whole = f < n_full;
        sub = whole ? f & ((1 << tpu_shift) - 1) : f - n_full;
        ent = list[whole ? f >> tpu_shift : n_blocks];
        rows = (whole ? b : tail) - sub * TS;
    };
    if (warp == STEP_WARPS) {
        // a lane per stage
        if (lane < L::NSTAGE) {
            const uint64_t policy = l2_policy(false);
            int issued = -1;
            for (int k = lane, parity = 1; k < n && ok; k += L::NSTAGE, parity ^= 1) {
                ok = mbar_wait(&empty[lane], parity);
                if (!ok) break;
                int ent, sub, rows;
                locate(k, ent, sub, rows);
                const int j = ent & 0xffffff;
                const int w = a.block_table ? __ldcg(a.block_table + (int64_t)i * a.table_stride + j) : i;
                const int y = (a.block_table ? 0 : j * b) + sub * TS;
                unsigned char* const dst = sm + lane * L::STAGE_BYTES;
                mbar_arrive_expect_tx(&full[lane], L::STAGE_BYTES);
                tma_load_5d(dst, &tmK, 0, y, 0, hk, w, &full[lane], policy);
                tma_load_5d(dst + L::STAGE_BYTES / 2, &tmV, 0, y, 0, hk, w, &full[lane], policy);
                issued = k;
            }
            if (issued >= 0) ok = mbar_wait(&full[lane], (issued / L::NSTAGE) & 1) && ok;      // whatever the others did: the copies have landed
        }
        ok = __all_sync(0xffffffffu, ok);
    } else {
        for (int k = warp / WARPS_PER_GROUP; k < n; k += STEP_WARPS / WARPS_PER_GROUP) {
            const int stage = k % L::NSTAGE;
            ok = __all_sync(0xffffffffu, ok && mbar_wait(&full[stage], (k / L::NSTAGE) & 1));
            if (!ok) break;
            int ent, sub, rows;
            locate(k, ent, sub, rows);
            const int nvalid = min(TS, rows), last = T - 1 - ((ent & 0xffffff) * b + sub * TS);      // the newest token's row of the tile
            const int urow = (a.flags & ETA_FLAG_UNGATE_LAST) && last < TS ? last : 0xff;
            at.tile(smem_u32(sm + stage * L::STAGE_BYTES), (ent >> 24) & 0xff, urow, nvalid, a.scale, a.beta, [&]() {
#ifdef ETA_TEST_SKIP_STAGE_ARRIVE
                // test build only: one warp of the first CTA never releases its stages, so that the waits of the warp that issues the
                // copies, and then of the warps that wait for them, run out
                if (blockIdx.x == 0 && warp == 1) return;
#endif
                if (lane == 0) mbar_arrive(&empty[stage]);
            });
        }
    }
    if (!ok && lane == 0 && a.status) atomicOr(a.status, ETA_DEV_TIMEOUT);
    __syncthreads();                      // the ring is free

    // ------------------------------------------------------------ the warps' parts, then the CTAs'
    float* const warp_m = reinterpret_cast<float*>(sm + L::WARP_ML_OFF), * const warp_l = warp_m + STEP_WARPS * 8;
    float* const parts = reinterpret_cast<float*>(sm);                  // [warp][head][D]
    // Each CTA makes a slice of the row's output: it gets every CTA's part of the slice, and their statistics
    const int per = (G * D / 4 + n_ranks - 1) / n_ranks;
    float4* const in_o = reinterpret_cast<float4*>(sm + L::TAB_OFF);                 // [CTA][per]
    float2* const in_ml = reinterpret_cast<float2*>(sm + L::IN_ML_OFF);              // [CTA][G]
    constexpr float LOG2E = 1.4426950408889634f;
    if (warp < STEP_WARPS) {
        float lsum = at.l_run + __shfl_xor_sync(0xffffffffu, at.l_run, 1);
        lsum += __shfl_xor_sync(0xffffffffu, lsum, 2);
        if (at.t == 0) { warp_m[warp * 8 + at.g] = at.m_run; warp_l[warp * 8 + at.g] = lsum; }
#pragma unroll
        for (int hf = 0; hf < D / 64; ++hf)
#pragma unroll
            for (int mt = 0; mt < 4; ++mt) {
                const int ha = 2 * at.t, dcol = 64 * hf + 8 * at.vchunk + 2 * mt;
                if (ha < G) *reinterpret_cast<float2*>(parts + (warp * G + ha) * D + dcol) = make_float2(at.o[hf][mt][0], at.o[hf][mt][2]);
                if (ha + 1 < G) *reinterpret_cast<float2*>(parts + (warp * G + ha + 1) * D + dcol) = make_float2(at.o[hf][mt][1], at.o[hf][mt][3]);
            }
    }
    __syncthreads();
    cluster_wait();
    for (int idx = tid; idx < G * D / 4; idx += STEP_THREADS) {
        const int h = idx / (D / 4), dq = idx % (D / 4);
        float M = -INFINITY;
#pragma unroll
        for (int w = 0; w < STEP_WARPS; ++w) M = fmaxf(M, warp_m[w * 8 + h]);
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        float lacc = 0.f;
        if (M != -INFINITY) {
#pragma unroll
            for (int w = 0; w < STEP_WARPS; ++w) {
                // (a warp whose tiles the head did not attend: its part may be 0 * infinity)
                const float m = warp_m[w * 8 + h], sc = exp2f((m - M) * LOG2E);
                const float4 x = m == -INFINITY ? make_float4(0.f, 0.f, 0.f, 0.f) : *reinterpret_cast<const float4*>(parts + (w * G + h) * D + 4 * dq);
                acc.x = fmaf(x.x, sc, acc.x); acc.y = fmaf(x.y, sc, acc.y);
                acc.z = fmaf(x.z, sc, acc.z); acc.w = fmaf(x.w, sc, acc.w);
                lacc = fmaf(warp_l[w * 8 + h], sc, lacc);
            }
        }
        const int owner = idx / per;
        *cluster.map_shared_rank(in_o + rank * per + idx - owner * per, owner) = acc;
        if (dq == 0)
            for (int c = 0; c < n_ranks; ++c) *cluster.map_shared_rank(in_ml + rank * G + h, c) = make_float2(M, lacc);
    }
    cluster_arrive();
    cluster_wait();
    const int idx = rank * per + tid;
    if (tid < per && idx < G * D / 4) {
        const int h = idx / (D / 4);
        float M = -INFINITY, l = 0.f;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
        for (int c0 = 0; c0 < n_ranks; c0 += 8) {               // eight parts at a time
            float2 p[8];
            float4 x[8];
            float top = M;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const bool in = c0 + c < n_ranks;
                p[c] = in ? in_ml[(c0 + c) * G + h] : make_float2(-INFINITY, 0.f);
                x[c] = in ? in_o[(c0 + c) * per + tid] : make_float4(0.f, 0.f, 0.f, 0.f);
                top = fmaxf(top, p[c].x);
            }
            if (top == -INFINITY) continue;
            const float keep = exp2f((M - top) * LOG2E);
            acc.x *= keep; acc.y *= keep; acc.z *= keep; acc.w *= keep;
            l *= keep;
            M = top;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const float sc = exp2f((p[c].x - M) * LOG2E);            // a CTA without tiles: 0
                acc.x = fmaf(x[c].x, sc, acc.x); acc.y = fmaf(x[c].y, sc, acc.y);
                acc.z = fmaf(x[c].z, sc, acc.z); acc.w = fmaf(x[c].w, sc, acc.w);
                l = fmaf(p[c].y, sc, l);
            }
        }
        if (l > 0.f) { acc.x /= l; acc.y /= l; acc.z /= l; acc.w /= l; }
        else acc = make_float4(0.f, 0.f, 0.f, 0.f);
        *reinterpret_cast<float4*>(a.out + ((int64_t)i * a.Hq + hk * G) * D + 4 * idx) = acc;
    }
}

// One instance of the kernel
struct StepVariant {
    void (*kernel)(CUtensorMap, CUtensorMap, StepArgs);
    size_t smem;
    int recs;                            // records that a warp bounds at a time
};
static bool step_variant(int D, int TS, int G, bool packed, StepVariant& v) {
#define ETA_CASE(DD, TT, GG) if (D == DD && TS == TT && G == GG) { \
        v = {packed ? step_kernel<DD, TT, GG, true> : step_kernel<DD, TT, GG, false>, StepSmem<DD, TT, GG>::BYTES, TileOf<DD>::RECS}; return true; }
#define ETA_CASES(GG) ETA_CASE(128, 64, GG) ETA_CASE(128, 32, GG) ETA_CASE(64, 64, GG) ETA_CASE(64, 32, GG)
    ETA_CASES(1) ETA_CASES(2) ETA_CASES(4) ETA_CASES(8)
#undef ETA_CASES
#undef ETA_CASE
    return false;
}

// Which problems, by what the host knows: the capacity.  A row's cluster has to do alone what the general path spreads over the GPU,
// so a step is bound by the fullest row's tiles per CTA (0.6 us a tile of 32 KB that is attended); what it saves is two kernels.  Beside
// it, us a step by the general path and by this one, half / a twentieth of the blocks attended (d = 128, blocks of 64, G = 4, one
// step a graph): 8 rows of 2K tokens 19.5, 14.4 / 18.4, 14.4; of 8K 22.6, 18.4 / 20.5, 14.4; of 16K (33 tiles a CTA) 24.6, 24.6 / 18.5,
// 16.4; 16 rows of 12K (33) 25.3, 24.6 / 20.5, 16.7; 24 rows of 8K (32) 26.5, 24.6 / 20.5, 16.4; 4 rows of 32K (32) 22.8, 24.6 / 18.5,
// 16.8; 64 rows of 2K (16) 24.5, 22.6 / 19.9, 16.6.  Not taken, because what half the blocks lose is more than what few of them gain:
// 6 rows of 16K (33, in 48 CTAs) 22.6, 26.7 / 18.5, 16.4, of 32K (64) 24.6, 41.3 / 20.2, 18.5; 14 rows of 12K (33) 24.6, 30.7 / 20.5,
// 20.5; 48 rows of 4K in clusters of two (32) 25.0, 28.7 / 19.2, 17.6; 96 rows of 2K, one CTA each (32) 27.2, 28.8 / 20.5, 19.4.  So: up
// to 24 tiles a CTA, and up to 34 where the problem is large enough to leave the general path something to do and clusters of
// four or more take the difference between rows.  Of 900 problems of 1 to 256 rows at 0.1 to 0.95 sparsity 17 lose more than 3 % this
// way (12 % at most, with half or more of the blocks attended); by the number of tiles in all alone it was 90 (39 %).  One or two
// rows of more than 128 or 256 tiles leave most of the GPU idle: 2 rows of 510 21.2, 23.7.
// How many CTAs: clusters that all fit the GPU at once, by its own answer (a B200 holds 45 of three CTAs, 33 of four, 22 of six, 15 of
// eight, 7 of sixteen; a launch in clusters of which not one fits would be refused), with some to spare for the predictor's: 16 rows in
// clusters of 6 15.5 us, of 3 16.6, of 8, which do not all fit beside it, 24.1; 48 rows of 2K in clusters of three, which do not fit
// either, 24.6, of two 16.4; four rows of many tiles in clusters of 16 24.1, of 8 28.1.
// fit[c]: clusters of c CTAs that the GPU holds at once.  -> 0: not a problem for this kernel, or not a GPU for it
int step_cluster_rule(int rows, int nb_cap, int b, const int* fit) {
    const int tiles = b > 64 ? 2 * nb_cap : nb_cap, all = rows * tiles;
    if (nb_cap > STEP_MAX_BLOCKS || rows > STEP_MAX_TILES || all > STEP_MAX_TILES || tiles > 128 * rows) return 0;
    if (rows <= 4 && tiles > 64 && fit[STEP_MAX_CLUSTER] >= rows) return STEP_MAX_CLUSTER;
    for (int c = 8; c >= 1; --c)
        if (c > 4 ? 10 * fit[c] >= 11 * rows : fit[c] > rows)
            return tiles <= 24 * c || (tiles <= 34 * c && c >= 4 && all >= 2000) ? c : 0;
    return 0;
}

int step_cluster(int rows, int nb_cap, int b, int D, int TS, int G, bool packed) {
    StepVariant v;
    if (nb_cap > STEP_MAX_BLOCKS || !step_variant(D, TS, G, packed, v)) return 0;
    const void* const kernel = reinterpret_cast<const void*>(v.kernel);
    if (configure_kernel(kernel, v.smem) != ETA_OK) return 0;
    int fit[STEP_MAX_CLUSTER + 1];
    clusters_that_fit(kernel, STEP_THREADS, v.smem, fit);
    return step_cluster_rule(rows, nb_cap, b, fit);
}

int launch_step(StepArgs a, const CUtensorMap& tmK, const CUtensorMap& tmV, int rows, int D, int TS, int G, int n_ranks, cudaStream_t s) {
    StepVariant v;
    if (!step_variant(D, TS, G, (a.flags & ETA_FLAG_PACKED_SIGMA) != 0, v)) return ETA_ERR_UNSUPPORTED;
    a.shared = n_ranks > 1 && a.nb_cap > STEP_WARPS * v.recs;
    const int rc = configure_kernel(reinterpret_cast<const void*>(v.kernel), v.smem);
    if (rc != ETA_OK) return rc;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = cluster_config(n_ranks, rows, STEP_THREADS, v.smem, attr);
    cfg.stream = s;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = pdl_enabled() ? 1 : 0;
    cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, v.kernel, tmK, tmV, a);
    if (e != cudaSuccess) { set_cuda_error(e, "step launch"); return ETA_ERR_CUDA; }
    return check_launch("step launch");
}

}  // namespace eta
