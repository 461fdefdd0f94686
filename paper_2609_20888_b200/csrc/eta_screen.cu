// Screening stage of eta_decode (Eq. dual_bound_eq; Algorithm 3, screening and
// rescue lines), and the diagnostic that returns its bounds.
//
// A warp bounds a tile of consecutive block records (8 KB of them) of one
// (sequence, KV head) row for all G query heads of the group.  Both sums of
// Score_dual are small dense contractions over head_dim and run on the tensor
// cores: <q, mu> in fp16, sum q^2 sigma^2 in tf32 with both factors split into
// two parts that hold them exactly.  The query side (A fragments) is prepared
// once per CTA in shared memory; a tile of records arrives in the warp's own
// piece of shared memory by one 1-D bulk copy, and the warps of a CTA do not
// wait for one another until the thresholds are needed.
//
// screen_kernel: a CTA of four warps takes a run of passes (four tiles each) of a
// row.  Phase 1 (bounds; needs neither thresholds nor the newest summary)
// never waits for a predecessor kernel; phase 2 (admission, pinning, mask,
// ballot + popc compaction) takes a warp per segment of SEG records after the
// dependency wait.  Nothing returns to the host.
//
// Top-1 rescue needs the whole rescue window of a head: the first CTA of a row
// takes at least the passes the window spans, and decides rescue before it
// writes its lists.  Where that would be more passes than the row's other CTAs
// take, every CTA leaves its largest bounds and rescue_kernel decides.
#include "eta_bounds.cuh"
#include "eta_timeline.h"

namespace eta {

// Shared memory of both kernels: the query table, two barriers per warp, the warps' tiles, bounds of `recs` records
template <int D, int G>
struct ScreenSmem {
    static constexpr int BAR_OFF = (int)((sizeof(QTab<D, G>) + 15) / 16 * 16);
    static constexpr int TILE_OFF = (BAR_OFF + 16 * SCR_WARPS + 127) / 128 * 128;
    static size_t bytes(int recs, int nbuf) {            // + slack for a 128-byte base
        return TILE_OFF + (size_t)nbuf * SCR_WARPS * TileOf<D>::BYTES + sizeof(float) * (size_t)recs * G + 112;
    }
};
// CTAs per SM the screening grid is sized for.  A fifth would fit an empty SM, but the append and predictor CTAs are still
// on some of them: with 5 the last CTAs only start when the first have had their thresholds (65536 blocks at d = 128: 71.7
// us a step, 4: 68.8, 3: 70.5, 2: 72.7; 128 rows at d = 64, G = 8: 118.4, 116.3, 120.4, 123.7; measured before the streaming
// kernel's changes that brought these steps to 59 and 90 us).
constexpr int SCR_SLOTS = 4;
constexpr int SCR_GROUP = 4;         // most passes whose bounds wait in shared memory for the thresholds
constexpr int SCR_WINDOW = 2;        // passes of a rescue window that a row's first CTA takes in any case

// Zeroes n bytes with the threads of a CTA: 16 at a time between the ends
__device__ __forceinline__ void zero_bytes(uint8_t* p, int n, int tid) {
    if (n <= 0) return;
    const int lead = min(n, (int)(-reinterpret_cast<uintptr_t>(p) & 15)), body = (n - lead) >> 4, rest = (n - lead) & 15;
    if (tid < lead) p[tid] = 0;
    for (int k = tid; k < body; k += 32 * SCR_WARPS) reinterpret_cast<uint4*>(p + lead)[k] = make_uint4(0, 0, 0, 0);
    if (tid < rest) p[lead + 16 * body + tid] = 0;
}

// What bounds it: HBM for the records (33.8 MB for 65536 blocks at d = 128, 5.2 us at the copy rate) once enough of them are
// requested; small CTAs, because the hardware then fills whatever the predecessor kernels leave of each SM, and all of them
// resident at once, because none can finish before the thresholds are there.  A step of 65536 blocks at d = 128, G = 4 took
// 68.8 us instead of 71.1 with it (two persistent CTAs per SM, the variance term on the fp32 pipe behind a shuffle tree and a CTA
// barrier per segment); 65536 blocks at d = 64, G = 8, where both terms were on that pipe, 116.3 instead of 126.9.
// Registers: CTAs start beside those of the append and the predictor, and with more registers fewer of them fit there.  The bound of
// six CTAs holds the instances to 80 that would take many more by themselves.  The others take 77 to 88 at five, at d = 64, G = 8
// 95 (packed 96 and 32 bytes spilled): six gives d = 128, G = 4 48.5 instead of 49.1 us at 32K x 8, but 57.9 instead of 57.6 at 128K x 4 and 41.9 instead of 41.5 at 512K x 1,
// and d = 64 32.8 instead of 31.8 at 64K x 4 (G = 1).
template <int D, int G, bool PACKED>
__global__ void __launch_bounds__(32 * SCR_WARPS, D == 128 && (G == 8 || (G == 4 && PACKED)) ? 6 : 5) screen_kernel(
    const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const ScreenArgs a) {
    using L = ScreenSmem<D, G>;
    using TL = TileOf<D>;
    constexpr int REC_BYTES = PACKED ? 3 * D : 4 * D;
    extern __shared__ unsigned char scr_raw[];
    unsigned char* sm = scr_raw + ((128u - (smem_u32(scr_raw) & 127u)) & 127u);
    QTab<D, G>& tab = *reinterpret_cast<QTab<D, G>*>(sm);
    float* const sbound_all = reinterpret_cast<float*>(sm + L::TILE_OFF + a.nbuf * SCR_WARPS * TL::BYTES);      // [record of the group][G]
    __shared__ uint32_t s_bkey[G];                      // per head: largest bound of the rescue window (as an ordered integer)
    __shared__ int s_best[G];                           // and the first block that attains it

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool dense = (a.flags & ETA_FLAG_DENSE) != 0;
    unsigned long long* const tl = ETA_TL((a.timeline && blockIdx.x < TL_SCREEN_N) ? a.timeline + (size_t)(TL_SCREEN + blockIdx.x) * 8 : nullptr);
    if (tl && tid == 0) tl[0] = globaltimer_ns();

    // The CTA's row and its passes [p_first, p_last) of it.  A row's first CTA takes `head` passes (its rescue window at
    // least), each further one `tp`.
    int i, hk, c, n_ctas = a.ctas_row, P = a.passes, tp = a.tp, Traw;    // P: passes of the row; n_ctas: CTAs of the row, c: this one
    bool by_capacity = true;
    if (a.by_length) {
        // Rows of one launch may differ in length, and the slowest CTA sets the kernel's end: every warp looks at the lengths (a
        // sequence per lane) and, unless all rows fill their capacity, works out the smallest tp with which all CTAs fit
        // the slots, and which of them it is.
        const bool seq = lane < a.batch;
        const int Tl = seq ? __ldg(a.seq_lens + lane) : 0;
        const int nb = min(max(min(Tl, a.t_cap), 0) >> a.b_shift, a.nb_cap);
        const int Pl = seq ? max(1, (nb + TL::PASS - 1) / TL::PASS) : 0;
        if (!__all_sync(0xffffffffu, !seq || Pl == a.passes)) {
            by_capacity = false;
            const int total = __reduce_add_sync(0xffffffffu, Pl) * a.Hkv;
            tp = a.div_slots.div(total + a.slots - 1);
            int k, incl;
            while (true) {
                // 1 + ceil((Pl - head) / tp), by a reciprocal: exact, the numbers are small
                const int over = max(0, Pl - max(tp, a.need)) + tp - 1;
                k = seq ? 1 + (int)(__fdividef((float)over + 0.5f, (float)tp)) : 0;
                incl = k * a.Hkv;
#pragma unroll
                for (int sft = 1; sft < 32; sft <<= 1) {
                    const int o = __shfl_up_sync(0xffffffffu, incl, sft);
                    if (lane >= sft) incl += o;
                }
                if (tp >= a.passes || __shfl_sync(0xffffffffu, incl, 31) <= a.slots) break;
                tp += max(1, tp >> 3);
            }
            const unsigned before = __ballot_sync(0xffffffffu, incl <= (int)blockIdx.x);
            if (before == 0xffffffffu) return;                // more CTAs than these lengths need
            i = __popc(before);
            n_ctas = __shfl_sync(0xffffffffu, k, i);
            P = __shfl_sync(0xffffffffu, Pl, i);
            Traw = __shfl_sync(0xffffffffu, Tl, i);
            const int rem = (int)blockIdx.x - (__shfl_sync(0xffffffffu, incl, i) - n_ctas * a.Hkv);
            hk = (int)__fdividef((float)rem + 0.5f, (float)n_ctas);
            c = rem - hk * n_ctas;
        }
    }
    if (by_capacity) {
        if ((int)blockIdx.x >= a.ctas_all) return;
        int rr;
        a.div_ctas.divmod(blockIdx.x, rr, c);
        a.div_hkv.divmod(rr, i, hk);
        Traw = __ldg(a.seq_lens + i);
    }
    const uint4 q_piece = dense ? make_uint4(0, 0, 0, 0) : load_qtab<D, G>(a.q + ((int64_t)i * a.Hq + hk * G) * D, tid);
    const int r = i * a.Hkv + hk, head = max(tp, a.need);
    const int p_first = c == 0 ? 0 : head + (c - 1) * tp, p_last = min(P, head + c * tp);
    const int T = Traw < 0 ? 0 : (Traw > a.t_cap ? a.t_cap : Traw);
    const int NB = min(T >> a.b_shift, a.nb_cap);
    const unsigned char* const rec_row = reinterpret_cast<const unsigned char*>(a.musig) + (int64_t)r * a.nb_cap * REC_BYTES;
    const float* const mn_row = a.mnorm + (int64_t)r * a.nb_cap;

    uint64_t* bars = reinterpret_cast<uint64_t*>(sm + L::BAR_OFF) + 2 * warp;
    if (lane == 0) { mbar_init(&bars[0], 1); mbar_init(&bars[1], 1); fence_barrier_init(); }
    if (tid < G) { s_bkey[tid] = 0u; s_best[tid] = 0; }
    __syncwarp();
    TileStream<D, G, PACKED> ts{sm + L::TILE_OFF + warp * a.nbuf * TL::BYTES, bars, rec_row, mn_row, dense ? 0 : NB, a.nbuf, 0, 0, 0u, true};
    for (int p = p_first; p < min(p_last, p_first + a.nbuf); ++p) ts.issue(p * TL::PASS + warp * TL::RECS);
    if (!dense) build_qtab<D, G>(tab, q_piece, tid);

    // an ungated newest token must be attended: when it closes a full block, that block counts as pinned
    const int lwb = ((a.flags & ETA_FLAG_UNGATE_LAST) && T > 0 && (T & (a.b - 1)) == 0 && a.lwb < 1) ? 1 : a.lwb;
    const int Wr = min(a.rescue_window, NB);
    float te_l = -INFINITY;               // lane gq < G: effective threshold of head gq
    // Top-1 rescue (Algorithm 3): a head that admits none of the first Wr blocks attends the first one with the largest
    // bound among them.  It admits none exactly when that bound is below its threshold and no block of the window is pinned
    // (a NaN bound admits), so the row's first CTA looks for the largest bounds ahead of the wait for the thresholds, a warp
    // per head, with bounds compared as order-preserving integers.
    const bool rescues = (c == 0 || a.resc) && !dense && Wr > 0 && !(lwb > 0 && NB - lwb < Wr);
    const bool stale = !dense && NB > 0 && (T & (a.b - 1)) == 0;      // the newest block's record may not have been final yet
    auto window_max = [&](int p0, int p1) {
        const int n_win = min(Wr, p1 * TL::PASS) - p0 * TL::PASS;
        for (int gq = warp; gq < G; gq += SCR_WARPS) {
            uint32_t key = 0;                     // 0: no record of the window in this lane
            int arg = 0x7fffffff;
            for (int rec = lane; rec < n_win; rec += 32) {                  // ascending: a lane keeps the first of equal bounds
                const uint32_t k2 = bound_key(sbound_all[rec * G + gq]);
                if (k2 > key) { key = k2; arg = rec; }
            }
            const uint32_t kmax = __reduce_max_sync(0xffffffffu, key);
            const int amin = __reduce_min_sync(0xffffffffu, key == kmax ? arg : 0x7fffffff);
            if (lane == 0 && kmax > s_bkey[gq]) { s_bkey[gq] = kmax; s_best[gq] = p0 * TL::PASS + amin; }
        }
        __syncthreads();
    };
    bool waited = false;
    unsigned missing = 0;                 // heads to rescue, known with the first group of passes where that holds the window
    const bool whole_window = Wr <= min(p_last, a.group) * TL::PASS;
    for (int p0 = p_first; p0 < p_last; p0 += a.group) {
        const int p1 = min(p_last, p0 + a.group);
        // -------------------------------------------------------- phase 1: bounds of a group of passes
        // The summaries and thresholds may still be in the making when this kernel starts (programmatic dependent
        // launch): the append kernel writes the record and the norm of a block that has just filled up, the predictor
        // writes tau.  Everything else this kernel reads is final.  Phase 1 therefore never waits: the one record per
        // row that may be stale (the newest block of a just-completed length) gets a bound there like any other, and
        // the warp that handles its segment in phase 2, after the wait, computes that bound again.
        for (int p = p0; p < p1; ++p) {
            const bool ok = ts.bounds(tab, p * TL::PASS + warp * TL::RECS, a.z, a.scale, sbound_all + ((p - p0) * TL::PASS + warp * TL::RECS) * G);
            if (!ok && lane == 0 && a.status) atomicOr(a.status, ETA_DEV_TIMEOUT);
            if (p + a.nbuf < p_last) ts.issue((p + a.nbuf) * TL::PASS + warp * TL::RECS);
            if (tl && tid == 0 && p == p_first) tl[1] = globaltimer_ns();
        }
        __syncthreads();
        const bool stale_in = stale && NB - 1 >= p0 * TL::PASS && NB - 1 < p1 * TL::PASS;
        if (rescues && p0 * TL::PASS < Wr && !stale_in) window_max(p0, p1);
        if (tl && tid == 0 && !waited) tl[2] = globaltimer_ns();
        // -------------------------------------------------------- phase 2: a warp per segment
        const int seg_0 = p0 * (TL::PASS / SEG), s_end = min(a.nseg, p1 * (TL::PASS / SEG));
        if (!waited) {
            pdl_wait();                   // the thresholds (and the newest summaries) are final now
            if (tl && tid == 0) tl[3] = globaltimer_ns();
            if (!dense && lane < G) {
                const int h = hk * G + lane;
                te_l = (a.tau ? __ldcg(a.tau + (int64_t)i * a.Hq + h) : __ldcg(a.head_const + h)) - a.a;
            }
        }
        // the newest block's bound again, while the thresholds are on their way
        if (stale_in) {
            if (((NB - 1) / SEG - seg_0) % SCR_WARPS == warp)
                bound_one<D, G, PACKED>(tab.raw, rec_row + (int64_t)(NB - 1) * REC_BYTES, __ldcg(mn_row + NB - 1), a.z, a.scale,
                                        sbound_all + (NB - 1 - p0 * TL::PASS) * G);
        }
        if (!waited && c == 0 && warp == 0) {
            if (lane < G) a.tau_eff[(int64_t)i * a.Hq + hk * G + lane] = te_l;
            if (lane == 0 && a.status) {
                if (Traw > a.t_cap) atomicOr(a.status, ETA_DEV_LEN_CLAMPED);
                if (Traw <= 0) atomicOr(a.status, ETA_DEV_EMPTY_ROW);
            }
        }
        waited = true;
        float te_g[G];
#pragma unroll
        for (int gq = 0; gq < G; ++gq) te_g[gq] = __shfl_sync(0xffffffffu, te_l, gq);
        // admission bits of records lane and lane + 32 of a segment
        auto admit = [&](int seg, unsigned (&m)[SEG / 32]) {
            const int j0 = seg * SEG, n_rec = min(SEG, NB - j0);
            const float (*sbound)[G] = reinterpret_cast<const float (*)[G]>(sbound_all + (j0 - p0 * TL::PASS) * G);
#pragma unroll
            for (int half = 0; half < SEG / 32; ++half) {
                const int rec = half * 32 + lane;
                m[half] = 0;
                if (rec < n_rec) {
                    const bool pinned = (j0 + rec) >= NB - lwb;
#pragma unroll
                    for (int gq = 0; gq < G; ++gq)
                        if (dense || pinned || !(sbound[rec][gq] < te_g[gq])) m[half] |= 1u << gq;
                }
            }
        };
        if (rescues && p0 * TL::PASS < Wr) {
            if (stale_in) { __syncthreads(); window_max(p0, p1); }
            if (!a.resc && p1 * TL::PASS >= Wr) {
#pragma unroll
                for (int gq = 0; gq < G; ++gq)
                    if (key_bound(s_bkey[gq]) < te_g[gq]) missing |= 1u << gq;
            }
        }
        for (int seg = seg_0 + warp; seg < s_end; seg += SCR_WARPS) {
            const int j0 = seg * SEG;
            unsigned m[SEG / 32];
            admit(seg, m);
            if (whole_window) {
                for (unsigned left = missing; left; left &= left - 1) {
                    const int gq = __ffs(left) - 1, rec = s_best[gq] - j0;
                    if (rec == lane) m[0] |= 1u << gq;
                    if (rec == lane + 32) m[1] |= 1u << gq;
                }
            }
            // user-visible bits; entries of this segment that are not full blocks read as "not attended"
#pragma unroll
            for (int half = 0; half < SEG / 32; ++half)
                if (j0 + half * 32 + lane < a.nb_cap) a.sel_mask[(int64_t)r * a.nb_cap + j0 + half * 32 + lane] = (uint8_t)m[half];
            // segment-local compaction of the union (ballot + popc prefix), ascending block order
            int carry = 0;
            int32_t* list = a.seg_list + ((int64_t)r * a.nseg + seg) * LSTRIDE;
#pragma unroll
            for (int half = 0; half < SEG / 32; ++half) {
                const unsigned nz = __ballot_sync(0xffffffffu, m[half] != 0);
                if (m[half]) list[carry + __popc(nz & ((1u << lane) - 1u))] = (j0 + half * 32 + lane) | (int)(m[half] << 24);
                carry += __popc(nz);
            }
            if (lane == 0) a.seg_cnt[((int64_t)r * a.gpr) * GRANULE + seg] = (uint8_t)carry;
            // The memory is idle from here until the streaming kernel's first copies, some 8 us: the segment's first survivors
            // start on their way into the L2.
            if (a.prefetch) {
                int rank = 0;
#pragma unroll
                for (int half = 0; half < SEG / 32; ++half) {
                    const unsigned nz = __ballot_sync(0xffffffffu, m[half] != 0);
                    if (m[half] && rank + __popc(nz & ((1u << lane) - 1u)) < a.prefetch) {
                        const int j = j0 + half * 32 + lane;
                        const int w4 = a.block_table ? __ldcg(a.block_table + (int64_t)i * a.table_stride + j) : i;
                        for (int k = 0; k < a.tiles; ++k) {
                            const int y = (a.block_table ? 0 : j * a.b) + k * a.tile_tokens;
                            tma_prefetch_5d(&tmK, 0, y, 0, hk, w4);
                            tma_prefetch_5d(&tmV, 0, y, 0, hk, w4);
                        }
                    }
                    rank += __popc(nz);
                }
            }
        }
        if (p1 < p_last) __syncthreads();          // the bounds of this group have been read: the next may overwrite them
    }
    // The successor may set up from here on (it waits for the end of this kernel before it reads anything).  After the stores
    // below, where warps leave one by one, a small eager step took up to a microsecond longer (2K x 1 17.5 -> 18.8).
    pdl_trigger();
    // what the row's passes do not reach: no survivors, nothing attended
    if (c == n_ctas - 1) {
        const int seg_n = min(a.nseg, P * (TL::PASS / SEG)), rec_n = min(a.nb_cap, P * TL::PASS);
        zero_bytes(a.seg_cnt + (int64_t)r * a.gpr * GRANULE + seg_n, a.gpr * GRANULE - seg_n, tid);
        zero_bytes(a.sel_mask + (int64_t)r * a.nb_cap + rec_n, a.nb_cap - rec_n, tid);
    }
    // A rescue window of several groups of passes: the rescued blocks join lists that are already written.  A block another
    // head fetches anyway gets the head's bit, any other goes to the end of its segment's list.
    if (missing && !whole_window) {
        __syncthreads();                  // lists, counts and mask of this CTA are written
        for (unsigned left = warp == 0 ? missing : 0u; left; left &= left - 1) {
            const int gq = __ffs(left) - 1, j = s_best[gq], seg = j / SEG;
            volatile uint8_t* mp = a.sel_mask + (int64_t)r * a.nb_cap + j;
            volatile uint8_t* np = a.seg_cnt + ((int64_t)r * a.gpr) * GRANULE + seg;
            volatile int32_t* list = a.seg_list + ((int64_t)r * a.nseg + seg) * LSTRIDE;
            const unsigned w = *mp, n = *np;
            __syncwarp();                 // every lane has read them
            if (w == 0) {
                if (lane == 0) { list[n] = j | (1 << (24 + gq)); *np = (uint8_t)(n + 1); }
            } else {
                for (unsigned k = lane; k < n; k += 32)
                    if ((list[k] & 0xffffff) == j) list[k] = list[k] | (1 << (24 + gq));
            }
            if (lane == 0) *mp = (uint8_t)(w | (1u << gq));
            __syncwarp();
        }
    }
    if (a.resc) {
        if (tid < G) a.resc[a.rows + (int64_t)blockIdx.x * G + tid] = make_int2((int)s_bkey[tid], s_best[tid]);
        if (c == 0 && tid == 0) a.resc[r] = make_int2(blockIdx.x, n_ctas);
    }
    if (tl && tid == 0) tl[5] = globaltimer_ns();
}

// Top-1 rescue of the rows whose window no single CTA of the screening kernel holds: a CTA per row, a warp per head (latency:
// two dependent reads, then as many for a head that needs rescue).  The largest of the CTAs' bounds decides; the rescued block
// joins lists that are already written.  A block another head fetches anyway gets the head's bit, any other goes to the end
// of its segment's list.
__global__ void __launch_bounds__(256) rescue_kernel(const int2* span, const int2* best, const float* tau_eff, int G, int nb_cap,
                                                     int nseg, int gpr, uint8_t* sel_mask, uint8_t* seg_cnt, int32_t* seg_list) {
    __shared__ int s_block[8];            // rescued block of each head, or -1
    const int r = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_trigger();
    pdl_wait();                           // the screening kernel's lists are complete
    if (warp < G) {
        const float te = __ldcg(tau_eff + (int64_t)r * G + warp);
        const int2 sp = __ldcg(span + r);
        uint32_t key = 0;
        int arg = 0x7fffffff;
        for (int c = lane; c < sp.y; c += 32) {            // ascending: a lane keeps the first of equal bounds
            const int2 e = __ldcg(best + (int64_t)(sp.x + c) * G + warp);
            if ((uint32_t)e.x > key) { key = (uint32_t)e.x; arg = e.y; }
        }
        const uint32_t kmax = __reduce_max_sync(0xffffffffu, key);
        const int amin = __reduce_min_sync(0xffffffffu, key == kmax ? arg : 0x7fffffff);
        if (lane == 0) s_block[warp] = key_bound(kmax) < te ? amin : -1;
    }
    __syncthreads();
    for (int gq = 0; gq < G && warp == 0; ++gq) {
        const int j = s_block[gq], seg = j / SEG;
        if (j < 0) continue;
        volatile uint8_t* mp = sel_mask + (int64_t)r * nb_cap + j;
        volatile uint8_t* np = seg_cnt + (int64_t)r * gpr * GRANULE + seg;
        volatile int32_t* list = seg_list + ((int64_t)r * nseg + seg) * LSTRIDE;
        const unsigned w = *mp, n = *np;
        __syncwarp();                     // every lane has read them
        if (w == 0) {
            if (lane == 0) { list[n] = j | (1 << (24 + gq)); *np = (uint8_t)(n + 1); }
        } else {
            for (unsigned k = lane; k < n; k += 32)
                if ((list[k] & 0xffffff) == j) list[k] = list[k] | (1 << (24 + gq));
        }
        if (lane == 0) *mp = (uint8_t)(w | (1u << gq));
        __syncwarp();
    }
}

// Eq. dual_bound_eq for every block, for its own sake: the tiles of the screening kernel, stored instead of compared.
// Bound by HBM (33.8 MB of records in, 1.05 MB of bounds out at 65536 blocks, d = 128, G = 4: 5.3 us at the copy rate) and by the two
// round trips of a CTA's two passes; a record is read once for all heads of its group.  8.2 us a call there as one of four nodes of a
// graph (9.2 before the records were the rows of the MMAs; of 65536 blocks at d = 64, 7.3 -> 5.5 for G = 1, 6.7 -> 5.6 for G = 4), some
// 10 queued eagerly, which is what the host takes for a call; 108 us with a warp per (head, block) that read every record G times in
// 2-byte pieces and reduced three sums over 32 lanes for each.
template <int D, int G, bool PACKED>
__global__ void __launch_bounds__(32 * SCR_WARPS, 5) score_dual_kernel(
    const __nv_bfloat16* q, const unsigned char* musig, const float* mnorm, const int32_t* seq_lens, int Hq, int Hkv, int b,
    int t_cap, int nb_cap, int per, int chunks, float z, float scale, float* __restrict__ bound) {
    using L = ScreenSmem<D, G>;
    using TL = TileOf<D>;
    extern __shared__ unsigned char scr_raw[];
    unsigned char* sm = scr_raw + ((128u - (smem_u32(scr_raw) & 127u)) & 127u);
    QTab<D, G>& tab = *reinterpret_cast<QTab<D, G>*>(sm);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint64_t* bars = reinterpret_cast<uint64_t*>(sm + L::BAR_OFF) + 2 * warp;
    float* const sb = reinterpret_cast<float*>(sm + L::TILE_OFF + SCR_WARPS * TL::BYTES) + warp * TL::RECS * G;
    const int r = blockIdx.x / chunks, i = r / Hkv, hk = r % Hkv;
    // Launched while the kernel before it ends, which it waits for before it reads anything.  That is worth the gap between two
    // kernels and no more: calls queued one after the other 12.3 -> 10.0 us each for 65536 blocks (9.9 -> 9.7 as nodes of a graph, 64
    // bounds 2.3 -> 2.2), a call by itself 14.4 between two events either way.  (It lets no successor start early: the screening kernel
    // reads its inputs without waiting for them.  The summary build, with CTAs by the ten thousand, is slower this way: 174 -> 218 us
    // for 1.07 GB, three inputs in turn.)
    pdl_wait();
    int T = __ldcg(seq_lens + i);
    const uint4 q_piece = load_qtab<D, G>(q + ((int64_t)i * Hq + hk * G) * D, tid);
    T = T < 0 ? 0 : (T > t_cap ? t_cap : T);
    const int NB = min(T / b, nb_cap);
    const int first = (blockIdx.x % chunks) * per * TL::PASS;
    if (first >= NB) return;
    if (lane == 0) { mbar_init(&bars[0], 1); mbar_init(&bars[1], 1); fence_barrier_init(); }
    __syncwarp();
    TileStream<D, G, PACKED> ts{sm + L::TILE_OFF + warp * TL::BYTES, bars, musig + (int64_t)r * nb_cap * TileStream<D, G, PACKED>::REC,
                                mnorm + (int64_t)r * nb_cap, NB, 1, 0, 0, 0u, true};
    const int last = min(NB, first + per * TL::PASS);
    ts.issue(first + warp * TL::RECS);
    build_qtab<D, G>(tab, q_piece, tid);
    for (int j0 = first + warp * TL::RECS; j0 < last; j0 += TL::PASS) {
        const int n = min(TL::RECS, NB - j0);
        ts.bounds(tab, j0, z, scale, sb);
        if (j0 + TL::PASS < last) ts.issue(j0 + TL::PASS);
        if (lane < n) {
#pragma unroll
            for (int g = 0; g < G; ++g) bound[((int64_t)i * Hq + hk * G + g) * nb_cap + j0 + lane] = sb[lane * G + g];
        }
        __syncwarp();
    }
}

// The same with a warp per (sequence, query head, block): for arrays that 16-byte loads cannot read (a caller's odd offset), and
// for few bounds, where warps fill the GPU and tiles do not (what counts is then the length of one tile's chain of steps).
__global__ void __launch_bounds__(128) score_dual_warp_kernel(
    const __nv_bfloat16* q, const unsigned char* musig, const float* mnorm, const int32_t* seq_lens, int B, int Hq, int Hkv,
    int d, int b, int t_cap, int nb_cap, float z, float scale, int packed, float* __restrict__ bound) {
    const int64_t wid = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    pdl_wait();
    if (wid >= (int64_t)B * Hq * nb_cap) return;
    const int j = (int)(wid % nb_cap);
    const int h = (int)((wid / nb_cap) % Hq);
    const int i = (int)(wid / ((int64_t)nb_cap * Hq));
    int T = __ldcg(seq_lens + i);
    T = T < 0 ? 0 : (T > t_cap ? t_cap : T);
    if (j >= T / b) return;
    const int G = Hq / Hkv;
    const int64_t rec = ((int64_t)i * Hkv + h / G) * nb_cap + j;
    const __nv_bfloat16* qv = q + ((int64_t)i * Hq + h) * d;
    float dot = 0.f, var = 0.f, n2 = 0.f;
    for (int c = lane; c < d; c += 32) {
        const float x = __bfloat162float(__ldcg(qv + c));
        const unsigned char* rp = musig + rec * (packed ? 3 * d : 4 * d);
        const float m = __half2float(__ldcg(reinterpret_cast<const __half*>(rp) + c));
        float s;
        if (packed) {
            const uint32_t h2 = e4m3x2_to_f16x2(__ldcg(rp + 2 * d + c));
            s = __half2float(*reinterpret_cast<const __half*>(&h2));
        } else {
            s = __half2float(__ldcg(reinterpret_cast<const __half*>(rp) + d + c));
        }
        dot = fmaf(x, m, dot);
        var = fmaf(x * x, s * s, var);
        n2 = fmaf(x, x, n2);
    }
    for (int s = 16; s >= 1; s >>= 1) {
        dot += __shfl_xor_sync(0xffffffffu, dot, s);
        var += __shfl_xor_sync(0xffffffffu, var, s);
        n2 += __shfl_xor_sync(0xffffffffu, n2, s);
    }
    if (lane == 0) bound[wid] = scale * min_keep_nan(dot + z * sqrtf(var), sqrtf(n2) * __ldcg(mnorm + rec));
}

// ------------------------------------------------------------------ launchers (host)

// Passes that all CTAs but a row's first take at full length, passes that the rescue window spans, and whether rescue_kernel settles
// rescue.  A window of more passes than a row's other CTAs take would be its first CTA's work alone, one pass after another: a kernel
// of its own settles rescue then, for 1 to 3 us a step.  128K x 4 (d = 128, two passes per CTA), windows of 128 blocks 58 us;
// 256 63.8 in the first CTA, 60.2 this way; 1024 90.9 and 60.5; all blocks 117.6 and 61.0 (512K x 1: 192 and 38.7; 64K, d = 64,
// G = 8: 76.0 and 32.6).
struct ScreenSplit { int tp, need; bool late; };
static ScreenSplit screen_split(int rows, int nseg, int nb_cap, int pass, int window, bool dense, int n_sm) {
    const int passes = (nseg + pass / SEG - 1) / (pass / SEG), slots = SCR_SLOTS * n_sm;
    ScreenSplit p;
    p.tp = (int)(((int64_t)rows * passes + slots - 1) / slots);
    p.need = ((window < nb_cap ? window : nb_cap) + pass - 1) / pass;
    p.late = !dense && p.need > (p.tp > SCR_WINDOW ? p.tp : SCR_WINDOW);
    return p;
}
int screen_launches(int rows, int nseg, int nb_cap, int D, int window, bool dense, int n_sm) {
    return screen_split(rows, nseg, nb_cap, D == 128 ? TileOf<128>::PASS : TileOf<64>::PASS, window, dense, n_sm).late ? 2 : 1;
}

template <int D, int G, bool PACKED>
static int launch_screen_t(const ScreenArgs& a, const CUtensorMap& tmK, const CUtensorMap& tmV, int rows, int n_sm, cudaStream_t s) {
    constexpr int SPP = TileOf<D>::PASS / SEG;
    ScreenArgs b2 = a;
    b2.passes = (a.nseg + SPP - 1) / SPP;
    b2.batch = rows / a.Hkv;
    b2.slots = SCR_SLOTS * n_sm;
    // the split at full length: what rows of any length stay below, and what is used where there are too many to look at
    const int64_t all = (int64_t)rows * b2.passes;
    const ScreenSplit split = screen_split(rows, a.nseg, a.nb_cap, TileOf<D>::PASS, a.rescue_window, (a.flags & ETA_FLAG_DENSE) != 0, n_sm);
    const bool late = split.late;
    b2.tp = split.tp;
    b2.need = late ? 0 : split.need;
    if (!late) b2.resc = nullptr;
    const int head = b2.tp > b2.need ? b2.tp : b2.need;
    b2.ctas_row = b2.passes <= head ? 1 : 1 + (b2.passes - head + b2.tp - 1) / b2.tp;
    b2.div_ctas = FastDiv(b2.ctas_row);
    b2.ctas_all = rows * b2.ctas_row;
    // by length where a warp can look at all sequences and there are enough passes for the split to matter
    b2.by_length = b2.batch > 1 && b2.batch <= 32 && all > b2.slots && rows <= b2.slots;
    b2.div_slots = FastDiv(b2.slots);
    const int grid = b2.by_length && b2.ctas_all < b2.slots ? b2.slots : b2.ctas_all;
    b2.group = head < b2.passes ? head : b2.passes;      // passes whose bounds wait in shared memory for the thresholds
    if (b2.group > SCR_GROUP) b2.group = SCR_GROUP;
    // A second buffer per warp (three CTAs per SM) where all CTAs are still resident at once: a CTA of two passes, such as
    // the one that holds the rescue window, then has both on their way from the start.
    b2.nbuf = (b2.group > 1 && all <= 3 * n_sm) ? 2 : 1;
    const int rc = launch_pdl("screen launch", screen_kernel<D, G, PACKED>, dim3((unsigned)grid), dim3(32 * SCR_WARPS),
                              ScreenSmem<D, G>::bytes(b2.group * TileOf<D>::PASS, b2.nbuf), s, tmK, tmV, b2);
    if (rc != ETA_OK || !late) return rc;
    return launch_pdl("rescue launch", rescue_kernel, dim3((unsigned)rows), dim3(256), 0, s, (const int2*)a.resc,
                      (const int2*)(a.resc + rows), (const float*)a.tau_eff, G, a.nb_cap, a.nseg, a.gpr, a.sel_mask, a.seg_cnt,
                      a.seg_list);
}

int launch_screen(const ScreenArgs& a, const CUtensorMap& tmK, const CUtensorMap& tmV, int rows, int D, int G, int n_sm, cudaStream_t s) {
    const bool packed = (a.flags & ETA_FLAG_PACKED_SIGMA) != 0;
#define ETA_CASE(DD, GG) if (D == DD && G == GG) return packed ? launch_screen_t<DD, GG, true>(a, tmK, tmV, rows, n_sm, s) \
                                                                : launch_screen_t<DD, GG, false>(a, tmK, tmV, rows, n_sm, s);
    ETA_CASE(128, 1) ETA_CASE(128, 2) ETA_CASE(128, 4) ETA_CASE(128, 8)
    ETA_CASE(64, 1) ETA_CASE(64, 2) ETA_CASE(64, 4) ETA_CASE(64, 8)
#undef ETA_CASE
    return ETA_ERR_UNSUPPORTED;
}

template <int D, int G, bool PACKED>
static int launch_score_t(const eta_cache_desc* desc, const __nv_bfloat16* q, const unsigned char* musig, const float* mnorm,
                          const int32_t* seq_lens, float z, float scale, float* bound, cudaStream_t s) {
    int dev = 0, n_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) { set_cuda_error(e, "device query"); return ETA_ERR_CUDA; }
    const int rows = desc->batch * desc->n_kv_heads, passes = (desc->nb_cap + TileOf<D>::PASS - 1) / TileOf<D>::PASS;
    const int64_t all = (int64_t)rows * passes;
    const int per = (int)((all + 5 * n_sm - 1) / (5 * n_sm)), chunks = (passes + per - 1) / per;      // about five CTAs per SM
    const size_t smem = ScreenSmem<D, G>::bytes(TileOf<D>::PASS, 1);
    return launch_pdl("eta_score_dual", score_dual_kernel<D, G, PACKED>, dim3((unsigned)(rows * chunks)), dim3(32 * SCR_WARPS), smem, s,
                      q, musig, mnorm, seq_lens, (int)desc->n_q_heads, (int)desc->n_kv_heads, (int)desc->block_size, (int)desc->t_cap,
                      (int)desc->nb_cap, per, chunks, z, scale, bound);
}

}  // namespace eta

extern "C" int eta_score_dual(const eta_cache_desc* desc, const eta_params* params, const void* q,
                              const int32_t* seq_lens, const void* musig, const float* mnorm, float* bound,
                              void* stream) {
    int rc = eta::validate_desc(desc);
    if (rc != ETA_OK) return rc;
    if (!params || !q || !seq_lens || !musig || !mnorm || !bound) return ETA_ERR_INVALID_ARG;
    const float scale = params->scale > 0.f ? params->scale : 1.0f / sqrtf((float)desc->head_dim);
    const bool packed = (params->flags & ETA_FLAG_PACKED_SIGMA) != 0;
    auto qp = static_cast<const __nv_bfloat16*>(q);
    auto mp = static_cast<const unsigned char*>(musig);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // Few bounds (counted by capacity), us with warps / with tiles: 256 2.9 / 4.0, 1024 2.9 / 4.0, 4096 3.7 / 3.9, 8192 5.7 / 3.9, 16384
    // 8.8 / 4.0 (d = 128; 64 alike, but 4.2 to 5.0 with tiles)
    const int64_t warps = (int64_t)desc->batch * desc->n_q_heads * desc->nb_cap;
    if (warps <= 4096 || ((reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(musig)) & 15)) {
        return eta::launch_pdl("eta_score_dual", eta::score_dual_warp_kernel, dim3((unsigned)((warps + 3) / 4)), dim3(128), 0, st, qp, mp,
                               mnorm, seq_lens, (int)desc->batch, (int)desc->n_q_heads, (int)desc->n_kv_heads, (int)desc->head_dim,
                               (int)desc->block_size, (int)desc->t_cap, (int)desc->nb_cap, params->z, scale, packed ? 1 : 0, bound);
    }
    const int D = desc->head_dim, G = desc->n_q_heads / desc->n_kv_heads;
#define ETA_CASE(DD, GG) if (D == DD && G == GG) return packed \
        ? eta::launch_score_t<DD, GG, true>(desc, qp, mp, mnorm, seq_lens, params->z, scale, bound, st) \
        : eta::launch_score_t<DD, GG, false>(desc, qp, mp, mnorm, seq_lens, params->z, scale, bound, st);
    ETA_CASE(128, 1) ETA_CASE(128, 2) ETA_CASE(128, 4) ETA_CASE(128, 8)
    ETA_CASE(64, 1) ETA_CASE(64, 2) ETA_CASE(64, 4) ETA_CASE(64, 8)
#undef ETA_CASE
    return ETA_ERR_UNSUPPORTED;
}
