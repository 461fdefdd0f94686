// Streaming stage of eta_decode: SiLU-gated attention over the surviving blocks
// (Algorithm 3, attention lines and tail phase; Eq. mult_attn at inference), the
// GQA-grouped execution of the fused-kernel appendix, and the associative
// (m, l, O) merge of its "two-stage reduction".
//
// decode_kernel is persistent, one CTA per SM.  Work is the flattened sequence
// of "units": for each (sequence, KV head) row its surviving blocks (the
// screening kernel's per-segment lists), then its tail.
// Every CTA finds its place in that sequence from the per-segment counts (a
// thread per 16 segments and one round trip to memory for up to 4096 of them)
// and takes an equal, contiguous share of its COST (units, plus a fixed charge for
// every row boundary inside the share: stream-K), so the load is balanced
// whatever the per-head survivor counts are; a share may cross rows, and a row
// may be split over CTAs; each (CTA, row) piece produces one partial (m, l, O)
// per query head and consumer group.
//
// Inside a CTA one producer warp walks the survivor lists and issues tiled TMA
// copies (5-D tensor maps, 128-byte swizzle) of K and V tiles into a ring of
// shared-memory stages; three consumer groups of four warps take the fills in
// rotation, each warp a quarter of a tile's tokens.  The G query heads of the
// group are packed on the M side of mma.m16n8k16 (bf16 in, fp32 out), tokens on
// N, so each K/V byte is read once from HBM and once from shared memory for all
// heads.  The head_dim and token orders fed to the MMAs are permuted (a dot
// product does not care) so that every shared-memory read is a conflict-free
// 16-byte load of the swizzled tile.  Softmax statistics and accumulators are
// fp32; P is fed to the second MMA as a bf16 high part plus a bf16 residual, so
// the product keeps fp32-level accuracy.  Every wait is bounded.
//
// merge_kernel folds the partials of a (row, head) in a fixed order: a CTA per
// (row, head, slice of head_dim).
#include <cuda.h>

#include "eta_attend.cuh"
#include "eta_step.h"
#include "eta_timeline.h"

namespace eta {

struct DecodeArgs {
    const __nv_bfloat16* q;
    const int32_t* seq_lens;
    const float* tau_eff;
    const int32_t* seg_list;
    const uint8_t* seg_cnt;
    int32_t* stats;
    int2* row_span;      // [rows] first streaming CTA that holds units of the row, number of such CTAs
    float2* part_ml;
    float* part_o;
    uint32_t* status;
    float beta, scale;
    int Hq, Hkv, G, b, t_cap, nb_cap, nseg, rows;
    int gpr, n_gran;     // granules (16 segments) of a row, of all rows
    int n_chunks, super; // chunks of 32 lanes x 8 granules; chunks whose sums share an entry in shared memory
    int ungate_last;     // the newest token of every sequence keeps its raw logit (ETA_FLAG_UNGATE_LAST)
    const int32_t* block_table;   // paged cache: [batch, table_stride] page of every block of tokens; null: contiguous
    int table_stride;
    int read_once;       // K and V leave the L2 first
    FastDiv div_gpr, div_hkv, div_grid;
    unsigned long long* timeline;
};

constexpr uint32_t UF_END = 1u;
// Tiles a row boundary inside a CTA's range is worth (flush of the partials, query reload, a pipeline that runs dry
// while a group flushes).  Measured: 3 left the CTAs with several pieces last by 8 us on the mixed-length
// configuration (128 rows); 6, 8, 10 and 14 are within noise of each other on every configuration.  Where that would
// leave SMs without work (a CTA needs more cost units than a row's padding) a boundary counts as one tile: a problem of
// 50 blocks then runs on 24 CTAs of two tiles instead of 6 of ten.
constexpr int PIECE_COST = 8, PIECE_COST_SMALL = 1;
constexpr int64_t LARGE_CACHE_BYTES = 256ll << 20, PREFETCH_BYTES = 32ll << 20;       // see decode_impl
constexpr int LGRAN = 8;               // granules per lane of a chunk
constexpr int CHUNK = 32 * LGRAN;      // granules of a chunk: what a warp reads in one round trip
constexpr int MAX_SUPER = 512;         // sums over `super` chunks each, kept in shared memory when there is more than one chunk
constexpr int SPAN_ROWS = 64;          // rows a CTA publishes at a time

// sum of the 16 survivor counts of a granule
__device__ __forceinline__ int granule_sum(const uint4& v) {
    return (int)__dp4a(v.x, 0x01010101u, __dp4a(v.y, 0x01010101u, __dp4a(v.z, 0x01010101u, __dp4a(v.w, 0x01010101u, 0u))));
}

template <int D, int TS, int NSTAGE, int NGROUPS>
struct DecodeSmem {
    static constexpr int HALVES = D / 64;
    static constexpr int TILE_BYTES = TS * 128;                 // one 64-column half tile
    static constexpr int STAGE_BYTES = 2 * HALVES * TILE_BYTES; // K halves then V halves
    static constexpr int BAR_OFF = NSTAGE * STAGE_BYTES;        // full[NSTAGE], empty[NSTAGE], flush[NGROUPS], layout
    static constexpr int DESC_OFF = (BAR_OFF + 8 * (2 * NSTAGE + NGROUPS + 1) + 15) / 16 * 16;
    static constexpr int WIN_OFF = DESC_OFF + 16 * NSTAGE;      // uint4 [32]: the producer's window of granules
    static constexpr int GRAN_OFF = WIN_OFF + 16 * 32;          // uint4 [CHUNK]: all granules (one chunk), else int2 [MAX_SUPER]: sums
    static constexpr int BEFORE_OFF = GRAN_OFF + 16 * CHUNK;    // int2 [CHUNK + 1] (+ pad): units and live rows before a granule (one chunk)
    static constexpr int SPAN_OFF = BEFORE_OFF + 8 * (CHUNK + 2);      // int2 [SPAN_ROWS + 1] (+ pad): units and live rows before a row
    static constexpr int INFO_OFF = SPAN_OFF + 8 * (SPAN_ROWS + 2);     // uint8 per row: bit 0 has tokens, bit 1 has a tail
    static constexpr int ML_OFF = INFO_OFF + MAX_ROWS;          // float m[NGROUPS][4][8], l[NGROUPS][4][8]
    static_assert(16 * CHUNK >= 8 * MAX_SUPER, "sums of the super-chunks share the granules' place");
    static constexpr int MO_OFF = ML_OFF + 4 * 2 * NGROUPS * WARPS_PER_GROUP * 8;
    // heads whose accumulators a flush parks at a time: eight heads of 128 columns would cost the ring a stage
    static constexpr int FLUSH_HEADS = 512 / D;
    static size_t bytes(int G) { return 1024 + MO_OFF + sizeof(float) * NGROUPS * WARPS_PER_GROUP * (G < FLUSH_HEADS ? G : FLUSH_HEADS) * D; }
};

// The streaming kernel.  Warp roles: NGROUPS consumer groups of four warps, then one producer warp.  Group k
// consumes the stage fills k, k + NGROUPS, ...; with two or three groups every scheduler holds several warps in
// different phases of a tile, which hides the fixed latencies of the MMA / shuffle / exp chains.  Each group
// keeps its own running (m, l, O) and writes its own partial per (CTA, row) piece.
template <int D, int TS, int NSTAGE, int NGROUPS>
__global__ void __launch_bounds__(32 * (WARPS_PER_GROUP * NGROUPS + 1), 1)
decode_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const DecodeArgs a) {
    using L = DecodeSmem<D, TS, NSTAGE, NGROUPS>;
    constexpr int HALVES = L::HALVES;
    constexpr int PRODUCER_WARP = WARPS_PER_GROUP * NGROUPS;

    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + L::BAR_OFF);
    uint64_t* empty = full + NSTAGE;
    uint64_t* flushbar = empty + NSTAGE;
    uint64_t* laybar = flushbar + NGROUPS;
    int4* desc = reinterpret_cast<int4*>(smem + L::DESC_OFF);
    uint8_t* rowinfo = smem + L::INFO_OFF;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned long long* const tl = ETA_TL(a.timeline ? a.timeline + (size_t)(TL_DECODE + blockIdx.x) * 8 : nullptr);
    unsigned long long* const tl2 = ETA_TL(a.timeline ? a.timeline + (size_t)(TL_DECODE2 + blockIdx.x) * 8 : nullptr);
    if (tl && tid == 0) tl[0] = globaltimer_ns();
    // A stage serves the same group in every round: a parity wait only tells the current phase of a barrier from the one
    // before it, and a group that ran ahead on a stage of another group could be told "done" too early.
    static_assert(NSTAGE % NGROUPS == 0, "stages must be a multiple of the consumer groups");
    if (tid == 0) {
        for (int s = 0; s < NSTAGE; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], WARPS_PER_GROUP); }
        for (int k = 0; k < NGROUPS; ++k) mbar_init(&flushbar[k], 32 * WARPS_PER_GROUP);
        mbar_init(laybar, 1);
        fence_barrier_init();
        prefetch_tmap(&tmK);
        prefetch_tmap(&tmV);
    }
    // what is known before the predecessor kernel is through: which rows have tokens and which a tail (a caller input)
    constexpr int NWARPS = WARPS_PER_GROUP * NGROUPS + 1;
    constexpr int NTHREADS = 32 * NWARPS;
    __shared__ int s_row0;                // row of the CTA's first unit; -1: no work
    for (int rr = tid; rr < a.rows; rr += NTHREADS) {
        int T = __ldg(a.seq_lens + a.div_hkv.div(rr));
        T = T < 0 ? 0 : (T > a.t_cap ? a.t_cap : T);
        rowinfo[rr] = (uint8_t)((T > 0 ? 1 : 0) | ((T & (a.b - 1)) ? 2 : 0));
    }
    __syncthreads();

    // ---- layout.  The flattened sequence of units is cut up by granules, 16 segments of a row each (the last one of a row
    // also holds its tail unit).  Up to 256 granules: a thread takes one, a scan over the threads gives it the units before it, and
    // the two threads whose granules hold the ends of the CTA's share say where it starts and ends.  More: lane l of a warp takes
    // eight consecutive granules of a chunk.  A row that starts inside a CTA's share costs that CTA a flush of its partials and
    // a query reload, worth `pc` tiles: row r spans the cost interval [units before + pc * live rows before, + pc (if it
    // has units) + its units).  Every live row has at least one unit (a tail, or what top-1 rescue leaves).
    // Bound by the number of instructions in a row, some four cycles each whatever they are: with one warp, eight granules to a
    // lane, it was 6300 to 8300 cycles from the wait to the first copy, with a thread per granule 4800 to 5300 (128K x 4 59.9 -> 58.4 us a
    // step, 32K x 8 50.8 -> 49.4, 512K 43.7 -> 42.7, 64K x 32 89.9 -> 88.3).
    uint32_t headm = 0, tailm = 0;        // bit m: the lane's granule m of the chunk is the first of a live row / ends a row with a tail
    auto lane_flags = [&](int ch) {
        headm = tailm = 0;
#pragma unroll 1
        for (int m = 0; m < LGRAN; ++m) {
            const int q = ch * CHUNK + lane * LGRAN + m;
            if (q >= a.n_gran) break;
            int r, pos;
            a.div_gpr.divmod(q, r, pos);
            const int info = rowinfo[r];
            headm |= (uint32_t)(pos == 0 && (info & 1)) << m;
            tailm |= (uint32_t)(pos == a.gpr - 1 && (info & 2)) << m;
        }
    };
    int us[LGRAN];                        // units of the lane's granules
    int lane_u = 0, lane_z = 0;           // units / live rows in the lane's granules
    const uint4* const gran = reinterpret_cast<const uint4*>(a.seg_cnt);
    uint4* const gran_s = reinterpret_cast<uint4*>(smem + L::GRAN_OFF);
    int2* const super_s = reinterpret_cast<int2*>(smem + L::GRAN_OFF);
    auto load_chunk = [&](int ch) {
        uint4 v[LGRAN];
#pragma unroll
        for (int m = 0; m < LGRAN; ++m) {
            const int q = ch * CHUNK + lane * LGRAN + m;
            v[m] = make_uint4(0, 0, 0, 0);
            if (q < a.n_gran) v[m] = __ldcg(gran + q);
        }
        lane_u = 0;
#pragma unroll
        for (int m = 0; m < LGRAN; ++m) {
            us[m] = granule_sum(v[m]) + (int)((tailm >> m) & 1);
            lane_u += us[m];
        }
        lane_z = __popc(headm);
    };
    int pre_u = 0, pre_z = 0, tot_u = 0, tot_z = 0;       // before the lane within the chunk; of the chunk
    auto scan_chunk = [&]() {
        uint32_t x = (uint32_t)lane_u | ((uint32_t)lane_z << 20);          // a chunk: < 2^19 units, <= 256 rows
#pragma unroll
        for (int sft = 1; sft < 32; sft <<= 1) {
            const uint32_t o = __shfl_up_sync(0xffffffffu, x, sft);
            if (lane >= sft) x += o;
        }
        const uint32_t t = __shfl_sync(0xffffffffu, x, 31);
        tot_u = (int)(t & 0xfffffu); tot_z = (int)(t >> 20);
        pre_u = (int)(x & 0xfffffu) - lane_u; pre_z = (int)(x >> 20) - lane_z;
    };
    const bool one_chunk = a.n_chunks == 1;
    const bool lays_out = warp == PRODUCER_WARP || warp == 0;              // the producer, and the warp that publishes
    // one chunk: a granule per thread
    static_assert(NTHREADS > CHUNK, "a thread per granule, and one for the end");
    int2* const before_s = reinterpret_cast<int2*>(smem + L::BEFORE_OFF);
    __shared__ uint32_t s_warp[CHUNK / 32];
    __shared__ int s_unit[2], s_gran;
    uint32_t my_head = 0, my_tail = 0;
    if (one_chunk && tid < a.n_gran) {
        int r, pos;
        a.div_gpr.divmod(tid, r, pos);
        const int info = rowinfo[r];
        my_head = pos == 0 && (info & 1);
        my_tail = pos == a.gpr - 1 && (info & 2);
    }
    pdl_wait();          // the screening kernel's lists and counts are complete from here on
    if (tl && tid == 0) tl[7] = globaltimer_ns();
    const unsigned long long clk0 = ETA_TL(reinterpret_cast<unsigned long long*>(1)) ? (unsigned long long)clock64() : 0ull;

    const int n_super = (a.n_chunks + a.super - 1) / a.super;
    if (!one_chunk) {
        for (int sc = warp; sc < n_super; sc += NWARPS) {
            int su = 0, sz = 0;
            for (int ch = sc * a.super; ch < min(a.n_chunks, (sc + 1) * a.super); ++ch) {
                lane_flags(ch);
                load_chunk(ch);
                su += lane_u; sz += lane_z;
            }
            su = __reduce_add_sync(0xffffffffu, su);
            sz = __reduce_add_sync(0xffffffffu, sz);
            if (lane == 0) super_s[sc] = make_int2(su, sz);
        }
        __syncthreads();
    }
    int U = 0, Z = 0;
    uint32_t my_n = 0, my_before = 0;        // one chunk: units (and, from bit 20, live rows) of the thread's granule, before it
    if (one_chunk) {
        const int n_warps = (a.n_gran + 31) / 32;
        uint32_t x = 0;
        if (warp < n_warps) {
            if (tid < a.n_gran) {
                const uint4 v = __ldcg(gran + tid);
                gran_s[tid] = v;
                my_n = (uint32_t)granule_sum(v) + my_tail;
            }
            x = my_n | (my_head << 20);          // all granules: < 2^19 units, <= 256 rows
#pragma unroll
            for (int sft = 1; sft < 32; sft <<= 1) {
                const uint32_t o = __shfl_up_sync(0xffffffffu, x, sft);
                if (lane >= sft) x += o;
            }
            if (lane == 31) s_warp[warp] = x;
            my_before = x - (my_n | (my_head << 20));
        }
        __syncthreads();
        uint32_t all = 0;
        for (int w = 0; w < n_warps; ++w) {
            const uint32_t t = s_warp[w];
            all += t;
            if (w < warp) my_before += t;
        }
        U = (int)(all & 0xfffffu); Z = (int)(all >> 20);
    } else if (lays_out) {
        for (int sc = lane; sc < n_super; sc += 32) { U += super_s[sc].x; Z += super_s[sc].y; }
        U = __reduce_add_sync(0xffffffffu, U);
        Z = __reduce_add_sync(0xffffffffu, Z);
    }
    // More cost units per CTA than a row's padding (fewer CTAs take part in a tiny problem): then no CTA's range lies
    // inside a padding; the CTAs that meet a row are exactly those between two ends that follow from the row's cost
    // interval in closed form (the merge kernel finds its candidates that way).
    const uint32_t grid = gridDim.x;
    const int pc = (uint32_t)U + (uint32_t)(PIECE_COST * Z) >= (PIECE_COST + 1) * grid ? PIECE_COST : PIECE_COST_SMALL;
    const uint32_t C = (uint32_t)U + (uint32_t)pc * (uint32_t)Z;
    const uint32_t P = min(grid, max(1u, C / (PIECE_COST_SMALL + 1)));
    // the CTA's share of the cost, [x0, x1)
    uint32_t x0 = C, x1 = C;
    if (blockIdx.x < P) {
        if (P == grid) {
            const uint32_t cq = (uint32_t)a.div_grid.div((int)C), cr = C - cq * grid;        // floor(c C / P): c cr < 2^16
            x0 = blockIdx.x * cq + (uint32_t)a.div_grid.div((int)(blockIdx.x * cr));
            x1 = (blockIdx.x + 1) * cq + (uint32_t)a.div_grid.div((int)((blockIdx.x + 1) * cr));
        } else {
            const uint32_t cq = C / P, cr = C - cq * P;
            x0 = blockIdx.x * cq + blockIdx.x * cr / P;
            x1 = (blockIdx.x + 1) * cq + (blockIdx.x + 1) * cr / P;
        }
    }
    if (one_chunk) {
        // whose granule holds an end of the share finds the unit it stands for (a position in a row's padding: the row's first)
        if (tid <= a.n_gran) {
            const int u = tid < a.n_gran ? (int)(my_before & 0xfffffu) : U, z = tid < a.n_gran ? (int)(my_before >> 20) : Z;
            before_s[tid] = make_int2(u, z);
            const uint32_t c = (uint32_t)u + (uint32_t)pc * (uint32_t)z, pad = my_head ? (uint32_t)pc : 0u;
            if (tid < a.n_gran) {
                if (x0 >= c && x0 < c + pad + my_n) { s_unit[0] = u + (x0 > c + pad ? (int)(x0 - c - pad) : 0); s_gran = tid; }
                if (x1 >= c && x1 < c + pad + my_n) s_unit[1] = u + (x1 > c + pad ? (int)(x1 - c - pad) : 0);
            }
        }
        __syncthreads();
    }
    if (warp == 0) {
        // ---- for the merge kernel and the caller, shared out over the CTAs (all of them find the same layout): the
        // streaming CTAs that hold units of each row, and the number of blocks fetched per row.  CTA c has the cost
        // interval [floor(c C / P), floor((c + 1) C / P)), row rr the interval [cs, ce) whose first pc units are
        // padding, and c holds units of the row exactly when its interval starts before ce and ends after the padding.
        int2* const span = reinterpret_cast<int2*>(smem + L::SPAN_OFF);
        const int r_end = (int)(((int64_t)(blockIdx.x + 1) * a.rows) / grid);
        for (int r_lo = (int)(((int64_t)blockIdx.x * a.rows) / grid); r_lo < r_end; r_lo += SPAN_ROWS) {
            const int r_hi = min(r_end, r_lo + SPAN_ROWS);
            if (lane == 0) span[r_hi - r_lo] = make_int2(U, Z);            // for the last row of all
            __syncwarp();
            auto store_rows = [&](int ch, int bu, int bz) {
                int u = bu + pre_u, z = bz + pre_z;
#pragma unroll
                for (int m = 0; m < LGRAN; ++m) {
                    const int q = ch * CHUNK + lane * LGRAN + m;
                    if (q < a.n_gran) {
                        int r, pos;
                        a.div_gpr.divmod(q, r, pos);
                        if (pos == 0 && r >= r_lo && r <= r_hi) span[r - r_lo] = make_int2(u, z);
                        u += us[m]; z += (int)((headm >> m) & 1);
                    }
                }
            };
            if (!one_chunk) {
                const int ch0 = (r_lo * a.gpr) / CHUNK, ch1 = min(a.n_chunks - 1, (r_hi * a.gpr) / CHUNK);
                int bu = 0, bz = 0, ch = 0;
                for (; ch + a.super <= ch0; ch += a.super) { bu += super_s[ch / a.super].x; bz += super_s[ch / a.super].y; }
                for (; ch <= ch1; ++ch) {
                    lane_flags(ch);
                    load_chunk(ch);
                    scan_chunk();
                    if (ch >= ch0) store_rows(ch, bu, bz);
                    bu += tot_u; bz += tot_z;
                }
            }
            __syncwarp();
            for (int k = lane; k < r_hi - r_lo; k += 32) {
                const int rr = r_lo + k;
                const int2 from = one_chunk ? before_s[rr * a.gpr] : span[k], to = one_chunk ? before_s[(rr + 1) * a.gpr] : span[k + 1];
                const int units = to.x - from.x;
                int c_lo = 0, n_span = 0;
                if (units > 0) {
                    const int64_t cs = (int64_t)from.x + (int64_t)pc * from.y, ce = cs + pc + units;
                    const int c_hi = (int)((ce * P - 1) / C);
                    c_lo = (int)(((cs + pc + 1) * P + C - 1) / C) - 1;
                    n_span = c_hi - c_lo + 1;
                }
                a.row_span[rr] = make_int2(c_lo, n_span);
                if (a.stats) a.stats[rr] = units - ((rowinfo[rr] >> 1) & 1);
            }
            __syncwarp();
        }
    }
    if (tl && tid == 0) tl[1] = globaltimer_ns();

    if (warp == PRODUCER_WARP) {
        // ------------------------------------------------------------ producer
        // cost position x < C -> unit, a granule at or before the one that holds it, units before that granule.  A position in a
        // row's padding stands for the row's first unit.
        auto locate = [&](uint32_t x, int& unit, int& gq, int& gu) {
            int bu = 0, bz = 0, ch = 0;
            for (int sc = 0; sc + 1 < n_super; ++sc) {
                const int2 t = super_s[sc];
                if (x < (uint32_t)(bu + t.x) + (uint32_t)pc * (uint32_t)(bz + t.y)) break;
                bu += t.x; bz += t.y; ch += a.super;
            }
            while (true) {
                lane_flags(ch);
                load_chunk(ch);
                scan_chunk();
                if (ch + 1 >= a.n_chunks || x < (uint32_t)(bu + tot_u) + (uint32_t)pc * (uint32_t)(bz + tot_z)) break;
                bu += tot_u; bz += tot_z; ++ch;
            }
            int u = bu + pre_u, fu = 0, fq = 0, fgu = 0;
            uint32_t c = (uint32_t)u + (uint32_t)pc * (uint32_t)(bz + pre_z);
            const int src = 31 - __clz(__ballot_sync(0xffffffffu, c <= x));      // the last lane that starts at or before x
            bool found = false;
#pragma unroll
            for (int m = 0; m < LGRAN; ++m) {
                const uint32_t pad = ((headm >> m) & 1) ? (uint32_t)pc : 0u;
                if (!found && x < c + pad + (uint32_t)us[m]) {
                    found = true;
                    fu = u + (x > c + pad ? (int)(x - c - pad) : 0);
                    fq = ch * CHUNK + lane * LGRAN + m; fgu = u;
                }
                c += pad + (uint32_t)us[m]; u += us[m];
            }
            unit = __shfl_sync(0xffffffffu, fu, src);
            gq = __shfl_sync(0xffffffffu, fq, src);
            gu = __shfl_sync(0xffffffffu, fgu, src);
        };
        int u0 = U, u1 = U, wq = 0, wu = 0;          // the CTA's units; the window's first granule, units before it
        if (x0 < C) {
            if (one_chunk) {
                u0 = s_unit[0];
                wq = s_gran;
                if (x1 < C) u1 = s_unit[1];
            } else {
                int nq, nu;
                if (x1 < C) locate(x1, u1, nq, nu);
                locate(x0, u0, wq, wu);
            }
        }
        if (tl2 && lane == 0) tl2[3] = (unsigned long long)clock64() - clk0;
        const int tpu_shift = a.b > TS ? 1 : 0, tpu = 1 << tpu_shift;          // tiles of a full unit: two for 128 tokens, else one
        // Window: granule wq + l in lane l, its counts in shared memory, the units before it in pre_w.
        uint4* const win = reinterpret_cast<uint4*>(smem + L::WIN_OFF);
        int pre_w = 0, wend = 0;
        auto load_window = [&]() {
            if (one_chunk) {
                pre_w = before_s[min(wq + lane, a.n_gran)].x;
                wend = before_s[min(wq + 32, a.n_gran)].x;
                return;
            }
            __syncwarp();
            const int q = wq + lane;
            uint4 v = make_uint4(0, 0, 0, 0);
            int tail = 0;
            if (q < a.n_gran) {
                v = __ldcg(gran + q);
                int r, pos;
                a.div_gpr.divmod(q, r, pos);
                tail = (pos == a.gpr - 1) ? (rowinfo[r] >> 1) & 1 : 0;
            }
            win[lane] = v;
            const int n = granule_sum(v) + tail;
            int incl = n;
#pragma unroll
            for (int sft = 1; sft < 32; sft <<= 1) {
                const int o = __shfl_up_sync(0xffffffffu, incl, sft);
                if (lane >= sft) incl += o;
            }
            pre_w = wu + incl - n;
            wend = wu + __shfl_sync(0xffffffffu, incl, 31);
            __syncwarp();
        };
        auto search = [&](int uu) {          // the last lane whose granule starts at or before unit uu
            int lo = 0;
#pragma unroll
            for (int step = 16; step >= 1; step >>= 1) {
                const int v = __shfl_sync(0xffffffffu, pre_w, lo + step);
                if (v <= uu) lo += step;
            }
            return lo;
        };
        // make the window hold the granule of unit ub; -> number of units of the batch starting at ub
        auto batch_size = [&](int ub) {
            while (true) {
                const int want = min((32 >> tpu_shift), u1 - ub);
                if (wq + 32 >= a.n_gran || wend >= ub + want) return want;
                if (wend <= ub) { wq += 32; wu = wend; load_window(); continue; }
                const int k0 = search(ub);
                if (k0 == 0) return min(want, wend - ub);
                wu = __shfl_sync(0xffffffffu, pre_w, k0);
                wq += k0;
                load_window();
            }
        };
        // per-lane description of unit ub + (lane >> tpu_shift) (row < 0: no such unit in this batch)
        auto fetch = [&](int ub, int nb, int& row, int& ent, int& nrows, int& page) {
            const int uu = ub + min((lane >> tpu_shift), nb - 1);
            const int k = search(uu);
            int off = uu - __shfl_sync(0xffffffffu, pre_w, k);
            row = -1; ent = 0; nrows = 0; page = 0;
            if ((lane >> tpu_shift) < nb) {
                const uint4 v = one_chunk ? gran_s[wq + k] : win[k];
                int r, pos;
                a.div_gpr.divmod(wq + k, r, pos);
                // the segment whose units include number `off` of the granule: first the word, then the byte
                const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
                int n4[4], sg = 0, first = 0;
#pragma unroll
                for (int j = 0; j < 4; ++j) n4[j] = (int)__dp4a(w4[j], 0x01010101u, 0u);
                uint32_t w = w4[0];
                int upto = n4[0];
#pragma unroll
                for (int j = 1; j < 4; ++j) {
                    if (off >= upto) { sg = 4 * j; w = w4[j]; first = upto; }
                    upto += n4[j];
                }
                const bool in = off < upto;
                off -= first;
                upto = 0;
                first = 0;
                int sub = 0;
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    upto += (int)((w >> (8 * j)) & 0xffu);
                    if (off >= upto) { sub = j + 1; first = upto; }
                }
                off -= first;
                sg += sub;
                row = r;
                int T = 0;
                if (!in || a.ungate_last) {
                    T = __ldg(a.seq_lens + a.div_hkv.div(r));
                    T = T < 0 ? 0 : (T > a.t_cap ? a.t_cap : T);
                }
                if (!in) {
                    const int NB = min(T / a.b, a.nb_cap);
                    ent = NB | (0xff << 24);           // the tail: every head attends it
                    nrows = T - NB * a.b;
                    if (a.ungate_last) nrows |= 0x10000;      // its last token is the sequence's newest
                } else {
                    ent = __ldcg(a.seg_list + ((int64_t)r * a.nseg + pos * GRANULE + sg) * LSTRIDE + off);
                    nrows = a.b;
                    if (a.ungate_last && ((ent & 0xffffff) + 1) * a.b == T) nrows |= 0x10000;   // the block the newest token closes
                }
                // paged cache: the page that holds the unit's block of tokens (one more dependent load per batch,
                // hidden like the list fetch behind the tiles already on their way)
                if (a.block_table)
                    page = __ldcg(a.block_table + (int64_t)a.div_hkv.div(r) * a.table_stride + (ent & 0xffffff));
            }
        };
        if (u0 >= u1) {
            if (lane == 0) { s_row0 = -1; mbar_arrive(laybar); }
            return;
        }
        load_window();
        int u = u0;
        int nb = batch_size(u);
        if (tl2 && lane == 0) tl2[6] = (unsigned long long)clock64() - clk0;
        int c_row, c_ent, c_nrows, c_page;
        fetch(u, nb, c_row, c_ent, c_nrows, c_page);
        if (lane == 0) { s_row0 = c_row; mbar_arrive(laybar); }
        if (tl2 && lane == 0) tl2[7] = (unsigned long long)clock64() - clk0 + (c_ent & 0);
        // A lane per tile: lane TPU j + sub is part `sub` of the batch's unit j.  Lanes whose stage is free issue their copies
        // together, so a tile costs the warp a fraction of a pass through this loop; with one tile per pass (its
        // description broadcast by shuffles) the producer took 550 ns a tile, which held every tile of less than 32 KB (64
        // columns or 32 tokens) below half of the copy rate.
        const int usub = (lane & (tpu - 1));
        const uint64_t once = l2_policy(a.read_once != 0);
        uint32_t fill = 0;
        int piece = -1, prev_row = -1;
        uint32_t piece_f0 = 0;
        bool ok = true;

        // groups that receive no tile of a piece never write its partial: mark those slots "absent" for the merge
        auto close_piece = [&](uint32_t end) {
            if (prev_row < 0) return;
            const uint32_t n = end - piece_f0;
            for (uint32_t k = n; k < (uint32_t)NGROUPS; ++k) {
                const int grp = (int)((piece_f0 + k) % NGROUPS);
                const int64_t slot = ((int64_t)blockIdx.x + prev_row) * NGROUPS + grp;
                if (lane < a.G) a.part_ml[slot * a.G + lane] = make_float2(-INFINITY, 0.f);
            }
        };
        while (u < u1 && ok) {
            const int un = u + nb;
            const int nrows = c_nrows & 0xffff;
            const bool valid = c_row >= 0 && usub * TS < nrows;
            const unsigned vmask = __ballot_sync(0xffffffffu, valid);
            const uint32_t my_fill = fill + (uint32_t)__popc(vmask & ((1u << lane) - 1u));
            // pieces: a new one starts where the row changes
            const int left = __shfl_up_sync(0xffffffffu, c_row, 1);
            unsigned starts = __ballot_sync(0xffffffffu, c_row >= 0 && c_row != (lane == 0 ? prev_row : left));
            const int my_piece = piece + __popc(starts & (0xffffffffu >> (31 - lane)));
            piece += __popc(starts);
            const int stage = (int)(my_fill % NSTAGE);
            const uint32_t parity = ((my_fill / NSTAGE) & 1) ^ 1;
            bool done = !valid;
            int my_i, my_hk;
            a.div_hkv.divmod(max(c_row, 0), my_i, my_hk);
            // The outermost coordinate is the sequence (contiguous cache: token offset in the sequence) or the page (paged
            // cache: token offset in the page)
            const int my_y = a.block_table ? usub * TS : (c_ent & 0xffffff) * a.b + usub * TS;
            const int my_w = a.block_table ? c_page : my_i;
            unsigned char* const my_smem = smem + stage * L::STAGE_BYTES;
            const int nvalid = min(TS, nrows - usub * TS);
            // bits 8..15: row of the tile whose token stays ungated, 0xff: none
            const int urow = ((c_nrows >> 16) != 0 && (usub + 1) * TS >= nrows) ? nvalid - 1 : 0xff;
            const int4 my_desc = make_int4(c_row, my_piece << 1, ((c_ent >> 24) & 0xff) | (urow << 8), nvalid);
            // One pass: lanes whose stage is free issue.  A lane looks at its stage's barrier only when the tile that used the
            // stage before it is on its way (parity tells two rounds apart, not three), that is, within NSTAGE tiles of
            // the first one that is not.
            auto issue_pass = [&]() {
                const unsigned open = __ballot_sync(0xffffffffu, !done);
                const int first = __ffs(open) - 1;
                const uint32_t f_first = __shfl_sync(0xffffffffu, my_fill, first < 0 ? 0 : first);
                const bool ready = !done && my_fill < f_first + NSTAGE && mbar_test(&empty[stage], parity);
                if (ready) {
                    done = true;
                    desc[stage] = my_desc;
                    mbar_arrive_expect_tx(&full[stage], L::STAGE_BYTES);
                }
                // one copy per tensor: 64 columns x TS tokens x HALVES half tiles, each half swizzled.  Tile after tile, so that
                // the first is complete as early as can be.
                for (unsigned rm = __ballot_sync(0xffffffffu, ready); rm; rm &= rm - 1) {
                    if (lane == __ffs(rm) - 1) {
                        tma_load_5d(my_smem, &tmK, 0, my_y, 0, my_hk, my_w, &full[stage], once);
                        tma_load_5d(my_smem + HALVES * L::TILE_BYTES, &tmV, 0, my_y, 0, my_hk, my_w, &full[stage], once);
                    }
                }
                return __any_sync(0xffffffffu, !done) != 0;
            };
            if (tl2 && lane == 0 && fill == 0) tl2[1] = (unsigned long long)clock64() - clk0;
            bool more = issue_pass();
            for (; starts; starts &= starts - 1) {
                const int sl = __ffs(starts) - 1;
                const uint32_t f = __shfl_sync(0xffffffffu, my_fill, sl);
                close_piece(f);
                prev_row = __shfl_sync(0xffffffffu, c_row, sl);
                piece_f0 = f;
            }
            // the next batch is fetched once what fits of this one is on its way
            int nbn = 0, n_row = -1, n_ent = 0, n_nrows = 0, n_page = 0;
            if (un < u1) {
                nbn = batch_size(un);
                fetch(un, nbn, n_row, n_ent, n_nrows, n_page);
            }
            for (uint32_t it = 0; more; ++it) {
                more = issue_pass();
                if (it >= WAIT_LIMIT) { ok = false; break; }
                if (more && it >= 2) __nanosleep(20);
            }
            if (!ok) {                    // give up: time for this batch's copies to land (those before it are waited for below)
                if (valid && done) mbar_wait(&full[stage], parity ^ 1);
                __syncwarp();
                break;
            }
            fill += (uint32_t)__popc(vmask);
            u = un;
            nb = nbn; c_row = n_row; c_ent = n_ent; c_nrows = n_nrows; c_page = n_page;
        }
        close_piece(fill);
        pdl_trigger();       // everything is issued: the merge kernel may start to set up
        // one end marker per group (no data): the next NGROUPS fills reach every group exactly once
        for (int k = 0; k < NGROUPS && ok; ++k) {
            const int stage = fill % NSTAGE;
            if (lane == 0) {
                if (!mbar_wait(&empty[stage], ((fill / NSTAGE) & 1) ^ 1)) {
                    ok = false;
                } else {
                    desc[stage] = make_int4(0, (int)UF_END, 0, 0);
                    mbar_arrive(&full[stage]);
                }
            }
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
            ++fill;
        }
        if (!ok) {
            // give up: report, then let copies already issued land before the CTA's shared memory is released
            if (lane == 0) {
                if (a.status) atomicOr(a.status, ETA_DEV_TIMEOUT);
                const uint32_t first_fill = fill > NSTAGE ? fill - NSTAGE : 0;
                for (uint32_t f = first_fill; f < fill; ++f) mbar_wait(&full[f % NSTAGE], (f / NSTAGE) & 1);
            }
        }
        return;
    }

    // ---------------------------------------------------------------- consumers
    const int group = warp / WARPS_PER_GROUP, wq = warp % WARPS_PER_GROUP;
    float* sm_m = reinterpret_cast<float*>(smem + L::ML_OFF) + group * 2 * WARPS_PER_GROUP * 8;
    float* sm_l = sm_m + WARPS_PER_GROUP * 8;
    const int fheads = min(a.G, L::FLUSH_HEADS);       // heads per round of a flush
    float* sm_o = reinterpret_cast<float*>(smem + L::MO_OFF) + group * WARPS_PER_GROUP * fheads * D;
    const int gtid = tid - group * 32 * WARPS_PER_GROUP;    // thread index inside the group
    const float LOG2E = 1.4426950408889634f;
    Attend<D, TS> at(lane, wq, a.G);
    int row = -1, piece = -1, q_row = -1;
    uint32_t flush_phase = 0;
    bool ok = true;

    // query fragments and threshold of a row: head g's slice in the permuted head_dim order of the MMA
    auto load_q = [&](int r) {
        int i, hk;
        a.div_hkv.divmod(r, i, hk);
        const int h = hk * a.G + (at.head ? at.g : 0);
        at.load_q(a.q + ((int64_t)i * a.Hq + h) * D);
        at.te = at.head ? __ldcg(a.tau_eff + (int64_t)i * a.Hq + h) : 0.f;
        q_row = r;
    };
    if (!mbar_wait(laybar, 0)) {
        if (lane == 0 && a.status) atomicOr(a.status, ETA_DEV_TIMEOUT);
        return;
    }
    if (s_row0 < 0) return;
    load_q(s_row0);       // the row of the CTA's first unit: fetched while its first tiles are on their way

    for (uint32_t fill = group;; fill += NGROUPS) {
        const int stage = fill % NSTAGE;
        if (!mbar_wait(&full[stage], (fill / NSTAGE) & 1)) { ok = false; break; }
        const int4 ds = desc[stage];
        const bool end = (ds.y & (int)UF_END) != 0;
        const int new_piece = ds.y >> 1;
        if (end) pdl_trigger();
        if (tl && warp == 0 && lane == 0) {
            if (fill == 0) tl[3] = globaltimer_ns();
            if (end) tl[4] = globaltimer_ns();
        }

        // the next piece's query is requested before the finished piece is flushed: the flush does not read the
        // query registers, and its barriers and stores hide the load's latency
        if (!end && new_piece != piece && ds.x != q_row) load_q(ds.x);
        if ((end || new_piece != piece) && piece >= 0) {
            // ---- this group's part of a piece is complete: combine its four warps and store (m, l, O) per head
            float lsum = at.l_run + __shfl_xor_sync(0xffffffffu, at.l_run, 1);
            lsum += __shfl_xor_sync(0xffffffffu, lsum, 2);
            if (at.t == 0) { sm_m[wq * 8 + at.g] = at.m_run; sm_l[wq * 8 + at.g] = lsum; }
            const int64_t slot = ((int64_t)blockIdx.x + row) * NGROUPS + group;
            for (int h0 = 0; h0 < a.G && ok; h0 += fheads) {
                const int ha = 2 * at.t - h0, hb = ha + 1;         // this lane's two heads within the round
#pragma unroll
                for (int hf = 0; hf < HALVES; ++hf)
#pragma unroll
                    for (int mt = 0; mt < 4; ++mt) {
                        const int dcol = 64 * hf + 8 * at.vchunk + 2 * mt;
                        if (ha >= 0 && ha < fheads)
                            *reinterpret_cast<float2*>(sm_o + ((wq * fheads + ha) * D + dcol)) = make_float2(at.o[hf][mt][0], at.o[hf][mt][2]);
                        if (hb >= 0 && hb < fheads)
                            *reinterpret_cast<float2*>(sm_o + ((wq * fheads + hb) * D + dcol)) = make_float2(at.o[hf][mt][1], at.o[hf][mt][3]);
                    }
#ifdef ETA_TEST_SKIP_FLUSH_ARRIVE
                // test build only: one warp of the first CTA never arrives, so that the group's bounded wait runs out and
                // the give-up path (status flag, orderly exit of the whole CTA) executes
                if (!(blockIdx.x == 0 && group == 0 && wq == 1))
#endif
                mbar_arrive(&flushbar[group]);
                if (!mbar_wait(&flushbar[group], flush_phase)) { ok = false; break; }
                flush_phase ^= 1;
                for (int idx = gtid; idx < fheads * D / 4; idx += 32 * WARPS_PER_GROUP) {
                    const int hr = idx / (D / 4), dq = idx % (D / 4), hh = h0 + hr;
                    float mw[WARPS_PER_GROUP], M = -INFINITY;
#pragma unroll
                    for (int w = 0; w < WARPS_PER_GROUP; ++w) { mw[w] = sm_m[w * 8 + hh]; M = fmaxf(M, mw[w]); }
                    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
                    float lacc = 0.f;
                    if (M != -INFINITY) {
#pragma unroll
                        for (int w = 0; w < WARPS_PER_GROUP; ++w) {
                            const float sc = exp2f((mw[w] - M) * LOG2E);
                            const float4 x = *reinterpret_cast<const float4*>(sm_o + (w * fheads + hr) * D + 4 * dq);
                            acc.x = fmaf(x.x, sc, acc.x); acc.y = fmaf(x.y, sc, acc.y);
                            acc.z = fmaf(x.z, sc, acc.z); acc.w = fmaf(x.w, sc, acc.w);
                            lacc = fmaf(sm_l[w * 8 + hh], sc, lacc);
                        }
                    }
                    *reinterpret_cast<float4*>(a.part_o + (slot * a.G + hh) * D + 4 * dq) = acc;
                    if (dq == 0) a.part_ml[slot * a.G + hh] = make_float2(M, lacc);
                }
                mbar_arrive(&flushbar[group]);
                if (!mbar_wait(&flushbar[group], flush_phase)) { ok = false; break; }
                flush_phase ^= 1;
            }
            if (!ok) break;
        }
        if (end) {
            if (tl && warp == 0 && lane == 0) tl[5] = globaltimer_ns();
            break;
        }

        const int hmask = ds.z & 0xff, urow = (ds.z >> 8) & 0xff, nvalid = ds.w;
        const uint32_t kbase = smem_u32(smem + stage * L::STAGE_BYTES);

        if (new_piece != piece) {
            piece = new_piece;
            row = ds.x;
            if (row != q_row) load_q(row);
            at.reset();
        }

        // the arrive (release) orders the warp's reads of the stage before the producer's next copy into it
        at.tile(kbase, hmask, urow, nvalid, a.scale, a.beta, [&]() { if (lane == 0) mbar_arrive(&empty[stage]); });
    }
    if (!ok && lane == 0 && a.status) atomicOr(a.status, ETA_DEV_TIMEOUT);
}

// Associative merge of the pieces of one (sequence, query head): Algorithm 3, global reduction.
struct MergeArgs {
    const int2* row_span;
    const float2* part_ml;
    const float* part_o;
    float* out;
    int Hq, Hkv, G, nseg, rows, ngroups;
    unsigned long long* timeline;
};

constexpr int MERGE_WARPS = 8;

// One CTA per (row, query head, slice of head_dim); DS slices of DW = D / DS coordinates each, chosen by the host so
// that a small batch still fills the GPU (with one sequence and four KV heads there are only 16 (row, head) pairs,
// each with up to 3 x 148 partials to fold).  The candidate parts are the (streaming CTA, consumer group) pairs of
// the streaming CTAs that hold units of the row, which the streaming kernel lists per row; a part marked absent
// weighs nothing.  Warp w takes a contiguous share of the candidates, MB warp instructions' worth a round (a row slice is
// DW / 4 lanes wide, so an instruction fetches 128 / DW candidates' slices): statistics and rows of a round are on their
// way together, and every lane weighs its own candidates, so a share of one round - the usual case - needs no exchange
// before the warps meet.  Lanes that hold the same coordinates, then the eight warps, are combined in a fixed order:
// o = sum_k O_k e^{m_k - m*} / sum_k l_k e^{m_k - m*},  m* = max_k m_k.
//
// Bound by latency: the chain wait - span - parts - output.  The span is read ahead of the wait as well (the streaming
// CTAs wrote it some 30 us earlier) and the parts it names are requested with the span itself, which is then checked.
template <int D, int DS>
__global__ void __launch_bounds__(32 * MERGE_WARPS) merge_kernel(const MergeArgs a) {
    constexpr int DW = D / DS;             // coordinates of this CTA's slice
    constexpr int LPC = DW / 4;            // lanes per candidate row slice (a float4 each)
    constexpr int CPW = 32 / LPC;          // candidates per warp instruction
    constexpr int MB = 4;                  // candidates per lane and round
    static_assert(DW >= 4 && LPC <= 32 && LPC * CPW == 32, "slice must be 4 .. 128 coordinates");
    __shared__ __align__(16) float s_acc[MERGE_WARPS][DW];
    __shared__ float s_l[MERGE_WARPS];
    __shared__ float s_m[MERGE_WARPS];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int pair = blockIdx.x / DS, dpart = blockIdx.x % DS;
    const int r = pair / a.G, gq = pair % a.G;
    const int i = r / a.Hkv, hk = r % a.Hkv;
    unsigned long long* const tl = ETA_TL((a.timeline && blockIdx.x < TL_MERGE_N) ? a.timeline + (size_t)(TL_MERGE + blockIdx.x) * 8 : nullptr);
    if (tl && tid == 0) tl[0] = globaltimer_ns();
    pdl_trigger();
    // what the span will most likely be; clamped, so that whatever is read here names slots of the scratch
    int2 guess = __ldcg(a.row_span + r);
    guess.x = min(max(guess.x, 0), MAX_CTAS - 1);
    guess.y = min(max(guess.y, 0), MAX_CTAS - guess.x);
    pdl_wait();          // every partial of the streaming kernel is in memory from here on
    if (tl && tid == 0) tl[1] = globaltimer_ns();
    const int sub = lane / LPC, dl = lane % LPC;        // candidate within a warp instruction, float4 within the slice
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    float m_w = -INFINITY, l_w = 0.f;                   // this lane's running maximum and weighted l
    const int2 span = __ldcg(a.row_span + r);
    auto fold_span = [&](const int2& sp, bool check) {
        const int n_cand = sp.y * a.ngroups;
        const int per = (n_cand + MERGE_WARPS - 1) / MERGE_WARPS;
        const int k_begin = warp * per, k_end = min(n_cand, k_begin + per);
        for (int k0 = k_begin + sub; k0 < k_end; k0 += MB * CPW) {
            float2 ml[MB];
            float4 x[MB];
#pragma unroll
            for (int u = 0; u < MB; ++u) {
                const int k = k0 + u * CPW;
                ml[u] = make_float2(-INFINITY, 0.f);
                x[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (k < k_end) {
                    const int64_t ph = (((int64_t)sp.x + r) * a.ngroups + k) * a.G + gq;
                    ml[u] = __ldcg(a.part_ml + ph);
                    x[u] = __ldcg(reinterpret_cast<const float4*>(a.part_o + ph * D + dpart * DW) + dl);
                }
            }
            if (check && (span.x != sp.x || span.y != sp.y)) return false;       // (the loads above are on their way)
            float m_new = m_w;
#pragma unroll
            for (int u = 0; u < MB; ++u) m_new = fmaxf(m_new, ml[u].x);
            if (m_new == -INFINITY) continue;
            const float keep = __expf(m_w - m_new);         // m_w = -inf gives 0
            acc.x *= keep; acc.y *= keep; acc.z *= keep; acc.w *= keep;
            l_w *= keep;
            m_w = m_new;
#pragma unroll
            for (int u = 0; u < MB; ++u) {
                if (ml[u].x != -INFINITY) {                 // an absent part's row is stale memory: never touch it
                    const float w = __expf(ml[u].x - m_new);
                    acc.x = fmaf(x[u].x, w, acc.x); acc.y = fmaf(x[u].y, w, acc.y);
                    acc.z = fmaf(x[u].z, w, acc.z); acc.w = fmaf(x[u].w, w, acc.w);
                    l_w = fmaf(ml[u].y, w, l_w);
                }
            }
        }
        return span.x == sp.x && span.y == sp.y;
    };
    if (!fold_span(guess, true)) {
        acc = make_float4(0.f, 0.f, 0.f, 0.f);
        m_w = -INFINITY; l_w = 0.f;
        fold_span(span, false);
    }
    // lanes that hold the same coordinates of different candidates
#pragma unroll
    for (int o = LPC; o < 32; o <<= 1) {
        const float m_o = __shfl_xor_sync(0xffffffffu, m_w, o), m_new = fmaxf(m_w, m_o);
        const float keep = m_w == -INFINITY ? 0.f : __expf(m_w - m_new), wo = m_o == -INFINITY ? 0.f : __expf(m_o - m_new);
        acc.x = acc.x * keep + __shfl_xor_sync(0xffffffffu, acc.x, o) * wo;
        acc.y = acc.y * keep + __shfl_xor_sync(0xffffffffu, acc.y, o) * wo;
        acc.z = acc.z * keep + __shfl_xor_sync(0xffffffffu, acc.z, o) * wo;
        acc.w = acc.w * keep + __shfl_xor_sync(0xffffffffu, acc.w, o) * wo;
        l_w = l_w * keep + __shfl_xor_sync(0xffffffffu, l_w, o) * wo;
        m_w = m_new;
    }
    if (tl && tid == 0) tl[3] = globaltimer_ns() + (__float_as_int(acc.x) & 0);
    if (sub == 0) *reinterpret_cast<float4*>(&s_acc[warp][dl * 4]) = acc;
    if (lane == 0) { s_l[warp] = l_w; s_m[warp] = m_w; }
    __syncthreads();
    if (tid < DW) {
        float M = -INFINITY;
#pragma unroll
        for (int w = 0; w < MERGE_WARPS; ++w) M = fmaxf(M, s_m[w]);
        float o = 0.f, l = 0.f;
        if (M != -INFINITY) {
#pragma unroll
            for (int w = 0; w < MERGE_WARPS; ++w) {
                const float sc = (s_m[w] == -INFINITY) ? 0.f : __expf(s_m[w] - M);
                o = fmaf(s_acc[w][tid], sc, o);
                l = fmaf(s_l[w], sc, l);
            }
        }
        a.out[((int64_t)i * a.Hq + hk * a.G + gq) * D + dpart * DW + tid] = l > 0.f ? o / l : 0.f;
    }
    if (tl && tid == 0) tl[4] = globaltimer_ns();
}

// ------------------------------------------------------------------ host side

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qr;
        cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qr);
        if (e != cudaSuccess || qr != cudaDriverEntryPointSuccess || !p) {
            set_cuda_error(e != cudaSuccess ? e : cudaErrorUnknown, "cuTensorMapEncodeTiled lookup");
            return nullptr;
        }
        fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// Tensor map of bf16 boxes in the 128-byte swizzle; what lies outside the tensor reads as zero
int encode_tiles(CUtensorMap* tm, const void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides,
                 const cuuint32_t* box) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return ETA_ERR_CUDA;
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    const CUresult rc = fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), dims, strides, box,
                           estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (rc != CUDA_SUCCESS) {
        set_cuda_error(cudaErrorInvalidValue, "cuTensorMapEncodeTiled");
        return ETA_ERR_CUDA;
    }
    return ETA_OK;
}

// K or V as a 5-D tensor (c within a 64-column half, t, half, hk, i) of bf16; a box is 64 columns x TS tokens x
// all halves: in shared memory, one 128-byte-swizzled [TS][64] tile per half, back to back.
// Tensor map of a K or V cache: 64 columns x tokens x column halves x KV heads x sequences, or, for a paged cache
// (n_pages > 0), ... x tokens of a page x ... x pages, with sb the stride between pages.
static int make_tmap(CUtensorMap* tm, const void* base, const eta_cache_desc* d, int64_t sb, int64_t sh, int64_t st,
                     int TS, int n_pages) {
    const cuuint32_t halves = (cuuint32_t)(d->head_dim / 64);
    cuuint64_t dims[5] = {64, (cuuint64_t)(n_pages > 0 ? d->block_size : d->t_cap), halves, (cuuint64_t)d->n_kv_heads,
                          (cuuint64_t)(n_pages > 0 ? n_pages : d->batch)};
    cuuint64_t strides[4] = {(cuuint64_t)st * 2, 128, (cuuint64_t)sh * 2, (cuuint64_t)sb * 2};
    cuuint32_t box[5] = {64, (cuuint32_t)TS, halves, 1, 1};
    return encode_tiles(tm, base, 5, dims, strides, box);
}

template <int D, int TS, int NSTAGE, int NGROUPS>
static int launch_decode_t(const CUtensorMap& tmK, const CUtensorMap& tmV, const DecodeArgs& a, int n_ctas,
                           cudaStream_t s) {
    const size_t smem = DecodeSmem<D, TS, NSTAGE, NGROUPS>::bytes(a.G);
    return launch_pdl("decode launch", decode_kernel<D, TS, NSTAGE, NGROUPS>, dim3(n_ctas),
                      dim3(32 * (WARPS_PER_GROUP * NGROUPS + 1)), smem, s, tmK, tmV, a);
}

// Streaming multiprocessors of the current device; negative: an eta_status
static int sm_count() {
    int dev = 0, n_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) { set_cuda_error(e, "device query"); return ETA_ERR_CUDA; }
    return n_sm;
}

// CTAs that a row gets in the one-kernel step; 0: the general path
static int step_ctas(const eta_cache_desc* desc, const eta_params* params) {
#ifdef ETA_TEST_GENERAL_PATH
    return 0;                           // test builds of the general path
#endif
    const int b = desc->block_size;
    if (params->flags & ETA_FLAG_DENSE) return 0;
    return step_cluster(desc->batch * desc->n_kv_heads, desc->nb_cap, b, desc->head_dim, b < 64 ? b : 64,
                        desc->n_q_heads / desc->n_kv_heads, (params->flags & ETA_FLAG_PACKED_SIGMA) != 0);
}

// eta_decode and eta_decode_paged: `pages` null selects the contiguous cache
static int decode_impl(const eta_cache_desc* desc, const eta_page_table* pages, const eta_params* params, const void* q,
                       const void* K, const void* V, const int32_t* seq_lens, const void* musig, const float* mnorm,
                       const float* tau, const float* head_const, float* out, uint8_t* sel_mask, int32_t* stats,
                       uint32_t* status_dev, void* workspace, size_t workspace_bytes, void* stream) {
    int rc = validate_desc(desc);
    if (rc != ETA_OK) return rc;
    if (pages && (rc = validate_pages(desc, pages)) != ETA_OK) return rc;
    if (!params || !q || !K || !V || !seq_lens || !out || !sel_mask) return ETA_ERR_INVALID_ARG;
    const bool dense = (params->flags & ETA_FLAG_DENSE) != 0;
    if (!dense && (!musig || !mnorm)) return ETA_ERR_INVALID_ARG;
    if ((tau != nullptr) == (head_const != nullptr)) return ETA_ERR_INVALID_ARG;
    if (params->rescue_window < 1 || params->lwb < 0) return ETA_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(K) | reinterpret_cast<uintptr_t>(V) | reinterpret_cast<uintptr_t>(q) |
         reinterpret_cast<uintptr_t>(musig) | reinterpret_cast<uintptr_t>(out)) & 15)
        return ETA_ERR_UNSUPPORTED;
    const WsLayout L = ws_layout(desc);
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) || workspace_bytes < L.total)
        return ETA_ERR_WORKSPACE;

    cudaStream_t s = static_cast<cudaStream_t>(stream);
    unsigned char* ws = static_cast<unsigned char*>(workspace);
    const int D = desc->head_dim, b = desc->block_size;
    const int G = desc->n_q_heads / desc->n_kv_heads;
    const float scale = params->scale > 0.f ? params->scale : 1.0f / sqrtf((float)D);

    const int n_sm = sm_count();
    if (n_sm < 0) return n_sm;
    const int TS = b < 64 ? b : 64;
    int n_ctas = n_sm;                  // one persistent CTA per SM; the shared-memory ring fills the SM
    if (n_ctas > MAX_CTAS) n_ctas = MAX_CTAS;

    ScreenArgs sa;
    sa.q = static_cast<const __nv_bfloat16*>(q);
    sa.musig = static_cast<const __half*>(musig);
    sa.mnorm = mnorm;
    sa.seq_lens = seq_lens;
    sa.tau = tau;
    sa.head_const = head_const;
    sa.z = params->z; sa.a = params->a; sa.scale = scale;
    sa.lwb = params->lwb; sa.rescue_window = params->rescue_window; sa.flags = params->flags;
    sa.Hq = desc->n_q_heads; sa.Hkv = desc->n_kv_heads; sa.b = b; sa.t_cap = desc->t_cap; sa.nb_cap = desc->nb_cap;
    sa.nseg = L.nseg; sa.rows = L.rows;
    sa.b_shift = (b == 32) ? 5 : (b == 64 ? 6 : 7);
    sa.div_hkv = FastDiv(desc->n_kv_heads);
    sa.seg_cnt = ws + L.seg_cnt;
    sa.gpr = L.gpr;
    sa.seg_list = reinterpret_cast<int32_t*>(ws + L.seg_list);
    sa.tau_eff = reinterpret_cast<float*>(ws + L.tau_eff);
    // at most rows + slots CTAs screen (launch_screen): with G entries each a small part of the partials' (MAX_CTAS + rows) * 3 G
    sa.resc = reinterpret_cast<int2*>(ws + L.resc);
    sa.sel_mask = sel_mask;
#ifdef ETA_TIMELINE
    sa.timeline = debug_timeline();
#endif
    sa.status = status_dev;
    CUtensorMap tmK, tmV;
    const int n_pages = pages ? pages->n_pages : 0;
    rc = make_tmap(&tmK, K, desc, desc->k_stride_b, desc->k_stride_h, desc->k_stride_t, TS, n_pages);
    if (rc != ETA_OK) return rc;
    rc = make_tmap(&tmV, V, desc, desc->v_stride_b, desc->v_stride_h, desc->v_stride_t, TS, n_pages);
    if (rc != ETA_OK) return rc;

    if (const int ctas = step_ctas(desc, params)) {
        StepArgs st;
        st.q = sa.q; st.musig = sa.musig; st.mnorm = mnorm; st.seq_lens = seq_lens; st.tau = tau; st.head_const = head_const;
        st.z = params->z; st.a = params->a; st.scale = scale; st.beta = params->beta;
        st.lwb = params->lwb; st.rescue_window = params->rescue_window; st.flags = params->flags;
        st.Hq = desc->n_q_heads; st.b_shift = sa.b_shift; st.t_cap = desc->t_cap; st.nb_cap = desc->nb_cap;
        st.block_table = pages ? pages->block_table : nullptr;
        st.table_stride = pages ? pages->table_stride : 0;
        st.div_hkv = sa.div_hkv;
        st.out = out; st.sel_mask = sel_mask; st.stats = stats; st.status = status_dev;
        profile_mark(2, s);
        profile_mark(3, s);
        rc = launch_step(st, tmK, tmV, L.rows, D, TS, G, ctas, s);
        profile_mark(4, s);
        profile_mark(5, s);
        return rc;
    }

    sa.tiles = b / TS; sa.tile_tokens = TS;
    sa.block_table = pages ? pages->block_table : nullptr;
    sa.table_stride = pages ? pages->table_stride : 0;
    // A cache well beyond the L2 (126 MB): what a step reads of it will not be there for the next step, so its lines leave
    // the L2 first, and the screening kernel starts the first survivors of every segment on their way, 32 MB in all (five of
    // the 8 us the memory would idle before the streaming kernel's first copies).  Batch 4 at 128K: 66.7 -> 60.5 us a step with
    // the first of the two, 58.4 with both (24, 48 and 80 MB within 1 us of 32); 32K x 8: 58.0 -> 51.2; 512K: 51.2 -> 43.4.
    // Where the cache fits, or nearly, both cost time: 50K x 1 with 4 KV heads (104 MB) 24.7 -> 27.8, 8K x 7 (30 MB) 24.7 -> 28.8;
    // between 140 and 330 MB the sign depends on how much survives (51.3 -> 45.0, 33.9 -> 33.2, 30.0 -> 32.4): the line lies
    // where most gain, it is not sharp.  It goes by the capacity, which the host knows; of a cache of 128K x 4 that holds little,
    // a step takes without and with both, 4K x 4 21.3, 21.4; 16K x 4 26.2, 27.1; 32K x 4 34.9, 32.7.  Lengths added up on the device
    // win the second and cost 0.5 to 2 us on the large steps, 8 where 183 MB are held in 419 (76.6 against 71.3 with both).
    const int64_t unit_bytes = (int64_t)4 * b * D, segs = (int64_t)L.rows * L.nseg;
    const bool large = (int64_t)L.rows * desc->nb_cap * unit_bytes > LARGE_CACHE_BYTES;
    const int64_t share = (PREFETCH_BYTES + segs * unit_bytes - 1) / (segs * unit_bytes);
    sa.prefetch = !large ? 0 : (int)(share < SEG ? share : SEG);
    profile_mark(2, s);
    rc = launch_screen(sa, tmK, tmV, L.rows, D, G, n_sm, s);
    profile_mark(3, s);
    if (rc != ETA_OK) return rc;

    DecodeArgs da;
    da.q = sa.q; da.seq_lens = seq_lens; da.tau_eff = sa.tau_eff; da.seg_list = sa.seg_list;
    da.seg_cnt = sa.seg_cnt; da.stats = stats;
    da.row_span = reinterpret_cast<int2*>(ws + L.row_span);
    da.part_ml = reinterpret_cast<float2*>(ws + L.part_ml);
    da.part_o = reinterpret_cast<float*>(ws + L.part_o);
    da.status = status_dev;
    da.beta = params->beta; da.scale = scale;
    da.Hq = desc->n_q_heads; da.Hkv = desc->n_kv_heads; da.G = G; da.b = b; da.t_cap = desc->t_cap;
    da.nseg = L.nseg; da.rows = L.rows; da.nb_cap = desc->nb_cap;
    da.gpr = L.gpr; da.n_gran = L.rows * L.gpr;
    da.n_chunks = (da.n_gran + CHUNK - 1) / CHUNK;
    da.super = (da.n_chunks + MAX_SUPER - 1) / MAX_SUPER;
    da.ungate_last = (!dense && (params->flags & ETA_FLAG_UNGATE_LAST)) ? 1 : 0;
    da.block_table = pages ? pages->block_table : nullptr;
    da.table_stride = pages ? pages->table_stride : 0;
    da.read_once = large ? 1 : 0;
    da.div_gpr = FastDiv(L.gpr); da.div_hkv = FastDiv(desc->n_kv_heads); da.div_grid = FastDiv(n_ctas);
    da.timeline = debug_timeline();
    if (D == 128 && TS == 64) {
        rc = launch_decode_t<128, 64, 6, DECODE_GROUPS>(tmK, tmV, da, n_ctas, s);
    } else if (D == 128 && TS == 32) {
        rc = launch_decode_t<128, 32, 12, DECODE_GROUPS>(tmK, tmV, da, n_ctas, s);
    } else if (D == 64 && TS == 64) {
        rc = launch_decode_t<64, 64, 12, DECODE_GROUPS>(tmK, tmV, da, n_ctas, s);
    } else {
        rc = launch_decode_t<64, 32, 24, DECODE_GROUPS>(tmK, tmV, da, n_ctas, s);
    }
    if (rc != ETA_OK) return rc;
    profile_mark(4, s);

    MergeArgs ma;
    ma.row_span = da.row_span; ma.part_ml = da.part_ml; ma.part_o = da.part_o; ma.out = out;
    ma.Hq = desc->n_q_heads; ma.Hkv = desc->n_kv_heads; ma.G = G; ma.nseg = L.nseg; ma.rows = L.rows; ma.ngroups = DECODE_GROUPS; ma.timeline = debug_timeline();
    // slices of head_dim per (row, head): enough CTAs to fill the GPU when the batch is small
    const int pairs = L.rows * G;
    const int DS = (pairs * 4 <= n_sm) ? 8 : (pairs * 2 <= n_sm ? 4 : (pairs <= n_sm / 2 ? 2 : 1));
    const dim3 mgrid((unsigned)(pairs * DS)), mblock(32 * MERGE_WARPS);
#define ETA_MERGE(DD, SS) launch_pdl("merge launch", merge_kernel<DD, SS>, mgrid, mblock, 0, s, ma)
    if (D == 128) rc = DS == 8 ? ETA_MERGE(128, 8) : (DS == 4 ? ETA_MERGE(128, 4) : (DS == 2 ? ETA_MERGE(128, 2) : ETA_MERGE(128, 1)));
    else rc = DS == 8 ? ETA_MERGE(64, 8) : (DS == 4 ? ETA_MERGE(64, 4) : (DS == 2 ? ETA_MERGE(64, 2) : ETA_MERGE(64, 1)));
#undef ETA_MERGE
    profile_mark(5, s);
    return rc;
}

}  // namespace eta

extern "C" {

int eta_decode_kernel_count(void) { return 3; }

int eta_decode_launches(const eta_cache_desc* desc, const eta_params* params) {
    using namespace eta;
    const int rc = validate_desc(desc);
    if (rc != ETA_OK) return rc;
    if (!params || params->rescue_window < 1 || params->lwb < 0) return ETA_ERR_INVALID_ARG;
    const int n_sm = sm_count();
    if (n_sm < 0) return n_sm;
    if (step_ctas(desc, params)) return 1;
    const WsLayout L = ws_layout(desc);
    return 2 + screen_launches(L.rows, L.nseg, desc->nb_cap, desc->head_dim, params->rescue_window, (params->flags & ETA_FLAG_DENSE) != 0, n_sm);
}

int eta_decode(const eta_cache_desc* desc, const eta_params* params, const void* q, const void* K, const void* V,
               const int32_t* seq_lens, const void* musig, const float* mnorm, const float* tau,
               const float* head_const, float* out, uint8_t* sel_mask, int32_t* stats, uint32_t* status_dev,
               void* workspace, size_t workspace_bytes, void* stream) {
    return eta::decode_impl(desc, nullptr, params, q, K, V, seq_lens, musig, mnorm, tau, head_const, out, sel_mask, stats,
                            status_dev, workspace, workspace_bytes, stream);
}

int eta_decode_paged(const eta_cache_desc* desc, const eta_page_table* pages, const eta_params* params, const void* q,
                     const void* K_pool, const void* V_pool, const int32_t* seq_lens, const void* musig,
                     const float* mnorm, const float* tau, const float* head_const, float* out, uint8_t* sel_mask,
                     int32_t* stats, uint32_t* status_dev, void* workspace, size_t workspace_bytes, void* stream) {
    if (!pages) return ETA_ERR_INVALID_ARG;
    return eta::decode_impl(desc, pages, params, q, K_pool, V_pool, seq_lens, musig, mnorm, tau, head_const, out, sel_mask,
                            stats, status_dev, workspace, workspace_bytes, stream);
}

}  // extern "C"
