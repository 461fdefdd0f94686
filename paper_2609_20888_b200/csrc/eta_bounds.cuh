// Bounds (Eq. dual_bound_eq) of tiles of block records, by one warp for all G query heads of a KV head: what the screening
// kernel, the diagnostic that returns bounds and the one-kernel step share.
#pragma once

#include "eta_common.cuh"

namespace eta {

// min that keeps a NaN (so that "not below the threshold" admits the block)
__device__ __forceinline__ float min_keep_nan(float g, float s) {
    return (g < s) ? g : ((s < g) ? s : ((g != g) ? g : s));
}

// Bounds as integers that ascend with them: 0xffffffff stands for a NaN, 0 for no bound at all (and reads as a NaN too: a
// comparison with it never holds)
__device__ __forceinline__ uint32_t bound_key(float bound) {
    const float bd = bound + 0.f;                                // (-0 counts as +0)
    const uint32_t u = __float_as_uint(bd);
    return bd != bd ? 0xffffffffu : ((u & 0x80000000u) ? ~u : (u | 0x80000000u));
}
__device__ __forceinline__ float key_bound(uint32_t k) { return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k); }

constexpr int SCR_WARPS = 4;

// A warp's tile: 8 KB of unpacked records, MT MMA tiles of 16 rows
template <int D>
struct TileOf {
    static constexpr int MT = 128 / D;                        // 1 at head_dim 128, 2 at 64
    static constexpr int RECS = 16 * MT;
    static constexpr int PASS = SCR_WARPS * RECS;             // records a CTA bounds at a time: 64 or 128
    static constexpr int BYTES = RECS * 4 * D;
    static_assert(PASS % SEG == 0, "a pass covers whole segments");
};

// D(16x8, fp32) += A(16x8, tf32, row) * B(8x8, tf32, col)
__device__ __forceinline__ void mma_tf32_1688(float (&c)[4], float a0, float a1, float a2, float a3, float b0, float b1) {
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(__float_as_uint(a0)), "r"(__float_as_uint(a1)), "r"(__float_as_uint(a2)), "r"(__float_as_uint(a3)),
                   "r"(__float_as_uint(b0)), "r"(__float_as_uint(b1)));
}
// the leading 11 significant bits of x: what a tf32 operand holds, so that x = tf32_hi(x) + (x - tf32_hi(x)) exactly and
// the rest of a 22-bit product fits tf32 too
__device__ __forceinline__ float tf32_hi(float x) { return __uint_as_float(__float_as_uint(x) & 0xffffe000u); }

// The query side of a row's bounds, in the order the MMAs want it.  Lane (hd = lane / 4, t = lane % 4) feeds column hd of B; in
// k-group j (32 coordinates) it holds coordinates 8 (4 j + t) .. + 7, the ones its 16-byte pieces of two records cover on the A
// side (a dot product does not care about the order of k).
template <int D, int G>
struct QTab {
    static constexpr int J = D / 32;
    static constexpr int NLO = (G == 8) ? 1 : 0;      // eight heads fill the columns of B: the second parts are another B
    uint4 f16[J][32];                                 // scaled q as fp16
    float4 sq[J][32][2];                              // q^2: columns 0-3 leading parts of heads 0-3, columns 4-7 the rest (G <= 4);
                                                      //      columns 0-7 leading parts (G = 8)
    float4 sq_lo[NLO ? J : 1][NLO ? 32 : 1][2];       // G = 8: the rest
    uint4 raw[G * D / 8];                             // the queries as they are (bf16)
    float n2[J][8];                                   // partial squared norms
    float norm[8];                                    // ||q_h||
};

// The power of two that puts a norm in [2^13, 2^14) is 2^qtab_shift.  fp16 holds neither the large nor the tiny end of
// bf16's range, so a head's query is scaled by it (every coordinate then fits, and one below fp16's normal range is below
// 2^-27 of the norm) and the sums are scaled back: both exact.  A norm that overflows fp32 gives NaN bounds (the block is
// admitted), one that underflows to zero a zero sum.
__device__ __forceinline__ int qtab_shift(float qn) { return min(max(140 - ((__float_as_int(qn) >> 23) & 0xff), -120), 120); }
__device__ __forceinline__ float qtab_scale(float qn) {
    const int ef = (__float_as_int(qn) >> 23) & 0xff;
    return ef == 255 ? __int_as_float(0x7fc00000) : (ef == 0 ? 0.f : __int_as_float((127 + qtab_shift(qn)) << 23));
}
__device__ __forceinline__ float qtab_unscale(float qn) {
    return ((__float_as_int(qn) >> 23) & 0xff) == 0 ? 0.f : __int_as_float((127 - qtab_shift(qn)) << 23);
}

// Thread tid's piece of the row's G queries, for build_qtab.  A load of its own, so that it can be on its way before anything waits
// for another one: from pinned host memory, or missing the L2, it is the longest one of a CTA's set-up (8 rows of 32K: 49.8 -> 49.4 us a
// step; 512K: 42.9 -> 42.5).
template <int D, int G>
__device__ __forceinline__ uint4 load_qtab(const __nv_bfloat16* q, int tid) {
    const int head = ((tid & 31) >> 2) & (G == 8 ? 7 : 3);         // columns 4-7 hold the second parts of heads 0-3
    uint4 v = make_uint4(0, 0, 0, 0);
    if (tid < D && head < G) v = __ldcg(reinterpret_cast<const uint4*>(q + head * D + 8 * (4 * (tid >> 5) + (tid & 3))));
    return v;
}

// Every thread of the CTA calls this with what load_qtab gave it; the first D threads (J warps) work.
template <int D, int G>
__device__ __forceinline__ void build_qtab(QTab<D, G>& tab, const uint4& v, int tid) {
    constexpr int J = D / 32;
    const bool mine = tid < D;
    const int j = tid >> 5, hd = (tid & 31) >> 2, t = tid & 3;
    float x[8];
    if (mine) {
        if (hd < G) tab.raw[hd * (D / 8) + 4 * j + t] = v;
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        float n2 = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) { x[2 * k] = bf16_lo(w[k]); x[2 * k + 1] = bf16_hi(w[k]); }
#pragma unroll
        for (int k = 0; k < 8; ++k) n2 = fmaf(x[k], x[k], n2);
        n2 += __shfl_xor_sync(0xffffffffu, n2, 1);
        n2 += __shfl_xor_sync(0xffffffffu, n2, 2);
        if (t == 0) tab.n2[j][hd] = n2;
    }
    __syncthreads();
    if (mine) {
        float n2 = 0.f;
#pragma unroll
        for (int k = 0; k < J; ++k) n2 += tab.n2[k][hd];
        const float qn = sqrtf(n2), sc = qtab_scale(qn);
        uint32_t h[4];
        float sq[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float a = x[2 * k] * sc, b = x[2 * k + 1] * sc;
            const __half2 hh = __floats2half2_rn(a, b);
            h[k] = (hd < G) ? *reinterpret_cast<const uint32_t*>(&hh) : 0u;
            sq[2 * k] = a * a; sq[2 * k + 1] = b * b;       // exact: q has 8 significant bits
        }
        tab.f16[j][tid & 31] = make_uint4(h[0], h[1], h[2], h[3]);
        const bool second = (G < 8) && hd >= 4;
        float hi[8], lo[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) { hi[k] = tf32_hi(sq[k]); lo[k] = sq[k] - hi[k]; }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const float4 a = make_float4(hi[4 * u], hi[4 * u + 1], hi[4 * u + 2], hi[4 * u + 3]);
            const float4 b = make_float4(lo[4 * u], lo[4 * u + 1], lo[4 * u + 2], lo[4 * u + 3]);
            tab.sq[j][tid & 31][u] = second ? b : a;
            if (G == 8) tab.sq_lo[j][tid & 31][u] = b;
        }
        if (j == 0 && t == 0 && hd < G) tab.norm[hd] = qn;
    }
    __syncthreads();
}

// One piece (eight coordinates) of a record's sigma as stored
template <bool PACKED> struct SigmaPiece { uint4 v; };
template <> struct SigmaPiece<true> { uint2 v; };
template <int D, bool PACKED>
__device__ __forceinline__ void load_sigma(SigmaPiece<PACKED>& s, const unsigned char* rec, int piece) {
    if constexpr (PACKED) s.v = __ldcg(reinterpret_cast<const uint2*>(rec + 2 * D + piece * 8));
    else s.v = __ldcg(reinterpret_cast<const uint4*>(rec + 2 * D + piece * 16));
}
template <int D, bool PACKED>
__device__ __forceinline__ void load_sigma_shared(SigmaPiece<PACKED>& s, uint32_t rec, int piece) {
    if constexpr (PACKED) asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(s.v.x), "=r"(s.v.y) : "r"(rec + 2 * D + piece * 8));
    else s.v = lds128(rec + 2 * D + piece * 16);
}
template <bool PACKED>
__device__ __forceinline__ void sigma_f32(const SigmaPiece<PACKED>& s, float (&out)[8]) {
    if constexpr (PACKED) {
        e4m3x8_to_f32(s.v, out);
    } else {
        const uint32_t w[4] = {s.v.x, s.v.y, s.v.z, s.v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[k]));
            out[2 * k] = f.x; out[2 * k + 1] = f.y;
        }
    }
}

// Bounds of a tile of records at `recs` in shared memory, for all heads of the group, by one warp: sb[record][head].  What
// the tile holds past its last record is computed like the rest and must not be read.  mn: the largest key norm of record
// `lane`.  sigma^2 has at most 22 significant bits (sigma is fp16) and q^2 sixteen: each is the sum of two tf32 values, every
// product of parts is exact and the accumulation is fp32, so the variance term is as good as one computed on the fp32
// pipe, without a shuffle tree and with a quarter of the fp32 instructions.
// -> whether some lane saw a NaN among the bounds of the first n records.
// What bounds it: an MMA of this kind takes a scheduler 8 cycles whatever its k, 21 in a chain.  So the records are the rows of A (16)
// and the queries the columns of B (eight heads, or four and their second parts): 40 MMAs for 8 KB of records at d = 128 and G <= 4
// where queries as rows, half of them empty, took 80, and the same sums in the same order.  us a step before and after: 16 rows of up
// to 64K tokens 131.8 -> 129.1, 512K x 1 43.0 -> 42.2, 128K x 4 58.9 -> 58.1, 16K x 1 17.4 -> 17.0.  Two accumulators for the variance
// term: a tile is a chain of dependent MMAs.  Unrolling the loop over j by two (129.8) or pairs in the packed fp32 instructions (130.0)
// gained nothing.
template <int D, int G, bool PACKED>
__device__ __forceinline__ bool bound_tile(const QTab<D, G>& tab, uint32_t recs, int n, float mn, float z, float scale,
                                           float* __restrict__ sb) {
    constexpr int J = D / 32, MT = TileOf<D>::MT, REC = PACKED ? 3 * D : 4 * D, NQ = G == 8 ? 2 : 1;
    const int lane = threadIdx.x & 31, n8 = lane >> 2, t = lane & 3;
    const uint32_t rp = recs + n8 * REC;
    float dot[MT][4], vhi[MT][NQ][4], vlo[MT][NQ][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            dot[mt][c] = 0.f;
#pragma unroll
            for (int p = 0; p < NQ; ++p) { vhi[mt][p][c] = 0.f; vlo[mt][p][c] = 0.f; }
        }
#pragma unroll 1
    for (int j = 0; j < J; ++j) {
        const uint4 qa = tab.f16[j][lane];
        float4 q2[NQ][2] = {{tab.sq[j][lane][0], tab.sq[j][lane][1]}};
        if constexpr (G == 8) { q2[1][0] = tab.sq_lo[j][lane][0]; q2[1][1] = tab.sq_lo[j][lane][1]; }
        uint4 mu[MT][2];
        SigmaPiece<PACKED> sg[MT][2];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int e = 0; e < 2; ++e) {             // records n8 and n8 + 8
                mu[mt][e] = lds128(rp + (mt * 16 + e * 8) * REC + (4 * j + t) * 16);
                load_sigma_shared<D, PACKED>(sg[mt][e], rp + (mt * 16 + e * 8) * REC, 4 * j + t);
            }
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            mma_f16_16816(dot[mt], mu[mt][0].x, mu[mt][1].x, mu[mt][0].y, mu[mt][1].y, qa.x, qa.y);
            mma_f16_16816(dot[mt], mu[mt][0].z, mu[mt][1].z, mu[mt][0].w, mu[mt][1].w, qa.z, qa.w);
            float hi[2][8], lo[2][8];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                sigma_f32<PACKED>(sg[mt][e], lo[e]);
#pragma unroll
                for (int k = 0; k < 8; ++k) { lo[e][k] *= lo[e][k]; hi[e][k] = tf32_hi(lo[e][k]); lo[e][k] -= hi[e][k]; }
            }
#pragma unroll
            for (int k = 0; k < 8; k += 2)
#pragma unroll
                for (int p = 0; p < NQ; ++p) {
                    const float4 b = q2[p][k / 4];
                    const float b0 = k % 4 ? b.z : b.x, b1 = k % 4 ? b.w : b.y;
                    mma_tf32_1688(vhi[mt][p], hi[0][k], hi[1][k], hi[0][k + 1], hi[1][k + 1], b0, b1);
                    mma_tf32_1688(vlo[mt][p], lo[0][k], lo[1][k], lo[0][k + 1], lo[1][k + 1], b0, b1);
                }
        }
    }
    // lane (n8, t) holds records n8 and n8 + 8 of columns 2 t and 2 t + 1
    const bool mine = 2 * t < G;
    float qn[2], un[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) { qn[c] = tab.norm[2 * t + c < G ? 2 * t + c : 0]; un[c] = qtab_unscale(qn[c]); }
    bool bad = false;
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int rec = mt * 16 + e * 8 + n8;
            const float m = __shfl_sync(0xffffffffu, mn, rec);
            float bound[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const float v = vhi[mt][0][2 * e + c] + vlo[mt][0][2 * e + c];
                const float v2 = v + (G == 8 ? vhi[mt][NQ - 1][2 * e + c] + vlo[mt][NQ - 1][2 * e + c] : __shfl_xor_sync(0xffffffffu, v, 2));
                bound[c] = scale * min_keep_nan((dot[mt][2 * e + c] + z * sqrtf(v2)) * un[c], qn[c] * m);
                bad = bad || (2 * t + c < G && rec < n && bound[c] != bound[c]);
            }
            if (mine) {
                if constexpr (G == 1) sb[rec] = bound[0];
                else *reinterpret_cast<float2*>(sb + rec * G + 2 * t) = make_float2(bound[0], bound[1]);
            }
        }
    __syncwarp();
    return __any_sync(0xffffffffu, bad);
}

// Bound of one record by one warp in plain fp32, for all heads of the group (queries in shared memory): 32 / (D / 8) heads
// side by side.
template <int D, int G, bool PACKED>
__device__ __forceinline__ void bound_one(const uint4* __restrict__ qw, const unsigned char* src,
                                          float mn, float z, float scale, float* __restrict__ sb) {
    constexpr int LPR = D / 8, HP = 32 / LPR;
    const int lane = threadIdx.x & 31, cl = lane % LPR, sub = lane / LPR;
    const uint4 m4 = __ldcg(reinterpret_cast<const uint4*>(src + cl * 16));
    SigmaPiece<PACKED> sp;
    load_sigma<D, PACKED>(sp, src, cl);
    const uint32_t mw[4] = {m4.x, m4.y, m4.z, m4.w};
    float mu[8], s2[8];
    sigma_f32<PACKED>(sp, s2);
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        const float2 mf = __half22float2(*reinterpret_cast<const __half2*>(&mw[kk]));
        mu[2 * kk] = mf.x; mu[2 * kk + 1] = mf.y;
    }
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) s2[kk] *= s2[kk];
#pragma unroll 1
    for (int g0 = 0; g0 < G; g0 += HP) {
        const int gq = g0 + sub;
        const uint4 qv = qw[min(gq, G - 1) * LPR + cl];
        const uint32_t qq[4] = {qv.x, qv.y, qv.z, qv.w};
        float dot = 0.f, var = 0.f, n2 = 0.f;
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
            const float x = (kk & 1) ? bf16_hi(qq[kk >> 1]) : bf16_lo(qq[kk >> 1]);
            n2 = fmaf(x, x, n2);
            dot = fmaf(x, mu[kk], dot);
            var = fmaf(x * x, s2[kk], var);
        }
#pragma unroll
        for (int sh = 1; sh < LPR; sh <<= 1) {
            n2 += __shfl_xor_sync(0xffffffffu, n2, sh);
            dot += __shfl_xor_sync(0xffffffffu, dot, sh);
            var += __shfl_xor_sync(0xffffffffu, var, sh);
        }
        if (cl == 0 && gq < G) sb[gq] = scale * min_keep_nan(dot + z * sqrtf(var), sqrtf(n2) * mn);
    }
    __syncwarp();
}

// A warp's stream of tiles: one or two bulk copies in flight, into the warp's own shared memory.
template <int D, int G, bool PACKED>
struct TileStream {
    static constexpr int REC = PACKED ? 3 * D : 4 * D;
    using T = TileOf<D>;
    unsigned char* bufs;               // nbuf tiles
    uint64_t* bars;                    // two barriers
    const unsigned char* rec_row;      // records and largest norms of the row
    const float* mn_row;
    int NB, nbuf;                      // full blocks of the row
    int in, out;                       // tiles issued and consumed so far
    uint32_t parity;                   // bit k: of buffer k
    bool alive;                        // false once a wait ran out: nothing is issued any more

    // starts the copy of the tile at record j (the buffer's previous tile has been read by the whole warp)
    __device__ __forceinline__ void issue(int j) {
        const int k = nbuf == 2 ? (in & 1) : 0, n = min(T::RECS, NB - j);
        ++in;
        if (n > 0 && alive && (threadIdx.x & 31) == 0) {
            mbar_arrive_expect_tx(bars + k, n * REC);
            tma_load_1d(bufs + k * T::BYTES, rec_row + (int64_t)j * REC, n * REC, bars + k);
        }
    }
    // Bounds of the oldest tile in flight, whose first record is j, into sb[record][head]; false when the copy did not arrive.
    // A wait that runs out admits the tile's blocks (NaN bounds: the safe direction).  What the tensor-core path cannot do
    // shows as a NaN bound too (an infinite sigma has no exact split, a query's norm may overflow) and is computed again in
    // fp32.
    __device__ __forceinline__ bool bounds(const QTab<D, G>& tab, int j, float z, float scale, float* __restrict__ sb) {
        const int lane = threadIdx.x & 31, k = nbuf == 2 ? (out & 1) : 0, n = min(T::RECS, NB - j);
        ++out;
        if (n <= 0) return true;
        const float mn = lane < n ? __ldcg(mn_row + j + lane) : 0.f;
        const bool was_alive = alive;
        if (alive) alive = __all_sync(0xffffffffu, mbar_wait(bars + k, (parity >> k) & 1));
        if (!alive) {
            for (int e = lane; e < n * G; e += 32) sb[e] = __int_as_float(0x7fc00000);
            if (was_alive) {                           // bounded: time for the copies to land before the CTA's memory is released
                mbar_wait(bars + k, (parity >> k) & 1);
                if (in > out) mbar_wait(bars + (k ^ 1), (parity >> (k ^ 1)) & 1);
            }
            __syncwarp();
            return false;
        }
        parity ^= 1u << k;
        if (bound_tile<D, G, PACKED>(tab, smem_u32(bufs + k * T::BYTES), n, mn, z, scale, sb)) {
            bool bad = false;
#pragma unroll
            for (int g = 0; g < G; ++g) bad = bad || (lane < n && sb[lane * G + g] != sb[lane * G + g]);
            unsigned todo = __ballot_sync(0xffffffffu, bad);
            while (todo) {
                const int rec = __ffs(todo) - 1;
                todo &= todo - 1;
                bound_one<D, G, PACKED>(tab.raw, rec_row + (int64_t)(j + rec) * REC, __shfl_sync(0xffffffffu, mn, rec), z, scale, sb + rec * G);
            }
        }
        return true;
    }
};

}  // namespace eta
