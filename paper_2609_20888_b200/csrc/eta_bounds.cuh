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

// A warp's tile: 8 KB of unpacked records, NT 8-column MMA tiles
template <int D>
struct TileOf {
    static constexpr int NT = 256 / D;                        // 2 at head_dim 128, 4 at 64
    static constexpr int RECS = 8 * NT;
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

// The query side of a row's bounds, in the order the MMAs want it.  Lane (hd = lane / 4, t = lane % 4) feeds row hd (and
// hd + 8) of A; in k-group j (32 coordinates) it holds coordinates 8 (4 j + t) .. + 7, the ones its 16-byte piece of a
// record covers on the B side (a dot product does not care about the order of k).
template <int D, int G>
struct QTab {
    static constexpr int J = D / 32;
    static constexpr int NLO = (G == 8) ? 1 : 0;      // eight heads fill rows 0-7 of A: the second parts go to rows 8-15
    uint4 f16[J][32];                                 // scaled q as fp16
    float4 sq[J][32][2];                              // q^2: rows 0-3 leading parts of heads 0-3, rows 4-7 the rest (G <= 4);
                                                      //      rows 0-7 leading parts (G = 8)
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
    const int head = ((tid & 31) >> 2) & (G == 8 ? 7 : 3);         // rows 4-7 hold the second parts of heads 0-3
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
// -> whether some lane saw a NaN among the bounds of the first n records.  Two accumulators for the variance term: a tile
// is a chain of dependent MMAs, and its latency is what a CTA of one or two tiles per warp takes (unrolling k gained nothing).
template <int D, int G, bool PACKED>
__device__ __forceinline__ bool bound_tile(const QTab<D, G>& tab, uint32_t recs, int n, float mn, float z, float scale,
                                           float* __restrict__ sb) {
    constexpr int J = D / 32, NT = TileOf<D>::NT, REC = PACKED ? 3 * D : 4 * D;
    const int lane = threadIdx.x & 31, n8 = lane >> 2, t = lane & 3;
    const uint32_t rp = recs + n8 * REC;
    float dot[NT][4], vhi[NT][4], vlo[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int c = 0; c < 4; ++c) { dot[nt][c] = 0.f; vhi[nt][c] = 0.f; vlo[nt][c] = 0.f; }
#pragma unroll 1
    for (int j = 0; j < J; ++j) {
        const uint4 qa = tab.f16[j][lane];
        const float4 sa = tab.sq[j][lane][0], sb4 = tab.sq[j][lane][1];
        float4 la = make_float4(0.f, 0.f, 0.f, 0.f), lb = la;
        if constexpr (G == 8) { la = tab.sq_lo[j][lane][0]; lb = tab.sq_lo[j][lane][1]; }
        uint4 mu[NT];
        SigmaPiece<PACKED> sg[NT];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            mu[nt] = lds128(rp + nt * 8 * REC + (4 * j + t) * 16);
            load_sigma_shared<D, PACKED>(sg[nt], rp + nt * 8 * REC, 4 * j + t);
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            mma_f16_16816(dot[nt], qa.x, 0u, qa.y, 0u, mu[nt].x, mu[nt].y);
            mma_f16_16816(dot[nt], qa.z, 0u, qa.w, 0u, mu[nt].z, mu[nt].w);
            float s[8], hi[8];
            sigma_f32<PACKED>(sg[nt], s);
#pragma unroll
            for (int k = 0; k < 8; ++k) { s[k] *= s[k]; hi[k] = tf32_hi(s[k]); s[k] -= hi[k]; }
            mma_tf32_1688(vhi[nt], sa.x, la.x, sa.y, la.y, hi[0], hi[1]);
            mma_tf32_1688(vlo[nt], sa.x, la.x, sa.y, la.y, s[0], s[1]);
            mma_tf32_1688(vhi[nt], sa.z, la.z, sa.w, la.w, hi[2], hi[3]);
            mma_tf32_1688(vlo[nt], sa.z, la.z, sa.w, la.w, s[2], s[3]);
            mma_tf32_1688(vhi[nt], sb4.x, lb.x, sb4.y, lb.y, hi[4], hi[5]);
            mma_tf32_1688(vlo[nt], sb4.x, lb.x, sb4.y, lb.y, s[4], s[5]);
            mma_tf32_1688(vhi[nt], sb4.z, lb.z, sb4.w, lb.w, hi[6], hi[7]);
            mma_tf32_1688(vlo[nt], sb4.z, lb.z, sb4.w, lb.w, s[6], s[7]);
        }
    }
    // lane (head n8, t) holds records 8 nt + 2 t and + 1
    const float qn = tab.norm[n8 < G ? n8 : 0], un = qtab_unscale(qn);
    bool bad = false;
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const float v = vhi[nt][c] + vlo[nt][c];
            const float v2 = v + (G == 8 ? vhi[nt][c + 2] + vlo[nt][c + 2] : __shfl_xor_sync(0xffffffffu, v, 16));
            const int rec = nt * 8 + 2 * t + c;
            const float m = __shfl_sync(0xffffffffu, mn, rec);
            const float bound = scale * min_keep_nan((dot[nt][c] + z * sqrtf(v2)) * un, qn * m);
            if (n8 < G) sb[rec * G + n8] = bound;
            bad = bad || (n8 < G && rec < n && bound != bound);
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
