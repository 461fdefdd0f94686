// Gated attention of one KV head's query heads over a tile of K and V in shared memory, by a group of four warps: what the
// streaming kernel and the one-kernel step share.
//
// The G query heads of the group are packed on the M side of mma.m16n8k16 (bf16 in, fp32 out), tokens on N, so each K/V byte is
// read once from shared memory for all heads.  The head_dim and token orders fed to the MMAs are permuted (a dot product does not
// care) so that every shared-memory read is a conflict-free 16-byte load of the 128-byte-swizzled tile.  Softmax statistics and
// accumulators are fp32; P is fed to the second MMA as a bf16 high part plus a bf16 residual, so the product keeps fp32-level
// accuracy.
#pragma once

#include "eta_common.cuh"

namespace eta {

constexpr int WARPS_PER_GROUP = 4;     // the four warps of a group each take a quarter of a tile's tokens

__device__ __forceinline__ uint32_t u4_get(const uint4& v, int i) {
    return i == 0 ? v.x : (i == 1 ? v.y : (i == 2 ? v.z : v.w));
}
// token row inside an 8-row group that MMA column n reads: bits 0 and 2 of n swapped, so that the two
// rows a quarter-warp touches in one 16-byte load sit in different halves of the swizzle pattern
__device__ __forceinline__ int rho(int n) { return (n & 2) | ((n & 1) << 2) | ((n >> 2) & 1); }
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// One warp's part.  Lane (g, t) = (lane / 4, lane % 4) holds head g's scores and statistics (its share of the sum l_run: tokens are
// spread over t), and heads 2 t and 2 t + 1 of the accumulators.  CHAINS = 2: a score is summed in two halves, so that a tile waits for
// half as many dependent MMAs (21 cycles each); for a kernel that is bound by a tile's latency (8 rows of 16K tokens 16.7 -> 16.2 us
// a step), not for one that streams (128K x 4 57.7 -> 58.0: registers).
template <int D, int TS, int CHAINS = 1>
struct Attend {
    static constexpr int HALVES = D / 64;
    static constexpr int WT = TS / WARPS_PER_GROUP;    // tokens per warp per tile (8 or 16)
    static constexpr int NT = WT / 8;                  // 8-token MMA column tiles per warp
    static constexpr int TILE_BYTES = TS * 128;        // one 64-column half tile; a stage holds K's halves, then V's
    static_assert(NT == 1 || NT == 2, "tile must give each warp 8 or 16 tokens");
    int g, t, rb, r0, r1, vchunk;
    bool head;
    // byte offsets inside a half tile of the 16-byte pieces this lane reads (fixed for the whole kernel)
    uint32_t koff[NT][2], voff[NT][2];
    uint32_t qa[HALVES][2][4];         // query fragments: head g's slice in the permuted head_dim order of the MMA
    float te;                          // head g's threshold
    float o[HALVES][4][4], m_run, l_run;

    __device__ __forceinline__ Attend(int lane, int warp, int G) {
        g = lane >> 2; t = lane & 3;
        head = g < G;
        rb = warp * WT;                                // first token row of this warp inside a tile
        r0 = rho(2 * t); r1 = rho(2 * t + 1);          // token rows (within an 8-group) of MMA columns 2t, 2t+1
        vchunk = ((g & 1) << 2) | (g >> 1);            // 16-byte chunk of a V half-row this lane reads
        te = 0.f;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const int krow = rb + nt * 8 + rho(g);
#pragma unroll
            for (int m = 0; m < 2; ++m) koff[nt][m] = krow * 128 + (((4 * m + t) ^ (krow & 7)) << 4);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int vrow = rb + nt * 8 + (c ? r1 : r0);
                voff[nt][c] = vrow * 128 + ((vchunk ^ (vrow & 7)) << 4);
            }
        }
        reset();
    }
    __device__ __forceinline__ void reset() {
        m_run = -INFINITY;
        l_run = 0.f;
#pragma unroll
        for (int hf = 0; hf < HALVES; ++hf)
#pragma unroll
            for (int mt = 0; mt < 4; ++mt)
#pragma unroll
                for (int c = 0; c < 4; ++c) o[hf][mt][c] = 0.f;
    }
    // q: head g's query (any valid row where there is no head g)
    __device__ __forceinline__ void load_q(const __nv_bfloat16* q) {
#pragma unroll
        for (int hf = 0; hf < HALVES; ++hf)
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                uint4 v = make_uint4(0, 0, 0, 0);
                if (head) v = __ldg(reinterpret_cast<const uint4*>(q + 64 * hf + 32 * m + 8 * t));
                qa[hf][m][0] = v.x; qa[hf][m][1] = v.y; qa[hf][m][2] = v.z; qa[hf][m][3] = v.w;
            }
    }
    // The tile at kbase: nvalid tokens of it are in the sequence, the heads of hmask attend it, token urow (0xff: none) keeps its
    // raw logit.  release() is called when the warp has read all of the tile.
    template <typename Release>
    __device__ __forceinline__ void tile(uint32_t kbase, int hmask, int urow, int nvalid, float scale, float beta, Release release) {
        constexpr float LOG2E = 1.4426950408889634f;
        const uint32_t vbase = kbase + HALVES * TILE_BYTES;
        // ---- S = q K^T for this warp's WT tokens: heads on M (rows 8..15 are padding), tokens on N
        float sacc[CHAINS][NT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int h = 0; h < CHAINS; ++h) sacc[h][nt][c] = 0.f;
        {
            uint4 kv[HALVES][2][NT];
#pragma unroll
            for (int hf = 0; hf < HALVES; ++hf)
#pragma unroll
                for (int m = 0; m < 2; ++m)
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) kv[hf][m][nt] = lds128(kbase + hf * TILE_BYTES + koff[nt][m]);
#pragma unroll
            for (int hf = 0; hf < HALVES; ++hf)
#pragma unroll
                for (int m = 0; m < 2; ++m)
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) {
                        mma_bf16_16816(sacc[0][nt], qa[hf][m][0], 0u, qa[hf][m][1], 0u, kv[hf][m][nt].x, kv[hf][m][nt].y);
                        mma_bf16_16816(sacc[CHAINS - 1][nt], qa[hf][m][2], 0u, qa[hf][m][3], 0u, kv[hf][m][nt].z, kv[hf][m][nt].w);
                    }
        }
        // V pieces are requested now so that their latency hides behind the softmax arithmetic
        uint4 v[HALVES][2 * NT];
#pragma unroll
        for (int hf = 0; hf < HALVES; ++hf)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int c = 0; c < 2; ++c) v[hf][nt * 2 + c] = lds128(vbase + hf * TILE_BYTES + voff[nt][c]);

        // ---- gate, mask, online softmax (lane (g,t) holds head g, tokens r0/r1 of each 8-group)
        const bool head_on = head && ((hmask >> g) & 1);
        float sg[NT][2];
        float bmax = -INFINITY;
        const bool gate_on = (te != -INFINITY);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int trow = rb + nt * 8 + (c ? r1 : r0);
                const float S = (CHAINS == 2 ? sacc[0][nt][c] + sacc[CHAINS - 1][nt][c] : sacc[0][nt][c]) * scale;
                float gated = S;
                if (gate_on) {
                    const float x = (beta == 0.f) ? 0.f : beta * (S - te);
                    gated = S * rcp_approx(1.f + exp2f(-x * LOG2E));      // S * sigmoid(x); exp2(+inf) -> rcp -> 0
                }
                if (trow == urow) gated = S;          // the query's own token (Eq. mult_attn, s = t)
                gated = (head_on && trow < nvalid) ? gated : -INFINITY;
                sg[nt][c] = gated;
                bmax = fmaxf(bmax, gated);
            }
        bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, 1));
        bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, 2));
        const float m_new = fmaxf(m_run, bmax);
        const float m_use = (m_new == -INFINITY) ? 0.f : m_new;
        const float alpha = (m_run == m_new) ? 1.f : exp2f((m_run - m_use) * LOG2E);   // m_run = -inf gives 0
        float p[NT][2], psum = 0.f;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                p[nt][c] = exp2f((sg[nt][c] - m_use) * LOG2E);   // -inf gives 0
                psum += p[nt][c];
            }
        l_run = l_run * alpha + psum;
        m_run = m_new;

        // accumulators hold heads 2t, 2t+1 in their columns: fetch those heads' rescale factors
        if (__any_sync(0xffffffffu, alpha != 1.f)) {
            const float al0 = __shfl_sync(0xffffffffu, alpha, 8 * t);
            const float al1 = __shfl_sync(0xffffffffu, alpha, 8 * t + 4);
#pragma unroll
            for (int hf = 0; hf < HALVES; ++hf)
#pragma unroll
                for (int mt = 0; mt < 4; ++mt) {
                    o[hf][mt][0] *= al0; o[hf][mt][1] *= al1; o[hf][mt][2] *= al0; o[hf][mt][3] *= al1;
                }
        }

        // ---- P as the B operand: bf16 high part and bf16 residual
        uint32_t pb_hi[2] = {0u, 0u}, pb_lo[2] = {0u, 0u};
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const __nv_bfloat162 hi = __floats2bfloat162_rn(p[nt][0], p[nt][1]);
            const float2 hf2 = __bfloat1622float2(hi);
            const __nv_bfloat162 lo = __floats2bfloat162_rn(p[nt][0] - hf2.x, p[nt][1] - hf2.y);
            pb_hi[nt] = *reinterpret_cast<const uint32_t*>(&hi);
            pb_lo[nt] = *reinterpret_cast<const uint32_t*>(&lo);
        }

        // ---- O^T += V^T P : head_dim on M, tokens on K, heads on N
        if (nvalid < TS) {
            // rows past the end of the sequence hold whatever the cache holds: keep them out of the product
#pragma unroll
            for (int hf = 0; hf < HALVES; ++hf)
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int c = 0; c < 2; ++c)
                        if (rb + nt * 8 + (c ? r1 : r0) >= nvalid) v[hf][nt * 2 + c] = make_uint4(0, 0, 0, 0);
        }
        // every shared-memory read of the tile has been issued before this point
        __syncwarp();
        release();
#pragma unroll
        for (int hf = 0; hf < HALVES; ++hf) {
#pragma unroll
            for (int mt = 0; mt < 4; ++mt) {
                const uint32_t xa = u4_get(v[hf][0], mt), xb = u4_get(v[hf][1], mt);
                const uint32_t a0 = __byte_perm(xa, xb, 0x5410), a1 = __byte_perm(xa, xb, 0x7632);
                uint32_t a2 = 0u, a3 = 0u;
                if (NT == 2) {
                    const uint32_t xc = u4_get(v[hf][2 * (NT - 1)], mt), xd = u4_get(v[hf][2 * (NT - 1) + 1], mt);
                    a2 = __byte_perm(xc, xd, 0x5410);
                    a3 = __byte_perm(xc, xd, 0x7632);
                }
                mma_bf16_16816(o[hf][mt], a0, a1, a2, a3, pb_hi[0], pb_hi[1]);
                mma_bf16_16816(o[hf][mt], a0, a1, a2, a3, pb_lo[0], pb_lo[1]);
            }
        }
    }
};

}  // namespace eta
