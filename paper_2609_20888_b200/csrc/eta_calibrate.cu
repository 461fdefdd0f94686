// Offline threshold calibration (appendix "Offline Threshold Calibration via
// 1/t-Weighted Histograms", Algorithm "Density-Matched Offline Threshold
// Calibration"): one pass over a calibration split builds, per query head, the
// 1/t-weighted histogram of the raw causal scores S_ts = s <q_t, k_s> and the
// density the dynamic thresholds realise; a bisection on the histogram then
// finds the static constant with the same density.
//
// calib_hist_kernel: a CTA per (128-query tile, head, sequence).  The scores of a
// 128 x 64 tile are a small dense contraction and go through the tensor cores
// (mma.m16n8k16, bf16 in, fp32 out; the whole pass is a few GFLOP, so nothing
// heavier is warranted); each score is binned into a histogram in shared memory.
// The causal row weight 1/t is added as the integer round(2^40 / t), so the
// histogram does not depend on the order in which the atomics land; the gates
// sigmoid(beta (S - tau_t)) are summed per row and reduced in a fixed order.
// calib_bisect_kernel: a CTA per head normalises the histogram and finds the root of
// g(c) = sum_b H[b] sigmoid(beta (s_b - c)) = dbar in double precision.
#include <type_traits>

#include "eta_common.cuh"

namespace eta {

constexpr int CAL_THREADS = 256;      // eight warps: 16 query rows each
constexpr int CAL_ROWS = CAL_THREADS / 2;       // queries per CTA
constexpr int CAL_KEYS = 64;          // keys per tile
constexpr int CAL_WSHIFT = 40;        // row weights are integers: round(2^40 / t)
constexpr int CAL_SPLIT = 16;         // bits of a weight that go to the histogram's low plane
constexpr int CAL_FLUSH = 512;        // keys after which the planes are emptied
constexpr int CAL_BISECT_THREADS = 512;

// Two fp32 values in a 64-bit register pair, as the packed fp32 instructions of sm_100 take them
__device__ __forceinline__ uint64_t pack2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t add2p(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t sub2p(uint64_t a, uint64_t b) {       // a - b as -1 * b + a: one rounding
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(b), "l"(pack2(-1.f, -1.f)), "l"(a));
    return r;
}
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_approx1(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// (no "memory" clobber: loads of the key tile may move across it; the histogram itself is only read behind barriers)
__device__ __forceinline__ void red_shared(uint32_t addr, uint32_t v) {
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(v));
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool in) {      // zeroes where !in
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
}

// What bounds it: latency and issue of c. 27 instructions per score (two of them atomics; 24 warps per SM at 80 registers,
// half of the issue slots used, tensor and special-function pipes at 30 %).  A row weight of up to 41 bits is added as two
// 32-bit numbers to two planes of the histogram, w mod 2^16 and w / 2^16: 32-bit shared atomics without a return value are
// native, a 64-bit one is a compare-and-swap loop.  Neither plane can wrap before it is emptied into the 64-bit histogram in
// memory: a row's weights sum to 2^40, so 128 rows put at most 2^31 into the high plane, and CAL_FLUSH = 512 keys of 128
// rows less than 2^32 into the low one.  16 x 1024 tokens, 32 heads, d = 128, 2048 bins: 470 us, against 1217 us with a
// 64-bit atomic, a double add and a true division per score.
template <int D>
__global__ void __launch_bounds__(CAL_THREADS, 3) calib_hist_kernel(
    const __nv_bfloat16* __restrict__ Q, const __nv_bfloat16* __restrict__ K, const float* __restrict__ tau,
    int Hq, int Hkv, int T, float c2, float scale, int n_bins, float s_min, float inv_w,
    unsigned long long* __restrict__ hist, double* __restrict__ dpart) {
    // padded row of the key tile: rows g and g + 1 start 64 bytes apart in the banks, so that the two rows a quarter-warp
    // touches in one 16-byte load never share a bank
    constexpr int KS = D + 32;
    constexpr int NP = D / 32;            // 16-byte pieces of a row per lane
    extern __shared__ __align__(16) unsigned char cal_raw[];
    __nv_bfloat16* sK = reinterpret_cast<__nv_bfloat16*>(cal_raw);               // two key tiles
    uint32_t* lo = reinterpret_cast<uint32_t*>(cal_raw + 2 * CAL_KEYS * KS * 2); // histogram: sums of w mod 2^16
    uint32_t* hi = lo + n_bins;                                                  // sums of w / 2^16
    __shared__ double s_red[CAL_THREADS / 32];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, tq = lane & 3;
    const int ttile = gridDim.x - 1 - blockIdx.x, h = blockIdx.y, x = blockIdx.z;      // the longest tiles start first
    const int hk = h / (Hq / Hkv);
    const int t0 = ttile * CAL_ROWS;
    const __nv_bfloat16* Qh = Q + (((int64_t)x * Hq + h) * T) * D;
    const __nv_bfloat16* Kh = K + (((int64_t)x * Hkv + hk) * T) * D;
    const float* tauh = tau + ((int64_t)x * Hq + h) * T;
    const int s_end = min(T, t0 + CAL_ROWS);          // keys of the CTA's longest row

    auto fetch = [&](int s0, int buf) {               // key tile -> shared memory; rows past the end read as zero
        const uint32_t dst = smem_u32(sK + buf * CAL_KEYS * KS);
#pragma unroll
        for (int u = 0; u < CAL_KEYS * (D / 8) / CAL_THREADS; ++u) {
            const int p = tid + u * CAL_THREADS, row = p / (D / 8), piece = p % (D / 8);
            const bool in = s0 + row < T;
            cp_async16(dst + (row * KS + piece * 8) * 2, Kh + (int64_t)(in ? s0 + row : 0) * D + piece * 8, in);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    fetch(0, 0);
    for (int b = tid; b < 2 * n_bins; b += CAL_THREADS) lo[b] = 0u;

    // this thread's two query rows and their A fragments: piece m of a lane is the coordinates 8 (4 m + tq) .. + 7, the
    // same ones its 16-byte load of a key covers (a dot product does not care about the order of k)
    const int rw = t0 + warp * 16, r0 = rw + g, r1 = r0 + 8;
    uint4 qa[NP], qb[NP];
#pragma unroll
    for (int m = 0; m < NP; ++m) {
        const int c = 8 * (4 * m + tq);
        qa[m] = (r0 < T) ? __ldg(reinterpret_cast<const uint4*>(Qh + (int64_t)r0 * D + c)) : make_uint4(0, 0, 0, 0);
        qb[m] = (r1 < T) ? __ldg(reinterpret_cast<const uint4*>(Qh + (int64_t)r1 * D + c)) : make_uint4(0, 0, 0, 0);
    }
    const float tau0 = (r0 < T) ? tauh[r0] : 0.f, tau1 = (r1 < T) ? tauh[r1] : 0.f;
    // t counts from 1: row index r is decoding step t = r + 1
    const unsigned long long w0 = (((1ull << CAL_WSHIFT) + (unsigned)(r0 + 1) / 2) / (unsigned)(r0 + 1));
    const unsigned long long w1 = (((1ull << CAL_WSHIFT) + (unsigned)(r1 + 1) / 2) / (unsigned)(r1 + 1));
    const uint32_t wl[2] = {(uint32_t)w0 & ((1u << CAL_SPLIT) - 1), (uint32_t)w1 & ((1u << CAL_SPLIT) - 1)};
    const uint32_t wh[2] = {(uint32_t)(w0 >> CAL_SPLIT), (uint32_t)(w1 >> CAL_SPLIT)};
    const uint64_t one2 = pack2(1.f, 1.f);
    // Sums of the two rows' gates (even and odd keys apart) as value + error: Dekker's sum, exact because the value starts
    // at 1 and never falls below a gate.  Twice fp32's precision on the fp32 pipe; a conversion to double and a double add
    // per gate would take four times as long.
    uint64_t gs[2] = {one2, one2}, ge[2] = {pack2(0.f, 0.f), pack2(0.f, 0.f)};
    const float b_max = (float)n_bins - 0.5f;
    const uint32_t lo_addr = smem_u32(lo) - (0x4B000000u << 2), hi_off = (uint32_t)n_bins * 4;

    auto add = [&](float y, int row) {
        // floor(y) sits in the low bits of 2^23 + y rounded down; the exponent bits are folded into lo_addr
        const float f = __fadd_rd(fminf(fmaxf(y, 0.f), b_max), 8388608.f);
        const uint32_t addr = lo_addr + (__float_as_uint(f) << 2);
        red_shared(addr, wl[row]);
        red_shared(addr + hi_off, wh[row]);
    };
    auto tile = [&](int s0, int buf, auto masked) {
        constexpr bool MASK = decltype(masked)::value;
        // two 8-key MMA tiles at a time: independent chains for the tensor cores and the arithmetic behind them
#pragma unroll 1
        for (int nn = 0; nn < CAL_KEYS / 8; nn += 2) {
            float acc[2][4];
            const __nv_bfloat16* krow = sK + (buf * CAL_KEYS + nn * 8 + g) * KS + 8 * tq;
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[u][c] = 0.f;
#pragma unroll
            for (int m = 0; m < NP; ++m) {
                const uint4 k0 = *reinterpret_cast<const uint4*>(krow + 32 * m);
                const uint4 k1 = *reinterpret_cast<const uint4*>(krow + 8 * KS + 32 * m);
                mma_bf16_16816(acc[0], qa[m].x, qb[m].x, qa[m].y, qb[m].y, k0.x, k0.y);
                mma_bf16_16816(acc[1], qa[m].x, qb[m].x, qa[m].y, qb[m].y, k1.x, k1.y);
                mma_bf16_16816(acc[0], qa[m].z, qb[m].z, qa[m].w, qb[m].w, k0.z, k0.w);
                mma_bf16_16816(acc[1], qa[m].z, qb[m].z, qa[m].w, qb[m].w, k1.z, k1.w);
            }
            // acc[u][0], acc[u][1]: row r0, keys col, col + 1; acc[u][2], acc[u][3]: row r1
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int col = s0 + (nn + u) * 8 + 2 * tq;
#pragma unroll
                for (int row = 0; row < 2; ++row) {
                    const int r = row ? r1 : r0;
                    const float tr = row ? tau1 : tau0;
                    const uint64_t S = mul2(pack2(acc[u][2 * row], acc[u][2 * row + 1]), pack2(scale, scale));
                    // the gate 1 / (1 + 2^y), y = -beta log2(e) (S - tau)
                    const float2 y = unpack2(mul2(sub2p(S, pack2(tr, tr)), pack2(c2, c2)));
                    float ma = rcp_approx1(1.f + ex2_approx(y.x)), mb = rcp_approx1(1.f + ex2_approx(y.y));
                    if (MASK) { ma = (r < T && col <= r) ? ma : 0.f; mb = (r < T && col + 1 <= r) ? mb : 0.f; }
                    const uint64_t m = pack2(ma, mb), sum = add2p(gs[row], m);
                    ge[row] = add2p(ge[row], sub2p(m, sub2p(sum, gs[row])));
                    gs[row] = sum;
                    const float2 bin = unpack2(mul2(sub2p(S, pack2(s_min, s_min)), pack2(inv_w, inv_w)));
                    if (!MASK || (r < T && col <= r)) add(bin.x, row);
                    if (!MASK || (r < T && col + 1 <= r)) add(bin.y, row);
                }
            }
        }
    };
    auto flush = [&]() {
        for (int b = tid; b < n_bins; b += CAL_THREADS) {
            const unsigned long long v = ((unsigned long long)hi[b] << CAL_SPLIT) + lo[b];
            if (v) {
                atomicAdd(&hist[(int64_t)h * n_bins + b], v);
                lo[b] = 0u; hi[b] = 0u;
            }
        }
    };
    for (int s0 = 0, buf = 0; s0 < s_end; s0 += CAL_KEYS, buf ^= 1) {
        // one barrier per tile: every thread's copies of this tile have landed, every warp is through with the one before,
        // whose buffer the next tile's copies may have
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        if (s0 && s0 % CAL_FLUSH == 0) { flush(); __syncthreads(); }
        if (s0 + CAL_KEYS < s_end) fetch(s0 + CAL_KEYS, buf ^ 1);
        // a warp whose rows all lie past the tile counts every score; one whose rows end before it none
        if (s0 + CAL_KEYS - 1 <= rw && rw + 16 <= T) tile(s0, buf, std::false_type{});
        else if (s0 <= rw + 15 && rw < T) tile(s0, buf, std::true_type{});
    }
    __syncthreads();
    // density contribution of this tile: sum over its rows of (1/t) * (sum of the row's gates), fixed order
    double dsum = 0.0;
#pragma unroll
    for (int row = 0; row < 2; ++row) {
        const float2 v = unpack2(gs[row]), e = unpack2(ge[row]);
        const int r = row ? r1 : r0;
        if (r < T) dsum += (((double)v.x - 1.0) + ((double)v.y - 1.0) + ((double)e.x + (double)e.y)) / (double)(r + 1);
    }
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) dsum += __shfl_xor_sync(0xffffffffu, dsum, s);
    if (lane == 0) s_red[warp] = dsum;
    flush();
    __syncthreads();
    if (tid == 0) {
        double tot = 0.0;
        for (int w = 0; w < CAL_THREADS / 32; ++w) tot += s_red[w];
        dpart[((int64_t)x * Hq + h) * gridDim.x + ttile] = tot;
    }
}

__device__ __forceinline__ double sigmoid_d(double v) {
    if (v >= 0) return 1.0 / (1.0 + exp(-v));
    const double e = exp(v);
    return e / (1.0 + e);
}

// Fixed-order sums of two values per thread over the block; every thread gets the results.
__device__ __forceinline__ double2 block_sum2_fixed(double a, double b, double2* scratch) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, s);
        b += __shfl_xor_sync(0xffffffffu, b, s);
    }
    __syncthreads();                       // the previous sums have been read
    if (lane == 0) scratch[warp] = make_double2(a, b);
    __syncthreads();
    double2 r = make_double2(0.0, 0.0);
#pragma unroll
    for (int w = 0; w < CAL_BISECT_THREADS / 32; ++w) { r.x += scratch[w].x; r.y += scratch[w].y; }
    return r;
}

// A serial chain of evaluations of g, each n_bins double-precision sigmoids: what counts is how many there are.  The root
// is found by Newton steps inside a bracket, with a halving wherever a step would leave the bracket or shrink too slowly:
// about eight evaluations to double precision where plain halving took eighty (177 -> 55 us; a first approximation in fp32 ahead of them gained nothing).
__global__ void __launch_bounds__(CAL_BISECT_THREADS) calib_bisect_kernel(
    const unsigned long long* __restrict__ hist, const double* __restrict__ dpart, int Hq, int n_seq, int n_ttiles,
    int T, int n_bins, double s_min, double s_max, double beta, int iters, float* __restrict__ head_const,
    float* __restrict__ dbar_out, double* __restrict__ head_const_d) {
    extern __shared__ unsigned char bis_raw[];
    double* Hn = reinterpret_cast<double*>(bis_raw);
    __shared__ double2 scratch[CAL_BISECT_THREADS / 32];
    __shared__ unsigned long long s_tot[CAL_BISECT_THREADS / 32];
    const int tid = threadIdx.x, h = blockIdx.x;
    const unsigned long long* Hh = hist + (int64_t)h * n_bins;

    // total weight (an integer: exact whatever the order), then the normalised histogram
    unsigned long long part = 0;
    for (int b = tid; b < n_bins; b += CAL_BISECT_THREADS) part += Hh[b];
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) part += __shfl_xor_sync(0xffffffffu, part, s);
    if ((tid & 31) == 0) s_tot[tid >> 5] = part;
    __syncthreads();
    part = 0;
#pragma unroll
    for (int w = 0; w < CAL_BISECT_THREADS / 32; ++w) part += s_tot[w];
    const double tot = (double)part;
    for (int b = tid; b < n_bins; b += CAL_BISECT_THREADS) Hn[b] = tot > 0.0 ? (double)Hh[b] / tot : 0.0;
    // target density: partial sums of every (sequence, tile) of this head, in a fixed order
    double d = 0.0;
    for (int k = tid; k < n_seq * n_ttiles; k += CAL_BISECT_THREADS) {
        const int x = k / n_ttiles, tt = k % n_ttiles;
        d += dpart[((int64_t)x * Hq + h) * n_ttiles + tt];
    }
    const double target = block_sum2_fixed(d, 0.0, scratch).x / ((double)n_seq * (double)T);

    // every thread follows the same iteration on the same sums
    const double w = (s_max - s_min) / n_bins;
    double lo = s_min - 40.0 / beta, hi = s_max + 40.0 / beta;
    double c = 0.5 * (lo + hi), dx_old = hi - lo, dx = dx_old;
    for (int it = 0; it < iters; ++it) {
        double gs = 0.0, ds = 0.0;
        for (int b = tid; b < n_bins; b += CAL_BISECT_THREADS) {
            const double sg = sigmoid_d(beta * (s_min + (b + 0.5) * w - c));
            gs += Hn[b] * sg;
            ds += Hn[b] * (sg * (1.0 - sg));
        }
        const double2 r = block_sum2_fixed(gs, ds, scratch);
        const double f = r.x - target, slope = beta * r.y;      // g falls with c: g' = -slope
        if (r.x > target) lo = c; else hi = c;
        const double cn = c + f / slope;
        double next;
        if (slope > 0.0 && cn > lo && cn < hi && 2.0 * fabs(f) <= fabs(dx_old * slope)) {
            dx_old = dx; dx = cn - c; next = cn;
        } else {
            dx_old = dx; dx = 0.5 * (hi - lo); next = lo + dx;
        }
        const bool done = next == c || fabs(dx) <= 1e-15 * (fabs(lo) + fabs(hi) + w);
        c = next;
        if (done) break;
    }
    if (tid == 0) {
        head_const[h] = (float)c;
        if (dbar_out) dbar_out[h] = (float)target;
        if (head_const_d) head_const_d[h] = c;
    }
}

static size_t cal_align(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace eta

extern "C" {

int eta_calibration_workspace_bytes(int32_t n_seq, int32_t seq_len, int32_t n_q_heads, int32_t n_bins,
                                    size_t* out_bytes) {
    if (!out_bytes || n_seq <= 0 || seq_len <= 0 || n_q_heads <= 0 || n_bins < 2) return ETA_ERR_INVALID_ARG;
    const size_t n_ttiles = (size_t)(seq_len + eta::CAL_ROWS - 1) / eta::CAL_ROWS;
    *out_bytes = eta::cal_align(sizeof(unsigned long long) * (size_t)n_q_heads * n_bins) +
                 eta::cal_align(sizeof(double) * (size_t)n_seq * n_q_heads * n_ttiles) +
                 eta::cal_align(sizeof(double) * (size_t)n_q_heads);
    return ETA_OK;
}

int eta_calibrate_head_const(int32_t n_seq, int32_t seq_len, int32_t n_q_heads, int32_t n_kv_heads, int32_t head_dim,
                             const void* Q, const void* K, const float* tau, float beta, float scale, int32_t n_bins,
                             float s_min, float s_max, float* head_const, float* dbar, void* workspace,
                             size_t workspace_bytes, void* stream) {
    using namespace eta;
    if (!Q || !K || !tau || !head_const) return ETA_ERR_INVALID_ARG;
    if (n_seq <= 0 || seq_len <= 0 || n_q_heads <= 0 || n_kv_heads <= 0 || n_q_heads % n_kv_heads != 0)
        return ETA_ERR_INVALID_ARG;
    if (!(beta > 0.f) || !(s_max > s_min) || n_bins < 2) return ETA_ERR_INVALID_ARG;
    if ((head_dim != 64 && head_dim != 128) || n_bins > 4096 || n_seq > 65535 || n_q_heads > 65535)
        return ETA_ERR_UNSUPPORTED;
    if ((int64_t)n_seq * seq_len > (1ll << 22)) return ETA_ERR_UNSUPPORTED;        // keeps the integer weights in 64 bits
    if ((reinterpret_cast<uintptr_t>(Q) | reinterpret_cast<uintptr_t>(K)) & 15) return ETA_ERR_UNSUPPORTED;
    size_t need = 0;
    int rc = eta_calibration_workspace_bytes(n_seq, seq_len, n_q_heads, n_bins, &need);
    if (rc != ETA_OK) return rc;
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) || workspace_bytes < need) return ETA_ERR_WORKSPACE;

    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int n_ttiles = (seq_len + CAL_ROWS - 1) / CAL_ROWS;
    unsigned char* ws = static_cast<unsigned char*>(workspace);
    unsigned long long* hist = reinterpret_cast<unsigned long long*>(ws);
    const size_t hist_bytes = cal_align(sizeof(unsigned long long) * (size_t)n_q_heads * n_bins);
    double* dpart = reinterpret_cast<double*>(ws + hist_bytes);
    double* hc_d = reinterpret_cast<double*>(ws + hist_bytes + cal_align(sizeof(double) * (size_t)n_seq * n_q_heads * n_ttiles));
    cudaError_t e = cudaMemsetAsync(hist, 0, hist_bytes, s);
    if (e != cudaSuccess) { set_cuda_error(e, "calibration memset"); return ETA_ERR_CUDA; }

    const float sc = scale > 0.f ? scale : 1.0f / sqrtf((float)head_dim);
    const float inv_w = (float)n_bins / (s_max - s_min);
    const dim3 grid((unsigned)n_ttiles, (unsigned)n_q_heads, (unsigned)n_seq);
    const float c2 = (float)(-(double)beta * 1.4426950408889634);      // exp(-beta x) = 2^(c2 x)
    const size_t smem = (size_t)2 * CAL_KEYS * (head_dim + 32) * 2 + sizeof(unsigned long long) * (size_t)n_bins;
    auto Qp = static_cast<const __nv_bfloat16*>(Q);
    auto Kp = static_cast<const __nv_bfloat16*>(K);
    if (head_dim == 128) {
        rc = configure_kernel(reinterpret_cast<const void*>(calib_hist_kernel<128>), 80 * 1024);
        if (rc != ETA_OK) return rc;
        calib_hist_kernel<128><<<grid, CAL_THREADS, smem, s>>>(Qp, Kp, tau, n_q_heads, n_kv_heads, seq_len, c2, sc,
                                                               n_bins, s_min, inv_w, hist, dpart);
    } else {
        rc = configure_kernel(reinterpret_cast<const void*>(calib_hist_kernel<64>), 80 * 1024);
        if (rc != ETA_OK) return rc;
        calib_hist_kernel<64><<<grid, CAL_THREADS, smem, s>>>(Qp, Kp, tau, n_q_heads, n_kv_heads, seq_len, c2, sc,
                                                              n_bins, s_min, inv_w, hist, dpart);
    }
    rc = check_launch("calibration histogram");
    if (rc != ETA_OK) return rc;
    calib_bisect_kernel<<<n_q_heads, CAL_BISECT_THREADS, sizeof(double) * (size_t)n_bins, s>>>(
        hist, dpart, n_q_heads, n_seq, n_ttiles, seq_len, n_bins, (double)s_min, (double)s_max, (double)beta, 160,
        head_const, dbar, hc_d);
    return check_launch("calibration bisection");
}

}  // extern "C"
