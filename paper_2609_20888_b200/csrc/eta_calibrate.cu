// Offline threshold calibration (appendix "Offline Threshold Calibration via
// 1/t-Weighted Histograms", Algorithm "Density-Matched Offline Threshold
// Calibration"): one pass over a calibration split builds, per query head, the
// 1/t-weighted histogram of the raw causal scores S_ts = s <q_t, k_s> and the
// density the dynamic thresholds realise; a root search on the histogram then
// finds the static constant with the same density.
//
// calib_hist_kernel: a CTA per (128-query tile, head, sequence).  The scores of a
// 128 x 64 tile are a small dense contraction and go through the tensor cores
// (tcgen05, bf16 in, fp32 accumulators in tensor memory); each score is binned into a histogram in shared memory.
// The causal row weight 1/t is added as the integer round(2^40 / t), so the
// histogram does not depend on the order in which the atomics land; the gates
// sigmoid(beta (S - tau_t)) are summed per row and reduced in a fixed order.
// calib_bisect_kernel: a CTA per head normalises the histogram and finds the root of
// g(c) = sum_b H[b] sigmoid(beta (s_b - c)) = dbar in double precision.
#include <type_traits>

#include "eta_common.cuh"

namespace eta {

constexpr int CAL_ROWS = 128;         // queries per CTA: the rows of an MMA tile
constexpr int CAL_WARPS = 8;          // warps that count: a thread has one row and half of a tile's keys
constexpr int CAL_THREADS = 32 * (CAL_WARPS + 1);       // ... and one that loads tiles and issues MMAs
constexpr int CAL_KEYS = 64;          // keys per tile
constexpr int CAL_TMEM = 128;         // columns of tensor memory: up to 64 for the queries, 64 for the scores of a tile
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

// ---- 5th-generation tensor core (one CTA): 128 query rows x CAL_KEYS keys, bf16 in, fp32 accumulators in tensor memory
// Shared-memory operand in the layout the copies leave: rows of 128 bytes, 128-byte swizzle, eight rows (1024 bytes) to a group
__device__ __forceinline__ uint64_t umma_operand(uint32_t addr) {
    return (uint64_t)((addr & 0x3ffffu) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// fp32 accumulator, bf16 x bf16, both operands with k contiguous, N = CAL_KEYS, M = CAL_ROWS; A in tensor memory
constexpr uint32_t CAL_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((CAL_KEYS >> 3) << 17) | ((CAL_ROWS >> 4) << 24);
__device__ __forceinline__ void umma_bf16(uint32_t acc, uint32_t a, uint64_t b, uint32_t idesc, bool accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(acc), "r"(a), "l"(b), "r"(idesc), "r"((uint32_t)accumulate) : "memory");
}
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
// mbar_wait for a warp that others wait for: no sleep between two polls
__device__ __forceinline__ bool mbar_spin(uint64_t* bar, uint32_t parity) {
    for (uint32_t it = 0; it < WAIT_LIMIT; ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
// arrives on the barrier when every MMA issued so far has completed
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tmem_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
// 16 lanes x 32 columns: rows lane / 4 and lane / 4 + 8; v[4 k + 0, 1] are columns 8 k + 2 (lane % 4) + 0, 1 of the first of
// the two rows, v[4 k + 2, 3] those of the second
__device__ __forceinline__ void tmem_load_16x32(uint32_t addr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]) : "r"(addr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int c = 0; c < 16; ++c) v[c] = __uint_as_float(r[c]);
}

// 32 bf16 of this thread's lane (32 lanes per warp) as 16 columns
__device__ __forceinline__ void tmem_store16(uint32_t addr, const uint4 (&q)[4]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(addr), "r"(q[0].x), "r"(q[0].y), "r"(q[0].z), "r"(q[0].w), "r"(q[1].x), "r"(q[1].y), "r"(q[1].z), "r"(q[1].w),
          "r"(q[2].x), "r"(q[2].y), "r"(q[2].z), "r"(q[2].w), "r"(q[3].x), "r"(q[3].y), "r"(q[3].z), "r"(q[3].w) : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

template <int D>
struct CalSmem {
    static constexpr int K_BYTES = CAL_KEYS * D * 2;
    static constexpr int copies(int n_bins) { return n_bins <= 2048 ? 2 : 1; }
    static constexpr size_t bytes(int n_bins) { return 1024 + 2 * K_BYTES + 8 * (size_t)n_bins * copies(n_bins); }
};

// Clears the histogram (512 KB at 32 heads x 2048 bins: latency).  A kernel of its own, not a memset: the next one is launched
// while it runs and waits for it only when it adds to the histogram.  Calibrations of 16 x 1024 tokens (32 / 8 heads, d = 128, 2048
// bins, as all figures here) 310.2 -> 307.2 us, 8 x 700 103.4 -> 101.6, 2 x 64 21.8 -> 20.2.  It is itself launched while the kernel
// before it ends, which counts where calibrations are queued one after the other (8 x 700 101.6 -> 99.6, 8 x 128 22.7 -> 20.7, 2 x 64
// 20.2 -> 18.1) and not for one by itself (22.5 for 2 x 64 either way).
__global__ void __launch_bounds__(256) calib_clear_kernel(uint4* __restrict__ p, int n16) {
    pdl_wait();          // the next kernel reads the call's inputs at once: all before this one has to be complete first
    pdl_trigger();
    const int k = blockIdx.x * 256 + threadIdx.x;
    if (k < n16) p[k] = make_uint4(0, 0, 0, 0);
}

// What bounds it: the shared-memory pipe (90 % of its passes), by the two atomics of a score: 3.55 passes each, which is what
// 32 lanes on random banks take.  A row weight of up to 41 bits is added as two 32-bit numbers to two planes of the histogram,
// w mod 2^16 and w / 2^16: 32-bit shared atomics without a return value are native, a 64-bit one is a compare-and-swap loop
// (19 cycles a warp and SM), and one that returns the sum, to pass on carries, is no faster than two that do not.  Neither
// plane can wrap before it is emptied into the 64-bit histogram in memory: a row's weights sum to 2^40, so 128 rows put at
// most 2^31 into the high plane, and CAL_FLUSH = 512 keys of 128 rows less than 2^32 into the low one.
// Everything else is kept off that pipe.  Fragments for mma.sync were 37 of its 102 million passes at 16 x 1024 tokens, 32
// heads, d = 128 (all of it 435 us): now keys go to the tensor core by bulk copy and descriptor, scores come back through
// tensor memory, and the queries sit there too (as an operand in shared memory they were read again for every tile: 14
// million passes, 4.7 are left).  One accumulator of 64 keys: the MMA of a tile runs while the second half of the tile before
// it is counted.  Two of 32 keys with a barrier each (347 us a calibration, against 313) cost more than they hide, two of 64
// do not fit the tensor memory of three CTAs beside the queries.  Four CTAs at 56 registers: 321.  Up to 2048 bins the planes have two
// copies, on even and on odd banks, for even and for odd lanes: 3.46 passes an atomic instead of 3.56 for scores spread over a
// hundred bins and more, and half as many where they crowd (all scores in one bin, 4 x 1024 tokens: 546 -> 288 us).  The MMAs are issued from
// a warp that walks along as a whole, their descriptors in uniform registers: 100 cycles a tile, not 600.  With 2048 bins: 515 -> 333
// (queries in shared memory) -> 313 us, of which the histogram 435 -> 290; with the launches and the root of today 305, with both of
// these 302.5.  Within 1 % of that: gates in fours over one reciprocal; two CTAs of three groups of warps that count tiles of their
// own.  What would count for more is fewer passes, but a byte per row and bin takes the shared memory of a whole SM.
template <int D, int COPIES>
__global__ void __launch_bounds__(CAL_THREADS, 3) calib_hist_kernel(
    const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, const float* __restrict__ tau,
    int Hq, int Hkv, int T, float c2, float scale, int n_bins, float s_min, float inv_w,
    unsigned long long* __restrict__ hist, double* __restrict__ dpart) {
    using L = CalSmem<D>;
    extern __shared__ unsigned char cal_raw[];
    unsigned char* sK = cal_raw + ((1024 - (smem_u32(cal_raw) & 1023)) & 1023);       // two key tiles, first of all the queries
    uint32_t* lo = reinterpret_cast<uint32_t*>(sK + 2 * L::K_BYTES);   // histogram: sums of w mod 2^16
    uint32_t* hi = lo + COPIES * n_bins;                                        // sums of w / 2^16
    __shared__ double s_red[CAL_WARPS];
    __shared__ __align__(8) uint64_t bar_q, bar_in[2], bar_acc, bar_free;      // queries, keys arrived; scores complete; ... read by all
    __shared__ uint32_t s_tmem;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int h = blockIdx.x, x = blockIdx.y, ttile = gridDim.z - 1 - blockIdx.z;      // the longest tiles start first
    const int t0 = ttile * CAL_ROWS;
    const int n_tiles = (min(T, t0 + CAL_ROWS) + CAL_KEYS - 1) / CAL_KEYS;              // up to the CTA's longest row

    if (warp == CAL_WARPS) {
        if (lane == 0) {
            for (uint64_t* b : {&bar_q, &bar_in[0], &bar_in[1], &bar_acc}) mbar_init(b, 1);
            mbar_init(&bar_free, CAL_WARPS);
            fence_barrier_init();
            mbar_arrive_expect_tx(&bar_q, 2 * L::K_BYTES);
            tma_load_4d(sK, &tmQ, 0, t0, 0, x * Hq + h, &bar_q);
        }
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&s_tmem)), "r"(CAL_TMEM) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int b = tid; b < 2 * COPIES * n_bins; b += CAL_THREADS) lo[b] = 0u;
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    const uint32_t tmem = s_tmem, tmem_acc = tmem + CAL_TMEM - CAL_KEYS;
    double dsum = 0.0;
    bool ok = true;
    if (warp < CAL_ROWS / 32) {             // the queries into tensor memory, a row per lane
        ok = __all_sync(0xffffffffu, mbar_wait(&bar_q, 0));
        const int row = warp * 32 + lane;
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
            uint4 q[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                q[u] = *reinterpret_cast<const uint4*>(sK + (c / 2) * (CAL_ROWS * 128) + row * 128 + ((((c & 1) * 4 + u) ^ (row & 7)) << 4));
            tmem_store16(tmem + ((uint32_t)(warp * 32) << 16) + 16 * c, q);
        }
        fence_proxy_async();
        tmem_fence_before();
    }
    __syncthreads();
    tmem_fence_after();

    // by threads that count only, all of them
    auto flush = [&]() {
        pdl_wait();          // the histogram in memory has been cleared
        for (int b = tid; b < n_bins; b += 32 * CAL_WARPS) {
            unsigned long long v;
            if constexpr (COPIES == 2) {
                const uint2 l = reinterpret_cast<const uint2*>(lo)[b], u = reinterpret_cast<const uint2*>(hi)[b];
                v = (((unsigned long long)u.x + u.y) << CAL_SPLIT) + l.x + l.y;
            } else {
                v = ((unsigned long long)hi[b] << CAL_SPLIT) + lo[b];
            }
            if (v) {
                atomicAdd(&hist[(int64_t)h * n_bins + b], v);
                if constexpr (COPIES == 2) reinterpret_cast<uint2*>(lo)[b] = reinterpret_cast<uint2*>(hi)[b] = make_uint2(0u, 0u);
                else lo[b] = hi[b] = 0u;
            }
        }
    };
    auto meet = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(32 * CAL_WARPS) : "memory"); };

    if (warp == CAL_WARPS) {
        // The whole warp walks along and one lane issues: what an MMA takes (its descriptors) is then computed by the uniform
        // datapath.
        const int hk = x * Hkv + h / (Hq / Hkv);
        const uint64_t keys_0 = umma_operand(smem_u32(sK));
        auto load = [&](int i) {
            mbar_arrive_expect_tx(&bar_in[i & 1], L::K_BYTES);
            tma_load_4d(sK + (i & 1) * L::K_BYTES, &tmK, 0, i * CAL_KEYS, 0, hk, &bar_in[i & 1]);
        };
        auto wait = [&](uint64_t* bar, uint32_t parity) { return __all_sync(0xffffffffu, mbar_spin(bar, parity)) != 0; };
        if (elect_one()) load(0);
        int issued = 0;                                // tiles whose MMAs are under way or complete
        for (int i = 0; i < n_tiles; ++i) {
            // a wait that runs out: nothing more is issued; what is still on its way gets as long again
            if (!wait(&bar_in[i & 1], (i >> 1) & 1)) { wait(&bar_in[i & 1], (i >> 1) & 1); break; }
            if (i > 0 && !wait(&bar_free, (i - 1) & 1)) break;
            tmem_fence_after();
            const uint64_t keys = keys_0 + (uint32_t)((i & 1) * (L::K_BYTES >> 4));
            if (elect_one()) {
#pragma unroll
                for (int k = 0; k < D / 16; ++k)       // 16 columns: 32 bytes along the swizzled row of a 64-column half
                    umma_bf16(tmem_acc, tmem + 8 * k, keys + (k / 4) * (CAL_KEYS * 128 >> 4) + (k % 4) * 2, CAL_IDESC, k > 0);
                umma_commit(&bar_acc);
                if (i + 1 < n_tiles) load(i + 1);      // the scores of the tile before are complete: its keys have been read
            }
            ++issued;
        }
        // the counting warps have waited for the last tile already, unless their wait ran out: the MMAs get as long again
        // before the tensor memory is given back
        if (issued) mbar_wait(&bar_acc, (issued - 1) & 1);
        __syncwarp();
    } else {
        const int l16 = (warp & 3) * 32 + (warp >> 2) * 16;      // the warp's 16 lanes of tensor memory
        const int rw = t0 + l16, r0 = rw + (lane >> 2), r1 = r0 + 8;
        const float* tauh = tau + ((int64_t)x * Hq + h) * T;
        const float tau0 = (r0 < T) ? tauh[r0] : 0.f, tau1 = (r1 < T) ? tauh[r1] : 0.f;
        // t counts from 1: row index r is decoding step t = r + 1
        const unsigned long long w0 = (((1ull << CAL_WSHIFT) + (unsigned)(r0 + 1) / 2) / (unsigned)(r0 + 1));
        const unsigned long long w1 = (((1ull << CAL_WSHIFT) + (unsigned)(r1 + 1) / 2) / (unsigned)(r1 + 1));
        const uint32_t wl[2] = {(uint32_t)w0 & ((1u << CAL_SPLIT) - 1), (uint32_t)w1 & ((1u << CAL_SPLIT) - 1)};
        const uint32_t wh[2] = {(uint32_t)(w0 >> CAL_SPLIT), (uint32_t)(w1 >> CAL_SPLIT)};
        // Sums of the two rows' gates (even and odd keys apart) as value + error: Dekker's sum, exact because the value
        // starts at 1 and never falls below a gate.  Twice fp32's precision on the fp32 pipe; a conversion to double and a
        // double add per gate would take four times as long.
        const uint64_t one2 = pack2(1.f, 1.f);
        uint64_t gs[2] = {one2, one2}, ge[2] = {pack2(0.f, 0.f), pack2(0.f, 0.f)};
        const float b_max = (float)n_bins - 0.5f;
        constexpr int SHIFT = COPIES == 2 ? 3 : 2;
        const uint32_t lo_addr = smem_u32(lo) + (COPIES == 2 ? 4 * (lane & 1) : 0) - (0x4B000000u << SHIFT), hi_off = (uint32_t)n_bins * 4 * COPIES;

        auto add = [&](float y, int row) {
            // floor(y) sits in the low bits of 2^23 + y rounded down; the exponent bits are folded into lo_addr
            const float f = __fadd_rd(fminf(fmaxf(y, 0.f), b_max), 8388608.f);
            const uint32_t addr = lo_addr + (__float_as_uint(f) << SHIFT);
            red_shared(addr, wl[row]);
            red_shared(addr + hi_off, wh[row]);
        };
        auto count = [&](const float (&acc)[16], int key, auto masked) {
            constexpr bool MASK = decltype(masked)::value;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int row = u & 1, r = row ? r1 : r0, col = key + (u / 2) * 8 + 2 * (lane & 3);
                const float tr = row ? tau1 : tau0;
                const uint64_t S = mul2(pack2(acc[2 * u], acc[2 * u + 1]), pack2(scale, scale));
                // the gate 1 / (1 + 2^y), y = -beta log2(e) (S - tau)
                const float2 y = unpack2(mul2(sub2p(S, pack2(tr, tr)), pack2(c2, c2)));
                float ma = rcp_approx1(1.f + ex2_approx(y.x)), mb = rcp_approx1(1.f + ex2_approx(y.y));
                const bool in_a = !MASK || (r < T && col <= r), in_b = !MASK || (r < T && col + 1 <= r);
                if (MASK) { ma = in_a ? ma : 0.f; mb = in_b ? mb : 0.f; }
                const uint64_t m = pack2(ma, mb), sum = add2p(gs[row], m);
                ge[row] = add2p(ge[row], sub2p(m, sub2p(sum, gs[row])));
                gs[row] = sum;
                const float2 bin = unpack2(mul2(sub2p(S, pack2(s_min, s_min)), pack2(inv_w, inv_w)));
                if (in_a) add(bin.x, row);
                if (in_b) add(bin.y, row);
            }
        };
        for (int i = 0; i < n_tiles; ++i) {
            if (i && i * CAL_KEYS % CAL_FLUSH == 0) { meet(); flush(); meet(); }
            ok = ok && mbar_wait(&bar_acc, i & 1);
            ok = __all_sync(0xffffffffu, ok);
            tmem_fence_after();
#pragma unroll 1
            for (int c = 0; c < CAL_KEYS; c += 32) {
                const int key = i * CAL_KEYS + c;
                const bool some = ok && key <= rw + 15 && rw < T;          // a warp whose rows end before the keys counts none
                float acc[16];
                if (some) tmem_load_16x32(tmem_acc + ((uint32_t)l16 << 16) + c, acc);
                if (c + 32 == CAL_KEYS) {          // the next tile's MMA runs while these are counted
                    tmem_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bar_free);
                }
                if (!some) continue;
                if (key + 31 <= rw && rw + 16 <= T) count(acc, key, std::false_type{});      // ... all past them: every score
                else count(acc, key, std::true_type{});
            }
        }
        meet();
        flush();
        pdl_trigger();       // the root search is launched while the last CTAs end: a calibration of 2 x 64 tokens 24.3 -> 21.8 us, 8 x 700 105.7 -> 103.4
        // density contribution of this tile: sum over its rows of (1/t) * (sum of the row's gates), fixed order
#pragma unroll
        for (int row = 0; row < 2; ++row) {
            const float2 v = unpack2(gs[row]), e = unpack2(ge[row]);
            const int r = row ? r1 : r0;
            if (r < T) dsum += (((double)v.x - 1.0) + ((double)v.y - 1.0) + ((double)e.x + (double)e.y)) / (double)(r + 1);
        }
        if (!ok) dsum = __longlong_as_double(0x7ff8000000000000ll);       // a wait ran out: the density becomes NaN
#pragma unroll
        for (int s = 16; s >= 1; s >>= 1) dsum += __shfl_xor_sync(0xffffffffu, dsum, s);
        if (lane == 0) s_red[warp] = dsum;
    }
    tmem_fence_before();
    __syncthreads();
    if (warp == CAL_WARPS) {
        tmem_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(CAL_TMEM) : "memory");
    }
    if (tid == 0) {
        double tot = 0.0;
        for (int w = 0; w < CAL_WARPS; ++w) tot += s_red[w];
        dpart[((int64_t)x * Hq + h) * gridDim.z + ttile] = tot;
    }
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
// is found by Newton steps inside a bracket, with a halving wherever a step would leave the bracket or shrink too slowly: four to
// seven evaluations for thresholds among the scores (twelve in their tail) where plain halving took eighty (177 us).  What matters most is
// to stop at the root: a step of less than the rounding of c leaves c at an end of the bracket, and the halving that used to
// follow started over, on the unluckiest head for eighty evaluations (54 -> 15 us).  1024 threads are 6 us slower than 512.
// Where g is so flat that its own rounding moves the root by more than float's rounding of c (a density of exactly 1 or 0, a
// gap between two clusters of scores), every c of the plateau solves the equation: only halvings are taken there, which end
// at the plateau's lower end, for a density of 1 at the bracket's.
__global__ void __launch_bounds__(CAL_BISECT_THREADS) calib_bisect_kernel(
    const unsigned long long* hist, const double* dpart, int Hq, int n_seq, int n_ttiles, int T, int n_bins, double s_min,
    double s_max, double beta, int iters, float* __restrict__ head_const, float* __restrict__ dbar_out,
    double* __restrict__ head_const_d) {
    extern __shared__ unsigned char bis_raw[];
    double* Hn = reinterpret_cast<double*>(bis_raw);
    __shared__ double2 scratch[CAL_BISECT_THREADS / 32];
    __shared__ unsigned long long s_tot[CAL_BISECT_THREADS / 32];
    const int tid = threadIdx.x, h = blockIdx.x;
    const unsigned long long* Hh = hist + (int64_t)h * n_bins;
    pdl_wait();          // the histogram and the densities are complete from here on

    // total weight (an integer: exact whatever the order), then the normalised histogram
    unsigned long long part = 0;
    for (int b = tid; b < n_bins; b += CAL_BISECT_THREADS) {
        const unsigned long long v = __ldcg(Hh + b);
        Hn[b] = (double)v;
        part += v;
    }
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) part += __shfl_xor_sync(0xffffffffu, part, s);
    if ((tid & 31) == 0) s_tot[tid >> 5] = part;
    __syncthreads();
    part = 0;
#pragma unroll
    for (int w = 0; w < CAL_BISECT_THREADS / 32; ++w) part += s_tot[w];
    const double tot = (double)part;
    for (int b = tid; b < n_bins; b += CAL_BISECT_THREADS) Hn[b] = tot > 0.0 ? Hn[b] / tot : 0.0;
    // target density: partial sums of every (sequence, tile) of this head, in a fixed order
    double d = 0.0;
    for (int k = tid; k < n_seq * n_ttiles; k += CAL_BISECT_THREADS) {
        const int x = k / n_ttiles, tt = k % n_ttiles;
        d += __ldcg(dpart + ((int64_t)x * Hq + h) * n_ttiles + tt);
    }
    const double target = block_sum2_fixed(d, 0.0, scratch).x / ((double)n_seq * (double)T);

    // every thread follows the same iteration on the same sums
    const double w = (s_max - s_min) / n_bins;
    double lo = s_min - 40.0 / beta, hi = s_max + 40.0 / beta;
    double c = 0.5 * (lo + hi), dx_old = hi - lo, dx = dx_old;
    // A NaN density (a NaN among the thresholds or scores, or a wait of the histogram kernel that ran out) has no root: the
    // constant is NaN too, since the density is an optional output.
    const bool bad = target != target;
    if (bad) c = target;
    for (int it = 0; it < iters && !bad; ++it) {
        double gs = 0.0, ds = 0.0;
        for (int b = tid; b < n_bins; b += CAL_BISECT_THREADS) {
            const double hb = Hn[b];
            if (hb == 0.0) continue;                       // (whole warps of empty bins beside the scores' range)
            const double v = beta * (s_min + (b + 0.5) * w - c), e = exp(-fabs(v)), r = 1.0 / (1.0 + e);
            gs += hb * (v >= 0.0 ? r : e * r);
            ds += hb * (e * r * r);
        }
        const double2 r = block_sum2_fixed(gs, ds, scratch);
        const double f = r.x - target, slope = beta * r.y;      // g falls with c: g' = -slope
        if (r.x > target) lo = c; else hi = c;
        const bool flat = slope * (fabs(c) + w) < 0x1p-26;      // rounding of g (2^-50 and better) against 2^-24 of c
        const double cn = c + f / slope, tol = 1e-15 * (fabs(lo) + fabs(hi) + w);
        // at the root, to rounding: c may now be an end of the bracket, which the step below must not leave by a halving
        // (|g''| <= beta |g'|, so a step of d leaves beta d^2 / 2: below a 2^-52 of 1 / beta here.  Going round once more to see the
        // step shrink below rounding cost an evaluation: a calibration of 8 x 700 tokens 107.8 -> 105.7 us, 2 x 300 33.3 -> 31.2.)
        if (!flat && (fabs(cn - c) <= tol || beta * fabs(cn - c) <= 2e-8)) { c = cn; break; }
        double next;
        if (!flat && cn > lo && cn < hi && 2.0 * fabs(f) <= fabs(dx_old * slope)) {
            dx_old = dx; dx = cn - c; next = cn;
        } else {
            dx_old = dx; dx = 0.5 * (hi - lo); next = lo + dx;
        }
        const bool done = next == c || fabs(dx) <= tol;
        c = next;
        if (done) break;
    }
    if (tid == 0) {
        head_const[h] = (float)c;
        if (dbar_out) dbar_out[h] = (float)target;
        if (head_const_d) head_const_d[h] = c;
    }
}

// [heads][T][D] bf16, dense: boxes of `rows` tokens, a 64-column half after the other in shared memory
static int cal_tmap(CUtensorMap* tm, const void* base, int64_t heads, int T, int D, int rows) {
    const cuuint64_t dims[4] = {64, (cuuint64_t)T, (cuuint64_t)(D / 64), (cuuint64_t)heads};
    const cuuint64_t strides[3] = {(cuuint64_t)D * 2, 128, (cuuint64_t)T * D * 2};
    const cuuint32_t box[4] = {64, (cuuint32_t)rows, (cuuint32_t)(D / 64), 1};
    return encode_tiles(tm, base, 4, dims, strides, box);
}

template <int D>
static int launch_hist(const CUtensorMap& tmQ, const CUtensorMap& tmK, const float* tau, int Hq, int Hkv, int T, int n_seq,
                       float c2, float scale, int n_bins, float s_min, float inv_w, unsigned long long* hist, double* dpart,
                       cudaStream_t s) {
    auto kernel = CalSmem<D>::copies(n_bins) == 2 ? calib_hist_kernel<D, 2> : calib_hist_kernel<D, 1>;
    const int rc = configure_kernel(reinterpret_cast<const void*>(kernel), CalSmem<D>::bytes(4096));
    if (rc != ETA_OK) return rc;
    const dim3 grid((unsigned)Hq, (unsigned)n_seq, (unsigned)((T + CAL_ROWS - 1) / CAL_ROWS));
    return launch_pdl("calibration histogram", kernel, grid, dim3(CAL_THREADS), CalSmem<D>::bytes(n_bins), s, tmQ, tmK,
                      tau, Hq, Hkv, T, c2, scale, n_bins, s_min, inv_w, hist, dpart);
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
    const int n16 = (int)(hist_bytes / 16);                            // at most 65535 heads x 4096 bins

    const float sc = scale > 0.f ? scale : 1.0f / sqrtf((float)head_dim);
    const float inv_w = (float)n_bins / (s_max - s_min);
    const float c2 = (float)(-(double)beta * 1.4426950408889634);      // exp(-beta x) = 2^(c2 x)
    CUtensorMap tmQ, tmK;
    rc = cal_tmap(&tmQ, Q, (int64_t)n_seq * n_q_heads, seq_len, head_dim, CAL_ROWS);
    if (rc == ETA_OK) rc = cal_tmap(&tmK, K, (int64_t)n_seq * n_kv_heads, seq_len, head_dim, CAL_KEYS);
    if (rc != ETA_OK) return rc;
    rc = launch_pdl("calibration clear", calib_clear_kernel, dim3((unsigned)(n16 + 255) / 256), dim3(256), 0, s, reinterpret_cast<uint4*>(hist), n16);
    if (rc != ETA_OK) return rc;
    rc = (head_dim == 128 ? launch_hist<128> : launch_hist<64>)(tmQ, tmK, tau, n_q_heads, n_kv_heads, seq_len, n_seq, c2, sc,
                                                               n_bins, s_min, inv_w, hist, dpart, s);
    if (rc != ETA_OK) return rc;
    return launch_pdl("calibration bisection", calib_bisect_kernel, dim3((unsigned)n_q_heads), dim3(CAL_BISECT_THREADS),
                      sizeof(double) * (size_t)n_bins, s, hist, dpart, (int)n_q_heads, (int)n_seq, n_ttiles, (int)seq_len,
                      (int)n_bins, (double)s_min, (double)s_max, (double)beta, 160, head_const, dbar, hc_d);
}

}  // extern "C"
