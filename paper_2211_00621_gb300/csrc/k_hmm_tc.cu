// Batched scaled HMM forward on the tensor cores, states on the lanes (K8).
//
// The forward recursion (map over states j of a reduce over states i inside a sequential
// loop over t; Appendix A patterns) for a tile of N sequences is one dense contraction per
// step.  The HMM itself is not in the paper; this is the textbook scaled forward algorithm,
// with the rescaling done by exact powers of two:
//   alpha~_t = (A^T X_{t-1}) o b(o_t),   s_t = sum_j alpha~_t(j),   X_t = alpha~_t 2^-k_t
//   logL     = ln2 * sum_{t<T-1} k_t + ln s_{T-1}
// Any integers k_t give the same logL exactly; they only keep X in range:
//   k_t = x_{t-2} - k_{t-1} - target,   x_t = log2 of the largest entry of X_t,
// which makes x_t = target + the growth of the last two steps.  The step before last is the
// newest whose maxima are not on the path from one step to the next.  Growth is at most 1 for
// probabilities, so the target sits high, at 2^60: two steps may shrink the vector by 2^-90 each.
// Emissions above 1 (densities) grow it: past 2^25 the target is low enough for two steps of the
// model's largest, up to 2^63 (target_of).
//
// A step's time is its latency (the sequences are long and a step depends on the last), so
// the tile is laid out for a short step, not for a full tensor core:
//  * the MMA computes D^T [128 states x N sequences] = A^T [128 x K] X [K x N], one block per
//    128 states: N is as small as the batch allows (16 to 128), and a step costs N columns
//    instead of the 128 rows a sequence-major tile pays for;
//  * A^T is the MMA's A operand and stays in tensor memory for the whole launch (K / 2 columns
//    per block of 128 states): an N = 32 product reads 1 KB of X per 16 states from shared
//    memory instead of 5 KB;
//  * X (BF16) is the B operand in the MN-major no-swizzle canonical layout, so the thread that
//    holds state j writes 8 sequences with one 16-byte store;
//  * each thread of the epilogue holds one state and CPT sequences: D comes from tensor
//    memory in one load, b(j, o) from a shared table of FP32 values (already rounded to BF16);
//  * X is double-buffered by step parity, so a block's epilogue writes X_t while the other
//    block's products still read X_{t-1};
//  * one warp per block of states does nothing but issue its MMAs;
//  * one warp keeps the books (lane s: sequence s): while the products of step i run it turns
//    the column maxima of X_{i-1} into the exponents of step i + 1 and publishes them with that
//    step's symbols.  For tiles of up to 32 sequences further warps read X_{i-1} back for the
//    maxima, which keeps their shuffles out of the epilogue warps' step; larger tiles form them
//    in the epilogue.  Row sums are needed at a sequence's last step alone, and only then do the
//    epilogue warps form them.
// Row sums: 32 states per warp, added in a fixed binary tree by a reduce-scatter over the
// lanes, then over the warps in order of states.
//
// Measured (GB300; K = 256, M = 64, 4,096 sequences of log-uniform 50 to 5,000 steps): 2.44 ms,
// 0.49 us a step of the longest sequence with tiles of 16.  One CTA per 128 sequences with the
// sequences on the lanes took 12.7 ms, and clusters of two CTAs splitting the states of 32
// sequences 8.8 ms: 2.5 and 1.75 us a step.  What is left of a step is a chain of latencies (the
// products 0.2 us, tensor memory to X 0.15 us, two mbarrier hand-offs), not a rate.
//
// Every wait is bounded (2 s); on expiry the kernel reports ACCEL_ERR_TIMEOUT.  A watchdog on
// the run time (accel_set_watchdog_ns) is checked at step boundaries, with no product in
// flight.
#include "common.cuh"
#include "hmm_internal.cuh"
#include "tc_ptx.cuh"

#include <cuda_bf16.h>

#include <type_traits>

namespace accel {
namespace hmm {

namespace {

constexpr int kMaxScale = 126;                // largest |k|
constexpr uint64_t kWaitNs = 2000000000ull;   // bounded mbarrier wait: 2 s of wall clock
// epilogue: column parts per lane quarter for tiles of N sequences
__host__ __device__ constexpr int col_parts(int N) { return N <= 16 ? 1 : 2; }
// warps that take the column maxima: 16 columns of a block of 128 states each (0: the epilogue's)
__host__ __device__ constexpr int max_warps(int K, int N) { return N <= 32 ? (K + 127) / 128 * (N / 16) : 0; }

// What a step is to the tile: the columns that start and that end a sequence, and whether the
// tile is done (the step is not run).
struct Ctl {
    uint32_t fresh[4], end[4], done, pad[3];
};

struct TileLayout {
    uint32_t x, x_bytes, e, scale, sym, ctl, mx, psum, bar, slot, bytes;
};

__host__ __device__ inline TileLayout tile_layout(int K, int M, int N, int esize) {
    TileLayout L;
    uint32_t o = 0;
    L.x_bytes = (uint32_t)N * (uint32_t)K * 2;
    L.x = o;      o += 2 * L.x_bytes;                               // [step parity]
    L.e = o;      o += (uint32_t)M * (uint32_t)K * (uint32_t)esize;
    o = (o + 15) & ~15u;
    L.scale = o;  o += 2 * (uint32_t)N * 4;                         // [step parity][N]: 2^-k
    L.sym = o;    o += 4 * (uint32_t)N * 4;                         // [step mod 4][N]: o_t K
    L.ctl = o;    o += 4 * 48;                                      // [step mod 4]: Ctl
    L.mx = o;     o += 2 * (uint32_t)(K / 32) * (uint32_t)N * 2;    // [step parity][K / 32][N]: BF16 maxima
    L.psum = o;   o += 2 * (uint32_t)(K / 32) * (uint32_t)N * 4;    // [step parity][K / 32][N]: row sums
    o = (o + 7) & ~7u;
    L.bar = o;    o += 10 * 8;
    L.slot = o;   o += 16;
    L.bytes = o;
    return L;
}

// log2 of X's target size for emissions of at most b (as bits) < 2^g: 60, or what leaves room for two of
// them, for sums over the states (2^8) and for the states' probability to meet in one (2^8) below 2^126.
__device__ __forceinline__ int32_t target_of(uint32_t b) {
    const int32_t g = (int32_t)(b >> 23) - 126;
    return g <= 25 ? 60 : 110 - 2 * g;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&h);
}

// Sums of C columns over the 32 lanes of a warp: lane l returns the sum of column *col, added
// as the binary tree over the lanes (pairs at distance 1, then 2, 4, 8, 16).  While more than
// one column is left, a level also halves the columns a lane keeps.
template <int C>
__device__ __forceinline__ float lane_sums(float (&v)[C], int lane, int* col) {
    int n = C, c = 0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        if (n > 1) {
            n >>= 1;
            const bool up = (lane & d) != 0;
#pragma unroll
            for (int i = 0; i < C / 2; ++i) {
                if (i < n) {
                    const float keep = up ? v[i + n] : v[i], send = up ? v[i] : v[i + n];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, d);
                }
            }
            c += up ? n : 0;
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], d);
        }
    }
    *col = c;
    return v[0];
}

template <int C>
__device__ __forceinline__ void tmem_ld_cols(uint32_t taddr, float (&v)[C]) {
    uint32_t r[C];
    if constexpr (C == 8) tc::tmem_ld8(taddr, r);
    else if constexpr (C == 16) tc::tmem_ld16(taddr, r);
    else tc::tmem_ld32(taddr, r);
#pragma unroll
    for (int i = 0; i < C; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ uint32_t max_bf16x2(uint32_t a, uint32_t b) {
    const __nv_bfloat162 m = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
    return *reinterpret_cast<const uint32_t*>(&m);
}

// Maxima of W words of two BF16 columns over the 32 lanes: lane l returns word *word (a
// reduce-scatter, as lane_sums).
template <int W>
__device__ __forceinline__ uint32_t lane_max(uint32_t (&v)[W], int lane, int* word) {
    int n = W, c = 0;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        if (n > 1) {
            n >>= 1;
            const bool up = (lane & d) != 0;
#pragma unroll
            for (int i = 0; i < W / 2; ++i) {
                if (i < n) {
                    const uint32_t keep = up ? v[i + n] : v[i], send = up ? v[i] : v[i + n];
                    v[i] = max_bf16x2(keep, __shfl_xor_sync(0xffffffffu, send, d));
                }
            }
            c += up ? n : 0;
        } else {
            v[0] = max_bf16x2(v[0], __shfl_xor_sync(0xffffffffu, v[0], d));
        }
    }
    *word = c;
    return v[0];
}

// A wait on a step's path.  The first poll suspends the warp until the phase completes, so it
// is nearly always the only one; `fail` is set when the wait gives up.
__device__ __noinline__ bool wait_slow(uint64_t* bar, uint32_t parity, volatile uint32_t* fail) {
    if (tc::mbar_wait_bounded(bar, parity, kWaitNs)) return true;
    *fail = 1;
    return false;
}
__device__ __forceinline__ bool wait_step(uint64_t* bar, uint32_t parity, volatile uint32_t* fail) {
    return tc::mbar_try_wait(bar, parity) || wait_slow(bar, parity, fail);
}

constexpr int tile_threads(int K, int N) {
    return 128 * ((K + 127) / 128) * col_parts(N) + 32 * ((K + 127) / 128 + 1 + max_warps(K, N));
}

// N = sequences of the tile, TE = emission table type.
template <int K, int N, typename TE>
__global__ void __launch_bounds__(tile_threads(K, N), 1)
k_hmm_tc(int M, const float* __restrict__ log_A, const float* __restrict__ log_B,
         const float* __restrict__ log_pi, const int32_t* __restrict__ obs, const int64_t* __restrict__ off,
         int64_t S, const int32_t* __restrict__ order, unsigned long long* __restrict__ next,
         const int32_t* __restrict__ pick, double* __restrict__ loglik, int32_t* __restrict__ status,
         uint64_t watchdog_ns, uint32_t tmem_cols) {
    if (pick && *pick != N) return;               // the other tile size runs this call
    constexpr int NH = (K + 127) / 128;           // blocks of 128 states
    constexpr int PARTS = col_parts(N);
    constexpr int NEPI = 4 * NH * PARTS;          // epilogue warps; then NH issuing, the bookkeeping and the max warps
    constexpr int CPT = N / PARTS;                // columns (sequences) of an epilogue thread
    constexpr int CH = CPT < 32 ? CPT : 32;       // ... taken CH at a time
    constexpr int NU = N < 32 ? 1 : N / 32;       // sequences of a bookkeeping lane
    constexpr int NMX = max_warps(K, N);
    constexpr int MXP = NMX > 0 ? NH : K / 32;    // maxima per column
    constexpr int kThreads = tile_threads(K, N);
    extern __shared__ __align__(1024) char smem[];
    const TileLayout L = tile_layout(K, M, N, (int)sizeof(TE));
    char* sX = smem + L.x;
    TE* sE = reinterpret_cast<TE*>(smem + L.e);
    float* s_scale = reinterpret_cast<float*>(smem + L.scale);
    int32_t* s_sym = reinterpret_cast<int32_t*>(smem + L.sym);
    Ctl* s_ctl = reinterpret_cast<Ctl*>(smem + L.ctl);
    uint16_t* s_mx = reinterpret_cast<uint16_t*>(smem + L.mx);
    float* s_ps = reinterpret_cast<float*>(smem + L.psum);
    uint64_t* bar_mma = reinterpret_cast<uint64_t*>(smem + L.bar);      // [2] per block of states: D ready
    // The rest are [2], per step parity: a warp may see a step's phase as late as the step after, so the
    // same barrier's next completion waits for it - of bar_x for the issuing and the max warps, through
    // D and through bar_mx and the bookkeeping.
    uint64_t* bar_x = bar_mma + 2;                                      // X written, D read
    uint64_t* bar_info = bar_mma + 4;                                   // scale, sym, ... written
    uint64_t* bar_ps = bar_mma + 6;                                     // row sums written
    uint64_t* bar_mx = bar_mma + 8;                                     // column maxima written
    uint32_t* slot = reinterpret_cast<uint32_t*>(smem + L.slot);
    volatile uint32_t* s_fail = slot + 1;         // set by a warp whose wait gave up
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int quarter = w & 3, half = (w >> 2) % NH, part = (w >> 2) / NH;
    const int j = 128 * half + 32 * quarter + lane;
    const bool valid = K % 128 == 0 || j < K;     // uniform over a warp: K is a multiple of 32

    if (w == NEPI) {
        tc::tmem_alloc(slot, tmem_cols);
        tc::tmem_relinquish();
        if (lane == 0) {
            for (int h = 0; h < 2; ++h) {
                tc::mbar_init(&bar_mma[h], 1);
                tc::mbar_init(&bar_x[h], NEPI);
                tc::mbar_init(&bar_info[h], 1);
                tc::mbar_init(&bar_ps[h], NEPI);
                tc::mbar_init(&bar_mx[h], NMX > 0 ? NMX : NEPI);
            }
            tc::fence_mbar_init();
            *s_fail = 0;
            slot[2] = 0;
        }
    }
    float top = 0.f;                              // the largest emission
    // b(j, o) = exp(log B[j, o]) rounded to BF16, symbol-major; X starts at zero (its columns
    // without a sequence are never read back)
    for (int idx = tid; idx < M * K; idx += kThreads) {
        const int o = idx / K, s = idx - o * K;
        const __nv_bfloat16 b = __float2bfloat16_rn(__expf(log_B[s * M + o]));
        top = fmaxf(top, __bfloat162float(b));
        if constexpr (sizeof(TE) == 4) sE[idx] = __bfloat162float(b); else sE[idx] = b;
    }
    for (int idx = tid; idx < (int)(2 * L.x_bytes / 16); idx += kThreads)
        reinterpret_cast<int4*>(sX)[idx] = make_int4(0, 0, 0, 0);
    tc::fence_proxy_async_smem();
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    top = warp_max_f32(top);
    if (lane == 0) atomicMax(slot + 2, __float_as_uint(top));
    const uint32_t tmem = *slot;
    const uint32_t tmem_a = tmem + (uint32_t)(NH * N);
    // A^T into tensor memory: lane j of block `half`, column c = (A[2c][j], A[2c+1][j])
    if (w < NEPI) {
        const int c1 = (part + 1) * (K / 2 / PARTS);
        for (int c0 = part * (K / 2 / PARTS); c0 < c1; c0 += 16) {
            uint32_t r[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const float* a = log_A + (int64_t)(2 * (c0 + e)) * K + j;
                r[e] = valid ? pack_bf16(__expf(a[0]), __expf(a[K])) : 0u;
            }
            tc::tmem_st16(tmem_a + (uint32_t)(half * (K / 2) + c0) + ((uint32_t)(32 * quarter) << 16), r);
        }
        tc::tmem_wait_st();
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();

    if (w >= NEPI && w < NEPI + NH) {
        // ---- an issuing warp: block h of D = A^T X_{t-1}
        const int h = w - NEPI;
        constexpr uint32_t idesc = tc::idesc_bf16_f32(128, N) | tc::kIdescBMnMajor;
        const uint64_t xdesc0 = tc::smem_desc_noswizzle(tc::smem_u32(sX), 128, 16u * (uint32_t)K);
        const uint32_t d = tmem + (uint32_t)(h * N), a = tmem_a + (uint32_t)(h * (K / 2));
        uint32_t issued = 0;
        for (uint32_t iter = 0;; ++iter) {
            const uint32_t par = iter & 1u, pprev = par ^ 1u;
            if (!wait_step(&bar_info[par], (iter >> 1) & 1u, s_fail) || s_ctl[iter & 3u].done != 0) break;
            if (iter > 0) wait_step(&bar_x[pprev], ((iter - 1) >> 1) & 1u, s_fail);
            tc::tc_fence_after();
            const uint64_t xd = xdesc0 + (uint64_t)(pprev * (L.x_bytes >> 4));
            if (tc::elect_one()) {
#pragma unroll
                for (int ks = 0; ks < K / 16; ++ks)
                    tc::mma_bf16_ts(d, a + ks * 8, xd + ks * 16, idesc, ks > 0 ? 1u : 0u);
                tc::mma_commit(&bar_mma[h]);
            }
            __syncwarp();
            issued = iter + 1;
        }
        // the products issued last complete before the tensor memory goes
        if (issued > 0) tc::mbar_wait_bounded(&bar_mma[h], (issued - 1) & 1u, kWaitNs);
    } else if (w == NEPI + NH) {
        // ---- the bookkeeping warp (lane l: columns l, l + 32, ...)
        const uint64_t t_launch = watchdog_ns != 0 ? tc::globaltimer_ns() : 0;
        const int64_t ncta = gridDim.x;
        const int32_t target = target_of(slot[2]);
        // the sequence on the column at the step last published, with the steps left after it
        int32_t seq[NU];
        int64_t left[NU];
        const int32_t* o[NU];                     // its next symbol
        int32_t nob[NU];                          // ... loaded one step ahead
        bool fresh[NU], dry[NU];
        auto start = [&](int u, int64_t q) {
            seq[u] = -1;
            if (q >= S) {
                dry[u] = true;
                return;
            }
            seq[u] = order ? order[q] : (int32_t)q;
            const int64_t o0 = off[seq[u]];
            left[u] = off[seq[u] + 1] - o0 - 1;
            o[u] = obs + o0 + 1;
            nob[u] = obs[o0];
            fresh[u] = true;
        };
        // what a step is to the column: 1 it has a sequence, 2 it begins, 4 it ends
        auto state = [&](int u) -> uint32_t {
            return seq[u] < 0 ? 0u : 1u | (fresh[u] ? 2u : 0u) | (left[u] <= 0 ? 4u : 0u);
        };
        auto publish = [&](int u, uint32_t step, uint32_t st) {     // all but the exponents
            if (u * 32 + lane < N) s_sym[(step & 3u) * N + u * 32 + lane] = st & 1u ? nob[u] * K : 0;
            if ((st & 5u) == 1u) nob[u] = *o[u]++;
            const uint32_t fm = __ballot_sync(0xffffffffu, st & 2u);
            const uint32_t em = __ballot_sync(0xffffffffu, st & 4u);
            if (lane == 0) {
                s_ctl[step & 3u].fresh[u] = fm;
                s_ctl[step & 3u].end[u] = em;
            }
            return em != 0;
        };
        // steps i - 1 and i: what they are to the column, their sequences, exponents and the
        // exponents before them
        uint32_t st1[NU], st0[NU];
        int32_t sq1[NU], sq0[NU], k1[NU], k0[NU];
        int64_t E1[NU], E0[NU];
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            dry[u] = u * 32 + lane >= N;
            seq[u] = -1;
            fresh[u] = false;
            left[u] = 0;
            nob[u] = 0;
            // the first N x grid positions are dealt out
            if (!dry[u]) start(u, blockIdx.x + (int64_t)(u * 32 + lane) * ncta);
            st1[u] = 0;
            sq1[u] = -1;
            k1[u] = k0[u] = 0;
            E1[u] = E0[u] = 0;
            st0[u] = state(u);
            sq0[u] = seq[u];
        }
        bool ended1 = false, ended0 = false;      // whether steps i - 1 and i end a sequence
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            ended0 = publish(u, 0, st0[u]) || ended0;
            if (u * 32 + lane < N) s_scale[u * 32 + lane] = 1.f;
        }
        if (lane == 0) s_ctl[0].done = 0;
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&bar_info[0]);
        uint32_t ps_phase = 0;                    // bit p: parity of the next completion of bar_ps[p]
        for (uint32_t iter = 0;; ++iter) {
            const uint32_t pprev = (iter & 1u) ^ 1u;
            // ---- step i + 1: what it is, and its symbols
            uint32_t st[NU];
            bool any = false, ended = false;
#pragma unroll
            for (int u = 0; u < NU; ++u) {
                if (st0[u] & 4u) {
                    seq[u] = -1;
                    if (next && !dry[u]) start(u, (int64_t)N * ncta + (int64_t)atomicAdd(next, 1ull));
                } else {
                    fresh[u] = false;
                    --left[u];
                }
                st[u] = state(u);
                any = any || ((st0[u] | st[u]) & 1u);
                ended = publish(u, iter + 1, st[u]) || ended;
            }
            bool stop = !__any_sync(0xffffffffu, any);
            if (watchdog_ns != 0 && tc::globaltimer_ns() - t_launch > watchdog_ns) *s_fail = 1;
            stop = __any_sync(0xffffffffu, stop || *s_fail != 0);
            if (lane == 0) s_ctl[(iter + 1) & 3u].done = stop ? 1u : 0u;
            // ---- its exponents, from the maxima of X_{i-1}
            if (iter > 0) wait_step(&bar_mx[pprev], ((iter - 1) >> 1) & 1u, s_fail);
            int32_t kn[NU];
#pragma unroll
            for (int u = 0; u < NU; ++u) {
                const int c = u * 32 + lane < N ? u * 32 + lane : 0;
                uint32_t m = 0;
#pragma unroll
                for (int q = 0; q < MXP; ++q) m = max(m, (uint32_t)s_mx[(pprev * MXP + q) * N + c]);
                // (at a sequence's second step X_{i-1} is not its own: 0 stands for log2 of 1)
                const int32_t x = st0[u] & 2u ? 0 : (int32_t)(m >> 7) - 127;
                int32_t k = x - k0[u] - target;
                k = k < -kMaxScale ? -kMaxScale : k > kMaxScale ? kMaxScale : k;
                kn[u] = (st[u] & 3u) == 1u ? k : 0;
                if (u * 32 + lane < N) s_scale[pprev * N + u * 32 + lane] = __uint_as_float((uint32_t)(127 - kn[u]) << 23);
            }
            // the row sums of the sequences that ended at step i - 1, before step i + 1 may write
            // its own in their place
            float sums[NU];
            if (ended1) {
                wait_step(&bar_ps[pprev], (ps_phase >> pprev) & 1u, s_fail);
                ps_phase ^= 1u << pprev;
#pragma unroll
                for (int u = 0; u < NU; ++u) {
                    sums[u] = 0.f;
                    if (st1[u] & 4u) {
                        // in the order of the states: chunks of 32, in K / 4 or K / 2 parts
                        constexpr int np = (K / 4) % 32 == 0 ? 4 : 2, cpp = K / 32 / np;
                        const float* ps = s_ps + (size_t)pprev * (K / 32) * N + u * 32 + lane;
                        float sum = 0.f;
#pragma unroll
                        for (int p = 0; p < np; ++p) {
                            float c = ps[p * cpp * N];
#pragma unroll
                            for (int q = 1; q < cpp; ++q) c += ps[(p * cpp + q) * N];
                            sum = p == 0 ? c : sum + c;
                        }
                        sums[u] = sum;
                    }
                }
            }
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&bar_info[pprev]);
            if (ended1 && *s_fail == 0) {
#pragma unroll
                for (int u = 0; u < NU; ++u)
                    if (st1[u] & 4u)
                        loglik[sq1[u]] = 0.6931471805599453 * (double)E1[u] + log(ldexp((double)sums[u], k1[u]));
            }
            if (stop) {
                // done, out of time, or a wait gave up
                if (lane == 0 && *s_fail != 0) report_status(status, ACCEL_ERR_TIMEOUT);
                break;
            }
#pragma unroll
            for (int u = 0; u < NU; ++u) {
                st1[u] = st0[u];
                sq1[u] = sq0[u];
                E1[u] = E0[u];
                k1[u] = k0[u];
                E0[u] = (st[u] & 3u) == 1u ? E0[u] + k0[u] : 0;
                k0[u] = kn[u];
                st0[u] = st[u];
                sq0[u] = seq[u];
            }
            ended1 = ended0;
            ended0 = ended;
        }
        __syncwarp();
    } else if (w > NEPI + NH) {
        // ---- the max warps: lanes 16 g .. 16 g + 15 take columns 8 g .. 8 g + 7 of the warp's 16,
        // every sixteenth state each
        const int h = (w - NEPI - NH - 1) % NH, c0 = (w - NEPI - NH - 1) / NH * 16;
        const int g = lane >> 4, kl = lane & 15;
        const int ns = K - 128 * h < 128 ? K - 128 * h : 128;
        const char* xr = sX + ((c0 >> 3) + g) * 16 * K + (128 * h + kl) * 16;
        for (uint32_t iter = 0;; ++iter) {
            const uint32_t par = iter & 1u;
            if (!wait_step(&bar_info[par], (iter >> 1) & 1u, s_fail) || s_ctl[iter & 3u].done != 0) break;
            wait_step(&bar_x[par], (iter >> 1) & 1u, s_fail);
            const uint4* v = reinterpret_cast<const uint4*>(xr + par * L.x_bytes);
            uint4 x[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = 16 * i < ns ? v[16 * i] : make_uint4(0, 0, 0, 0);
            uint32_t m[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                auto wd = [&](int i) { return r == 0 ? x[i].x : r == 1 ? x[i].y : r == 2 ? x[i].z : x[i].w; };
                m[r] = max_bf16x2(max_bf16x2(max_bf16x2(wd(0), wd(1)), max_bf16x2(wd(2), wd(3))),
                                  max_bf16x2(max_bf16x2(wd(4), wd(5)), max_bf16x2(wd(6), wd(7))));
            }
            // over the 16 lanes: two halving levels (4 -> 2 -> 1 words), then two full ones
            const bool up1 = (kl & 8) != 0, up2 = (kl & 4) != 0;
#pragma unroll
            for (int r = 0; r < 2; ++r)
                m[r] = max_bf16x2(up1 ? m[r + 2] : m[r], __shfl_xor_sync(0xffffffffu, up1 ? m[r] : m[r + 2], 8));
            m[0] = max_bf16x2(up2 ? m[1] : m[0], __shfl_xor_sync(0xffffffffu, up2 ? m[0] : m[1], 4));
            m[0] = max_bf16x2(m[0], __shfl_xor_sync(0xffffffffu, m[0], 2));
            m[0] = max_bf16x2(m[0], __shfl_xor_sync(0xffffffffu, m[0], 1));
            if ((kl & 3) == 0)
                *reinterpret_cast<uint32_t*>(s_mx + (par * MXP + h) * N + c0 + 8 * g + 2 * (kl >> 2)) = m[0];
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&bar_mx[par]);
        }
    } else {
        // ---- the epilogue warps
        const float pij = valid ? __expf(log_pi[j]) : 0.f;
        const uint32_t lane_base = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(half * N + part * CPT);
        char* const xw = sX + (j >> 3) * 128 + (j & 7) * 16;
        const TE* const ej = sE + j;
        for (uint32_t iter = 0;; ++iter) {
            const uint32_t par = iter & 1u;
            const Ctl& ctl = s_ctl[iter & 3u];
            if (!wait_step(&bar_info[par], (iter >> 1) & 1u, s_fail) || ctl.done != 0) break;
            bool ends = false;                    // some column of the tile ends a sequence
#pragma unroll
            for (int u = 0; u < NU; ++u) ends = ends || ctl.end[u] != 0;
#pragma unroll
            for (int ch = 0; ch < CPT / CH; ++ch) {
                const int s0 = part * CPT + ch * CH;
                // this step's emissions, scaled by 2^-k (exact), while the products run
                float bs[CH];
                uint32_t fm = 0;
                if (valid) {
                    fm = ctl.fresh[s0 >> 5] >> (s0 & 31);
#pragma unroll
                    for (int c = 0; c < CH; c += 4) {
                        const int4 sy = *reinterpret_cast<const int4*>(s_sym + (iter & 3u) * N + s0 + c);
                        const float4 sc = *reinterpret_cast<const float4*>(s_scale + par * N + s0 + c);
                        float e0, e1, e2, e3;
                        if constexpr (sizeof(TE) == 4) {
                            e0 = ej[sy.x]; e1 = ej[sy.y]; e2 = ej[sy.z]; e3 = ej[sy.w];
                        } else {
                            e0 = __bfloat162float(ej[sy.x]); e1 = __bfloat162float(ej[sy.y]);
                            e2 = __bfloat162float(ej[sy.z]); e3 = __bfloat162float(ej[sy.w]);
                        }
                        const float2 p0 = __fmul2_rn(make_float2(e0, e1), make_float2(sc.x, sc.y));
                        const float2 p1 = __fmul2_rn(make_float2(e2, e3), make_float2(sc.z, sc.w));
                        bs[c] = p0.x; bs[c + 1] = p0.y; bs[c + 2] = p1.x; bs[c + 3] = p1.y;
                    }
                }
                if (ch == 0) {
                    wait_step(&bar_mma[half], par, s_fail);
                    tc::tc_fence_after();
                }
                if (valid) {
                    float v[CH];
                    tmem_ld_cols<CH>(lane_base + (uint32_t)(ch * CH), v);
                    const uint32_t mask = CH == 32 ? 0xffffffffu : (1u << (CH & 31)) - 1u;
                    if ((fm & mask) != 0) {
                        // columns that start a sequence: alpha~_0 = pi o b(o_0)
#pragma unroll
                        for (int c = 0; c < CH; ++c) v[c] = (fm >> c) & 1u ? pij : v[c];
                    }
#pragma unroll
                    for (int c = 0; c < CH; c += 2) {
                        const float2 p = __fmul2_rn(make_float2(v[c], v[c + 1]), make_float2(bs[c], bs[c + 1]));
                        v[c] = p.x;
                        v[c + 1] = p.y;
                    }
                    uint32_t pk[CH / 2];
#pragma unroll
                    for (int c = 0; c < CH / 2; ++c) pk[c] = pack_bf16(v[2 * c], v[2 * c + 1]);
#pragma unroll
                    for (int c = 0; c < CH; c += 8)
                        *reinterpret_cast<uint4*>(xw + par * L.x_bytes + ((s0 + c) >> 3) * 16 * K) =
                            make_uint4(pk[c / 2], pk[c / 2 + 1], pk[c / 2 + 2], pk[c / 2 + 3]);
                    if (ch == CPT / CH - 1) {
                        tc::fence_proxy_async_smem();
                        tc::tc_fence_before();
                        __syncwarp();
                        if (lane == 0) tc::mbar_arrive(&bar_x[par]);
                    }
                    if constexpr (NMX == 0) {
                        int word;
                        const uint32_t top = lane_max<CH / 2>(pk, lane, &word);
                        if ((lane & (64 / CH - 1)) == 0)
                            *reinterpret_cast<uint32_t*>(s_mx + (par * MXP + (j >> 5)) * N + s0 + 2 * word) = top;
                    }
                    if (ends) {
                        int col;
                        const float sum = lane_sums<CH>(v, lane, &col);
                        if (CH == 32 || (lane & ~(CH - 1)) == 0) s_ps[(par * (K / 32) + (j >> 5)) * N + s0 + col] = sum;
                    }
                } else if (ch == CPT / CH - 1) {
                    if (lane == 0) tc::mbar_arrive(&bar_x[par]);
                }
            }
            if (NMX == 0 || ends) {
                __syncwarp();
                if (lane == 0) {
                    if (NMX == 0) tc::mbar_arrive(&bar_mx[par]);
                    if (ends) tc::mbar_arrive(&bar_ps[par]);
                }
            }
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (w == NEPI) tc::tmem_dealloc(tmem, tmem_cols);
}

using Kernel = void (*)(int, const float*, const float*, const float*, const int32_t*, const int64_t*, int64_t,
                        const int32_t*, unsigned long long*, const int32_t*, double*, int32_t*, uint64_t, uint32_t);

template <int K>
Kernel kernel_k(int n, int esize) {
    if constexpr (K <= 128)
        if (esize == 2) return n == 16 ? k_hmm_tc<K, 16, __nv_bfloat16> : k_hmm_tc<K, 32, __nv_bfloat16>;
    return n == 16 ? k_hmm_tc<K, 16, float> : n == 32 ? k_hmm_tc<K, 32, float>
         : n == 64 ? k_hmm_tc<K, 64, float> : k_hmm_tc<K, 128, float>;
}

// A tile of n sequences: the size of a table entry, or 0 if no kernel takes it.  The BF16 table
// is for the models whose FP32 table does not fit even beside 32 sequences (K <= 128, M > 400).
int table_esize(int K, int M, int n) {
    if ((int)tile_layout(K, M, n, 4).bytes <= max_smem_optin()) return 4;
    return K <= 128 && n <= 32 && (int)tile_layout(K, M, n, 2).bytes <= max_smem_optin() ? 2 : 0;
}

// One of two tile sizes, picked on the device where the lengths are: *pick = lo or hi, the one with
// the smaller estimated time.  A launch of tiles of N on g CTAs takes about
//   t_N max(T_max, sum(T) / (N g) + 0.3 mean(T))
// (the longest sequence, or the columns' load with part of a last sequence); t_hi / t_lo is
// measured (GB300, us a step at N = 16 / 32 / 64: K = 256 0.49 / 0.76 / 1.27, K = 128 0.40 /
// 0.51 / 0.87, K = 64 0.42 / 0.48 / 0.84).
__global__ void __launch_bounds__(1024) k_pick_tile(const int64_t* __restrict__ off, int64_t S, int lo, int hi, int g,
                                                    float ratio, int32_t* __restrict__ pick) {
    __shared__ int64_t s_max[32];
    int64_t m = 0;
    for (int64_t s = threadIdx.x; s < S; s += blockDim.x) m = max(m, off[s + 1] - off[s]);
    for (int d = 16; d > 0; d >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, d));
    if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < 32; ++q) m = max(m, s_max[q]);
        const float total = (float)(off[S] - off[0]), tail = 0.3f * total / (float)S;
        const float t_lo = fmaxf((float)m, total / ((float)lo * g) + tail);
        const float t_hi = fmaxf((float)m, total / ((float)hi * g) + tail) * ratio;
        *pick = t_hi < t_lo ? hi : lo;
    }
}

// the largest tile of at most n sequences that some kernel takes, or 0
int tile_fit(int K, int M, int n) {
    while (n >= 16 && table_esize(K, M, n) == 0) n >>= 1;
    return n >= 16 ? n : 0;
}

accel_status launch_tiles(const accel_hmm_model* m, const int32_t* obs, const int64_t* off, int64_t S, int n, int grid,
                          const int32_t* order, unsigned long long* next, const int32_t* pick, double* loglik,
                          int32_t* d_status, cudaStream_t st) {
    const int K = m->K, M = m->M;
    const int es = table_esize(K, M, n), nh = (K + 127) / 128;
    const TileLayout L = tile_layout(K, M, n, es);
    const int need = nh * n + nh * (K / 2);                         // tensor memory: D, and A
    uint32_t cols = 32;
    while ((int)cols < need) cols <<= 1;
    const Kernel kern = K == 64 ? kernel_k<64>(n, es) : K == 128 ? kernel_k<128>(n, es)
                      : K == 192 ? kernel_k<192>(n, es) : kernel_k<256>(n, es);
    ACCEL_CUDA_TRY(allow_smem((const void*)kern, L.bytes));
    kern<<<grid, tile_threads(K, n), L.bytes, st>>>(M, m->log_A, m->log_B, m->log_pi, obs, off, S, order, next, pick,
                                                    loglik, d_status, watchdog_ns(), cols);
    return ACCEL_OK;
}

constexpr size_t kPickOff = 24;          // in the status block: the tile size picked on the device

}  // namespace

// The shapes taken: K a multiple of 64 whose transition matrix, emission table and a tile of 128
// sequences fit shared memory together in BF16 (every such shape has a tile of 16 that fits).
bool tc_supported(int K, int M) {
    if (K < 64 || K > 256 || K % 64 != 0 || M < 1 || M > 32767) return false;
    const size_t bytes = (size_t)K * K * 2 + (size_t)128 * K * 2 + (((size_t)M * K * 2 + 15) & ~(size_t)15) + 2576;
    return bytes <= (size_t)max_smem_optin() && tile_fit(K, M, 16) != 0;
}

// workspace: the status block, the order by length and its scratch
size_t tc_ws_bytes(int K, int M, int64_t S) {
    (void)K; (void)M;
    return align_up(kStatusBytes, 256) + order_ws_bytes(S);
}

// rows and split of a tile of n sequences: n = 2 rows / split
TcConfig tile_config(int n) { return n >= 32 ? TcConfig{2, n, 0, 0} : TcConfig{4, 32, 0, 0}; }

// The tile without a tuned configuration, by size alone: every sequence on a column of its own
// where tiles of 16 allow it (the shortest step), else the larger size that k_pick_tile weighs.
TcConfig default_config(int64_t S) {
    const int64_t g = num_sms();
    return tile_config(S <= 16 * g ? 16 : S <= 32 * g ? 32 : 64);
}

accel_status tc_forward_cfg(const accel_hmm_model* mdl, const int32_t* obs, const int64_t* off, int64_t S,
                            double* loglik, char* ws, int32_t* d_status, const TcConfig* cfg, cudaStream_t st) {
    const int K = mdl->K, M = mdl->M;
    ACCEL_REQUIRE(tc_supported(K, M), ACCEL_ERR_UNSUPPORTED,
                  "hmm_forward(bf16): K must be a multiple of 64 in [64, 256] and the tables must fit shared "
                  "memory (K=%d, M=%d)", K, M);
    const TcConfig c = cfg ? *cfg : default_config(S);
    const int rows = c.rows < 32 || c.rows > 128 ? 128 : c.rows;
    const int n = tile_fit(K, M, c.split == 4 ? rows / 2 : rows);
    int lo = n;
    if (!cfg && n > 16) lo = n / 2;                                  // weighed on the device
    const int64_t tiles = (S + lo - 1) / lo;
    int grid = (int)(tiles < num_sms() ? tiles : num_sms());
    const int64_t ctas = (int64_t)c.units * (c.pair == 1 ? 2 : c.pair == 2 ? 4 : 1);
    if (ctas > 0 && ctas < grid) grid = (int)ctas;
    // every sequence on a column of its own from the start needs neither an order nor a queue
    int32_t* order = nullptr;
    unsigned long long* next = nullptr;
    int nk = 1;
    if (S > (int64_t)lo * grid) {
        next = (unsigned long long*)(ws + kQueueOff);               // inside the status block
        order = (int32_t*)(ws + align_up(kStatusBytes, 256));
        ACCEL_CUDA_TRY(cudaMemsetAsync(next, 0, 8, st));
        accel_status r = order_by_length(off, S, order, (char*)order + align_up((size_t)S * 4, 256), st);
        if (r != ACCEL_OK) return r;
        nk += 3;
    }
    int32_t* pick = nullptr;
    if (lo != n) {
        pick = (int32_t*)(ws + kPickOff);
        const float ratio = n > 32 ? 1.7f : K > 128 ? 1.54f : 1.25f;
        k_pick_tile<<<1, 1024, 0, st>>>(off, S, lo, n, grid, ratio, pick);
        accel_status r = launch_tiles(mdl, obs, off, S, lo, grid, order, next, pick, loglik, d_status, st);
        if (r != ACCEL_OK) return r;
        nk += 2;
    }
    accel_status r = launch_tiles(mdl, obs, off, S, n, grid, order, next, pick, loglik, d_status, st);
    if (r != ACCEL_OK) return r;
    return after_launch(st, "hmm_forward(bf16 tcgen05)", nk);
}

accel_status tc_forward(const accel_hmm_model* mdl, const int32_t* obs, const int64_t* off, int64_t S,
                        double* loglik, char* ws, int32_t* d_status, cudaStream_t st) {
    TcConfig c;
    return tc_forward_cfg(mdl, obs, off, S, loglik, ws, d_status, tuned_entry(mdl->K, mdl->M, S, &c) ? &c : nullptr, st);
}

}  // namespace hmm
}  // namespace accel
