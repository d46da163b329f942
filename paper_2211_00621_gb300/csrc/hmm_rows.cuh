// The recurrences of the SIMT HMM kernels on CTAs (K <= 128) or CTA pairs (K <= 256) that keep the
// step matrix in registers: one step of up to 8 sequences is out[g][j] = sum_i x[g][i] Mx[i][j].
//
// States are padded to KP = 64, 128 or 256 (zero probabilities add exact zeros); a CTA owns Kh = KP /
// NC of them.  It has 8 contraction warps and 8 epilogue warps.
//  * Contraction warp w takes WC = Kh / 8 columns, lane 4 ip + cg part ip of the rows (eight
//    contiguous parts, see Contraction) and CW = WC / 4 columns: the thread's KP / 8 x CW block of Mx
//    is loaded once per kernel.  The vectors come from shared memory (8 x 16 consecutive bytes a
//    load); the rows' partial sums meet in a part of shared memory of the warp's own.
//  * Epilogue warp g owns sequence slot g: all of a slot's bookkeeping is uniform over a warp, a row of
//    the CTA's columns is one vector access, and its sum one warp reduction.  (4 warps of two slots
//    each: a warp that waits for one half is late for the other.)
//
// The 8 slots are two halves of 4 that run as two interleaved recurrences: a phase is one step of one
// half, and the halves take turns, so that the epilogue, the hand-overs between the warps and the
// exchange between the CTAs of a pair (st.async on an mbarrier per half and step parity) of one half
// hide behind the other half's products.  A half whose slots have all finished is left out.  In one
// group of warps that did both (and a CTA barrier per step) a step took 5,300 cycles at K = 256, of
// which the FMA pipe was busy 2,350: two warps per scheduler cannot cover the epilogue's latencies.
// Now a step of both halves takes about 3,700 cycles, of which the FMA pipe needs 2,048.
//
// Slots and sequences: slot sl = cluster + clusters * g of n = 8 * clusters runs the sequences
// k n + sl (k even) and k n + n - 1 - sl (k odd) of the order (by decreasing length), one after the
// other with no gap: a fixed assignment, balanced like the greedy one for sorted lengths, that needs
// neither a queue nor any agreement between the CTAs of a pair.
#pragma once
#include "hmm_internal.cuh"
#include "tc_ptx.cuh"

#include <cooperative_groups.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

namespace accel {
namespace hmm {
namespace rows {

constexpr int kCon = 256;       // contraction threads
constexpr int kEpi = 256;       // epilogue threads
constexpr int kT = kCon + kEpi;
constexpr int kG = 8;           // slots per cluster
constexpr uint64_t kWaitNs = 2000000000ull;

template <int KP>
struct Cfg {
    static constexpr int NC = KP == 256 ? 2 : 1;
    static constexpr int Kh = KP / NC;
    static constexpr int WC = Kh / 8;
    static constexpr int CW = WC / 4;
    static constexpr int NQ = KP / 32;
    static constexpr int OC = CW / 2;
    static constexpr int EC = Kh / 32;             // columns of an epilogue lane
    static constexpr int ST = KP + 16;             // row stride of the vectors
    static constexpr int SO = Kh + 16;             // ... of the products
    static constexpr int MINB = KP == 64 ? 2 : 1;  // CTAs per SM
};

template <int KP>
struct Smem {
    float x[2][kG][Cfg<KP>::ST];                   // vectors [step parity][slot]
    float out[2][4][Cfg<KP>::SO];                  // products [half][slot]
    float peer[2][kG];                             // the peer's scalar of the slot's vector [step parity][slot]
    int64_t tot[kG];
    uint64_t x_own[2][2];                          // [half][step parity]: the CTA's columns of x written
    uint64_t x_peer[2][2];                         // ... the peer's have arrived
    uint64_t out_full[2];                          // [half]: products written
};

template <int N>
struct Vec {
    float v[N];
    __device__ __forceinline__ void load(const float* p) {
        if constexpr (N == 4) { const float4 t = *reinterpret_cast<const float4*>(p); v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w; }
        else if constexpr (N == 2) { const float2 t = *reinterpret_cast<const float2*>(p); v[0] = t.x; v[1] = t.y; }
        else v[0] = *p;
    }
    __device__ __forceinline__ void store(float* p) const {
        if constexpr (N == 4) *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
        else if constexpr (N == 2) *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
        else *p = v[0];
    }
    __device__ __forceinline__ void send(uint32_t a, uint32_t bar) const {
        if constexpr (N == 4) tc::st_async4(a, make_float4(v[0], v[1], v[2], v[3]), bar);
        else if constexpr (N == 2) tc::st_async2(a, make_float2(v[0], v[1]), bar);
        else tc::st_async1(a, v[0], bar);
    }
};

// Registers of the two kinds of warps (K = 256: the launch gives 128 each).
template <int KP> __device__ __forceinline__ void regs_contraction() {
    if constexpr (KP == 256) asm volatile("setmaxnreg.inc.sync.aligned.u32 192;");
}
template <int KP> __device__ __forceinline__ void regs_epilogue() {
    if constexpr (KP == 256) asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
}

// Bounded waits.  One that gives up reports and is not repeated: the kernel then finishes with
// unusable values.
struct Waits {
    int32_t* status;
    bool dead = false;
    template <typename Poll>
    __device__ __forceinline__ void until(Poll&& poll) {
        if (dead || poll()) return;
        const uint64_t t0 = tc::globaltimer_ns();
        while (!poll()) {
            if (tc::globaltimer_ns() - t0 > kWaitNs) {
                dead = true;
                report_status(status, ACCEL_ERR_TIMEOUT);
                return;
            }
        }
    }
    __device__ __forceinline__ void local(uint64_t* bar, uint32_t ph) {
        until([&]() { return tc::mbar_try_wait(bar, ph); });
    }
    __device__ __forceinline__ void cluster(uint64_t* bar, uint32_t ph) {
        until([&]() { return tc::mbar_try_wait_cluster(bar, ph); });
    }
};
// the parity of the phase of step i's barrier of parity i & 1
__device__ __forceinline__ uint32_t step_phase(uint32_t i) { return (i >> 1) & 1u; }

template <int KP>
__device__ __forceinline__ void init_bars(Smem<KP>& sm, int out_warps = kCon / 32) {
    if (threadIdx.x == 0) {
        for (int q = 0; q < 4; ++q) {
            tc::mbar_init(&sm.x_own[q >> 1][q & 1], 4);
            tc::mbar_init(&sm.x_peer[q >> 1][q & 1], 1);
        }
        tc::mbar_init(&sm.out_full[0], out_warps);
        tc::mbar_init(&sm.out_full[1], out_warps);
        tc::fence_mbar_init();
    }
}

// ---------------------------------------------------------------- slots
__device__ __forceinline__ int64_t slot_at(int64_t n, int32_t sl, int64_t k) { return k * n + ((k & 1) ? n - 1 - sl : sl); }

// The sequences of one slot, one after the other.
struct Slot {
    int32_t k, sl;
    int32_t seq;           // -1: none left
    int64_t o0, T;         // its first row (from the first sequence's offset), its length
};

// Advance the slot to its next sequence that is neither empty nor refused by `ok` (first row, length).
template <typename Ok>
__device__ __forceinline__ void next_seq(Slot& s, int64_t S, int64_t n, const int32_t* order, const int64_t* off, Ok&& ok) {
    for (;;) {
        ++s.k;
        if ((int64_t)s.k * n >= S) {
            s.seq = -1;
            return;
        }
        const int64_t q = slot_at(n, s.sl, s.k);
        if (q >= S) continue;
        s.seq = order ? order[q] : (int32_t)q;
        const int64_t o0 = off[s.seq];
        s.o0 = o0 - off[0];
        s.T = off[s.seq + 1] - o0;
        if (s.T > 0 && ok(s.o0, s.T)) return;
    }
}

// The steps of the slots: half[h] = the largest of half h's (the first 8 warps count a slot each).
template <typename Ok, typename I>
__device__ __forceinline__ void slot_totals(int64_t* tot, int64_t S, int64_t n, int32_t cid, int32_t ncl,
                                            const int32_t* order, const int64_t* off, Ok&& ok, I (&half)[2]) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (w < kG) {
        int64_t sum = 0;
        for (int64_t k = lane; k * n < S; k += 32) {
            const int64_t q = slot_at(n, cid + ncl * w, k);
            if (q >= S) continue;
            const int64_t sq = order ? (int64_t)order[q] : q;
            const int64_t T = off[sq + 1] - off[sq];
            if (T > 0 && ok(off[sq] - off[0], T)) sum += T;
        }
        for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
        if (lane == 0) tot[w] = sum;
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        half[h] = 0;
        for (int g = 0; g < 4; ++g) half[h] = (I)tot[4 * h + g] > half[h] ? (I)tot[4 * h + g] : half[h];
    }
}

// ---------------------------------------------------------------- contraction warps
// A product's sum over the rows is eight contiguous parts of NQ chunks of four, each part in the order of
// the positions p (chunk pos_swap(p)), even and odd rows apart, and the parts are added one after the other:
// the order of the checkpointed form's pairs of CTAs, so that both forms give the same bits for K = 64, 128
// and 256.  Row lane ip takes part ip; chunk c of a vector lies at chunk vec_pos(c), where the eight lanes'
// chunks of a step are next to each other.
__device__ __forceinline__ int pos_swap(int p) { return p ^ ((p >> 3) & 1); }
template <int KP>
__device__ __forceinline__ int vec_pos(int c) {
    const int p = pos_swap(c);
    return 8 * (p % Cfg<KP>::NQ) + p / Cfg<KP>::NQ;
}

template <int KP>
struct Contraction {
    using C = Cfg<KP>;
    int rank, w, lane, ip, cg;
    float2 a[2 * C::NQ][C::CW];                    // (rows 2k, 2k + 1) of the lane's 4 per q

    __device__ __forceinline__ void load(const float* __restrict__ Mx, int r) {
        rank = r;
        w = threadIdx.x >> 5;
        lane = threadIdx.x & 31;
        ip = lane >> 2;
        cg = lane & 3;
#pragma unroll
        for (int q = 0; q < C::NQ; ++q)
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const float* p = Mx + (size_t)(4 * pos_swap(C::NQ * ip + q) + 2 * k) * KP + rank * C::Kh + w * C::WC + cg * C::CW;
#pragma unroll
                for (int h = 0; h < C::CW; ++h) a[2 * q + k][h] = make_float2(p[h], p[KP + h]);
            }
    }
    // the products of the four vectors at x, added to acc
    __device__ __forceinline__ void add(const float* x, float2 (&acc)[4][C::CW]) const {
#pragma unroll
        for (int q = 0; q < C::NQ; ++q) {
            const float* xq = x + 32 * q + 4 * ip;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const float4 v = *reinterpret_cast<const float4*>(xq + g * C::ST);
#pragma unroll
                for (int h = 0; h < C::CW; ++h) {
                    acc[g][h] = __ffma2_rn(make_float2(v.x, v.y), a[2 * q][h], acc[g][h]);
                    acc[g][h] = __ffma2_rn(make_float2(v.z, v.w), a[2 * q + 1][h], acc[g][h]);
                }
            }
        }
    }
    // the sums over the 8 row lanes, in their order, into out (row stride SO), by way of the warp's `part`
    static constexpr int PS = 16 * C::CW + 4 * C::CW;              // row lane stride: conflict-free
    __device__ __forceinline__ void reduce(const float2 (&acc)[4][C::CW], float* part, float* out) const {
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            Vec<C::CW> v;
#pragma unroll
            for (int h = 0; h < C::CW; ++h) v.v[h] = acc[g][h].x + acc[g][h].y;
            v.store(part + ip * PS + g * C::WC + cg * C::CW);
        }
        __syncwarp();
        const int at = (ip >> 1) * C::WC + cg * C::CW + (ip & 1) * C::OC;
        Vec<C::OC> o, v[8];
#pragma unroll
        for (int l = 0; l < 8; ++l) v[l].load(part + l * PS + at);
        o = v[0];
#pragma unroll
        for (int l = 1; l < 8; ++l)
#pragma unroll
            for (int h = 0; h < C::OC; ++h) o.v[h] += v[l].v[h];
        o.store(out + (ip >> 1) * C::SO + w * C::WC + cg * C::CW + (ip & 1) * C::OC);
    }
};

// The contraction warps' part of a kernel: steps 1 .. half[u] - 1 of both halves.
template <int KP, typename I>
__device__ __forceinline__ void contraction_loop(const Contraction<KP>& m, Smem<KP>& sm, const I (&half)[2], Waits& wt) {
    using C = Cfg<KP>;
    __shared__ __align__(16) float part[kCon / 32][8 * Contraction<KP>::PS];
    const I iters = half[0] > half[1] ? half[0] : half[1];
    for (I it = 1; it < iters; ++it) {
        const int pb = (int)(it & 1) ^ 1;
        const uint32_t ph = step_phase(it - 1);
#pragma unroll 1
        for (int u = 0; u < 2; ++u) {
            if (it >= (u ? half[1] : half[0])) continue;
            float2 acc[4][C::CW];
#pragma unroll
            for (int g = 0; g < 4; ++g)
#pragma unroll
                for (int h = 0; h < C::CW; ++h) acc[g][h] = make_float2(0.f, 0.f);
            const float* x = &sm.x[pb][4 * u][0];
            wt.local(&sm.x_own[u][pb], ph);
            // (products of the own columns before this wait: a second bubble a phase, 3% slower)
            if constexpr (C::NC == 2) wt.cluster(&sm.x_peer[u][pb], ph);
            m.add(x, acc);
            m.reduce(acc, part[m.w], &sm.out[u][0][0]);
            __syncwarp();
            if (m.lane == 0) tc::mbar_arrive(&sm.out_full[u]);
        }
    }
}

// ---------------------------------------------------------------- products in the order of the rows
// A thread owns a column, and its sum runs over the rows one by one.  Two stages of four warps take half of
// the rows each (four of two warps a quarter, for 64 columns); while one works on a half of the slots,
// another works on the other half.
template <int KP>
struct Mid {
    static constexpr int Kh = Cfg<KP>::Kh, NS = kCon / Kh, W = Kh / 32;
    uint64_t full[2][NS - 1][W];                   // [half][stage][warp of columns]
    float sum[2][4][Kh];                           // [half][slot][column]: over the rows so far
    __device__ __forceinline__ void init() {
        if (threadIdx.x == 0)
            for (int q = 0; q < 2 * (NS - 1) * W; ++q) tc::mbar_init(&full[0][0][0] + q, 1);
    }
};
template <int KP, typename I>
__device__ __forceinline__ void products_in_order(const float* __restrict__ A, int rank, Smem<KP>& sm, Mid<KP>& mid,
                                                  const I (&half)[2], Waits& wt) {
    using C = Cfg<KP>;
    constexpr int NS = Mid<KP>::NS, R = KP / NS;
    const int col = threadIdx.x % C::Kh, stage = threadIdx.x / C::Kh, w = col >> 5, lane = threadIdx.x & 31;
    float a[R];
#pragma unroll
    for (int i = 0; i < R; ++i) a[i] = A[(size_t)(stage * R + i) * KP + rank * C::Kh + col];
    const I iters = half[0] > half[1] ? half[0] : half[1];
    for (I it = 1; it < iters; ++it) {
        const int pb = (int)(it & 1) ^ 1;
        const uint32_t ph = step_phase((uint32_t)(it - 1));
#pragma unroll 1
        for (int u = 0; u < 2; ++u) {
            if (it >= (u ? half[1] : half[0])) continue;
            const float* x = &sm.x[pb][4 * u][stage * R];
            wt.local(&sm.x_own[u][pb], ph);
            if constexpr (C::NC == 2) wt.cluster(&sm.x_peer[u][pb], ph);
            float acc[4] = {};
            if (stage > 0) {
                wt.local(&mid.full[u][stage - 1][w], (uint32_t)(it - 1) & 1u);
#pragma unroll
                for (int g = 0; g < 4; ++g) acc[g] = mid.sum[u][g][col];
            }
#pragma unroll
            for (int q = 0; q < R / 4; ++q) {
                float4 v[4];
#pragma unroll
                for (int g = 0; g < 4; ++g) v[g] = *reinterpret_cast<const float4*>(x + g * C::ST + 4 * q);
#pragma unroll
                for (int g = 0; g < 4; ++g) acc[g] = fmaf(v[g].x, a[4 * q], acc[g]);
#pragma unroll
                for (int g = 0; g < 4; ++g) acc[g] = fmaf(v[g].y, a[4 * q + 1], acc[g]);
#pragma unroll
                for (int g = 0; g < 4; ++g) acc[g] = fmaf(v[g].z, a[4 * q + 2], acc[g]);
#pragma unroll
                for (int g = 0; g < 4; ++g) acc[g] = fmaf(v[g].w, a[4 * q + 3], acc[g]);
            }
            const bool last = stage == NS - 1;
#pragma unroll
            for (int g = 0; g < 4; ++g) (last ? sm.out[u][g][col] : mid.sum[u][g][col]) = acc[g];
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(last ? &sm.out_full[u] : &mid.full[u][last ? 0 : stage][w]);
        }
    }
}

// ---------------------------------------------------------------- epilogue warps
template <int KP>
struct Epilogue {
    using C = Cfg<KP>;
    Smem<KP>& sm;
    int rank, g, u, lane;                          // the warp's slot and its half
    int col;                                       // the lane's first column within the CTA's
    int xcol;                                      // where it lies in a vector
    uint32_t peer_x, peer_s, peer_bar;             // the peer's buffers (shared::cluster addresses)
    // (in_order: vectors in the order of the states, not by vec_pos)
    __device__ __forceinline__ Epilogue(Smem<KP>& s, int r, bool in_order) : sm(s), rank(r) {
        g = (threadIdx.x - kCon) >> 5;
        u = g >> 2;
        lane = threadIdx.x & 31;
        col = C::EC * lane;
        const int c = r * C::Kh + col;
        xcol = in_order ? c : 4 * vec_pos<KP>(c >> 2) + (c & 3);
        if constexpr (C::NC == 2) {
            const uint32_t pr = (uint32_t)(r ^ 1);
            peer_x = tc::cluster_addr(&s.x[0][0][0], pr);
            peer_s = tc::cluster_addr(&s.peer[0][0], pr);
            peer_bar = tc::cluster_addr(&s.x_peer[0][0], pr);
        } else {
            peer_x = peer_s = peer_bar = 0;
        }
    }
    // The slot's new vector (and a scalar of it) into parity b of both CTAs, and the end of the phase.
    __device__ __forceinline__ void put(int b, const Vec<C::EC>& v, bool scalar, float s) {
        v.store(&sm.x[b][g][xcol]);
        if constexpr (C::NC == 2) {
            const uint32_t bar = peer_bar + 8u * (uint32_t)(2 * u + b);
            v.send(peer_x + 4u * (uint32_t)((b * kG + g) * C::ST + xcol), bar);
            if (scalar && lane == 0) tc::st_async1(peer_s + 4u * (uint32_t)(b * kG + g), s, bar);
        }
        __syncwarp();
        if (lane == 0) {
            tc::mbar_arrive(&sm.x_own[u][b]);
            if (C::NC == 2 && (g & 3) == 0)              // the peer's bytes of this step
                tc::mbar_arrive_expect_tx(&sm.x_peer[u][b], (uint32_t)(4 * C::Kh * 4 + (scalar ? 4 * 4 : 0)));
        }
    }
    // The sums of 32 columns each (e[k]: columns 32 k ..), by a butterfly, the highest bit of the column first
    __device__ __forceinline__ void sums_by32(const Vec<C::EC>& v, float (&e)[4]) const {
        Vec<C::EC> t = v;
#pragma unroll
        for (int d = 16 / C::EC; d > 0; d >>= 1)
#pragma unroll
            for (int h = 0; h < C::EC; ++h) t.v[h] += __shfl_xor_sync(0xffffffffu, t.v[h], d);
        float s;
        if constexpr (C::EC == 4) s = (t.v[0] + t.v[2]) + (t.v[1] + t.v[3]);
        else s = t.v[0] + t.v[1];
#pragma unroll
        for (int k = 0; k < 4; ++k) e[k] = k < C::Kh / 32 ? __shfl_sync(0xffffffffu, s, (32 / C::EC * k) & 31) : 0.f;
    }
    // K > 128, as 16 threads of eight columns each add: eight columns in order, then the threads pairwise
    __device__ __forceinline__ float warp_sum_by8(const Vec<C::EC>& v) const {
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const float before = __shfl_xor_sync(0xffffffffu, s, 1);
            if ((lane & 1) == k) {
                s = k ? before + v.v[0] : v.v[0];
#pragma unroll
                for (int h = 1; h < C::EC; ++h) s += v.v[h];
            }
        }
        s = __shfl_sync(0xffffffffu, s, lane | 1);
#pragma unroll
        for (int d = 2; d < 32; d <<= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
        return s;
    }
    __device__ __forceinline__ float warp_sum(const Vec<C::EC>& v) const {
        float s = v.v[0];
#pragma unroll
        for (int h = 1; h < C::EC; ++h) s += v.v[h];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
        return s;
    }
};

// ---------------------------------------------------------------- launches
// Clusters of the recurrences resident at once on the device (cached per device and kernel).
template <typename Kern>
int max_clusters(Kern kern, int nc) {
    static std::mutex mu;
    static std::map<std::pair<int, const void*>, int> cache;
    int dev = 0;
    cudaGetDevice(&dev);
    const auto key = std::make_pair(dev, reinterpret_cast<const void*>(kern));
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    int n = 0;
    if (nc == 2) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3((unsigned)(num_sms() / 2 * 2), 1, 1);
        cfg.blockDim = dim3(kT, 1, 1);
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) n = 0;
    } else if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, kT, 0) == cudaSuccess) {
        n *= num_sms();
    }
    cudaGetLastError();
    if (n < 1) n = num_sms() / nc;
    cache[key] = n;
    return n;
}

// Clusters of a launch: all that are resident, but no more than there are sequences; with a budget
// of SMs, those that fit it.
template <typename Kern>
int clusters_for(Kern kern, int KP, int64_t S, int budget) {
    const int nc = KP == 256 ? 2 : 1;
    int64_t n = max_clusters(kern, nc);
    if (budget > 0) n = std::min<int64_t>(n, std::max<int64_t>(1, n * budget / num_sms()));
    return (int)std::max<int64_t>(1, std::min(n, S));
}

}  // namespace rows
}  // namespace hmm
}  // namespace accel
