// U = X^T Q over all rows of the adjoint (hmm_adj_rows.cu), on the tensor cores: a K x K result of a
// long reduction.  A CTA takes a 128 x 128 tile of U and a contiguous range of the rows, in
// tcgen05.mma kind::f16 on BF16 (16 rows of the reduction per instruction).
//
// FP32 accuracy from BF16 products: x = hi + mid + lo, each the BF16 rounding of what is left (24
// bits), and a b = hi hi + (hi mid + mid hi + mid mid + hi lo + lo hi), which drops terms below
// 2^-24.  The tensor core truncates when it adds to an accumulator, so a sum of n products loses
// about n 2^-25 of itself.  Two things keep that down: the five small products have an accumulator of
// their own (their truncation is relative to their own size), and after kBlock rows the accumulators
// are added, rounded to nearest, to sums in registers: 8 truncations, about 3e-7.
//
// Pipeline: 512 splitter threads, one piece of a 16-row chunk each (eight rows of one column, loaded
// two chunks ahead straight from global memory), write the three parts into a stage (no-swizzle
// K-major canonical layout, 16-byte stores); the stage's mbarrier counts them; one warp issues the
// chunk's six MMAs under elect.sync (in a divergent branch each costs about 100 cycles) and commits
// them to the stage's second mbarrier, which the splitters wait on before they refill it.  The
// accumulators are double-buffered in tensor memory (all 512 columns), so the splitters take a
// block's sums while the next block's products run.  Every wait is bounded.
//
// What bounds it: the splitters' instructions (about 650 issue slots a chunk and scheduler); DRAM and
// the tensor cores are at a third.  1.13M rows at K = 256: 1.13 ms (2.3 GB of operands, 0.34 ms at the
// copy rate).  One chunk in flight and an arrival per thread and stage: 1.50 ms.
#include "hmm_adj_rows.cuh"
#include "tc_ptx.cuh"

#include <cuda_bf16.h>

namespace accel {
namespace hmm {
namespace rows {

namespace {

constexpr int kSplitThreads = 512;              // warps 0-15: loads, operand split, register sums
constexpr int kThreads = kSplitThreads + 32;    // + warp 16: issues the MMAs
constexpr int kKC = 16;                         // rows per chunk (one MMA's reduction)
constexpr int kBlock = 128;                     // rows between flushes
constexpr int kChunks = kBlock / kKC;
constexpr int kStages = 4;
constexpr int kPrefetch = 12;                   // chunks brought into L2 ahead
constexpr uint64_t kWait = 2000000000ull;

// Canonical K-major offset of the 16 bytes (n, k = 8 kq .. + 7) of a [rows][kKC] BF16 block: core
// matrices of 8 n x 8 k, LBO = 128 (along k), SBO = 256 (along n).
__device__ __forceinline__ uint32_t canon(int n, int kq) {
    return (uint32_t)(n >> 3) * 256 + (uint32_t)kq * 128 + (uint32_t)(n & 7) * 16;
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float lo_f(uint32_t x) { return __uint_as_float(x << 16); }
__device__ __forceinline__ float hi_f(uint32_t x) { return __uint_as_float(x & 0xffff0000u); }

// The BF16 rounding of eight values, which are replaced by what is left of them.
__device__ __forceinline__ uint4 take_part(float (&v)[8]) {
    uint32_t p[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        p[i] = pack2(v[2 * i], v[2 * i + 1]);
        v[2 * i] -= lo_f(p[i]);
        v[2 * i + 1] -= hi_f(p[i]);
    }
    return make_uint4(p[0], p[1], p[2], p[3]);
}

constexpr int tile(int K) { return K < 128 ? K : 128; }
constexpr uint32_t part_bytes(int K) { return 2u * tile(K) * kKC * 2; }       // X and Q columns of one part
constexpr uint32_t stage_bytes(int K) { return 3 * part_bytes(K); }
constexpr uint32_t smem_bytes(int K) { return kStages * stage_bytes(K); }

// (with the bounded loop out of line behind a first poll: 1.23 ms, 1.13 so)
__device__ __forceinline__ bool wait(uint64_t* bar, uint32_t parity) { return tc::mbar_wait_bounded(bar, parity, kWait); }

template <int K>
__global__ void __launch_bounds__(kThreads, 1) k_rows_xi(const float* __restrict__ X, const float* __restrict__ Q,
                                                         const int32_t* __restrict__ d_rows, int nsplit,
                                                         float* __restrict__ U, int32_t* __restrict__ status) {
    constexpr int TN = tile(K), NB = K / TN;              // tile edge; tiles along i and j
    constexpr uint32_t kQOff = TN * kKC * 2;              // Q's columns within a part
    constexpr uint32_t kBuf = 2 * TN;                     // columns of an accumulator pair
    extern __shared__ __align__(1024) char smem[];
    __shared__ __align__(8) uint64_t s_bar[kStages];      // stage s: its MMAs done
    __shared__ __align__(8) uint64_t s_full[kStages];     // stage s: operands written
    __shared__ __align__(8) uint64_t s_read[2];           // accumulator pair b has been read
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_fail;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tl = (int)blockIdx.x % (NB * NB), sp = (int)blockIdx.x / (NB * NB);
    const int i0 = tl / NB * TN, j0 = tl % NB * TN;
    const int64_t rows = *d_rows;
    const int64_t r0 = rows * sp / nsplit, r1 = rows * (sp + 1) / nsplit;
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            tc::mbar_init(&s_bar[s], 1);
            tc::mbar_init(&s_full[s], kSplitThreads / 32);
        }
        tc::mbar_init(&s_read[0], kSplitThreads / 32);
        tc::mbar_init(&s_read[1], kSplitThreads / 32);
        tc::fence_mbar_init();
        s_fail = 0;
    }
    if (warp == 0) {
        tc::tmem_alloc(&s_tmem, 2 * kBuf);
        tc::tmem_relinquish();
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = s_tmem;
    const int nchunks = r1 > r0 ? (int)((r1 - r0 + kKC - 1) / kKC) : 0;
    // chunk c's products have completed (its stage is c mod kStages)
    auto done = [&](int c) {
        return wait(&s_bar[c % kStages], (uint32_t)(c / kStages) & 1u);
    };
    if (warp == kSplitThreads / 32) {
        // ---- the issuing warp
        constexpr uint32_t id = tc::idesc_bf16_f32(TN, TN);
        constexpr uint64_t P = part_bytes(K) >> 4;
        const uint64_t desc0 = tc::smem_desc_noswizzle(tc::smem_u32(smem), 128, 256);
        int issued = 0;
        for (int q = 0; q < nchunks; ++q) {
            const int s = q % kStages, blk = q / kChunks;
            const bool first = q % kChunks == 0;
            bool ok = wait(&s_full[s], (uint32_t)(q / kStages) & 1u);
            // the pair's last block has been taken
            if (first && blk >= 2) ok = wait(&s_read[blk & 1], (uint32_t)(blk / 2 - 1) & 1u) && ok;
            if (!ok || s_fail != 0) {
                s_fail = 1;
                break;
            }
            tc::tc_fence_after();
            const uint64_t a = desc0 + (uint64_t)(s * (stage_bytes(K) >> 4)), b = a + (kQOff >> 4);
            const uint32_t d = tmem + (uint32_t)(blk & 1) * kBuf, acc = first ? 0u : 1u;
            if (tc::elect_one()) {
                tc::mma_bf16(d, a, b, id, acc);                          // hi hi
                tc::mma_bf16(d + TN, a, b + P, id, acc);                 // hi mid
                tc::mma_bf16(d + TN, a + P, b, id, 1u);                  // mid hi
                tc::mma_bf16(d + TN, a + P, b + P, id, 1u);              // mid mid
                tc::mma_bf16(d + TN, a, b + 2 * P, id, 1u);              // hi lo
                tc::mma_bf16(d + TN, a + 2 * P, b, id, 1u);              // lo hi
                tc::mma_commit(&s_bar[s]);
            }
            __syncwarp();
            issued = q + 1;
        }
        // the MMAs issued last complete before the tensor memory goes
        if (issued > 0) done(issued - 1);
    } else {
        // ---- the splitters: columns 0 .. TN - 1 are X's, TN .. 2 TN - 1 Q's, two row octets each
        const int col = tid % (2 * TN), kq = tid / (2 * TN);
        const bool mine = kq < 2;                                         // (K = 64: half the threads)
        const float* src = (col < TN ? X + i0 + col : Q + j0 + (col - TN)) + (r0 + 8 * (mine ? kq : 0)) * K;
        const uint32_t dst = (col < TN ? canon(col, kq) : kQOff + canon(col - TN, kq));
        const int qd = warp & 3, part = warp >> 2;                        // the thread's part of D
        const bool sums = 32 * part < TN;
        const uint32_t at = tmem + ((uint32_t)(32 * qd) << 16) + (uint32_t)(32 * part);
        auto load = [&](float (&v)[8], int q) {
            if (q >= nchunks || !mine) return;
            const float* p = src + (int64_t)q * (kKC * K);
            if (q + 1 < nchunks) {                                        // a whole chunk
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] = __ldcg(p + i * K);
            } else {
                const int left = (int)(r1 - r0) - q * kKC - 8 * kq;       // rows from the piece's first
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] = i < left ? __ldcg(p + i * K) : 0.f;
            }
        };
        auto prefetch = [&](int q) {
            if (q >= nchunks) return;
            const int64_t row0 = r0 + (int64_t)q * kKC;
            const uint32_t bytes = (uint32_t)(r1 - row0 < kKC ? r1 - row0 : kKC) * K * 4;
            tc::bulk_prefetch_l2(Q + row0 * K, bytes);
            tc::bulk_prefetch_l2(X + row0 * K, bytes);
        };
        float acc[32];
#pragma unroll
        for (int e = 0; e < 32; ++e) acc[e] = 0.f;
        // take the sums of block blk, whose products have completed
        auto flush = [&](int blk) {
            tc::tc_fence_after();
            if (sums) {
                uint32_t v[32];
                tc::tmem_ld32(at + (uint32_t)(blk & 1) * kBuf, v);
#pragma unroll
                for (int e = 0; e < 32; ++e) acc[e] += __uint_as_float(v[e]);
                tc::tmem_ld32(at + (uint32_t)(blk & 1) * kBuf + TN, v);
#pragma unroll
                for (int e = 0; e < 32; ++e) acc[e] += __uint_as_float(v[e]);
            }
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&s_read[blk & 1]);
        };
        // write chunk c from v and load chunk c + 2 into it; false: a wait gave up
        auto step = [&](float (&v)[8], int c) -> bool {
            const int s = c % kStages;
            char* st = smem + s * stage_bytes(K) + dst;
            if (tid == 0) prefetch(c + kPrefetch);
            // the stage's previous MMAs (chunk c - kStages) have completed
            if (c >= kStages && !done(c - kStages)) return false;
            if (mine) {
                *reinterpret_cast<uint4*>(st) = take_part(v);
                *reinterpret_cast<uint4*>(st + part_bytes(K)) = take_part(v);
                *reinterpret_cast<uint4*>(st + 2 * part_bytes(K)) = take_part(v);
            }
            load(v, c + 2);
            tc::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&s_full[s]);
            // a block's sums, when the wait above was for its last chunk
            if (c >= kChunks && c % kChunks == kStages - 1) flush(c / kChunks - 1);
            return s_fail == 0;
        };
        if (tid == 0)
            for (int q = 0; q < kPrefetch; ++q) prefetch(q);
        float v0[8], v1[8];
        load(v0, 0);
        load(v1, 1);
        bool ok = true;
        for (int c = 0; c < nchunks && ok; c += 2) {
            ok = step(v0, c);
            if (ok && c + 1 < nchunks) ok = step(v1, c + 1);
        }
        if (ok) {
            // the blocks not taken yet: the last one, and the one before it if it ended less than a
            // stage's depth before the end
            const int lastb = nchunks > 0 ? (nchunks - 1) / kChunks : 0;
            if (lastb >= 1 && (nchunks - 1) % kChunks < kStages - 1 && (ok = done(lastb * kChunks - 1))) flush(lastb - 1);
            if (nchunks > 0 && ok && (ok = done(nchunks - 1))) flush(lastb);
            // row r of the tile: lane r (TN = 128) or lane 32 (r / 16) + r % 16 (TN = 64)
            if (sums && (TN == 128 || lane < 16)) {
                const int row = TN == 128 ? 32 * qd + lane : 16 * qd + lane;
                float4* out = reinterpret_cast<float4*>(U + ((int64_t)sp * K + i0 + row) * K + j0 + 32 * part);
#pragma unroll
                for (int e = 0; e < 8; ++e) out[e] = make_float4(acc[4 * e], acc[4 * e + 1], acc[4 * e + 2], acc[4 * e + 3]);
            }
        }
        if (!ok) s_fail = 1;
    }
    tc::tc_fence_before();
    __syncthreads();
    if (s_fail != 0 && tid == 0) report_status(status, ACCEL_ERR_TIMEOUT);
    if (warp == 0) tc::tmem_dealloc(tmem, 2 * kBuf);
}

}  // namespace

// Row ranges (and partials) of a launch: one CTA per SM over the tiles, fewer where the rows are few
// (at least a block each).
int xi_parts(int KP, int64_t rows) {
    const int nt = (KP / tile(KP)) * (KP / tile(KP));
    int64_t n = num_sms() / nt;
    if (n > rows / kBlock) n = rows / kBlock;
    return (int)(n < 1 ? 1 : n);
}

accel_status xi_rows(const float* X, const float* Q, const int32_t* d_rows, int KP, int parts, float* U,
                     int32_t* status, cudaStream_t st) {
    auto kern = KP == 64 ? k_rows_xi<64> : KP == 128 ? k_rows_xi<128> : k_rows_xi<256>;
    const uint32_t smem = KP == 64 ? smem_bytes(64) : smem_bytes(128);
    const int nt = (KP / tile(KP)) * (KP / tile(KP));
    ACCEL_CUDA_TRY(allow_smem((const void*)kern, smem));
    kern<<<(unsigned)(parts * nt), kThreads, smem, st>>>(X, Q, d_rows, parts, U, status);
    return ACCEL_OK;
}

}  // namespace rows
}  // namespace hmm
}  // namespace accel
