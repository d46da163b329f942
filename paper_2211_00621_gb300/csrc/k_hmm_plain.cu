// Plain FP32 log-space HMM forward recursion (K7).
//
// The recursion is a map over states j of a reduce over states i inside a sequential
// loop over t (Appendix A patterns; Listing 1's loop/reduce pairing).  The paper does
// not discuss HMMs; the arithmetic is the textbook forward algorithm in log space:
//     la_1(j) = log pi_j + log B[j, o_1]
//     la_t(j) = LSE_i(la_{t-1}(i) + log A[i, j]) + log B[j, o_t],   logL = LSE_j la_T(j)
// evaluated as la_t(j) = m + log sum_i exp(la_{t-1}(i) - m) A[i, j] + log B[j, o_t] with
// m = max_i la_{t-1}(i) (max-shifted sum of exponentials; A = exp(log A) precomputed).
// Each sequence keeps la = c + r with r in FP32 and the running offset c (the sum of the
// per-step maxima, a sum of log scale factors) in FP64.
//
// k_plain_warp<J> (K <= 32 J, J <= 2): one warp per sequence, no block-wide synchronisation; exp(log A)
// in registers, the emission table log B^T in shared memory.  More states: k_hmm_rows_log.cu.
//
// What bounds it: with a few hundred sequences a scheduler has one warp, and a step is the chain
// maximum - exp - exchange through shared memory - products - log.  Each half warp takes every other
// four rows and 2 J columns a lane (so a step reads half the shared memory that J columns of all rows
// would: the four warps of an SM share one path), then the halves exchange J sums.  The products are
// FFMA2 in 2 J chains, the maximum is one redux, the next step's emission is fetched a step ahead, and
// a lane keeps the shift of one step in 32, so that the FP64 sum takes one addition per 32 steps.
// 512 sequences of 1,000 steps, K = 64: 217 us, 420 cycles a step (128 of them FFMA2 issue); with J
// chains of 64 dependent FMAs, a shuffle tree and an FP64 addition a step: 398 us.  Two blocks an SM:
// ptxas aims at three otherwise, with 168 registers instead of 192, and a step takes 570 cycles
// (4,096 sequences, where occupancy could help: 1.05 ms, 1.11 with three).
#include "common.cuh"
#include "hmm_internal.cuh"

namespace accel {
namespace hmm {

namespace rows {
size_t log_ws_bytes(int K, int M, int64_t S);
accel_status log_forward(const accel_hmm_model* m, const int32_t* obs, const int64_t* off, int64_t S, double* loglik,
                         char* ws, int32_t* d_status, cudaStream_t st);
}

// ---------------------------------------------------------------- warp per sequence
template <int J>
__global__ void __launch_bounds__(128, 2)
k_plain_warp(const float* __restrict__ logA, const float* __restrict__ logB, const float* __restrict__ logpi,
             int K, int M, const int32_t* __restrict__ obs, const int64_t* __restrict__ off, int64_t S,
             double* __restrict__ loglik) {
    constexpr int CW = 2 * J;                // columns of a lane's products; J of them are its own
    extern __shared__ float smem[];
    float* sB = smem;                                  // [M][K]  log B^T
    float* sP = smem + (((size_t)M * K + 3) & ~(size_t)3);   // [4][32 J] per-warp, 16-byte aligned
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll 4
    for (int idx = threadIdx.x; idx < M * K; idx += blockDim.x) {
        int j = idx / M, k = idx - j * M;
        sB[k * K + j] = logB[idx];
    }
    __syncthreads();
    const int64_t s = blockIdx.x * 4 + w;
    if (s >= S) return;

    const int h = lane >> 4, l = lane & 15;
    const int j0 = CW * l + J * h;           // the lane's own columns: j0 .. j0 + J - 1
    // rows 8 i + 4 h + 2 k and the one after (i < 4 J, k < 2), columns CW l + c.  The loads are
    // unconditional: behind a test each one waits for the one before.
    float2 a[4 * J][2][CW];
#pragma unroll
    for (int i = 0; i < 4 * J; ++i)
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int c = 0; c < CW; ++c) {
                const int row = 8 * i + 4 * h + 2 * k, col = min(CW * l + c, K - 1);
                a[i][k][c] = make_float2(logA[min(row, K - 1) * K + col], logA[min(row + 1, K - 1) * K + col]);
            }
#pragma unroll
    for (int i = 0; i < 4 * J; ++i)
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int c = 0; c < CW; ++c) {
                const int row = 8 * i + 4 * h + 2 * k, col = CW * l + c;
                a[i][k][c].x = col < K && row < K ? __expf(a[i][k][c].x) : 0.f;
                a[i][k][c].y = col < K && row + 1 < K ? __expf(a[i][k][c].y) : 0.f;
            }
    float* P = sP + w * 32 * J;
    const int64_t o0 = off[s];
    const int64_t T = off[s + 1] - o0;
    const int32_t* o = obs + o0;
    bool own[J];
    int jc[J];                               // (a column within the table for those beyond it)
#pragma unroll
    for (int jj = 0; jj < J; ++jj) {
        own[jj] = j0 + jj < K;
        jc[jj] = min(j0 + jj, K - 1);
    }

    float r[J], lb[J];
    int32_t ob = o[0];
#pragma unroll
    for (int jj = 0; jj < J; ++jj) r[jj] = own[jj] ? logpi[j0 + jj] + sB[ob * K + j0 + jj] : -INFINITY;
    double c = 0.0;                          // the lane's share of the shifts: steps with t mod 32 = lane
    int32_t ochunk = lane < T ? o[lane] : 0;           // lane l holds o[32 floor(t / 32) + l]
    ob = __shfl_sync(0xffffffffu, ochunk, 1);
#pragma unroll
    for (int jj = 0; jj < J; ++jj) lb[jj] = sB[ob * K + jc[jj]];
    for (int64_t tb = 0; tb < T; tb += 32) {
        const int32_t next = tb + 32 + lane < T ? o[tb + 32 + lane] : 0;
        const int t0 = tb == 0 ? 1 : 0, t1 = T - tb < 32 ? (int)(T - tb) : 32;
        float shift = 0.f;
#pragma unroll 1
        for (int t = t0; t < t1; ++t) {
            float m = r[0];
#pragma unroll
            for (int jj = 1; jj < J; ++jj) m = fmaxf(m, r[jj]);
            m = warp_max_f32(m);
            if (J == 2) *reinterpret_cast<float2*>(P + j0) = make_float2(__expf(r[0] - m), __expf(r[J - 1] - m));
            else P[j0] = __expf(r[0] - m);
            __syncwarp();
            float2 acc[CW];
#pragma unroll
            for (int k = 0; k < CW; ++k) acc[k] = make_float2(0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 4 * J; ++i) {
                const float4 p = reinterpret_cast<const float4*>(P)[2 * i + h];
#pragma unroll
                for (int k = 0; k < CW; ++k) acc[k] = __ffma2_rn(make_float2(p.x, p.y), a[i][0][k], acc[k]);
#pragma unroll
                for (int k = 0; k < CW; ++k) acc[k] = __ffma2_rn(make_float2(p.z, p.w), a[i][1][k], acc[k]);
            }
            // the other 16 lanes' rows: each lane of a pair gives the columns that are the other's
            float sum[J];
#pragma unroll
            for (int jj = 0; jj < J; ++jj) {
                const float u = acc[jj].x + acc[jj].y, v = acc[jj + J].x + acc[jj + J].y;
                sum[jj] = (h ? v : u) + __shfl_xor_sync(0xffffffffu, h ? u : v, 16);
            }
#pragma unroll
            for (int jj = 0; jj < J; ++jj) r[jj] = own[jj] ? __logf(sum[jj]) + lb[jj] : -INFINITY;
            shift = lane == t ? m : shift;
            // the next step's symbol
            ob = __shfl_sync(0xffffffffu, t == 31 ? next : ochunk, (t + 1) & 31);
#pragma unroll
            for (int jj = 0; jj < J; ++jj) lb[jj] = sB[ob * K + jc[jj]];
        }
        c += (double)shift;
        ochunk = next;
    }
    float m = r[0];
#pragma unroll
    for (int jj = 1; jj < J; ++jj) m = fmaxf(m, r[jj]);
    m = warp_max_f32(m);
    float e = 0.f;
#pragma unroll
    for (int jj = 0; jj < J; ++jj) e += __expf(r[jj] - m);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) e += __shfl_xor_sync(0xffffffffu, e, d);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
    if (lane == 0) loglik[s] = c + (double)m + log((double)e);
}

size_t plain_ws_bytes(int K, int M, int64_t S) { return K <= 64 ? 0 : rows::log_ws_bytes(K, M, S); }

accel_status plain_forward(const accel_hmm_model* m, const int32_t* obs, const int64_t* off, int64_t S,
                           double* loglik, char* ws, int32_t* d_status, cudaStream_t st) {
    const int K = m->K, M = m->M;
    if (K <= 64) {
        size_t smem = ((((size_t)M * K + 3) & ~(size_t)3) + 4 * 64) * sizeof(float);
        ACCEL_REQUIRE(smem <= (size_t)max_smem_optin(), ACCEL_ERR_UNSUPPORTED, "hmm_forward: M*K too large for the FP32 kernel");
        unsigned grid = (unsigned)((S + 3) / 4);
        if (K <= 32) {
            ACCEL_CUDA_TRY(cudaFuncSetAttribute(k_plain_warp<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            k_plain_warp<1><<<grid, 128, smem, st>>>(m->log_A, m->log_B, m->log_pi, K, M, obs, off, S, loglik);
        } else {
            ACCEL_CUDA_TRY(cudaFuncSetAttribute(k_plain_warp<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            k_plain_warp<2><<<grid, 128, smem, st>>>(m->log_A, m->log_B, m->log_pi, K, M, obs, off, S, loglik);
        }
        return after_launch(st, "hmm_forward(fp32 warp)", 1);
    }
    // the models taken: a K x K stream ring, the emission table and eight vectors within shared memory
    const size_t Kp = (size_t)((K + 3) & ~3);
    const size_t bytes = align_up(3 * 32 * Kp * 4 + 24, 16) + ((((size_t)M * K + 3) & ~(size_t)3) + 8 * Kp) * sizeof(float);
    ACCEL_REQUIRE(bytes <= (size_t)max_smem_optin(), ACCEL_ERR_UNSUPPORTED, "hmm_forward: M*K too large for the FP32 kernel");
    return rows::log_forward(m, obs, off, S, loglik, ws, d_status, st);
}

}  // namespace hmm
}  // namespace accel
