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
// k_plain_warp<J> (K <= 32 J, J <= 2): one warp per sequence, no block-wide synchronisation; lane l owns
// states l and l + 32, their columns of exp(log A) in registers, the emission table log B^T in shared
// memory.  More states: k_hmm_rows_log.cu.
//
// What bounds it: with a few hundred sequences a scheduler has one warp, and a step is the chain
// maximum - exp - exchange through shared memory - products - log.  The products are J chains of K FMAs in
// the order of the rows.  (Four chains a column and half the shared-memory reads take 420 cycles a step
// instead of 470, but r is rounded at a magnitude of several units, so another order of the sum moves logL
// by up to 1e-8 of itself in short sequences of few symbols.)  The maximum is one redux, the next step's
// emission is fetched a step ahead, and a lane keeps the shift of one step in 32, so that the FP64 sum
// takes one addition per 32 steps.  512 sequences of 1,000 steps, K = 64: 242 us; with a shuffle tree and
// an FP64 addition a step, and one load of A after the other, 398 us.  Two blocks an SM: ptxas aims at
// three otherwise, with 168 registers.
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

    // a[jj][i] = A[i, lane + 32 jj].  The loads are unconditional: behind a test each one waits for the one
    // before.
    float a[J][32 * J];
    bool own[J];
    int jc[J];                               // (a column within the table for those beyond it)
#pragma unroll
    for (int jj = 0; jj < J; ++jj) {
        own[jj] = lane + 32 * jj < K;
        jc[jj] = min(lane + 32 * jj, K - 1);
#pragma unroll
        for (int i = 0; i < 32 * J; ++i) a[jj][i] = logA[min(i, K - 1) * K + jc[jj]];
    }
#pragma unroll
    for (int jj = 0; jj < J; ++jj)
#pragma unroll
        for (int i = 0; i < 32 * J; ++i) a[jj][i] = own[jj] && i < K ? __expf(a[jj][i]) : 0.f;
    float* P = sP + w * 32 * J;
    const int64_t o0 = off[s];
    const int64_t T = off[s + 1] - o0;
    const int32_t* o = obs + o0;

    float r[J], lb[J];
    int32_t ob = o[0];
#pragma unroll
    for (int jj = 0; jj < J; ++jj) r[jj] = own[jj] ? logpi[jc[jj]] + sB[ob * K + jc[jj]] : -INFINITY;
    double c = 0.0;
    int32_t ochunk = lane < T ? o[lane] : 0;           // lane l holds o[32 floor(t / 32) + l]
    ob = __shfl_sync(0xffffffffu, ochunk, 1);
#pragma unroll
    for (int jj = 0; jj < J; ++jj) lb[jj] = sB[ob * K + jc[jj]];
    for (int64_t tb = 0; tb < T; tb += 32) {
        const int32_t next = tb + 32 + lane < T ? o[tb + 32 + lane] : 0;
        const int t0 = tb == 0 ? 1 : 0, t1 = T - tb < 32 ? (int)(T - tb) : 32;
        float shift = 0.f;                   // lane l keeps the shift of step tb + l
        for (int t = t0; t < t1; ++t) {
            float m = r[0];
#pragma unroll
            for (int jj = 1; jj < J; ++jj) m = fmaxf(m, r[jj]);
            m = warp_max_f32(m);
#pragma unroll
            for (int jj = 0; jj < J; ++jj) P[lane + 32 * jj] = __expf(r[jj] - m);
            __syncwarp();
            float acc[J];
#pragma unroll
            for (int jj = 0; jj < J; ++jj) acc[jj] = 0.f;
#pragma unroll
            for (int i4 = 0; i4 < 8 * J; ++i4) {
                const float4 p = reinterpret_cast<const float4*>(P)[i4];
#pragma unroll
                for (int jj = 0; jj < J; ++jj) acc[jj] = fmaf(p.x, a[jj][4 * i4 + 0], acc[jj]);
#pragma unroll
                for (int jj = 0; jj < J; ++jj) acc[jj] = fmaf(p.y, a[jj][4 * i4 + 1], acc[jj]);
#pragma unroll
                for (int jj = 0; jj < J; ++jj) acc[jj] = fmaf(p.z, a[jj][4 * i4 + 2], acc[jj]);
#pragma unroll
                for (int jj = 0; jj < J; ++jj) acc[jj] = fmaf(p.w, a[jj][4 * i4 + 3], acc[jj]);
            }
            __syncwarp();
#pragma unroll
            for (int jj = 0; jj < J; ++jj) r[jj] = own[jj] ? __logf(acc[jj]) + lb[jj] : -INFINITY;
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
            ACCEL_CUDA_TRY(allow_smem((const void*)k_plain_warp<1>, smem));
            k_plain_warp<1><<<grid, 128, smem, st>>>(m->log_A, m->log_B, m->log_pi, K, M, obs, off, S, loglik);
        } else {
            ACCEL_CUDA_TRY(allow_smem((const void*)k_plain_warp<2>, smem));
            k_plain_warp<2><<<grid, 128, smem, st>>>(m->log_A, m->log_B, m->log_pi, K, M, obs, off, S, loglik);
        }
        return after_launch(st, "hmm_forward(fp32 warp)", 1);
    }
    // The models taken: those whose rows ring, emission table and eight vectors once fitted shared memory.  The
    // kernel needs none of it (the table is read from global memory); the limit stays as the call's contract.
    const size_t Kp = (size_t)((K + 3) & ~3);
    const size_t bytes = align_up(3 * 32 * Kp * 4 + 24, 16) + ((((size_t)M * K + 3) & ~(size_t)3) + 8 * Kp) * sizeof(float);
    ACCEL_REQUIRE(bytes <= (size_t)max_smem_optin(), ACCEL_ERR_UNSUPPORTED, "hmm_forward: M*K too large for the FP32 kernel");
    return rows::log_forward(m, obs, off, S, loglik, ws, d_status, st);
}

}  // namespace hmm
}  // namespace accel
