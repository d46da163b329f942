// Internal interfaces shared by the HMM kernels and the hmm_forward / hmm_adjoint entry
// points (not part of the C ABI).
#pragma once
#include "common.cuh"

namespace accel {
namespace hmm {

// Layout of the status block at the start of every HMM workspace.
constexpr size_t kDebugScratchOff = 0;   // 8 bytes for debug-mode checks
constexpr size_t kStatusOff = 8;         // int32 device status (ACCEL_OK or an error code)
constexpr size_t kQueueOff = 16;         // uint64 sequence-queue counter

// Sequence order by decreasing length (approximate: 1024 logarithmic length buckets), so
// that long sequences start first and groups of consecutive sequences have similar
// lengths.  order[q] = sequence index.  Scratch: order_ws_bytes(S) - S*4 bytes after order.
size_t order_ws_bytes(int64_t S);
accel_status order_by_length(const int64_t* d_off, int64_t S, int32_t* d_order, char* scratch, cudaStream_t st);

// The largest of the warp's values (one instruction; NaNs are left out, as by fmaxf).
__device__ __forceinline__ float warp_max_f32(float v) {
    float m;
    asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(v));
    return m;
}

// FP32 log-space forward (k_hmm_plain.cu, k_hmm_rows_log.cu).
size_t plain_ws_bytes(int K, int M, int64_t S);
accel_status plain_forward(const accel_hmm_model* m, const int32_t* obs, const int64_t* off, int64_t S,
                           double* loglik, char* ws, int32_t* d_status, cudaStream_t st);

// Launch configuration of the BF16 tensor-core forward, chosen by the autotuner
// (hmm_autotune.cu): one CTA takes tiles of 2 rows / split sequences (split 2 or 4, rows 32, 64 or
// 128: tiles of 16 to 128).  `pair` is kept for configurations saved by earlier versions, which
// split a tile over a cluster of two (1) or four (2) CTAs: it says what their units were.
struct TcConfig {
    int split;
    int rows;
    int pair;
    int units;      // persistent CTAs launched, or pairs or fours of them (pair); 0: all that fit
};
TcConfig tile_config(int n);             // the configuration of a tile of n sequences
TcConfig default_config(int64_t S);      // ... used without a tuned one
bool tuned_entry(int K, int M, int64_t S, TcConfig* out);    // the tuned configuration, if there is one

// BF16 tensor-core scaled forward (k_hmm_tc.cu); cfg null: the tile is chosen from S and, past
// tiles of 16, from the lengths on the device.
accel_status tc_forward_cfg(const accel_hmm_model* m, const int32_t* obs, const int64_t* off, int64_t S,
                            double* loglik, char* ws, int32_t* d_status, const TcConfig* cfg, cudaStream_t st);
size_t tc_ws_bytes(int K, int M, int64_t S);
accel_status tc_forward(const accel_hmm_model* m, const int32_t* obs, const int64_t* off, int64_t S,
                        double* loglik, char* ws, int32_t* d_status, cudaStream_t st);
bool tc_supported(int K, int M);

// Tensor-core (TF32, hi/lo split) accumulation of the adjoint's transition and emission
// counts over the row buffers of one backward round (k_xi_tc.cu):
//   Upart[g] += P^T Q over rows [0, *rows_r), and, when cntp is not null,
//   cntp[g][i][k] += sum_rows G[row][i] [osym[row] == k].
// The rows are divided into xi_tc_splits(K) contiguous ranges; clusters of consecutive
// ranges add their sums together, so there are xi_tc_partials(K) partials g.
constexpr int kXiSplitMax = 160;
bool xi_tc_supported(int K);
bool xi_tc_counts_supported(int K, int M);
int xi_tc_splits(int K, int M, bool counts);
int xi_tc_partials(int K, int M, bool counts);   // partials the splits leave (one per cluster)
accel_status xi_tc_round(const float* P, const float* Q, const float* G, const int32_t* osym, const int32_t* rows_r,
                         int K, int M, float* Upart, float* cntp, int32_t* status, cudaStream_t st);

}  // namespace hmm
}  // namespace accel
