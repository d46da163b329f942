// The adjoint with every alpha kept (hmm_adj_rows.cu), as hmm_adjoint.cu calls it.
#pragma once
#include "hmm_internal.cuh"

namespace accel {
namespace hmm {
namespace rows {

struct RowsArgs {
    const accel_hmm_model* m;
    const int32_t* obs;
    const int64_t* off;
    int64_t S, total_T;
    int Cmax;               // ceil(sqrt(max_T)): a sequence whose own is larger, or that lies past total_T, is
                            // reported, not computed
    void* ws;
    int32_t* status;
};

// U[part] = X^T Q over the part's share of *d_rows rows (k_rows_xi.cu): xi_parts(KP, rows) partials of
// KP x KP.
int xi_parts(int KP, int64_t rows);
accel_status xi_rows(const float* X, const float* Q, const int32_t* d_rows, int KP, int parts, float* U,
                     int32_t* status, cudaStream_t st);

// Workspace bytes of these sizes, 0 where their rows are not kept.
size_t rows_ws_bytes(int K, int M, int64_t S, int64_t total_T);
accel_status rows_forward(const RowsArgs& a, double* d_loglik, cudaStream_t st, int& nlaunch);
accel_status rows_backward(const RowsArgs& a, const double* d_weights, float* gA, float* gB, float* gpi,
                           cudaStream_t st, int& nlaunch);

}  // namespace rows
}  // namespace hmm
}  // namespace accel
