// FP32 log-space forward of the models with more than 64 states (K7): the recursion
//     la_t(j) = m + log sum_i exp(la_{t-1}(i) - m) A[i, j] + log B[j, o_t]
// on the CTAs and CTA pairs of hmm_rows.cuh, which keep exp(log A) in registers.  A sequence's
// la = c + r, r in FP32 and the offset c (the sum of the shifts m) in FP64.
//
// The shift is the largest r.  An epilogue warp holds a slot's row of the CTA's columns, so its maximum
// is one warp reduction; the warps of a pair's CTAs exchange theirs (a word and an mbarrier per slot
// and step parity) before the exponentials, and the other half's products hide the way.
//
// A column's sum runs over the rows in order, one FMA after the other, like the sum of the kernel for
// fewer states: r is rounded at a magnitude of several units, so any other order moves logL by up to
// 1e-8 of itself in short sequences of few symbols.  For the same reason log(sum) + log B is one FMA.
//
// What bounds it: the shared-memory reads of the vectors (a thread has one column, so 16 bytes serve four
// FMAs) beside the FMAs.  1,024 sequences of 200 to 2,000 steps (1.13M steps) at K = 256: 5.4 ms, 2.0 ms of
// them FMAs; with the products of the other recurrences (16 FMAs for 16 bytes, eight partial sums a
// column) 3.9 ms, but 5e-9 of logL away.  One CTA per 8 sequences that streamed A from L2 every step:
// 31.5 ms, and the same results.
#include "hmm_rows.cuh"

namespace accel {
namespace hmm {
namespace rows {

namespace cg = cooperative_groups;

namespace {

struct LogPrm {
    int64_t S;
    int32_t ncl;
    const float *A, *logBT, *logpi;         // padded: exp(log A) [KP][KP], log B^T [M][KP], log pi [KP]
    const int32_t* obs;
    const int64_t* off;
    const int32_t* order;
    double* loglik;
    int32_t* status;
};

// Padded parameters; padded states have log-probability -inf.  An empty sequence, which no slot takes,
// has no log-likelihood.
__global__ void k_log_prep(const int64_t* __restrict__ off, int64_t S, double* __restrict__ loglik,
                           const float* __restrict__ logA, const float* __restrict__ logB, const float* __restrict__ logpi,
                           int K, int KP, int M, float* __restrict__ A, float* __restrict__ logBT,
                           float* __restrict__ lpi) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < S; s += (int64_t)gridDim.x * blockDim.x)
        if (off[s + 1] <= off[s]) loglik[s] = NAN;
    const int64_t nA = (int64_t)KP * KP, nB = (int64_t)M * KP;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < nA + nB + KP;
         idx += (int64_t)gridDim.x * blockDim.x) {
        if (idx < nA) {
            const int r = (int)(idx / KP), c = (int)(idx % KP);
            A[idx] = r < K && c < K ? __expf(logA[(int64_t)r * K + c]) : 0.f;
        } else if (idx < nA + nB) {
            const int64_t q = idx - nA;
            const int k = (int)(q / KP), j = (int)(q % KP);
            logBT[q] = j < K ? logB[(int64_t)j * M + k] : -INFINITY;
        } else {
            const int j = (int)(idx - nA - nB);
            lpi[j] = j < K ? logpi[j] : -INFINITY;
        }
    }
}

template <int N>
__device__ __forceinline__ float warp_max(const Vec<N>& v) {
    float m = v.v[0];
#pragma unroll
    for (int h = 1; h < N; ++h) m = fmaxf(m, v.v[h]);
    return warp_max_f32(m);
}

// Shared memory beside the engine's: the maxima of the peer's columns.
template <int KP>
struct LogSmem {
    Smem<KP> s;
    uint64_t max_full[2][kG];                      // [step parity][slot]
    float max_peer[2][kG];
    Mid<KP> mid;
};

// Step i of a slot forms r_t; its exponentials, shifted by the largest, are the next vector.
template <int KP>
__device__ __forceinline__ void log_epilogue(const LogPrm& p, int rank, int cid, LogSmem<KP>& ls, const uint32_t (&half)[2],
                                             Waits& wt) {
    using C = Cfg<KP>;
    Smem<KP>& sm = ls.s;
    Epilogue<KP> ep(sm, rank, true);
    const int u = ep.u;
    const int64_t n = (int64_t)p.ncl * kG;
    const int32_t* obs = p.obs + p.off[0];
    const int c = rank * C::Kh + ep.col;
    const bool lead = rank == C::NC - 1 && ep.lane == 0;
    uint32_t peer_max = 0, peer_full = 0;        // shared::cluster addresses of the peer's
    if constexpr (C::NC == 2) {
        peer_max = tc::cluster_addr(&ls.max_peer[0][0], (uint32_t)(rank ^ 1));
        peer_full = tc::cluster_addr(&ls.max_full[0][0], (uint32_t)(rank ^ 1));
    }
    auto any = [](int64_t, int64_t) { return true; };
    Vec<C::EC> pi;
    pi.load(p.logpi + c);
    Slot s;
    int64_t row, left;
    int32_t sym, nsym;
    bool fresh;
    double off_c;                             // c: the shifts of the sequence so far
    // the sequence that ended with the step before (-1: none): its c and the sums of the exponentials of
    // the CTA's columns, 32 by 32
    int32_t pseq;
    double pc;
    float psum[4];
    auto begin = [&]() {
        next_seq(s, p.S, n, p.order, p.off, any);
        fresh = true;
        off_c = 0.0;
        if (s.seq < 0) return;
        row = s.o0;
        left = s.T - 1;
        sym = obs[row];
        nsym = left > 0 ? obs[row + 1] : 0;
    };
    s.k = -1;
    s.sl = cid + p.ncl * ep.g;
    row = left = 0;
    sym = nsym = 0;
    pseq = -1;
    pc = 0.0;
    psum[0] = psum[1] = psum[2] = psum[3] = 0.f;
    begin();
    auto finish = [&](int32_t ended, uint32_t it) {
        if (ended < 0) return;
        const int pb = (int)(it & 1) ^ 1;
        if (C::NC == 2) wt.cluster(&sm.x_peer[u][pb], step_phase(it - 1));
        if (!lead) return;
        float sum = rank == 1 ? sm.peer[pb][ep.g] : 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) sum += psum[k];
        p.loglik[ended] = pc + log((double)sum);
    };
    const uint32_t steps = half[u];
    for (uint32_t it = 0; it <= steps; ++it) {
        const int b = (int)(it & 1);
        const bool on = s.seq >= 0;
        const int32_t ended = pseq;
        pseq = -1;
        if (it < steps) {
            Vec<C::EC> lb, r, x;
            if (on) lb.load(p.logBT + (size_t)sym * KP + c);
            if (it > 0) {
                wt.local(&sm.out_full[u], (uint32_t)(it - 1) & 1u);
                r.load(&sm.out[u][ep.g & 3][ep.col]);
            }
#pragma unroll
            for (int h = 0; h < C::EC; ++h)       // (not one sum of a choice: log + lb is to stay one FMA)
                r.v[h] = !on ? -INFINITY : fresh ? __fadd_rn(pi.v[h], lb.v[h]) : __logf(r.v[h]) + lb.v[h];
            float m = warp_max(r);
            if constexpr (C::NC == 2) {
                if (ep.lane == 0) {
                    const uint32_t q = (uint32_t)(b * kG + ep.g);
                    tc::st_async1(peer_max + 4u * q, m, peer_full + 8u * q);
                    tc::mbar_arrive_expect_tx(&ls.max_full[b][ep.g], 4u);
                }
                wt.cluster(&ls.max_full[b][ep.g], step_phase(it));
                m = fmaxf(m, ls.max_peer[b][ep.g]);
            }
#pragma unroll
            for (int h = 0; h < C::EC; ++h) x.v[h] = on ? __expf(r.v[h] - m) : 0.f;
            // At the end of a sequence the sum of the exponentials is wanted, too: 32 columns by a butterfly
            // (the highest bit of the column first), these sums in the order of the columns, so the second
            // CTA goes on from the first one's.
            float e4[4] = {};
            if (on && left == 0) {
                Vec<C::EC> e = x;
#pragma unroll
                for (int d = 4; d > 0; d >>= 1)
#pragma unroll
                    for (int h = 0; h < C::EC; ++h) e.v[h] += __shfl_xor_sync(0xffffffffu, e.v[h], d);
                const float sum = (e.v[0] + e.v[2]) + (e.v[1] + e.v[3]);
#pragma unroll
                for (int k = 0; k < 4; ++k) e4[k] = __shfl_sync(0xffffffffu, sum, 8 * k);
            }
            ep.put(b, x, true, ((e4[0] + e4[1]) + e4[2]) + e4[3]);
            finish(ended, it);
            // on to the next step
            if (on) {
                off_c += (double)m;
                if (left == 0) {
                    pseq = s.seq;
                    pc = off_c;
#pragma unroll
                    for (int k = 0; k < 4; ++k) psum[k] = e4[k];
                    begin();
                } else {
                    fresh = false;
                    ++row;
                    --left;
                    sym = nsym;
                    nsym = left > 0 ? obs[row + 1] : 0;
                }
            }
        } else {
            finish(ended, it);
        }
    }
}

template <int KP>
__device__ __forceinline__ void log_body(const LogPrm& p, int rank, int cid, LogSmem<KP>& ls, cg::cluster_group* cl) {
    if (threadIdx.x == 0)
        for (int q = 0; q < 2 * kG; ++q) tc::mbar_init(&ls.max_full[0][0] + q, 1);
    ls.mid.init();
    init_bars(ls.s, Mid<KP>::W);
    uint32_t half[2];          // (a slot's steps fit 32 bits: 2^32 of them would take two hours)
    slot_totals(ls.s.tot, p.S, (int64_t)p.ncl * kG, cid, p.ncl, p.order, p.off, [](int64_t, int64_t) { return true; }, half);
    if constexpr (Cfg<KP>::NC == 2) cl->sync();  // the peer's barriers exist before any remote store
    Waits wt{p.status};
    if (threadIdx.x < kCon) {
        regs_contraction<KP>();
        products_in_order<KP>(p.A, rank, ls.s, ls.mid, half, wt);
    } else {
        regs_epilogue<KP>();
        log_epilogue<KP>(p, rank, cid, ls, half, wt);
    }
    if constexpr (Cfg<KP>::NC == 2) cl->sync();  // the peer no longer addresses this CTA's shared memory
}

__global__ void __launch_bounds__(kT, Cfg<128>::MINB) k_rows_log(LogPrm p) {
    __shared__ __align__(16) LogSmem<128> ls;
    log_body<128>(p, 0, (int)blockIdx.x, ls, nullptr);
}
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kT, 1) k_rows_log_pair(LogPrm p) {
    __shared__ __align__(16) LogSmem<256> ls;
    cg::cluster_group cl = cg::this_cluster();
    log_body<256>(p, (int)cl.block_rank(), (int)(blockIdx.x >> 1), ls, &cl);
}

struct LogLayout {
    size_t A, lbt, pi, order, total;
    int KP;
};
LogLayout log_layout(int K, int M, int64_t S) {
    LogLayout L;
    L.KP = K <= 128 ? 128 : 256;
    size_t o = 0;
    auto take = [&](size_t bytes) { size_t r = o; o = align_up(o + bytes, 256); return r; };
    L.A = take((size_t)L.KP * L.KP * 4);
    L.lbt = take((size_t)M * L.KP * 4);
    L.pi = take((size_t)L.KP * 4);
    L.order = o;
    L.total = o + order_ws_bytes(S);
    return L;
}

}  // namespace

size_t log_ws_bytes(int K, int M, int64_t S) { return log_layout(K, M, S).total; }

accel_status log_forward(const accel_hmm_model* m, const int32_t* obs, const int64_t* off, int64_t S, double* loglik,
                         char* ws, int32_t* d_status, cudaStream_t st) {
    const LogLayout L = log_layout(m->K, m->M, S);
    LogPrm p{};
    p.S = S;
    p.A = (float*)(ws + L.A);
    p.logBT = (float*)(ws + L.lbt);
    p.logpi = (float*)(ws + L.pi);
    p.obs = obs;
    p.off = off;
    p.order = (int32_t*)(ws + L.order);
    p.loglik = loglik;
    p.status = d_status;
    k_log_prep<<<num_sms() * 2, 256, 0, st>>>(off, S, loglik, m->log_A, m->log_B, m->log_pi, m->K, L.KP, m->M, (float*)p.A,
                                              (float*)p.logBT, (float*)p.logpi);
    accel_status r = order_by_length(off, S, (int32_t*)(ws + L.order), ws + L.order + align_up((size_t)S * 4, 256), st);
    if (r != ACCEL_OK) return r;
    auto kern = L.KP == 128 ? k_rows_log : k_rows_log_pair;
    p.ncl = clusters_for(kern, L.KP, S, 0);
    kern<<<(unsigned)(p.ncl * (L.KP == 256 ? 2 : 1)), kT, 0, st>>>(p);
    return after_launch(st, "hmm_forward(fp32 rows)", 5);
}

}  // namespace rows
}  // namespace hmm
}  // namespace accel
