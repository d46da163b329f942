// The adjoint of the scaled HMM forward recursion with every alpha kept (K9, the default form).
//
//   forward:   X_t = (X_{t-1} 2^-e_{t-1} A) o b(o_t),  X_0 = pi o b(o_0),  c_t = sum_j X_t(j) = f 2^e_t
//              logL = ln2 sum_{t<T-1} e_t + ln c_{T-1}
//   backward:  R_{T-1} = 1 / c_{T-1},  v_{t+1} = 2^-e_t b(o_{t+1}) o R_{t+1},  R_t = A v_{t+1}
//   counts:    xi(i,j) = A_ij sum_t X_t(i) w v_{t+1}(j),   gamma_t = w X_t o R_t
//
// The rows X_t, w v_{t+1} and gamma_t of every step go to memory (12 KP bytes a step, at the row
// off[s] + t of the flat observations), so nothing is recomputed and one launch runs all steps of
// all sequences forward, one backward, and one contracts the rows on the tensor cores
// (k_rows_xi.cu).  The checkpointed form (hmm_adjoint.cu) recomputes X segment by segment in
// sqrt(T) rounds: it needs 5 to 6 times less memory and is kept for calls whose rows would not
// fit kRowBytesMax or the caller's workspace.  Rows count from the first sequence's offset.
#include "hmm_adj_rows.cuh"
#include "hmm_rows.cuh"

#include <algorithm>

namespace accel {
namespace hmm {
namespace rows {

namespace cg = cooperative_groups;

struct RowsPrm {
    int64_t S, rows;                        // sequences; rows there is room for
    int32_t ncl, K, M, Cmax;
    const float *A, *At, *BT, *pi;          // padded: [KP][KP], its transpose, [M][KP], [KP]
    const int32_t* obs;
    const int64_t* off;
    const int32_t* order;                   // null: the sequences as given
    const double* w;                        // weights or null
    float *X, *Q, *Gm;                      // rows [total_T][KP]
    int32_t* e;                             // exponents [total_T]
    float* clast;                           // c_{T-1} [S]
    double* loglik;                         // [S] or null
    int32_t* status;
};

// Padded parameters.
__global__ void k_rows_prep(const float* __restrict__ logA, const float* __restrict__ logB,
                            const float* __restrict__ logpi, int K, int KP, int M, float* __restrict__ A,
                            float* __restrict__ At, float* __restrict__ BT, float* __restrict__ pi,
                            const int64_t* __restrict__ off, int64_t S, int64_t room, int32_t* __restrict__ d_rows) {
    const int64_t nA = (int64_t)KP * KP, nB = (int64_t)M * KP;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < 2 * nA + nB + KP;
         idx += (int64_t)gridDim.x * blockDim.x) {
        if (idx < 2 * nA) {
            const int64_t q = idx < nA ? idx : idx - nA;
            const int r = (int)(q / KP), c = (int)(q % KP);
            const float v = r < K && c < K ? __expf(idx < nA ? logA[(int64_t)r * K + c] : logA[(int64_t)c * K + r]) : 0.f;
            (idx < nA ? A : At)[q] = v;
        } else if (idx < 2 * nA + nB) {
            const int64_t q = idx - 2 * nA;
            const int k = (int)(q / KP), j = (int)(q % KP);
            BT[q] = j < K ? __expf(logB[(int64_t)j * M + k]) : 0.f;
        } else {
            const int j = (int)(idx - 2 * nA - nB);
            pi[j] = j < K ? __expf(logpi[j]) : 0.f;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *d_rows = (int32_t)min(off[S] - off[0], room);
}

// The scale exponent of a sum c = m 2^e, m in [0.5, 1), and 2^-e.
__device__ __forceinline__ int scale_exp(float c) {
    const int f = (int)((__float_as_uint(c) >> 23) & 0xffu);
    if (f == 0 || f == 0xff) {
        int e = 0;
        frexpf(c, &e);
        return e;
    }
    return f - 126;
}
__device__ __forceinline__ float pow2_scale(int e) {
    return (e > -127 && e < 127) ? __uint_as_float((uint32_t)(127 - e) << 23) : ldexpf(1.0f, -e);
}

__device__ __forceinline__ int seg_len(int64_t T) {       // ceil(sqrt(T)), as the checkpointed form
    int c = (int)ceil(sqrt((double)T));
    while ((int64_t)c * c < T) ++c;
    while (c > 1 && (int64_t)(c - 1) * (c - 1) >= T) --c;
    return c < 1 ? 1 : c;
}

// A sequence that the call's sizes have room for: of max_T, and within the rows (offsets past total_T).
__device__ __forceinline__ bool fits(const RowsPrm& p, int64_t o0, int64_t T) {
    return seg_len(T) <= p.Cmax && o0 >= 0 && o0 + T <= p.rows;
}

// Step i of a slot computes one X_t; the sum of X_{t-1}, and with it e_{t-1}, is complete by then.  A
// last step only finishes the last ones' books.
template <int KP, bool ORD>
__device__ __forceinline__ void fwd_epilogue(const RowsPrm& p, int rank, int cid, Smem<KP>& sm, const int32_t (&half)[2],
                                             Waits& wt) {
    using C = Cfg<KP>;
    Epilogue<KP> ep(sm, rank, ORD);
    const int u = ep.u;
    const int64_t n = (int64_t)p.ncl * kG;
    const int32_t* obs = p.obs + p.off[0];       // rows and symbols count from the first sequence
    const int c = rank * C::Kh + ep.col;
    const bool lead = rank == 0 && ep.lane == 0;
    auto ok = [&](int64_t o0, int64_t T) {
        if (fits(p, o0, T)) return true;
        report_status(p.status, ACCEL_ERR_SHAPE);
        return false;
    };
    Vec<C::EC> pi;
    pi.load(p.pi + c);
    // the warp's slot: the sequence, the step to compute (row, steps left after it), its symbol and
    // the one after
    Slot s;
    int32_t row, left, sym, nsym;
    bool fresh;
    // the step computed last: whether there was one, whether it ended its sequence, the CTA's sum of it
    int32_t pseq;
    bool pon, plast;
    float psum, e4[4] = {};
    int64_t E;
    auto begin = [&]() {
        next_seq(s, p.S, n, p.order, p.off, ok);
        fresh = true;
        if (s.seq < 0) return;
        row = (int32_t)s.o0;
        left = (int32_t)s.T - 1;
        sym = obs[row];
        nsym = left > 0 ? obs[row + 1] : 0;
    };
    s.k = -1;
    s.sl = cid + p.ncl * ep.g;
    row = left = sym = nsym = 0;
    pon = plast = false;
    pseq = -1;
    psum = 0.f;
    E = 0;
    begin();
    const int32_t steps = half[u];
    for (int32_t it = 0; it <= steps; ++it) {
        const int b = (int)(it & 1), pb = b ^ 1;
        const bool on = s.seq >= 0;
        Vec<C::EC> em, o;
        if (on) em.load(p.BT + (size_t)sym * KP + c);
        float sum = psum, peer_sum = 0.f;
        const float last4[4] = {e4[0], e4[1], e4[2], e4[3]};
        if (it > 0) {
            if (C::NC == 2) {                // the peer's sum: in the order of the columns
                wt.cluster(&sm.x_peer[u][pb], step_phase(it - 1));
                const float q = sm.peer[pb][ep.g];
                peer_sum = q;
                sum = rank == 0 ? sum + q : q + sum;
            }
            if (it < steps) {
                wt.local(&sm.out_full[u], (uint32_t)(it - 1) & 1u);
                o.load(&sm.out[u][ep.g & 3][ep.col]);
            }
        }
        const int ex = scale_exp(sum);
        if (it < steps) {
            const float sc = pow2_scale(ex);
            Vec<C::EC> x;
#pragma unroll
            for (int h = 0; h < C::EC; ++h) x.v[h] = on ? (fresh ? pi.v[h] : o.v[h] * sc) * em.v[h] : 0.f;
            // (the last step's sum is the sequence's c: in the checkpointed form's order)
            if (ORD && left == 0) {
                ep.sums_by32(x, e4);
                psum = ((e4[0] + e4[1]) + e4[2]) + e4[3];
            } else {
                psum = C::NC == 2 && left == 0 ? ep.warp_sum_by8(x) : ep.warp_sum(x);
            }
            ep.put(b, x, true, psum);
            if (on) x.store(p.X + (size_t)row * KP + c);
        }
        // the books of the step before
        if (pon) {
            if (plast) {
                float c_last = sum;
                if (ORD && C::NC == 2) {         // CTA 1 goes on from CTA 0's
                    c_last = peer_sum;
#pragma unroll
                    for (int k = 0; k < 4; ++k) c_last += last4[k];
                }
                if (ep.lane == 0 && rank == (ORD ? C::NC - 1 : 0)) {
                    p.clast[pseq] = c_last;
                    if (p.loglik) p.loglik[pseq] = 0.6931471805599453 * (double)E + log((double)c_last);
                }
                E = 0;
            } else {
                if (lead) p.e[row - 1] = ex;      // the sequence goes on: the row before this one
                E += ex;
            }
        }
        // on to the next step
        pon = on;
        plast = left == 0;
        pseq = s.seq;
        if (on) {
            if (left == 0) {
                begin();
            } else {
                fresh = false;
                ++row;
                --left;
                sym = nsym;
                nsym = left > 0 ? obs[row + 1] : 0;
            }
        }
    }
}

// Step i of a slot computes R_t (t from T - 1 down), gamma_t and v_t.
template <int KP>
__device__ __forceinline__ void bwd_epilogue(const RowsPrm& p, int rank, int cid, Smem<KP>& sm, const int32_t (&half)[2],
                                             Waits& wt) {
    using C = Cfg<KP>;
    Epilogue<KP> ep(sm, rank, false);
    const int u = ep.u;
    const int64_t n = (int64_t)p.ncl * kG;
    const int32_t* obs = p.obs + p.off[0];
    const int c = rank * C::Kh + ep.col;
    auto ok = [&](int64_t o0, int64_t T) { return fits(p, o0, T); };
    // the warp's slot: the step to compute (row, steps left below it), its symbol and the one
    // below, the exponents of the two steps below, the sequence's weight and 1 / c_{T-1}
    Slot s;
    int32_t row, left, sym, nsym, eb, neb;
    float wgt, cinv;
    bool fresh;
    auto begin = [&]() {
        next_seq(s, p.S, n, p.order, p.off, ok);
        fresh = true;
        if (s.seq < 0) return;
        left = (int32_t)s.T - 1;
        row = (int32_t)s.o0 + left;
        sym = obs[row];
        eb = left > 0 ? p.e[row - 1] : 0;
        nsym = left > 0 ? obs[row - 1] : 0;
        neb = left > 1 ? p.e[row - 2] : 0;
        wgt = p.w ? (float)p.w[s.seq] : 1.f;
        cinv = 1.f / p.clast[s.seq];
    };
    {
        s.k = -1;
        s.sl = cid + p.ncl * ep.g;
        row = left = sym = nsym = eb = neb = 0;
        wgt = cinv = 0.f;
        begin();
    }
    const int32_t steps = half[u];
    for (int32_t it = 0; it < steps; ++it) {
        const int b = (int)(it & 1);
        const bool on = s.seq >= 0, more = on && left > 0;
        Vec<C::EC> em, xr, o;
        if (on) {
            em.load(p.BT + (size_t)sym * KP + c);
            xr.load(p.X + (size_t)row * KP + c);
            // the rows of the coming steps on their way into L2
            if ((ep.lane & 7) == 0 && left >= 4)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(p.X + (size_t)(row - 4) * KP + c));
        }
        if (it > 0) {
            wt.local(&sm.out_full[u], (uint32_t)(it - 1) & 1u);
            o.load(&sm.out[u][ep.g & 3][ep.col]);
        }
        const float sc = pow2_scale(eb);
        Vec<C::EC> R, v;
#pragma unroll
        for (int h = 0; h < C::EC; ++h) {
            R.v[h] = fresh ? cinv : o.v[h];
            v.v[h] = more ? em.v[h] * R.v[h] * sc : 0.f;
        }
        ep.put(b, v, false, 0.f);
        if (on) {
            Vec<C::EC> g, q;
#pragma unroll
            for (int h = 0; h < C::EC; ++h) {
                g.v[h] = wgt * xr.v[h] * R.v[h];
                q.v[h] = wgt * v.v[h];
            }
            const size_t at = (size_t)row * KP + c;
            g.store(p.Gm + at);
            if (more) q.store(p.Q + at - KP);
            if (fresh) {
                Vec<C::EC> z;
#pragma unroll
                for (int h = 0; h < C::EC; ++h) z.v[h] = 0.f;
                z.store(p.Q + at);           // no transition leaves the last step
            }
            if (!more) {
                begin();
            } else {
                fresh = false;
                --row;
                --left;
                sym = nsym;
                eb = neb;
                nsym = left > 0 ? obs[row - 1] : 0;
                neb = left > 1 ? p.e[row - 2] : 0;
            }
        }
    }
    // the last steps' parts have landed before this CTA's shared memory goes
    if (C::NC == 2 && steps > 0) wt.cluster(&sm.x_peer[u][(steps - 1) & 1], step_phase(steps - 1));
}

// ORD: products in the order of the rows (forward, K other than 64, 128 and 256: the order of the
// checkpointed form there).
template <int KP, bool BWD, bool ORD>
__device__ __forceinline__ void rows_body(const RowsPrm& p, int rank, int cid, Smem<KP>& sm, Mid<KP>* mid,
                                          cg::cluster_group* cl) {
    if constexpr (ORD) mid->init();
    init_bars(sm, ORD ? Mid<KP>::W : kCon / 32);
    int32_t half[2];
    slot_totals(sm.tot, p.S, (int64_t)p.ncl * kG, cid, p.ncl, p.order, p.off,
                [&](int64_t o0, int64_t T) { return fits(p, o0, T); }, half);
    if constexpr (Cfg<KP>::NC == 2) cl->sync();  // the peer's barriers exist before any remote store
    Waits wt{p.status};
    if (threadIdx.x < kCon) {
        regs_contraction<KP>();
        if constexpr (ORD) {
            products_in_order<KP>(p.A, rank, sm, *mid, half, wt);
        } else {
            Contraction<KP> m;
            m.load(BWD ? p.At : p.A, rank);
            contraction_loop(m, sm, half, wt);
        }
    } else {
        regs_epilogue<KP>();
        if constexpr (BWD) bwd_epilogue<KP>(p, rank, cid, sm, half, wt);
        else fwd_epilogue<KP, ORD>(p, rank, cid, sm, half, wt);
    }
    if constexpr (Cfg<KP>::NC == 2) cl->sync();  // the peer no longer addresses this CTA's shared memory
}

template <int KP, bool BWD, bool ORD>
__global__ void __launch_bounds__(kT, Cfg<KP>::MINB) k_rows(RowsPrm p) {
    __shared__ __align__(16) Smem<KP> sm;
    if constexpr (ORD) {
        __shared__ __align__(16) Mid<KP> mid;
        rows_body<KP, BWD, ORD>(p, 0, (int)blockIdx.x, sm, &mid, nullptr);
    } else {
        rows_body<KP, BWD, ORD>(p, 0, (int)blockIdx.x, sm, nullptr, nullptr);
    }
}
template <bool BWD, bool ORD>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kT, 1) k_rows_pair(RowsPrm p) {
    __shared__ __align__(16) Smem<256> sm;
    cg::cluster_group cl = cg::this_cluster();
    if constexpr (ORD) {
        __shared__ __align__(16) Mid<256> mid;
        rows_body<256, BWD, ORD>(p, (int)cl.block_rank(), (int)(blockIdx.x >> 1), sm, &mid, &cl);
    } else {
        rows_body<256, BWD, ORD>(p, (int)cl.block_rank(), (int)(blockIdx.x >> 1), sm, nullptr, &cl);
    }
}

// Block q of kPiParts: pig[q][j] = sum of gamma_0(j) over its share of the sequences, in order.  The
// rows of a sequence that the call has no room for (reported, not computed) are cleared.
constexpr int kPiParts = 64;
__global__ void __launch_bounds__(256) k_rows_pi(RowsPrm p, int KP, float* __restrict__ pig) {
    const int j = threadIdx.x;
    const int64_t s0 = p.S * blockIdx.x / kPiParts, s1 = p.S * (blockIdx.x + 1) / kPiParts;
    const int64_t base = p.off[0];
    float sum = 0.f;
    for (int64_t s = s0; s < s1; ++s) {
        const int64_t o0 = p.off[s] - base, T = p.off[s + 1] - base - o0;
        if (T <= 0) continue;
        if (!fits(p, o0, T)) {
            const int64_t a = max(o0, (int64_t)0) * KP, z = min(o0 + T, p.rows) * KP;
            for (int64_t i = a + j; i < z; i += blockDim.x) {
                p.X[i] = 0.f;
                p.Q[i] = 0.f;
                p.Gm[i] = 0.f;
            }
        } else if (j < KP) {
            sum += p.Gm[o0 * KP + j];
        }
    }
    if (j < KP) pig[blockIdx.x * KP + j] = sum;
}

// Emission counts: block (split, window of symbols, 256 states) sums its rows' gammas by symbol in
// shared memory, thread j owning column j (no conflicts, in row order).  Bound by the latency of a row's
// read-add-write chain, so eight rows' gammas and symbols are loaded ahead and the grid holds as many
// CTAs as the tables of its window allow (64 KB at M = 64: three an SM).
constexpr int kCntSplit = 456, kWin = 64;
__global__ void __launch_bounds__(256) k_rows_counts(const float* __restrict__ Gm, const int32_t* __restrict__ obs,
                                                     const int64_t* __restrict__ off, int64_t S, int64_t room, int KP,
                                                     int M, int nsplit, float* __restrict__ cntp) {
    extern __shared__ float sc[];                 // [window][KP]
    const int64_t rows = min(off[S] - off[0], room);
    obs += off[0];
    const int sp = blockIdx.x % nsplit, m0 = blockIdx.x / nsplit * kWin, nm = min(kWin, M - m0);
    const int64_t r0 = rows * sp / nsplit, r1 = rows * (sp + 1) / nsplit;
    const int j = threadIdx.x;
    for (int k = 0; k < nm; ++k) sc[k * KP + j] = 0.f;
    constexpr int U = 8;
    int64_t r = r0;
    for (; r + U <= r1; r += U) {
        float g[U];
        int o[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            g[u] = __ldcs(Gm + (r + u) * KP + j);
            o[u] = obs[r + u] - m0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if ((unsigned)o[u] < (unsigned)nm) sc[o[u] * KP + j] += g[u];
    }
    for (; r < r1; ++r) {
        const int o = obs[r] - m0;
        if ((unsigned)o < (unsigned)nm) sc[o * KP + j] += Gm[r * KP + j];
    }
    float* dst = cntp + (int64_t)sp * KP * M;
    for (int k = 0; k < nm; ++k) dst[(int64_t)(m0 + k) * KP + j] = sc[k * KP + j];      // [M][KP]
}

// grad_log_A = A o sum U, grad_log_B = sum of the counts, grad_log_pi = sum of pig, each over its
// partials in order, without the padding.
__global__ void k_rows_finish(const float* __restrict__ A, const float* __restrict__ U, const float* __restrict__ cnt,
                              const float* __restrict__ pig, int K, int KP, int M, int nU, int nC,
                              float* __restrict__ gA, float* __restrict__ gB, float* __restrict__ gpi) {
    const int64_t nA = (int64_t)K * K, nB = (int64_t)K * M;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < nA + nB + K;
         idx += (int64_t)gridDim.x * blockDim.x) {
        // (the partials are many: summed in float64, so their number adds no rounding)
        double x = 0.0;
        if (idx < nA) {
            const int64_t q = idx / K * KP + idx % K;
#pragma unroll 8
            for (int s = 0; s < nU; ++s) x += (double)U[(int64_t)s * KP * KP + q];
            gA[idx] = A[q] * (float)x;
        } else if (idx < nA + nB) {
            const int64_t q = idx - nA, c = q % M * KP + q / M;          // counts are symbol-major
#pragma unroll 8
            for (int s = 0; s < nC; ++s) x += (double)cnt[(int64_t)s * KP * M + c];
            gB[q] = (float)x;
        } else if (gpi) {
            const int64_t q = idx - nA - nB;
            for (int s = 0; s < kPiParts; ++s) x += (double)pig[s * KP + q];
            gpi[q] = (float)x;
        }
    }
}

namespace {

int pad_states(int K) { return K <= 64 ? 64 : K <= 128 ? 128 : 256; }

// Rows of at most 32 GiB in all (an eighth of the device's memory): 10M steps at K = 256.
constexpr size_t kRowBytesMax = (size_t)32 << 30;

struct Layout {
    size_t A, At, BT, pi, X, Q, Gm, e, clast, U, cnt, pig, rows, order, total;
    int KP, nU, nC;
};

Layout layout(int K, int M, int64_t S, int64_t total_T) {
    Layout L;
    L.KP = pad_states(K);
    const size_t KP = (size_t)L.KP;
    size_t o = kStatusBytes;
    auto take = [&](size_t bytes) { size_t r = o; o = align_up(o + bytes, 256); return r; };
    L.A = take(KP * KP * 4);
    L.At = take(KP * KP * 4);
    L.BT = take((size_t)M * KP * 4);
    L.pi = take(KP * 4);
    L.X = take((size_t)total_T * KP * 4);
    L.Q = take((size_t)total_T * KP * 4);
    L.Gm = take((size_t)total_T * KP * 4);
    L.e = take((size_t)total_T * 4);
    L.clast = take((size_t)S * 4);
    L.nU = xi_parts(L.KP, total_T);
    L.nC = (int)std::max<int64_t>(1, std::min<int64_t>(kCntSplit, total_T / 64));
    L.U = take((size_t)L.nU * KP * KP * 4);
    L.cnt = take((size_t)L.nC * KP * M * 4);
    L.pig = take((size_t)kPiParts * KP * 4);
    L.rows = take(4);
    L.order = o;
    L.total = o + order_ws_bytes(S);
    return L;
}

using Kern = void (*)(RowsPrm);
Kern fwd_kernel(int K, int KP) {
    if (K == KP) return KP == 64 ? k_rows<64, false, false> : KP == 128 ? k_rows<128, false, false> : k_rows_pair<false, false>;
    return KP == 64 ? k_rows<64, false, true> : KP == 128 ? k_rows<128, false, true> : k_rows_pair<false, true>;
}
Kern bwd_kernel(int KP) { return KP == 64 ? k_rows<64, true, false> : KP == 128 ? k_rows<128, true, false> : k_rows_pair<true, false>; }

void fill(RowsPrm& p, const Layout& L, const RowsArgs& a) {
    char* ws = (char*)a.ws;
    p = RowsPrm{};
    p.S = a.S;
    p.rows = a.total_T;
    p.K = a.m->K;
    p.M = a.m->M;
    p.Cmax = a.Cmax;
    p.A = (float*)(ws + L.A);
    p.At = (float*)(ws + L.At);
    p.BT = (float*)(ws + L.BT);
    p.pi = (float*)(ws + L.pi);
    p.obs = a.obs;
    p.off = a.off;
    p.X = (float*)(ws + L.X);
    p.Q = (float*)(ws + L.Q);
    p.Gm = (float*)(ws + L.Gm);
    p.e = (int32_t*)(ws + L.e);
    p.clast = (float*)(ws + L.clast);
    p.status = a.status;
}

}  // namespace

// Whether the rows of these sizes are kept (else 0), and the workspace that takes.
size_t rows_ws_bytes(int K, int M, int64_t S, int64_t total_T) {
    if (K < 1 || K > 256 || M < 1 || M > 1024 || S < 1 || S > INT32_MAX || total_T < 1) return 0;
    const int64_t KP = pad_states(K);
    if ((uint64_t)total_T > kRowBytesMax / (12 * (uint64_t)KP)) return 0;
    return layout(K, M, S, total_T).total;
}

accel_status rows_forward(const RowsArgs& a, double* d_loglik, cudaStream_t st, int& nlaunch) {
    const int K = a.m->K, M = a.m->M;
    const Layout L = layout(K, M, a.S, a.total_T);
    char* ws = (char*)a.ws;
    RowsPrm p;
    fill(p, L, a);
    p.loglik = d_loglik;
    k_rows_prep<<<num_sms() * 2, 256, 0, st>>>(a.m->log_A, a.m->log_B, a.m->log_pi, K, L.KP, M, (float*)p.A,
                                               (float*)p.At, (float*)p.BT, (float*)p.pi, a.off, a.S,
                                               a.total_T, (int32_t*)(ws + L.rows));
    // the order by length (kept for the backward): the slots' loads balance, and the halves of a
    // cluster's slots finish together
    accel_status r = order_by_length(a.off, a.S, (int32_t*)(ws + L.order), ws + L.order + align_up((size_t)a.S * 4, 256), st);
    if (r != ACCEL_OK) return r;
    p.order = (int32_t*)(ws + L.order);
    const Kern kern = fwd_kernel(K, L.KP);
    p.ncl = clusters_for(kern, L.KP, a.S, sm_budget());
    kern<<<(unsigned)(p.ncl * (L.KP == 256 ? 2 : 1)), kT, 0, st>>>(p);
    nlaunch += 5;
    return ACCEL_OK;
}

accel_status rows_backward(const RowsArgs& a, const double* d_weights, float* gA, float* gB, float* gpi,
                           cudaStream_t st, int& nlaunch) {
    const int K = a.m->K, M = a.m->M;
    const Layout L = layout(K, M, a.S, a.total_T);
    char* ws = (char*)a.ws;
    RowsPrm p;
    fill(p, L, a);
    p.w = d_weights;
    p.order = (int32_t*)(ws + L.order);
    float* U = (float*)(ws + L.U);
    float* cnt = (float*)(ws + L.cnt);
    float* pig = (float*)(ws + L.pig);
    const Kern kern = bwd_kernel(L.KP);
    p.ncl = clusters_for(kern, L.KP, a.S, 0);
    kern<<<(unsigned)(p.ncl * (L.KP == 256 ? 2 : 1)), kT, 0, st>>>(p);
    k_rows_pi<<<kPiParts, 256, 0, st>>>(p, L.KP, pig);
    accel_status r = xi_rows(p.X, p.Q, (const int32_t*)(ws + L.rows), L.KP, L.nU, U, p.status, st);
    if (r != ACCEL_OK) return r;
    const size_t sm = (size_t)std::min(M, kWin) * L.KP * 4;
    ACCEL_CUDA_TRY(allow_smem((const void*)k_rows_counts, sm));
    k_rows_counts<<<(unsigned)(L.nC * ((M + kWin - 1) / kWin)), L.KP, sm, st>>>(p.Gm, p.obs, p.off, a.S, a.total_T, L.KP, M,
                                                                              L.nC, cnt);
    k_rows_finish<<<num_sms() * 4, 256, 0, st>>>(p.A, U, cnt, pig, K, L.KP, M, L.nU, L.nC, gA, gB, gpi);
    nlaunch += 5;
    return ACCEL_OK;
}

}  // namespace rows
}  // namespace hmm
}  // namespace accel
