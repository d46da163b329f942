// All-pairs histogram of angular separations (the two-point angular correlation shape the
// paper names as its tpacf workload, Table 1): a map over point pairs of a bin lookup,
// reduced into a histogram.  For unit vectors p_i, p_j the separation enters through the dot
// product d = (x_i x_j + y_i y_j) + z_i z_j, computed in FP32 with every product and sum
// rounded separately (no fused multiply-add), and the bin of d is the number of edges
// e_k >= d of a descending edge list (the cosines of increasing angles): bin 0 holds pairs
// closer than the first edge, bin n_edges those beyond the last one.
//
// Self mode (B is A) counts the unordered pairs i < j; cross mode all pairs (i in A, j in B).
//
// k_pairhist_rows: the bin by one table row.  The key of d - the octave, or half octave, of (1 - d)
// scaled and clamped - is monotone in d, so whether an edge e_k >= d is decided by the keys alone unless
// they are equal.  Where no two edges share a key, a pair takes one compare, with its row's edge; the row
// and the outcome are counted, and rows are mapped to bins only at the end.  The host looks for a scale
// with one edge an octave, then half octave: the cosines of log-spaced angles have one up to about 35
// bins over the 26 octaves that FP32 can tell apart.  Any other edge list takes k_pairhist_search,
// binary lifting over the edges.
//
// What bounds it: issue slots, 11 to 12 a pair and warp.  A row is 32 counters (one a lane number) and 32
// copies of the edge, so one address, put together by one byte permutation, serves both, without
// conflicts between lanes; a counter holds the two outcomes in 16 bits each (emptied before they can run
// over) and is shared by the block's warps by shared-memory reductions, which have no result to wait
// for.  A thread has four points of A in registers, so a point of B is read once for four pairs, and the
// arithmetic is packed over two points of B.  32,768 points, 20 bins: 254 us (2.1G pairs/ms); the search
// over the edges, with 10 shared-memory accesses a pair: 651 us.
#include "common.cuh"

#include <math.h>
#include <string.h>

#include <algorithm>

namespace accel {
namespace pairhist {

constexpr int kThreads = 256;
constexpr int kTile = 256;
constexpr int kMaxBins = 32;             // n_edges + 1 <= 32

struct HistPrm {
    const float *ax, *ay, *az;
    const float *bx, *by, *bz;
    int64_t NA, NB;
    int self;                          // 1: B is A, count i < j
    int nbins;                         // n_edges + 1
    float edges[kMaxBins];             // descending, padded with -inf
    unsigned long long* hist;          // [nbins]
    int64_t ti, tj, ntiles;            // tiles along A, along B, tiles in the launch
};

// Tile q of the launch -> (tile of A, tile of B).  Self mode enumerates the upper triangle
// (tb >= ta) row by row.
__device__ __forceinline__ void tile_of(const HistPrm& p, int64_t q, int64_t& ta, int64_t& tb) {
    if (!p.self) {
        ta = q / p.tj;
        tb = q - ta * p.tj;
        return;
    }
    // row ta holds ti - ta tiles; find ta with prefix(ta) <= q < prefix(ta + 1),
    // prefix(a) = a ti - a (a - 1) / 2
    int64_t lo = 0, hi = p.ti - 1;
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        const int64_t pre = mid * p.ti - mid * (mid - 1) / 2;
        if (pre <= q) lo = mid; else hi = mid - 1;
    }
    ta = lo;
    tb = ta + (q - (lo * p.ti - lo * (lo - 1) / 2));
}

// Tiles of 256 x 256 pairs: one CTA holds its 256 points of A in registers (one per thread) and streams
// the tile's points of B through shared memory (read as broadcasts).  The edges, padded to 32 with -inf,
// are 32 words (conflict-free); each thread counts into its own column of a shared [bin][thread] array;
// at the end a CTA sums its columns and adds them to the global int64 histogram.
__global__ void __launch_bounds__(kThreads) k_pairhist_search(HistPrm p) {
    __shared__ float sx[kTile], sy[kTile], sz[kTile];
    __shared__ float se[kMaxBins];
    __shared__ unsigned int cnt[kMaxBins][kThreads];
    const int tid = threadIdx.x;
    if (tid < kMaxBins) se[tid] = p.edges[tid];
    for (int b = 0; b < kMaxBins; ++b) cnt[b][tid] = 0u;
    for (int64_t q = blockIdx.x; q < p.ntiles; q += gridDim.x) {
        int64_t ta, tb;
        tile_of(p, q, ta, tb);
        const int64_t i = ta * kTile + tid;
        const bool has_i = i < p.NA;
        const float xi = has_i ? p.ax[i] : 0.f, yi = has_i ? p.ay[i] : 0.f, zi = has_i ? p.az[i] : 0.f;
        const int64_t j0 = tb * kTile;
        int64_t nj = p.NB - j0;
        if (nj > kTile) nj = kTile;
        __syncthreads();                  // the previous tile's points are no longer read
        if (tid < nj) {
            sx[tid] = p.bx[j0 + tid];
            sy[tid] = p.by[j0 + tid];
            sz[tid] = p.bz[j0 + tid];
        }
        __syncthreads();
        if (has_i) {
            // self mode, diagonal tile: only j > i
            const int jstart = (p.self && ta == tb) ? tid + 1 : 0;
            auto bin_of = [&](int jj) {
                const float d = __fadd_rn(__fadd_rn(__fmul_rn(xi, sx[jj]), __fmul_rn(yi, sy[jj])), __fmul_rn(zi, sz[jj]));
                int b = 0;
#pragma unroll
                for (int step = 16; step > 0; step >>= 1)
                    if (se[b + step - 1] >= d) b += step;
                return b;
            };
            int jj = jstart;
            // four independent lookups in flight, then their counts
            for (; jj + 4 <= (int)nj; jj += 4) {
                const int b0 = bin_of(jj), b1 = bin_of(jj + 1), b2 = bin_of(jj + 2), b3 = bin_of(jj + 3);
                cnt[b0][tid] += 1u;
                cnt[b1][tid] += 1u;
                cnt[b2][tid] += 1u;
                cnt[b3][tid] += 1u;
            }
            for (; jj < (int)nj; ++jj) cnt[bin_of(jj)][tid] += 1u;
        }
    }
    __syncthreads();
    // sum the columns: warp w sums bins w, w + 8, ... (d = -inf passes the padding, too)
    const int w = tid >> 5, lane = tid & 31;
    for (int b = w; b < kMaxBins; b += kThreads / 32) {
        unsigned long long s = 0;
        for (int t = lane; t < kThreads; t += 32) s += cnt[b][t];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
        if (lane == 0 && s) atomicAdd(&p.hist[b < p.nbins ? b : p.nbins - 1], s);
    }
}

// ---------------------------------------------------------------- by table row
constexpr int kRowThreads = 128;
constexpr int kPer = 4;                           // points of A per thread
constexpr int kTileA = kRowThreads * kPer;
constexpr int kMaxTileB = 256;

// key(d) = the top byte of w: w = u^2 + 2^-54 (N = 1) or u^4 + 2^-108 (N = 2), u = scale (1 - d) clamped to
// [0, 1]; one byte permutation makes a row's address of it.
template <int N> __host__ __device__ __forceinline__ float key_word(float u) {
    const float t = N == 1 ? u : u * u;
    return fmaf(t, t, N == 1 ? 5.5511151231257827e-17f : 3.0814879110195774e-33f);
}
template <int N> struct Keys {
    static constexpr int first = (127 - 54 * N) >> 1, rows = (127 >> 1) - first + 1;
};
constexpr int kMaxRows = Keys<2>::rows;

struct RowPrm {
    HistPrm h;                                    // (ti, tj in tiles of this kernel; edges unused)
    int tileB;
    float scale;                                  // of the key, in [1/4, 1/2)
    float one;                                    // 1: see the sums of the products
    float edge[kMaxRows];                         // the row's edge, -inf: none
    unsigned char bin[kMaxRows], has[kMaxRows];   // edges of smaller keys; whether the row has one
};

// Unit q -> (tile of A, tile of B); self mode: the tiles of B from the tile of A's first point on.
__device__ __forceinline__ void unit_of(const RowPrm& p, int64_t q, int64_t& ta, int64_t& tb) {
    if (!p.h.self) {
        ta = q / p.h.tj;
        tb = q - ta * p.h.tj;
        return;
    }
    const int64_t per = kTileA / p.tileB;         // prefix(a) = a tj - per a (a - 1) / 2
    int64_t lo = 0, hi = p.h.ti - 1;
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (mid * p.h.tj - per * (mid * (mid - 1) / 2) <= q) lo = mid; else hi = mid - 1;
    }
    ta = lo;
    tb = ta * per + (q - (lo * p.h.tj - per * (lo * (lo - 1) / 2)));
}

template <int N>
__global__ void __launch_bounds__(kRowThreads) k_pairhist_rows(RowPrm p) {
    constexpr int R = Keys<N>::rows;
    __shared__ __align__(256) unsigned int rows[R * 64];
    __shared__ __align__(16) float sb[3][kMaxTileB];
    __shared__ unsigned int s_bin[kMaxBins];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    for (int r = w; r < R; r += kRowThreads / 32) {
        rows[r * 64 + lane] = 0u;
        rows[r * 64 + 32 + lane] = __float_as_uint(p.edge[r]);
    }
    if (tid < kMaxBins) s_bin[tid] = 0u;
    // a lane's counter in row r: base + 256 (r + first)
    const char* base = reinterpret_cast<const char*>(rows) - Keys<N>::first * 256;
    const float scale = p.scale;
    // the bin of d, counted: the row's edge says which half of its counter
    auto count = [&](float d) {
        const float word = key_word<N>(__saturatef(fmaf(-scale, d, scale)));
        const uint32_t at = __byte_perm(__float_as_uint(word), (uint32_t)lane * 4u, 0x5534);   // [0, 0, key, 4 lane]
        const float e = *reinterpret_cast<const float*>(base + at + 128);
        atomicAdd(reinterpret_cast<unsigned int*>(const_cast<char*>(base + at)), e >= d ? 0x10000u : 1u);
    };
    // the counters into the bins, the bins into the histogram
    auto empty = [&]() {
        __syncthreads();
        for (int r = w; r < R; r += kRowThreads / 32) {
            const unsigned int c = rows[r * 64 + lane];
            rows[r * 64 + lane] = 0u;
            const unsigned int far = __reduce_add_sync(0xffffffffu, c & 0xffffu);
            const unsigned int near = __reduce_add_sync(0xffffffffu, c >> 16);
            if (lane == 0) {
                if (far) atomicAdd(&s_bin[p.bin[r]], far);
                if (near) atomicAdd(&s_bin[p.bin[r] + p.has[r]], near);
            }
        }
        __syncthreads();
        if (tid < p.h.nbins && s_bin[tid]) {
            atomicAdd(&p.h.hist[tid], (unsigned long long)s_bin[tid]);
            s_bin[tid] = 0u;
        }
    };
    // A packed product and sum become one FMA, even as explicitly rounded PTX instructions, and d would
    // be rounded differently; a sum as p * 1 + q, the 1 unknown to the compiler, stays as written.
    const float2 one = {p.one, p.one};
    const int per_unit = kTileA / 32 * p.tileB;   // pairs of a lane number in a tile
    int used = 0;                                 // ... since the counters were empty
    for (int64_t q = blockIdx.x; q < p.h.ntiles; q += gridDim.x) {
        if (used + per_unit > 0xffff) {
            empty();
            used = 0;
        }
        used += per_unit;
        int64_t ta, tb;
        unit_of(p, q, ta, tb);
        const int64_t i0 = ta * kTileA + tid, j0 = tb * p.tileB;
        float ax[kPer], ay[kPer], az[kPer];
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int64_t i = i0 + k * kRowThreads;
            const bool has = i < p.h.NA;
            ax[k] = has ? p.h.ax[i] : 0.f;
            ay[k] = has ? p.h.ay[i] : 0.f;
            az[k] = has ? p.h.az[i] : 0.f;
        }
        const int nj = p.h.NB - j0 < p.tileB ? (int)(p.h.NB - j0) : p.tileB;
        __syncthreads();                          // the last tile's points are no longer read
        for (int j = tid; j < nj; j += kRowThreads) {
            sb[0][j] = p.h.bx[j0 + j];
            sb[1][j] = p.h.by[j0 + j];
            sb[2][j] = p.h.bz[j0 + j];
        }
        __syncthreads();
        const bool whole = nj == p.tileB && (ta + 1) * kTileA <= p.h.NA && !(p.h.self && j0 < (ta + 1) * kTileA);
        if (whole) {
#pragma unroll 2
            for (int j = 0; j < nj; j += 4) {
                const float4 x = *reinterpret_cast<const float4*>(&sb[0][j]);
                const float4 y = *reinterpret_cast<const float4*>(&sb[1][j]);
                const float4 z = *reinterpret_cast<const float4*>(&sb[2][j]);
                const float2 bx[2] = {{x.x, x.y}, {x.z, x.w}}, by[2] = {{y.x, y.y}, {y.z, y.w}}, bz[2] = {{z.x, z.y}, {z.z, z.w}};
#pragma unroll
                for (int k = 0; k < kPer; ++k) {
                    const float2 kx = {ax[k], ax[k]}, ky = {ay[k], ay[k]}, kz = {az[k], az[k]};
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const float2 d = __ffma2_rn(__ffma2_rn(__fmul2_rn(kx, bx[e]), one, __fmul2_rn(ky, by[e])), one,
                                                    __fmul2_rn(kz, bz[e]));
                        count(d.x);
                        count(d.y);
                    }
                }
            }
        } else {
            for (int j = 0; j < nj; ++j) {
                const float x = sb[0][j], y = sb[1][j], z = sb[2][j];
#pragma unroll
                for (int k = 0; k < kPer; ++k) {
                    const int64_t i = i0 + k * kRowThreads;
                    if (i >= p.h.NA || (p.h.self && i >= j0 + j)) continue;
                    const float d = __fadd_rn(__fadd_rn(__fmul_rn(ax[k], x), __fmul_rn(ay[k], y)), __fmul_rn(az[k], z));
                    count(d);
                }
            }
        }
    }
    empty();
}

// The rows of an edge list; false: two edges share one, whichever of 16 scales the keys have.
template <int N>
bool make_rows(const float* edges, int n, RowPrm& p) {
    constexpr int R = Keys<N>::rows;
    for (int c = 0; c < 16; ++c) {
        p.scale = 0.25f * (float)(16 + c) / 16.f;
        for (int r = 0; r < R; ++r) {
            p.edge[r] = -INFINITY;
            p.has[r] = p.bin[r] = 0;
        }
        int k = 0;
        for (; k < n; ++k) {
            const float u = fmaf(-p.scale, edges[k], p.scale);
            const float word = key_word<N>(u > 0.f ? (u < 1.f ? u : 1.f) : 0.f);
            uint32_t bits;
            memcpy(&bits, &word, 4);
            const int r = (int)(bits >> 24) - Keys<N>::first;
            if (p.has[r]) break;
            p.has[r] = 1;
            p.edge[r] = edges[k];
        }
        if (k < n) continue;
        for (int r = 1; r < R; ++r) p.bin[r] = p.bin[r - 1] + p.has[r - 1];
        return true;
    }
    return false;
}

template <int N>
accel_status run_rows(RowPrm& p, cudaStream_t st) {
    auto kern = k_pairhist_rows<N>;
    int per = 0;
    ACCEL_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, kRowThreads, 0));
    const int64_t slots = (int64_t)std::max(per, 1) * num_sms();
    // the largest tiles of B that leave every block eight of them, or the smallest
    p.h.ti = (p.h.NA + kTileA - 1) / kTileA;
    for (p.tileB = kMaxTileB;; p.tileB /= 2) {
        p.h.tj = (p.h.NB + p.tileB - 1) / p.tileB;
        p.h.ntiles = p.h.self ? p.h.ti * p.h.tj - (kTileA / p.tileB) * (p.h.ti * (p.h.ti - 1) / 2) : p.h.ti * p.h.tj;
        if (p.tileB == 8 || p.h.ntiles >= 8 * slots) break;
    }
    kern<<<(unsigned)std::min(slots, p.h.ntiles), kRowThreads, 0, st>>>(p);
    return after_launch(st, "accel_pair_histogram", 1);
}

}  // namespace pairhist
}  // namespace accel

using namespace accel;
using namespace accel::pairhist;

extern "C" {

accel_status accel_pair_histogram(const float* d_ax, const float* d_ay, const float* d_az, int64_t NA,
                                  const float* d_bx, const float* d_by, const float* d_bz, int64_t NB,
                                  const float* h_edges, int32_t n_edges, int64_t* d_hist, void* stream) {
    ACCEL_REQUIRE(NA >= 0 && NB >= 0, ACCEL_ERR_INVALID_ARG, "accel_pair_histogram: negative size");
    ACCEL_REQUIRE(n_edges >= 1 && n_edges <= kMaxBins - 1, ACCEL_ERR_UNSUPPORTED,
                  "accel_pair_histogram: n_edges=%d outside [1, %d]", n_edges, kMaxBins - 1);
    ACCEL_REQUIRE(h_edges && d_hist, ACCEL_ERR_INVALID_ARG, "accel_pair_histogram: null pointer");
    // self mode: B is A (the same arrays and count)
    const bool self = d_bx == d_ax && d_by == d_ay && d_bz == d_az && NB == NA;
    ACCEL_REQUIRE(NA == 0 || (d_ax && d_ay && d_az), ACCEL_ERR_INVALID_ARG, "accel_pair_histogram: null point array");
    ACCEL_REQUIRE(NB == 0 || (d_bx && d_by && d_bz), ACCEL_ERR_INVALID_ARG, "accel_pair_histogram: null point array");
    HistPrm p{};
    for (int k = 0; k < n_edges; ++k) {
        ACCEL_REQUIRE(!isnan(h_edges[k]), ACCEL_ERR_INVALID_ARG, "accel_pair_histogram: edge %d is NaN", k);
        ACCEL_REQUIRE(k == 0 || h_edges[k] < h_edges[k - 1], ACCEL_ERR_SHAPE,
                      "accel_pair_histogram: edges must be strictly decreasing (edge %d)", k);
        p.edges[k] = h_edges[k];
    }
    for (int k = n_edges; k < kMaxBins; ++k) p.edges[k] = -INFINITY;
    p.nbins = n_edges + 1;
    p.self = self ? 1 : 0;
    p.ax = d_ax; p.ay = d_ay; p.az = d_az;
    p.NA = NA;
    p.bx = d_bx; p.by = d_by; p.bz = d_bz;
    p.NB = NB;
    p.hist = (unsigned long long*)d_hist;
    p.ti = (p.NA + kTile - 1) / kTile;
    p.tj = (p.NB + kTile - 1) / kTile;
    p.ntiles = self ? p.ti * (p.ti + 1) / 2 : p.ti * p.tj;
    cudaStream_t st = as_stream(stream);
    ACCEL_CUDA_TRY(cudaMemsetAsync(d_hist, 0, (size_t)p.nbins * sizeof(int64_t), st));
    if (p.ntiles == 0) return after_launch(st, "accel_pair_histogram", 0);
    RowPrm rp;
    rp.h = p;
    rp.one = 1.f;
    if (make_rows<1>(h_edges, n_edges, rp)) return run_rows<1>(rp, st);
    if (make_rows<2>(h_edges, n_edges, rp)) return run_rows<2>(rp, st);
    // a thread counts at most 256 pairs per tile in uint32: at most 2^24 tiles per CTA
    int64_t grid = 4LL * num_sms();
    const int64_t min_grid = (p.ntiles + (1LL << 24) - 1) >> 24;
    if (grid < min_grid) grid = min_grid;
    if (grid > p.ntiles) grid = p.ntiles;
    k_pairhist_search<<<(unsigned)grid, kThreads, 0, st>>>(p);
    return after_launch(st, "accel_pair_histogram", 1);
}

}  // extern "C"
