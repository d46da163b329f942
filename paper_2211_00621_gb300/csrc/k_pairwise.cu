// All-pairs map-of-reduce (K10): for every body i a reduce over all bodies j
// (Appendix A: a map whose function is a reduce; the paper's tpacf / mri-q workloads,
// Table 1, have this shape).  Softened gravity, G = 1, FP32:
//     a_i = sum_j m_j (p_j - p_i) / (|p_j - p_i|^2 + eps^2)^(3/2)
//
// FP32-pipe bound (12 FP32 operations + 1 MUFU rsqrt per interaction), no tensor cores.
// The FP32 work is issued as packed pairs (add/mul/fma .f32x2, one instruction for two
// lanes' worth of operations): with scalar FFMAs the FP32 pipe alone needs one issue slot per
// cycle, so every shared-memory load, MUFU and loop instruction came out of its time; with
// pairs the pipe keeps its rate at half the issue slots.  A pair is two j bodies against one
// i body, so the i coordinates are duplicated into both halves once, and the j bodies are
// staged in shared memory as a structure of arrays, read four at a time as float4 warp
// broadcasts.  The reciprocal square root is the MUFU approximation with denormal inputs
// flushed: r >= eps^2, and the host accepts only eps whose eps^2 is a normal float, so no
// input of it is denormal and the flush never applies.
//
// Decomposition: a CTA owns 64 bodies (lane l holds bodies l and l + 32) and its four warps
// take the four quarters of every j tile.  A cluster of P CTAs (P in {1, 2, 4, 8}) shares one
// group of 64 bodies and splits the j range P ways; the P partial sums are added through
// distributed shared memory, so nothing leaves the cluster before the final sums.  The host
// picks P so that the grid holds about six waves of resident CTAs (eight per SM at <= 64
// registers) -- finer work units, so that every SM stays full to the end instead of running
// a partial last wave.
// Each body's sums are kept per parity of j (the two halves of a pair) and added in a fixed
// order: the halves, the four quarters, then the P cluster ranks -- results are
// deterministic for a given N and P.
#include "common.cuh"

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cooperative_groups.h>

namespace cg = cooperative_groups;

namespace accel {
namespace pair {

constexpr int kThreads = 128;
constexpr int kBodies = 64;   // bodies per CTA (per cluster)
constexpr int kSplit = 4;     // j quarters per tile, one per warp
constexpr int kTile = 512;    // j bodies per shared-memory tile
constexpr int kMaxCluster = 8;

__device__ __forceinline__ float rsqrt_ftz(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// One pair of interactions: the j pair (xj, yj, zj, mj) against body i, whose negated
// coordinates are duplicated in (nx, ny, nz).  The arithmetic of each half is that of the
// scalar form: d = p_j - p_i, r = dx^2 + (dy^2 + (dz^2 + eps^2)), s = m r^(-1/2)^3,
// a += s d.
__device__ __forceinline__ void interact2(float2 xj, float2 yj, float2 zj, float2 mj, float2 nx, float2 ny,
                                          float2 nz, float2 e2, float2& ax, float2& ay, float2& az) {
    const float2 dx = __fadd2_rn(xj, nx), dy = __fadd2_rn(yj, ny), dz = __fadd2_rn(zj, nz);
    float2 r = __ffma2_rn(dz, dz, e2);
    r = __ffma2_rn(dy, dy, r);
    r = __ffma2_rn(dx, dx, r);
    const float2 inv = make_float2(rsqrt_ftz(r.x), rsqrt_ftz(r.y));
    const float2 s = __fmul2_rn(__fmul2_rn(__fmul2_rn(mj, inv), inv), inv);
    ax = __ffma2_rn(s, dx, ax);
    ay = __ffma2_rn(s, dy, ay);
    az = __ffma2_rn(s, dz, az);
}

// Launched in clusters of P CTAs along x: cluster c owns bodies [64 c, 64 c + 64), its rank r
// the j range [r per, min(n, (r + 1) per)).
__global__ void __launch_bounds__(kThreads, 8)
k_gravity(const float* __restrict__ X, const float* __restrict__ Y, const float* __restrict__ Z,
          const float* __restrict__ Mass, int64_t n, int64_t per, float eps2, float* __restrict__ AX,
          float* __restrict__ AY, float* __restrict__ AZ) {
    __shared__ __align__(16) float s_x[kTile];
    __shared__ __align__(16) float s_y[kTile];
    __shared__ __align__(16) float s_z[kTile];
    __shared__ __align__(16) float s_m[kTile];
    __shared__ float3 s_part[kSplit][kBodies];
    __shared__ float3 s_sum[kBodies];
    cg::cluster_group cluster = cg::this_cluster();
    const int P = (int)cluster.num_blocks();
    const int rank = (int)cluster.block_rank();
    const int t = threadIdx.x;
    const int w = t >> 5;
    const int l = t & 31;
    const int64_t ib = (int64_t)(blockIdx.x / P) * kBodies;
    const int64_t jbeg = rank * per;
    const int64_t jend = jbeg + per < n ? jbeg + per : n;
    const int64_t i0 = ib + l, i1 = ib + l + 32;
    float x0 = 0, y0 = 0, z0 = 0, x1 = 0, y1 = 0, z1 = 0;
    if (i0 < n) { x0 = X[i0]; y0 = Y[i0]; z0 = Z[i0]; }
    if (i1 < n) { x1 = X[i1]; y1 = Y[i1]; z1 = Z[i1]; }
    const float2 nx0 = make_float2(-x0, -x0), ny0 = make_float2(-y0, -y0), nz0 = make_float2(-z0, -z0);
    const float2 nx1 = make_float2(-x1, -x1), ny1 = make_float2(-y1, -y1), nz1 = make_float2(-z1, -z1);
    const float2 e2 = make_float2(eps2, eps2);
    float2 ax0 = make_float2(0.f, 0.f), ay0 = ax0, az0 = ax0, ax1 = ax0, ay1 = ax0, az1 = ax0;

    for (int64_t jb = jbeg; jb < jend; jb += kTile) {
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kTile / kThreads; ++k) {
            // padding bodies (past the range) sit at the origin with zero mass
            const int s = t + k * kThreads;
            const int64_t j = jb + s;
            const bool in = j < jend;
            s_x[s] = in ? X[j] : 0.f;
            s_y[s] = in ? Y[j] : 0.f;
            s_z[s] = in ? Z[j] : 0.f;
            s_m[s] = in ? Mass[j] : 0.f;
        }
        __syncthreads();
        const int q0 = w * (kTile / kSplit);
        const float4* px = reinterpret_cast<const float4*>(s_x + q0);
        const float4* py = reinterpret_cast<const float4*>(s_y + q0);
        const float4* pz = reinterpret_cast<const float4*>(s_z + q0);
        const float4* pm = reinterpret_cast<const float4*>(s_m + q0);
#pragma unroll 2
        for (int g = 0; g < kTile / kSplit / 4; ++g) {
            const float4 bx = px[g], by = py[g], bz = pz[g], bm = pm[g];
            const float2 xa = make_float2(bx.x, bx.y), ya = make_float2(by.x, by.y);
            const float2 za = make_float2(bz.x, bz.y), ma = make_float2(bm.x, bm.y);
            const float2 xb = make_float2(bx.z, bx.w), yb = make_float2(by.z, by.w);
            const float2 zb = make_float2(bz.z, bz.w), mb = make_float2(bm.z, bm.w);
            interact2(xa, ya, za, ma, nx0, ny0, nz0, e2, ax0, ay0, az0);
            interact2(xa, ya, za, ma, nx1, ny1, nz1, e2, ax1, ay1, az1);
            interact2(xb, yb, zb, mb, nx0, ny0, nz0, e2, ax0, ay0, az0);
            interact2(xb, yb, zb, mb, nx1, ny1, nz1, e2, ax1, ay1, az1);
        }
    }
    // this CTA's sums: the two halves of each pair, then the four quarters in order
    s_part[w][l] = make_float3(ax0.x + ax0.y, ay0.x + ay0.y, az0.x + az0.y);
    s_part[w][l + 32] = make_float3(ax1.x + ax1.y, ay1.x + ay1.y, az1.x + az1.y);
    __syncthreads();
    if (t < kBodies) {
        float3 a = s_part[0][t];
#pragma unroll
        for (int r = 1; r < kSplit; ++r) {
            const float3 b = s_part[r][t];
            a.x += b.x; a.y += b.y; a.z += b.z;
        }
        s_sum[t] = a;
    }
    // the cluster's ranks in order; rank r finishes bodies [r 64/P, (r + 1) 64/P)
    cluster.sync();
    const int nb = kBodies / P;
    if (t < nb) {
        const int b = rank * nb + t;
        float3 a = cluster.map_shared_rank(s_sum, 0)[b];
        for (int r = 1; r < P; ++r) {
            const float3 c = cluster.map_shared_rank(s_sum, r)[b];
            a.x += c.x; a.y += c.y; a.z += c.z;
        }
        const int64_t i = ib + b;
        if (i < n) { AX[i] = a.x; AY[i] = a.y; AZ[i] = a.z; }
    }
    cluster.sync();   // no CTA leaves while a peer still reads its sums
}

// Cluster size for n bodies: double P while the grid holds under six waves of resident CTAs
// and every rank keeps at least two j tiles (the best measured P at N = 16,384, 65,536 and
// 262,144 bodies: 8, 8 and 2).
int choose_cluster(int64_t n) {
    static int slots = -1;
    if (slots < 0) {
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gravity, kThreads, 0) != cudaSuccess) {
            cudaGetLastError();
            per_sm = 1;
        }
        slots = (per_sm > 0 ? per_sm : 1) * num_sms();
    }
    const int64_t groups = (n + kBodies - 1) / kBodies;
    int P = 1;
    while (P < kMaxCluster && groups * P < 6 * (int64_t)slots && n >= (int64_t)2 * P * 2 * kTile) P *= 2;
    return P;
}

accel_status launch_gravity(const float* d_x, const float* d_y, const float* d_z, const float* d_m, int64_t n,
                            float eps, float* d_ax, float* d_ay, float* d_az, int P, cudaStream_t st) {
    const int64_t groups = (n + kBodies - 1) / kBodies;
    const int64_t per = (n + P - 1) / P;
    cudaLaunchConfig_t lc = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)P;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    lc.gridDim = dim3((unsigned)(groups * P), 1, 1);
    lc.blockDim = dim3(kThreads, 1, 1);
    lc.dynamicSmemBytes = 0;
    lc.stream = st;
    lc.attrs = attr;
    lc.numAttrs = 1;
    ACCEL_CUDA_TRY(cudaLaunchKernelEx(&lc, k_gravity, d_x, d_y, d_z, d_m, n, per, eps * eps, d_ax, d_ay, d_az));
    return after_launch(st, "pairwise_mapreduce", 1);
}

// ---------------------------------------------------------------- each pair of bodies once
// With room for partial sums, d, r and r^(-3/2) of a pair serve both of its bodies: 16 FP32 operations
// and one rsqrt for two interactions, instead of 24 and two.  A unit is 1,024 bodies I (a CTA of 8 warps
// of 128, four bodies a lane) against 512 bodies J, J not before I; the units within I itself (J < I + 1,024)
// take both directions one by one and give sums to I only.
//  * A warp goes through the 64-body groups of J in turn, warp w starting at group w, with a barrier
//    between turns, so that a group's sums have one writer at a time and a fixed order.
//  * In a group, a lane holds the sums of two bodies of J (a packed pair), which move on by one lane after
//    each of 32 steps; the bodies' coordinates are read from shared memory at the moving index.
//  * Sums over I go to partial[unit], those over J to partial[I block]; k_pairs_sum adds a body's
//    partial sums in a fixed order: results are deterministic for a given n.
// What bounds it: the FP32 pipe (packed: 128 cycles for 4 x 2 pairs a lane, beside about 90 issue slots).
// Against k_gravity, which evaluates both directions: n = 24,576 253 -> 193 us, 65,536 1,660 -> 1,162,
// 131,072 6,598 -> 4,466; the error against 64 bits is about half as large (more, shorter sums).  From
// kPairsMin on, where the units (594) give every SM two rounds of two CTAs; at 16,384 there is less than
// one.  Up to kPairsMax: the partial sums grow as n^2 (385 MB there).
constexpr int kPT = 256;
constexpr int kPI = 1024, kPJ = 512;
constexpr int64_t kPairsMin = 24576, kPairsMax = 131072;
// The inverse cube of a distance is formed once for both bodies where it stays a normal float, for
// (softened) distances up to 2^42: all that bodies within 2^40 of the origin can have.  Past that it is denormal
// (and 0 from 1e15 on) however large the masses are, so a unit with such bodies is left to k_pairs_far, which
// multiplies each mass on its own: one operation more (all units so: 1,245 us at 65,536).  In one kernel
// the two loops take 1,204 us and more; so, 1,162 (1,155 with no far form at all).
constexpr float kPNear = 1099511627776.f;

struct PairsPrm {
    const float *X, *Y, *Z, *M;
    int64_t n;
    int ni, nj;              // blocks of I, of J
    float eps2;
    float *pi, *pj;          // [3][units][kPI], [3][ni][nj kPJ]
    int32_t* far;            // [units]
    float *AX, *AY, *AZ;
};

// Units of the I blocks before i: sum of nj - 2 i'.
__host__ __device__ __forceinline__ int units_before(int i, int nj) { return i * nj - i * (i - 1); }

// FAR: a unit that the other form has marked.
template <bool FAR>
__device__ __forceinline__ void pairs_unit(const PairsPrm& p, int u) {
    __shared__ __align__(16) float4 s_xy[kPJ / 2], s_zm[kPJ / 2];   // pairs: (x, x', y, y'), (z, z', m, m')
    __shared__ float2 s_a[3][kPJ / 2];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int units = units_before(p.ni, p.nj);
    int lo = 0, hi = p.ni - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (units_before(mid, p.nj) <= u) lo = mid; else hi = mid - 1;
    }
    const int I = lo, J = 2 * I + u - units_before(I, p.nj);
    const bool both = J >= 2 * (I + 1);
    {
        // bodies past the end sit at the origin with zero mass
        const int64_t j = (int64_t)J * kPJ + 2 * t;
        const bool in0 = j < p.n, in1 = j + 1 < p.n;
        s_xy[t] = make_float4(in0 ? p.X[j] : 0.f, in1 ? p.X[j + 1] : 0.f, in0 ? p.Y[j] : 0.f, in1 ? p.Y[j + 1] : 0.f);
        s_zm[t] = make_float4(in0 ? p.Z[j] : 0.f, in1 ? p.Z[j + 1] : 0.f, in0 ? p.M[j] : 0.f, in1 ? p.M[j + 1] : 0.f);
#pragma unroll
        for (int c = 0; c < 3; ++c) s_a[c][t] = make_float2(0.f, 0.f);
    }
    auto is_far = [](float x, float y, float z) { return !(fabsf(x) <= kPNear && fabsf(y) <= kPNear && fabsf(z) <= kPNear); };
    bool far = p.eps2 > kPNear * kPNear || is_far(s_xy[t].x, s_xy[t].z, s_zm[t].x) || is_far(s_xy[t].y, s_xy[t].w, s_zm[t].y);
    float2 nx[4], ny[4], nz[4], nm[4], ax[4], ay[4], az[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int64_t i = (int64_t)I * kPI + w * 128 + k * 32 + lane;
        const bool in = i < p.n;
        const float x = in ? -p.X[i] : 0.f, y = in ? -p.Y[i] : 0.f, z = in ? -p.Z[i] : 0.f, m = in ? -p.M[i] : 0.f;
        far = far || is_far(x, y, z);
        nx[k] = make_float2(x, x);
        ny[k] = make_float2(y, y);
        nz[k] = make_float2(z, z);
        nm[k] = make_float2(m, m);
        ax[k] = ay[k] = az[k] = make_float2(0.f, 0.f);
    }
    const float2 e2 = make_float2(p.eps2, p.eps2);
    if constexpr (FAR) {
        __syncthreads();
    } else {
        far = __syncthreads_or(far) != 0;
        if (t == 0) p.far[u] = far;
        if (far) return;
    }
    for (int turn = 0; turn < 8; ++turn) {
        const int g = ((turn + w) & 7) * 32;      // the group's first pair
        if (both) {
            float2 bx = make_float2(0.f, 0.f), by = bx, bz = bx;
#pragma unroll 2
            for (int step = 0; step < 32; ++step) {
                const int q = g + ((lane + step) & 31);
                const float4 xy = s_xy[q], zm = s_zm[q];
                const float2 xj = make_float2(xy.x, xy.y), yj = make_float2(xy.z, xy.w), zj = make_float2(zm.x, zm.y),
                             mj = make_float2(zm.z, zm.w);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float2 dx = __fadd2_rn(xj, nx[k]), dy = __fadd2_rn(yj, ny[k]), dz = __fadd2_rn(zj, nz[k]);
                    float2 r = __ffma2_rn(dz, dz, e2);
                    r = __ffma2_rn(dy, dy, r);
                    r = __ffma2_rn(dx, dx, r);
                    const float2 inv = make_float2(rsqrt_ftz(r.x), rsqrt_ftz(r.y));
                    float2 si, sj;
                    if constexpr (FAR) {
                        const float2 inv2 = __fmul2_rn(inv, inv);
                        si = __fmul2_rn(__fmul2_rn(mj, inv), inv2);
                        sj = __fmul2_rn(__fmul2_rn(nm[k], inv), inv2);
                    } else {
                        const float2 c3 = __fmul2_rn(__fmul2_rn(inv, inv), inv);
                        si = __fmul2_rn(c3, mj);
                        sj = __fmul2_rn(c3, nm[k]);
                    }
                    ax[k] = __ffma2_rn(si, dx, ax[k]);
                    ay[k] = __ffma2_rn(si, dy, ay[k]);
                    az[k] = __ffma2_rn(si, dz, az[k]);
                    bx = __ffma2_rn(sj, dx, bx);
                    by = __ffma2_rn(sj, dy, by);
                    bz = __ffma2_rn(sj, dz, bz);
                }
                // the sums move on with their bodies
                const int from = (lane + 1) & 31;
                bx = make_float2(__shfl_sync(0xffffffffu, bx.x, from), __shfl_sync(0xffffffffu, bx.y, from));
                by = make_float2(__shfl_sync(0xffffffffu, by.x, from), __shfl_sync(0xffffffffu, by.y, from));
                bz = make_float2(__shfl_sync(0xffffffffu, bz.x, from), __shfl_sync(0xffffffffu, bz.y, from));
            }
            const float2 sx = s_a[0][g + lane], sy = s_a[1][g + lane], sz = s_a[2][g + lane];
            s_a[0][g + lane] = make_float2(sx.x + bx.x, sx.y + bx.y);
            s_a[1][g + lane] = make_float2(sy.x + by.x, sy.y + by.y);
            s_a[2][g + lane] = make_float2(sz.x + bz.x, sz.y + bz.y);
        } else {
#pragma unroll 2
            for (int step = 0; step < 32; ++step) {
                const float4 xy = s_xy[g + step], zm = s_zm[g + step];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    interact2(make_float2(xy.x, xy.y), make_float2(xy.z, xy.w), make_float2(zm.x, zm.y),
                              make_float2(zm.z, zm.w), nx[k], ny[k], nz[k], e2, ax[k], ay[k], az[k]);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float* at = p.pi + (int64_t)u * kPI + w * 128 + k * 32 + lane;
        const int64_t plane = (int64_t)units * kPI;
        at[0] = ax[k].x + ax[k].y;
        at[plane] = ay[k].x + ay[k].y;
        at[2 * plane] = az[k].x + az[k].y;
    }
    if (both) {
        const int64_t row = (int64_t)p.nj * kPJ, plane = p.ni * row;
        float* at = p.pj + I * row + (int64_t)J * kPJ + 2 * t;
#pragma unroll
        for (int c = 0; c < 3; ++c) *reinterpret_cast<float2*>(at + c * plane) = s_a[c][t];
    }
}

__global__ void __launch_bounds__(kPT, 2) k_pairs(PairsPrm p) { pairs_unit<false>(p, blockIdx.x); }

// The marked units, on CTAs that are resident at once: there are none but in units far from 1.
__global__ void __launch_bounds__(kPT, 2) k_pairs_far(PairsPrm p) {
    const int units = units_before(p.ni, p.nj);
    for (int base = blockIdx.x; base < units; base += gridDim.x * kPT) {
        const int64_t mine = base + (int64_t)threadIdx.x * gridDim.x;
        if (!__syncthreads_or(mine < units && p.far[mine])) continue;
        for (int k = 0; k < kPT; ++k) {
            const int64_t u = base + (int64_t)k * gridDim.x;
            if (u < units && p.far[u]) pairs_unit<true>(p, (int)u);
        }
    }
}

// A body's sums: over the units of its I block, then over the I blocks before it.
__global__ void __launch_bounds__(256) k_pairs_sum(PairsPrm p) {
    const int64_t b = blockIdx.x * (int64_t)256 + threadIdx.x;
    if (b >= p.n) return;
    const int I = (int)(b / kPI), u0 = units_before(I, p.nj), nu = p.nj - 2 * I;
    const int64_t pl_i = (int64_t)units_before(p.ni, p.nj) * kPI, row = (int64_t)p.nj * kPJ, pl_j = p.ni * row;
    float* const out[3] = {p.AX, p.AY, p.AZ};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float* fi = p.pi + c * pl_i + (int64_t)u0 * kPI + b % kPI;
        const float* fj = p.pj + c * pl_j + b;
        float a[8] = {};                      // (eight sums, added in pairs: fewer roundings)
        auto add = [&](const float* f, int n, int64_t stride) {
            int q = 0;
            for (; q + 8 <= n; q += 8)
#pragma unroll
                for (int k = 0; k < 8; ++k) a[k] += f[(q + k) * stride];
            for (; q < n; ++q) a[0] += f[q * stride];
        };
        add(fi, nu, kPI);
        add(fj, I, row);
        out[c][b] = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
    }
}

size_t pairs_ws(int64_t n) {
    if (n < kPairsMin || n > kPairsMax) return 0;
    const int64_t ni = (n + kPI - 1) / kPI, nj = (n + kPJ - 1) / kPJ;
    const int64_t units = units_before((int)ni, (int)nj);
    return (size_t)(3 * (units * kPI + ni * nj * kPJ) + units) * sizeof(float);
}

accel_status launch_pairs(const float* d_x, const float* d_y, const float* d_z, const float* d_m, int64_t n, float eps,
                          float* d_ax, float* d_ay, float* d_az, void* ws, cudaStream_t st) {
    PairsPrm p{d_x, d_y, d_z, d_m, n, (int)((n + kPI - 1) / kPI), (int)((n + kPJ - 1) / kPJ), eps * eps,
               nullptr, nullptr, nullptr, d_ax, d_ay, d_az};
    const int units = units_before(p.ni, p.nj);
    p.pi = (float*)ws;
    p.pj = p.pi + 3 * (int64_t)units * kPI;
    p.far = (int32_t*)(p.pj + 3 * (int64_t)p.ni * p.nj * kPJ);
    k_pairs<<<units, kPT, 0, st>>>(p);
    k_pairs_far<<<std::min(units, 2 * num_sms()), kPT, 0, st>>>(p);
    k_pairs_sum<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(p);
    return after_launch(st, "pairwise_mapreduce", 3);
}

}  // namespace pair
}  // namespace accel

using namespace accel;

extern "C" {

size_t pairwise_mapreduce_workspace_size(int32_t op, int64_t n) {
    return op == ACCEL_PAIR_GRAVITY_SOFTENED ? pair::pairs_ws(n) : 0;
}

accel_status pairwise_mapreduce(int32_t op, const float* d_x, const float* d_y, const float* d_z, const float* d_m,
                                int64_t n, float eps, float* d_ax, float* d_ay, float* d_az, void* stream) {
    return pairwise_mapreduce_ws(op, d_x, d_y, d_z, d_m, n, eps, d_ax, d_ay, d_az, nullptr, 0, stream);
}

accel_status pairwise_mapreduce_ws(int32_t op, const float* d_x, const float* d_y, const float* d_z, const float* d_m,
                                   int64_t n, float eps, float* d_ax, float* d_ay, float* d_az, void* d_ws,
                                   size_t ws_bytes, void* stream) {
    ACCEL_REQUIRE(op == ACCEL_PAIR_GRAVITY_SOFTENED, ACCEL_ERR_INVALID_ARG, "pairwise_mapreduce: bad op %d", op);
    ACCEL_REQUIRE(n >= 0, ACCEL_ERR_INVALID_ARG, "pairwise_mapreduce: n < 0");
    // the j = i term (and a padding body's) is 0 * r^(-3/2) with r >= eps^2: it stays 0 only
    // while eps^-3 is finite in FP32, with a margin for the rounding of r and the rsqrt
    ACCEL_REQUIRE(eps > 0.f && std::isfinite(eps) && 1.0 / ((double)eps * eps * eps) <= FLT_MAX / 4.0,
                  ACCEL_ERR_INVALID_ARG, "pairwise_mapreduce: eps must be positive and finite with eps^-3 < FLT_MAX/4 (eps = %g)",
                  (double)eps);
    if (n == 0) return ok();
    ACCEL_REQUIRE(d_x && d_y && d_z && d_m && d_ax && d_ay && d_az, ACCEL_ERR_INVALID_ARG, "pairwise_mapreduce: null pointer");
    ACCEL_REQUIRE((n + pair::kBodies - 1) / pair::kBodies * pair::kMaxCluster <= (int64_t)INT32_MAX,
                  ACCEL_ERR_UNSUPPORTED, "pairwise_mapreduce: n too large");
    ACCEL_REQUIRE(((uintptr_t)d_ws % 16) == 0, ACCEL_ERR_INVALID_ARG, "pairwise_mapreduce: d_ws must be 16-byte aligned");
    const size_t need = pair::pairs_ws(n);
    if (d_ws && need > 0 && ws_bytes >= need)
        return pair::launch_pairs(d_x, d_y, d_z, d_m, n, eps, d_ax, d_ay, d_az, d_ws, as_stream(stream));
    return pair::launch_gravity(d_x, d_y, d_z, d_m, n, eps, d_ax, d_ay, d_az, pair::choose_cluster(n),
                                as_stream(stream));
}

}  // extern "C"
