// Charge update q = S (G psi - b) (Eq. electrode-wise, Sec. II.B, in the library's sign of b),
// followed by the FP64 neutrality fix q <- q - u (e^T q), u = A^-1 e / (e^T A^-1 e), and the
// total charge e^T q.  In exact arithmetic S e = 0 already (Eq. S); the fix removes the
// rounding left by a single-precision S.
#include <cooperative_groups.h>

#include "common.cuh"

namespace cpm {

namespace cg = cooperative_groups;

// S is symmetric, so q_i = sum_j S_ji b_j: one thread per output i reads column i of S (row
// j = column j, coalesced across the block), the b_j are broadcast from shared memory, and the
// rows j are split over blocks (partial sums reduced in FP64 in a fixed order).
//
// Single precision: the sum is centred per output, sum_j S_ij (b_j - b_i), which equals S b
// because the rows of S sum to zero (Eq. S); without the projection (symm = 0, S = A^-1) the
// reduction adds b_i sum_j S_ij back, from the FP64 row sums of the stored single-precision S.  S rounded to FP32 then only perturbs the
// products where b_j differs from b_i, i.e. mostly far sites where S_ij is small; b enters as
// an FP32 hi + lo pair so the differences are formed to about 2^-24 of themselves, and each
// thread's partial sum is Kahan-compensated.
constexpr int GT_COLS = 128;   // outputs (threads) per block
constexpr int GT_JT = 64;      // rows of S staged per iteration
constexpr int GT_MR = 8;       // replicas per block

template <typename TS> struct LaneSum;
template <> struct LaneSum<float> {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x) {
        float y = x - c;
        float t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

// bhl[t] = (hi, lo) with hi = float(b[t]) and lo = float(b[t] - hi)
__global__ void k_split_b(const double* __restrict__ b, int64_t cnt, float2* __restrict__ bhl) {
    grid_go();
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= cnt) return;
    double v = b[t];
    float hi = (float)v;
    bhl[t] = make_float2(hi, (float)(v - (double)hi));
}

// FP64: part[split][r][i] = sum over this split's rows j of S_ji b_j for MR replicas, two columns per thread
// (16-byte loads, n even) or one, sixteen rows of S in flight.  Compiled for the replica count: tested per
// element instead, one replica of 4,320 sites took 299 us where S streams from HBM in 22 and the FP64 pipe
// needs 31.
constexpr int G6_T = 128, G6_U = 16;
template <int MR, int NC>
__global__ void __launch_bounds__(G6_T) k_gemv64(const double* __restrict__ S, const double* __restrict__ bv, int64_t n,
                                                 int m, int64_t jchunk, double* __restrict__ part) {
    grid_wait();
    __shared__ double bs[GT_JT][MR];
    const int64_t i0 = ((int64_t)blockIdx.x * G6_T + threadIdx.x) * NC;
    const int split = blockIdx.y, r0 = blockIdx.z * MR;
    const int64_t jb = (int64_t)split * jchunk, je = min(n, jb + jchunk);
    const bool live = i0 < n;
    double acc[MR][NC];
#pragma unroll
    for (int t = 0; t < MR; ++t)
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[t][c] = 0.0;
    auto row = [&](int64_t j, double* v) {
        // volatile: all rows of the unrolled group are requested before the first is used
        if (NC == 2)
            asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[NC - 1]) : "l"(S + j * n + i0));
        else
            asm volatile("ld.global.nc.f64 %0, [%1];" : "=d"(v[0]) : "l"(S + j * n + i0));
    };
    for (int64_t j0 = jb; j0 < je; j0 += GT_JT) {
        const int jn = (int)min((int64_t)GT_JT, je - j0);
        __syncthreads();
        for (int e = threadIdx.x; e < MR * GT_JT; e += G6_T) {
            const int t = e / GT_JT, jj = e % GT_JT;
            bs[jj][t] = (r0 + t < m && jj < jn) ? bv[(int64_t)(r0 + t) * n + j0 + jj] : 0.0;
        }
        __syncthreads();
        if (!live) continue;
        int jj = 0;
        for (; jj + G6_U <= jn; jj += G6_U) {
            double v[G6_U][NC];
#pragma unroll
            for (int u = 0; u < G6_U; ++u) row(j0 + jj + u, v[u]);
#pragma unroll
            for (int u = 0; u < G6_U; ++u)
#pragma unroll
                for (int t = 0; t < MR; ++t)
#pragma unroll
                    for (int c = 0; c < NC; ++c) acc[t][c] = fma(v[u][c], bs[jj + u][t], acc[t][c]);
        }
        for (; jj < jn; ++jj) {
            double v[NC];
            row(j0 + jj, v);
#pragma unroll
            for (int t = 0; t < MR; ++t)
#pragma unroll
                for (int c = 0; c < NC; ++c) acc[t][c] = fma(v[c], bs[jj][t], acc[t][c]);
        }
    }
    if (!live) return;
#pragma unroll
    for (int t = 0; t < MR; ++t)
        if (r0 + t < m)
#pragma unroll
            for (int c = 0; c < NC; ++c) part[((int64_t)split * m + r0 + t) * n + i0 + c] = acc[t][c];
}

// Single precision: the hi/lo pairs of b are staged jj-major in shared memory so
// one 16-byte load serves two replicas, and eight loads of S are in flight before use.  Each tile
// of GT_JT terms is summed plainly in FP32 as S_ij (hi_j - hi_i) + S_ij lo_j (the hi difference
// is exact; centring the tiny lo part would change nothing), and the tile sums are added with
// compensation.
__global__ void __launch_bounds__(GT_COLS) k_gemv32(const float* __restrict__ S, const float2* __restrict__ bv,
                                                   int64_t n, int m, int64_t jchunk, double* __restrict__ part) {
    grid_wait();
    __shared__ __align__(16) float2 bs[GT_JT][GT_MR];
    const int64_t i = (int64_t)blockIdx.x * GT_COLS + threadIdx.x;
    const int split = blockIdx.y;
    const int r0 = blockIdx.z * GT_MR;
    const int mm = min(GT_MR, m - r0);
    const int64_t jb = (int64_t)split * jchunk, je = min(n, jb + jchunk);
    float2 bi[GT_MR];
    LaneSum<float> acc[GT_MR];
#pragma unroll
    for (int t = 0; t < GT_MR; ++t) bi[t] = (t < mm && i < n) ? bv[(int64_t)(r0 + t) * n + i] : make_float2(0.f, 0.f);
    for (int64_t j0 = jb; j0 < je; j0 += GT_JT) {
        for (int e = threadIdx.x; e < GT_MR * GT_JT; e += GT_COLS) {
            const int t = e / GT_JT, jj = e % GT_JT;
            const int64_t j = j0 + jj;
            bs[jj][t] = (t < mm && j < je) ? bv[(int64_t)(r0 + t) * n + j] : make_float2(0.f, 0.f);
        }
        __syncthreads();
        const int jn = (int)min((int64_t)GT_JT, je - j0);
        if (i < n) {
            float tile[GT_MR];
#pragma unroll
            for (int t = 0; t < GT_MR; ++t) tile[t] = 0.f;
            int jj = 0;
            for (; jj + 8 <= jn; jj += 8) {
                float sv[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) sv[u] = S[(j0 + jj + u) * n + i];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const float4* row = reinterpret_cast<const float4*>(bs[jj + u]);
#pragma unroll
                    for (int tp = 0; tp < GT_MR / 2; ++tp) {
                        const float4 v = row[tp];
                        tile[2 * tp] = fmaf(sv[u], v.x - bi[2 * tp].x, tile[2 * tp]);
                        tile[2 * tp] = fmaf(sv[u], v.y, tile[2 * tp]);
                        tile[2 * tp + 1] = fmaf(sv[u], v.z - bi[2 * tp + 1].x, tile[2 * tp + 1]);
                        tile[2 * tp + 1] = fmaf(sv[u], v.w, tile[2 * tp + 1]);
                    }
                }
            }
            for (; jj < jn; ++jj) {
                const float sv = S[(j0 + jj) * n + i];
#pragma unroll
                for (int t = 0; t < GT_MR; ++t) {
                    tile[t] = fmaf(sv, bs[jj][t].x - bi[t].x, tile[t]);
                    tile[t] = fmaf(sv, bs[jj][t].y, tile[t]);
                }
            }
#pragma unroll
            for (int t = 0; t < GT_MR; ++t) acc[t].add(tile[t]);
        }
        __syncthreads();
    }
    if (i < n) {
#pragma unroll
        for (int t = 0; t < GT_MR; ++t)
            if (t < mm) part[((int64_t)split * m + r0 + t) * n + i] = acc[t].value();
    }
}

// k_gemv32 with two output columns per thread (8-byte loads of S, n even) and sixteen rows of S
// in flight, so that enough bytes are outstanding to stream S at HBM speed.
constexpr int G2_T = 256;
__global__ void __launch_bounds__(G2_T, 2) k_gemv32x2(const float* __restrict__ S, const float2* __restrict__ bv,
                                                      int64_t n, int m, int64_t jchunk, double* __restrict__ part) {
    grid_wait();
    __shared__ __align__(16) float2 bs[GT_JT][GT_MR];
    const int64_t i0 = ((int64_t)blockIdx.x * G2_T + threadIdx.x) * 2;
    const int split = blockIdx.y;
    const int r0 = blockIdx.z * GT_MR;
    const int mm = min(GT_MR, m - r0);
    const int64_t jb = (int64_t)split * jchunk, je = min(n, jb + jchunk);
    const bool live = i0 < n;
    float bh[2][GT_MR];
    LaneSum<float> acc[2][GT_MR];
#pragma unroll
    for (int t = 0; t < GT_MR; ++t) {
        bh[0][t] = (t < mm && live) ? bv[(int64_t)(r0 + t) * n + i0].x : 0.f;
        bh[1][t] = (t < mm && live) ? bv[(int64_t)(r0 + t) * n + i0 + 1].x : 0.f;
    }
    for (int64_t j0 = jb; j0 < je; j0 += GT_JT) {
        for (int e = threadIdx.x; e < GT_MR * GT_JT; e += G2_T) {
            const int t = e / GT_JT, jj = e % GT_JT;
            const int64_t j = j0 + jj;
            bs[jj][t] = (t < mm && j < je) ? bv[(int64_t)(r0 + t) * n + j] : make_float2(0.f, 0.f);
        }
        __syncthreads();
        const int jn = (int)min((int64_t)GT_JT, je - j0);
        if (live) {
            float tile[2][GT_MR];
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int t = 0; t < GT_MR; ++t) tile[c][t] = 0.f;
            int jj = 0;
            for (; jj + 16 <= jn; jj += 16) {
                float2 sv[16];
#pragma unroll
                for (int u = 0; u < 16; ++u) sv[u] = *reinterpret_cast<const float2*>(S + (j0 + jj + u) * n + i0);
#pragma unroll
                for (int u = 0; u < 16; ++u) {
                    const float4* row = reinterpret_cast<const float4*>(bs[jj + u]);
#pragma unroll
                    for (int tp = 0; tp < GT_MR / 2; ++tp) {
                        const float4 v = row[tp];   // (hi, lo) of replicas 2 tp and 2 tp + 1
                        tile[0][2 * tp] = fmaf(sv[u].x, v.x - bh[0][2 * tp], tile[0][2 * tp]);
                        tile[0][2 * tp] = fmaf(sv[u].x, v.y, tile[0][2 * tp]);
                        tile[1][2 * tp] = fmaf(sv[u].y, v.x - bh[1][2 * tp], tile[1][2 * tp]);
                        tile[1][2 * tp] = fmaf(sv[u].y, v.y, tile[1][2 * tp]);
                        tile[0][2 * tp + 1] = fmaf(sv[u].x, v.z - bh[0][2 * tp + 1], tile[0][2 * tp + 1]);
                        tile[0][2 * tp + 1] = fmaf(sv[u].x, v.w, tile[0][2 * tp + 1]);
                        tile[1][2 * tp + 1] = fmaf(sv[u].y, v.z - bh[1][2 * tp + 1], tile[1][2 * tp + 1]);
                        tile[1][2 * tp + 1] = fmaf(sv[u].y, v.w, tile[1][2 * tp + 1]);
                    }
                }
            }
            for (; jj < jn; ++jj) {
                const float2 sv = *reinterpret_cast<const float2*>(S + (j0 + jj) * n + i0);
#pragma unroll
                for (int t = 0; t < GT_MR; ++t) {
                    tile[0][t] = fmaf(sv.x, bs[jj][t].x - bh[0][t], tile[0][t]);
                    tile[0][t] = fmaf(sv.x, bs[jj][t].y, tile[0][t]);
                    tile[1][t] = fmaf(sv.y, bs[jj][t].x - bh[1][t], tile[1][t]);
                    tile[1][t] = fmaf(sv.y, bs[jj][t].y, tile[1][t]);
                }
            }
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int t = 0; t < GT_MR; ++t) acc[c][t].add(tile[c][t]);
        }
        __syncthreads();
    }
    if (live) {
#pragma unroll
        for (int t = 0; t < GT_MR; ++t)
            if (t < mm) {
                part[((int64_t)split * m + r0 + t) * n + i0] = acc[0][t].value();
                part[((int64_t)split * m + r0 + t) * n + i0 + 1] = acc[1][t].value();
            }
    }
}

template <typename P> struct PartSum;
template <> struct PartSum<double> { using type = PartSumD; };
template <> struct PartSum<float2> { using type = PartSumF2; };
template <> struct PartSum<float> { using type = PartSumF; };   // partials of the tensor-core product

// q = SG psi - sum of the split partials (tensor-core product: - SZ gmean, the share of the group means taken out
// of its operand), then the neutrality fix of Sec. II.B: q <- q - u (e^T q) with symm, and qtot[r] = e^T q of the
// result (plain FP64 sums in a fixed order: the rounding, about n eps max|q|, is far below the 1e-12 e the total
// is held to).
//
// Grid (cluster of up to sixteen blocks, m): one cluster per replica, one thread per site (slices beyond 640 sites take
// several passes), the block sums exchanged through distributed shared memory, so that every thread still holds
// its q when e^T q is known.  With a replica's last block (a ticket) doing the fix, that block read the whole q
// back.  Whole steps, before and now: 4,320 sites x 8 replicas 158.3 and 155.4 us, the product alone x 64 80.0 and
// 74.5, 512 sites x 4 54.0 and 51.2, 256 small replicas 184 and 178.  Bounded by the latency of the loads and of
// two cluster barriers, and FP64 at sixteen clocks a warp and SM: one warp adds a block's values (the product x 64
// 67.9 with a tree per warp, 65.5 without).  48 registers let two blocks of 640 threads share an SM (with 64, one: the
// product took 89 us).
constexpr int NB_CLUSTER = 16;  // blocks per replica, at most; more than eight where the replicas are few
constexpr int NB_T = 640;      // threads per block, at most
constexpr int NB_LEAST = 64;    // sites per block that a cluster of several blocks has at least
template <typename P>
__global__ void __launch_bounds__(NB_T, 2) k_gemv_reduce(const P* __restrict__ part, int splits,
                                                      const double* __restrict__ SG, int ng,
                                                      const double* __restrict__ psi, int64_t n, int m,
                                                      double* __restrict__ q, const double* __restrict__ u, int symm,
                                                      double* __restrict__ qtot, const double* __restrict__ b,
                                                      const double* __restrict__ srow, const double* __restrict__ SZ,
                                                      const double* __restrict__ gmean, int ngrp) {
    cluster_arrive();   // matched in front of the first store to another block, which must have started by then
    grid_wait();
    __shared__ double sh[NB_T];
    __shared__ double csum[2][NB_CLUSTER];   // block sums of the cluster before and after the fix
    const cg::cluster_group cluster = cg::this_cluster();
    const int r = blockIdx.y, cl = gridDim.x, rank = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t slice = (n + cl - 1) / cl, lo = rank * slice, hi = min(n, lo + slice);
    double* qr = q + (int64_t)r * n;
    auto exchange = [&](double a, int which) {   // fixed order: lanes over the block's values, a warp tree, blocks in order
        sh[threadIdx.x] = a;
        __syncthreads();
        if (warp == 0) {   // one warp: an FP64 instruction occupies the SM for sixteen clocks whatever its lanes do
            double t = sh[lane];
            for (int k = lane + 32; k < (int)blockDim.x; k += 32) t += sh[k];
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane < cl) *cluster.map_shared_rank(&csum[which][rank], lane) = t;
        }
        cluster.sync();
        double t = csum[which][0];
        for (int k = 1; k < cl; ++k) t += csum[which][k];
        return t;
    };
    double q0 = 0.0, u0 = 0.0, a = 0.0;   // this thread's first site
    if (symm && lo + threadIdx.x < hi) u0 = u[lo + threadIdx.x];
    for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
        typename PartSum<P>::type v;
        const P* pi = part + (int64_t)r * n + i;
        const int64_t stride = (int64_t)m * n;
        constexpr int LD = sizeof(P) == 4 ? 16 : 8;   // loads in flight, added in split order
        for (int sp = 0; sp < splits; sp += LD) {
            P x[LD];
#pragma unroll
            for (int k = 0; k < LD; ++k) x[k] = sp + k < splits ? pi[(int64_t)(sp + k) * stride] : P{};
#pragma unroll
            for (int k = 0; k < LD; ++k)
                if (sp + k < splits) v.add(x[k]);
        }
        double vs = v.value();
        if constexpr (std::is_same<P, float>::value)
            if (!isfinite(vs)) vs = sum_fp64(pi, stride, splits);
        double sv = 0.0;
        for (int g = 0; g < ng; ++g) sv += SG[i * ng + g] * psi[(int64_t)r * ng + g];
        for (int g = 0; g < ngrp; ++g) sv -= SZ[i * ngrp + g] * gmean[(int64_t)r * ngrp + g];
        // the centred products give sum_j S_ij (b_j - b_i): add b_i sum_j S_ij back where rows do not sum to zero
        const double qi = sv - (srow ? vs + b[(int64_t)r * n + i] * srow[i] : vs);
        if (i == lo + threadIdx.x) q0 = qi;
        else qr[i] = qi;                        // read back by this thread alone
        a += qi;
    }
    cluster_wait();
    const double s = exchange(a, 0);
    a = 0.0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
        const bool first = i == lo + threadIdx.x;
        double v = first ? q0 : qr[i];
        if (symm) v -= (first ? u0 : u[i]) * s;
        qr[i] = v;
        a += v;
    }
    if (!qtot) return;   // uniform
    const double tot = exchange(a, 1);
    if (rank == 0 && threadIdx.x == 0) qtot[r] = tot;
}

// out[r][i] = sum of the split partials, one output per thread over the whole GPU
template <typename P>
__global__ void __launch_bounds__(256) k_sum_splits(const P* __restrict__ part, int splits, int64_t cnt,
                                                    double* __restrict__ out) {
    grid_wait();
    grid_go();
    const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (t >= cnt) return;
    typename PartSum<P>::type v;
    for (int sp = 0; sp < splits; sp += 16) {   // sixteen loads in flight, added in split order
        P x[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) x[k] = sp + k < splits ? part[(int64_t)(sp + k) * cnt + t] : P{};
#pragma unroll
        for (int k = 0; k < 16; ++k)
            if (sp + k < splits) v.add(x[k]);
    }
    out[t] = v.value();
}

// Blocks per replica.  Sixteen up to four replicas (one replica of 4,320 sites: 20.9 us an update against 22.8 with
// eight); beyond, eight while the replicas' blocks are one wave of two per SM, and fewer after that: with eight for
// every batch, 256 replicas of 4,320 sites took 566 us an update, with one block each 507; of 1,031 sites 113 and 101;
// 64 of 4,320 on the tensor cores 66 and 56 with four.
// wide: the device places clusters of sixteen
static int reduce_cluster(int64_t n, int m, bool wide) {
    int cl = m <= 4 && wide ? NB_CLUSTER : 8;
    while (cl > 1 && (m > 4 && (int64_t)m * cl > 2 * 152)) cl /= 2;
    while (cl > 1 && n < (int64_t)cl * (cl > 8 ? 2 * NB_LEAST : NB_LEAST)) cl /= 2;
    return cl;
}
// A replica of more sites than sixteen blocks have threads, its partials in many splits, and fewer blocks of eight
// than SMs: most of the GPU would wait while a few SMs read the partials, so k_sum_splits adds them beforehand.  16,384
// sites, 86 splits: one replica 193 -> 181 us an update, five 248 -> 234, eight 261 -> 247, sixteen 463 -> 456, but 32
// replicas 839 -> 857; 8,192 sites x 8 86 -> 89; 16,384 sites x 8 in the tensor-core product's few splits 280 -> 290.
static bool reduce_sums_first(int64_t n, int m, int64_t splits) {
    return n > (int64_t)NB_CLUSTER * NB_T && splits >= 32 && 8 * m <= 152;
}

template <typename P>
static cpm_status launch_reduce(cpm_ctx* c, const void* part, int splits, int m, const double* psi, double* q, double* qtot,
                                const double* b, const double* srow, const double* SZ, const double* gmean, int ngrp) {
    // clusters beyond eight blocks are not portable: asked once per context whether the largest blocks can be placed
    signed char& wide = c->wide_reduce[std::is_same<P, double>::value ? 0 : std::is_same<P, float2>::value ? 1 : 2];
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = NB_CLUSTER;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    if (m <= 4 && wide < 0) {
        int fit = 0;
        cfg.gridDim = dim3(NB_CLUSTER);
        cfg.blockDim = dim3(NB_T);
        cfg.numAttrs = 1;
        wide = cudaFuncSetAttribute(k_gemv_reduce<P>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
               cudaOccupancyMaxActiveClusters(&fit, k_gemv_reduce<P>, &cfg) == cudaSuccess && fit > 0;
        cudaGetLastError();   // a refusal is an answer
    }
    const int cl = reduce_cluster(c->n, m, wide > 0);
    const int64_t slice = (c->n + cl - 1) / cl;
    cfg.gridDim = dim3((unsigned)cl, (unsigned)m);
    cfg.blockDim = dim3((unsigned)std::min<int64_t>(NB_T, (slice + 31) / 32 * 32));
    cfg.stream = c->stream;
    at[0].val.clusterDim.x = (unsigned)cl;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // as launch_after()
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
    CPM_CUDA(c, cudaLaunchKernelEx(&cfg, k_gemv_reduce<P>, (const P*)part, splits, (const double*)upd_sg(c), (int)upd_ng(c), psi,
                                   c->n, m, q, (const double*)c->u, (int)c->p.symm, qtot, b, srow, SZ, gmean, ngrp));
    return CPM_OK;
}

// the streamed products: with the splits added first where that is faster (the sums are the same)
template <typename P>
static cpm_status reduce_streamed(cpm_ctx* c, const void* part, double* sums, int splits, int m, const double* psi, double* q,
                                  double* qtot, const double* b, const double* srow) {
    if (!reduce_sums_first(c->n, m, splits)) return launch_reduce<P>(c, part, splits, m, psi, q, qtot, b, srow, nullptr, nullptr, 0);
    const int64_t cnt = (int64_t)m * c->n;
    CPM_CUDA(c, launch_after(k_sum_splits<P>, dim3((unsigned)((cnt + 255) / 256)), dim3(256), 0, c->stream, (const P*)part,
                             splits, cnt, sums));
    c->launches += 1;
    return launch_reduce<double>(c, sums, 1, m, psi, q, qtot, b, srow, nullptr, nullptr, 0);
}

// split count and row chunk of the centred product; grows the scratch when needed
static bool gemv_pairs(const cpm_ctx* c) { return c->p.s_prec == CPM_PREC_FP32 && c->n % 2 == 0; }
static bool gemv_fp64(const cpm_ctx* c) { return c->p.s_prec == CPM_PREC_FP64; }
static int gemv64_mr(int m) { return m >= 5 ? 8 : m >= 3 ? 4 : m; }
static int64_t gemv_colblocks(const cpm_ctx* c) {
    if (gemv_fp64(c)) return c->n % 2 == 0 ? (c->n + 2 * G6_T - 1) / (2 * G6_T) : (c->n + G6_T - 1) / G6_T;
    return gemv_pairs(c) ? (c->n + 2 * G2_T - 1) / (2 * G2_T) : (c->n + GT_COLS - 1) / GT_COLS;
}

// FP64: rows per split in steps of the rows in flight.  The FP64 pipe is what bounds the product, so the time is the rows
// that the busiest SM takes: blocks per SM times rows per block while all blocks fit at once (four per SM), their mean
// and half a block beyond; one to three blocks of four warps keep the pipe less than busy (the factors are fitted to
// 25 split counts at each of 42 sizes).  About one wave of blocks whatever their remainder, the rule before: 2,050 sites
// x 8 87.5 us an update, 77.5 now, x 64 621 and 509; 8,192 x 16 2,124 and 1,781, x 64 8,286 and 6,950; 16,384 x 1 567
// and 493.  The fewest splits within 1 % (their partial sums are memory).
static void gemv64_plan(int64_t n, int64_t blocks, int lean, int64_t* splits, int64_t* jchunk) {
    const double busy[5] = {0.0, 0.5, 0.9, 0.95, 1.0};
    const int64_t most = std::min<int64_t>(lean > 1 ? 1 : 64 >> (2 * lean), (n + G6_U - 1) / G6_U);
    double cost[65], best = 1e300;
    for (int64_t s = 1; s <= most; ++s) {
        const int64_t j = ((n + s - 1) / s + G6_U - 1) / G6_U * G6_U, nb = blocks * ((n + j - 1) / j), k = (nb + 151) / 152;
        cost[s] = (k <= 4 ? (double)k / busy[k] : (double)nb / 152 + 0.5) * (double)j;
        best = std::min(best, cost[s]);
    }
    int64_t s = 1;
    while (cost[s] > 1.01 * best) ++s;
    *jchunk = ((n + s - 1) / s + G6_U - 1) / G6_U * G6_U;
    *splits = (n + *jchunk - 1) / *jchunk;
}

static cpm_status reserve_update_lean(cpm_ctx* c, int m, int64_t* splits_out, int64_t* jchunk_out) {
    const int64_t n = c->n;
    const int64_t colblocks = gemv_colblocks(c);
    const int mr = gemv_fp64(c) ? gemv64_mr(m) : GT_MR;
    const int rchunks = (m + mr - 1) / mr;
    const int64_t want = gemv_pairs(c) ? 2 * 152 : 4 * 152;   // resident blocks: about one wave
    int64_t splits = (want + colblocks * rchunks - 1) / (colblocks * rchunks);   // rows per split in whole tiles
    splits = std::max<int64_t>(1, std::min<int64_t>(splits, (n + GT_JT - 1) / GT_JT));
    int64_t jchunk = (((n + splits - 1) / splits + GT_JT - 1) / GT_JT) * GT_JT;
    splits = (n + jchunk - 1) / jchunk;
    if (gemv_fp64(c)) gemv64_plan(n, colblocks * rchunks, c->lean, &splits, &jchunk);
    if (gemv_tma_supported(c)) {
        int64_t cb;
        gemv_tma_plan(n, m, &cb, &splits, &jchunk);
    }
    // the partials, then the two-float split of b, whose place the sums of the splits take after the product
    const size_t need = ((sizeof(double) * splits * m * n + 255) & ~(size_t)255) + sizeof(float2) * m * n;
    if (c->ubuf_bytes < need) {
        dev_free(c, c->ubuf);
        c->ubuf = nullptr;
        c->ubuf_bytes = 0;
        c->graph_valid = false;
        CPM_TRY(dev_alloc(c, &c->ubuf, need));
        c->ubuf_bytes = need;
    }
    *splits_out = splits;
    *jchunk_out = jchunk;
    return CPM_OK;
}

static cpm_status reserve_update_plan(cpm_ctx* c, int m, int64_t* splits, int64_t* jchunk) {
    return reserve_within_budget(c, [&] { return reserve_update_lean(c, m, splits, jchunk); });
}

cpm_status reserve_update(cpm_ctx* c, int m) {
    if (c->p.s_prec == CPM_PREC_BF16X3) return tc_reserve(c, m);
    int64_t s, j;
    return reserve_update_plan(c, m, &s, &j);
}

float2* update_bhl(cpm_ctx* c, int m) {
    if (c->p.s_prec != CPM_PREC_FP32) return nullptr;
    int64_t splits = 0, jchunk = 0;
    if (reserve_update_plan(c, m, &splits, &jchunk) != CPM_OK) return nullptr;
    return (float2*)((char*)c->ubuf + ((sizeof(double) * splits * m * c->n + 255) & ~(size_t)255));
}

cpm_status update(cpm_ctx* c, int m, const double* psi, const double* b, double* q, double* qtot, bool bhl_ready) {
    const int64_t n = c->n;
    cudaStream_t st = c->stream;
    if (c->p.s_prec == CPM_PREC_BF16X3) {
        const float* part = nullptr;
        const double* gmean = nullptr;
        int splits = 0;
        prof_begin(c, CPM_K_GEMV);
        CPM_TRY(tc_product(c, m, b, &part, &splits, &gmean));
        prof_end(c, CPM_K_GEMV);
        prof_begin(c, CPM_K_NEUTRAL);
        CPM_TRY(launch_reduce<float>(c, part, splits, m, psi, q, qtot, b, nullptr, c->SZ, gmean, c->tc_ngrp));
        prof_end(c, CPM_K_NEUTRAL);
        CPM_LAUNCH(c, "k_gemv_reduce");
        c->launches += 1;
        return CPM_OK;
    }
    const bool f32 = c->p.s_prec == CPM_PREC_FP32;
    int64_t splits = 0, jchunk = 0;
    CPM_TRY(reserve_update_plan(c, m, &splits, &jchunk));
    const int64_t colblocks = gemv_colblocks(c);
    const int rchunks = (m + GT_MR - 1) / GT_MR;
    double* part = (double*)c->ubuf;
    float2* bhl = (float2*)((char*)c->ubuf + ((sizeof(double) * splits * m * n + 255) & ~(size_t)255));
    bhl_ready = bhl_ready && f32;
    c->launches += (f32 && !bhl_ready) ? 3 : 2;
    // profiled stages: the split of b with the combination of b, the S stream alone, the reduction
    // of the split partial sums with the neutrality fix
    dim3 grid((unsigned)colblocks, (unsigned)splits, (unsigned)rchunks);
    if (f32) {
        if (!bhl_ready) {
            prof_begin(c, CPM_K_COMBINE);
            k_split_b<<<(unsigned)((m * n + 255) / 256), 256, 0, st>>>(b, (int64_t)m * n, bhl);
            prof_end(c, CPM_K_COMBINE);
        }
        prof_begin(c, CPM_K_GEMV);
        if (gemv_tma_supported(c)) CPM_TRY(gemv_tma(c, m, bhl, (float2*)part, splits, jchunk));
        else if (gemv_pairs(c)) CPM_CUDA(c, launch_after(k_gemv32x2, dim3(grid), dim3(G2_T), 0, st, c->S32, bhl, n, m, jchunk, part));
        else CPM_CUDA(c, launch_after(k_gemv32, dim3(grid), dim3(GT_COLS), 0, st, c->S32, bhl, n, m, jchunk, part));
    } else {
        prof_begin(c, CPM_K_GEMV);
        const int mr = gemv64_mr(m);
        dim3 g6((unsigned)colblocks, (unsigned)splits, (unsigned)((m + mr - 1) / mr));
        if (n % 2 == 0) {
            if (mr == 1) CPM_CUDA(c, launch_after(k_gemv64<1, 2>, dim3(g6), dim3(G6_T), 0, st, c->S, b, n, m, jchunk, part));
            else if (mr == 2) CPM_CUDA(c, launch_after(k_gemv64<2, 2>, dim3(g6), dim3(G6_T), 0, st, c->S, b, n, m, jchunk, part));
            else if (mr == 4) CPM_CUDA(c, launch_after(k_gemv64<4, 2>, dim3(g6), dim3(G6_T), 0, st, c->S, b, n, m, jchunk, part));
            else CPM_CUDA(c, launch_after(k_gemv64<8, 2>, dim3(g6), dim3(G6_T), 0, st, c->S, b, n, m, jchunk, part));
        } else {
            if (mr == 1) CPM_CUDA(c, launch_after(k_gemv64<1, 1>, dim3(g6), dim3(G6_T), 0, st, c->S, b, n, m, jchunk, part));
            else if (mr == 2) CPM_CUDA(c, launch_after(k_gemv64<2, 1>, dim3(g6), dim3(G6_T), 0, st, c->S, b, n, m, jchunk, part));
            else if (mr == 4) CPM_CUDA(c, launch_after(k_gemv64<4, 1>, dim3(g6), dim3(G6_T), 0, st, c->S, b, n, m, jchunk, part));
            else CPM_CUDA(c, launch_after(k_gemv64<8, 1>, dim3(g6), dim3(G6_T), 0, st, c->S, b, n, m, jchunk, part));
        }
    }
    prof_end(c, CPM_K_GEMV);
    prof_begin(c, CPM_K_NEUTRAL);
    const double* srow = (f32 && !c->p.symm) ? c->dvec : nullptr;
    if (f32 && gemv_tma_supported(c))
        CPM_TRY(reduce_streamed<float2>(c, part, (double*)bhl, (int)splits, m, psi, q, qtot, b, srow));
    else
        CPM_TRY(reduce_streamed<double>(c, part, (double*)bhl, (int)splits, m, psi, q, qtot, b, srow));
    prof_end(c, CPM_K_NEUTRAL);
    CPM_LAUNCH(c, "k_gemv");
    return CPM_OK;
}

}  // namespace cpm
