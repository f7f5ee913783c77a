// Dense FP64 linear algebra of the one-time setup: Cholesky factorisation A = L L^T,
// the inverse A^-1 = L^-T L^-1, and the charge-neutral capacitance matrix of
// Eq. (S), Sec. II.A:  S = A^-1 - d d^T / (e^T d),  d = A^-1 e.
// Also the electrode response SG = S G (Sec. II.B) and the neutraliser u = d / (e^T d).
#include "common.cuh"

namespace cpm {

// ----------------------------------------------------------------------------- DGEMM
// C = alpha op(A) op(B) + beta C, row-major, BM x BN tiles, 256 threads (BM / 16 x BN / 16 each).
// lower: skip tiles strictly above the diagonal of C.  tri & 1: op(A)[i][k] = 0 for k < i;
// tri & 2: op(B)[k][j] = 0 for k < j (triangular operands; the K loop starts past the zeros).
// status: when non-null and nonzero the kernel returns without touching C.
//
// The FP64 pipe retires two multiply-adds per clock and SM, so even a 2 x 2 block of accumulators per
// thread is not load-bound once the next K step is fetched while the current one is multiplied; what
// matters is that every SM has a tile: 64 x 64 x 64 takes 68 us on one.  64 x 64 tiles are taken from DG_MANY of
// them on (four per SM), 32 x 32 below.
constexpr int DG_LARGE = 64, DG_SMALL = 32, DG_BK = 16, DG_T = 256, DG_MANY = 4 * 152;

// one tile at (r0, c0), K range [kbeg, kend), kbeg a multiple of DG_BK
template <bool TA, bool TB, int BM, int BN>
__device__ __forceinline__ void dgemm_tile(int r0, int c0, int M, int N, int K, int kbeg, int kend, double alpha,
                                           const double* A, int64_t lda, const double* B, int64_t ldb, double beta,
                                           double* C, int64_t ldc) {
    constexpr int TM = BM / 16, TN = BN / 16, PA = DG_BK * BM / DG_T, PB = DG_BK * BN / DG_T;
    __shared__ double As[DG_BK][BM + 1];
    __shared__ double Bs[DG_BK][BN + 1];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    double acc[TM][TN];
#pragma unroll
    for (int p = 0; p < TM; ++p)
#pragma unroll
        for (int q = 0; q < TN; ++q) acc[p][q] = 0.0;
    kend = min(kend, K);
    double va[PA], vb[PB];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int u = 0; u < PA; ++u) {
            const int e = threadIdx.x + u * DG_T;
            int m, kk;
            if (TA) { m = e % BM; kk = e / BM; } else { kk = e % DG_BK; m = e / DG_BK; }
            const int gi = r0 + m, gk = k0 + kk;
            va[u] = (gi < M && gk < kend) ? (TA ? A[(int64_t)gk * lda + gi] : A[(int64_t)gi * lda + gk]) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < PB; ++u) {
            const int e = threadIdx.x + u * DG_T;
            int nn, kk;
            if (TB) { kk = e % DG_BK; nn = e / DG_BK; } else { nn = e % BN; kk = e / BN; }
            const int gj = c0 + nn, gk = k0 + kk;
            vb[u] = (gj < N && gk < kend) ? (TB ? B[(int64_t)gj * ldb + gk] : B[(int64_t)gk * ldb + gj]) : 0.0;
        }
    };
    if (kbeg < kend) fetch(kbeg);
    for (int k0 = kbeg; k0 < kend; k0 += DG_BK) {
#pragma unroll
        for (int u = 0; u < PA; ++u) {
            const int e = threadIdx.x + u * DG_T;
            if (TA) As[e / BM][e % BM] = va[u]; else As[e % DG_BK][e / DG_BK] = va[u];
        }
#pragma unroll
        for (int u = 0; u < PB; ++u) {
            const int e = threadIdx.x + u * DG_T;
            if (TB) Bs[e % DG_BK][e / DG_BK] = vb[u]; else Bs[e / BN][e % BN] = vb[u];
        }
        __syncthreads();
        if (k0 + DG_BK < kend) fetch(k0 + DG_BK);
#pragma unroll
        for (int kk = 0; kk < DG_BK; ++kk) {
            double a[TM], b[TN];
#pragma unroll
            for (int p = 0; p < TM; ++p) a[p] = As[kk][ty + 16 * p];
#pragma unroll
            for (int q = 0; q < TN; ++q) b[q] = Bs[kk][tx + 16 * q];
#pragma unroll
            for (int p = 0; p < TM; ++p)
#pragma unroll
                for (int q = 0; q < TN; ++q) acc[p][q] = fma(a[p], b[q], acc[p][q]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int p = 0; p < TM; ++p) {
        int i = r0 + ty + 16 * p;
        if (i >= M) continue;
#pragma unroll
        for (int q = 0; q < TN; ++q) {
            int j = c0 + tx + 16 * q;
            if (j >= N) continue;
            double* cp = C + (int64_t)i * ldc + j;
            *cp = beta == 0.0 ? alpha * acc[p][q] : fma(beta, *cp, alpha * acc[p][q]);
        }
    }
}

template <bool TA, bool TB, int BM, int BN>
__global__ void __launch_bounds__(DG_T) k_dgemm(int M, int N, int K, double alpha, const double* A,
                                               int64_t lda, const double* B, int64_t ldb, double beta,
                                               double* C, int64_t ldc, int lower, int tri, const unsigned* status) {
    if (status && *status) return;
    const int r0 = blockIdx.y * BM, c0 = blockIdx.x * BN;
    if (lower && c0 > r0 + BM - 1) return;
    int kbeg = 0;
    if (tri & 1) kbeg = max(kbeg, r0);
    if (tri & 2) kbeg = max(kbeg, c0);
    dgemm_tile<TA, TB, BM, BN>(r0, c0, M, N, K, (kbeg / DG_BK) * DG_BK, K, alpha, A, lda, B, ldb, beta, C, ldc);
}

// One level of the blocked inverse of a lower-triangular W whose diagonal blocks of size s are inverted:
// for every pair of blocks (rows [r, r + s2) below columns [r - s, r), s2 the rows that exist),
//   step 1: T = W_21 W_11,   step 2: W_21 <- -W_22 T      (W_11, W_22 lower triangular: K skips their zeros).
// grid (s / BM, s / BM, pairs); T is an n x n scratch, used at the place of W_21.  Every level is two launches
// over all pairs; block row by block row the inverse of 2,048 rows was 62 launches of at most 32 tiles each
// (36 of the 62 ms of an inversion).
template <int BM>
__global__ void __launch_bounds__(DG_T) k_trinv_level(double* W, double* T, int64_t n, int s, int step,
                                                      const unsigned* status) {
    if (status && *status) return;
    const int64_t c = (int64_t)blockIdx.z * 2 * s, r = c + s;
    const int s2 = (int)min((int64_t)s, n - r);
    const int r0 = blockIdx.y * BM, c0 = blockIdx.x * BM;
    if (r0 >= s2) return;
    double* W21 = W + r * n + c;
    double* T21 = T + r * n + c;
    if (step == 1) dgemm_tile<false, false, BM, BM>(r0, c0, s2, s, s, c0, s, 1.0, W21, n, W + c * n + c, n, 0.0, T21, n);
    else dgemm_tile<false, false, BM, BM>(r0, c0, s2, s, s2, 0, r0 + BM, -1.0, W + r * n + r, n, T21, n, 0.0, W21, n);
}

template <bool TA, bool TB>
static void dgemm_tiles(cudaStream_t s, int M, int N, int K, double alpha, const double* A, int64_t lda, const double* B,
                        int64_t ldb, double beta, double* C, int64_t ldc, int lower, int tri, const unsigned* status) {
    const int64_t tm = (M + DG_LARGE - 1) / DG_LARGE, tn = (N + DG_LARGE - 1) / DG_LARGE, tiles = lower ? tm * (tm + 1) / 2 : tm * tn;
    if (tiles >= DG_MANY)
        k_dgemm<TA, TB, DG_LARGE, DG_LARGE><<<dim3((unsigned)tn, (unsigned)tm), DG_T, 0, s>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc,
                                                                                 lower, tri, status);
    else
        k_dgemm<TA, TB, DG_SMALL, DG_SMALL><<<dim3((N + DG_SMALL - 1) / DG_SMALL, (M + DG_SMALL - 1) / DG_SMALL), DG_T, 0, s>>>(M, N, K, alpha, A, lda, B, ldb, beta, C,
                                                                                   ldc, lower, tri, status);
}

cpm_status launch_dgemm(cudaStream_t s, bool ta, bool tb, int M, int N, int K, double alpha, const double* A,
                        int64_t lda, const double* B, int64_t ldb, double beta, double* C, int64_t ldc, int lower,
                        int tri, const unsigned* status) {
    if (M <= 0 || N <= 0) return CPM_OK;
    if (ta && tb) dgemm_tiles<true, true>(s, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, lower, tri, status);
    else if (ta) dgemm_tiles<true, false>(s, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, lower, tri, status);
    else if (tb) dgemm_tiles<false, true>(s, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, lower, tri, status);
    else dgemm_tiles<false, false>(s, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, lower, tri, status);
    return cudaGetLastError() == cudaSuccess ? CPM_OK : CPM_E_CUDA;
}

// ----------------------------------------------------------------------------- diagonal blocks
constexpr int NB = 64;

// Unblocked Cholesky of one kb x kb diagonal block (in place, lower), and the inverse of
// its factor written to Linv (NB x NB, zero above the diagonal).  A pivot that is not
// positive and finite sets ST_NOT_SPD and stops the factorisation.
// One pass eliminates both: after column j, row i > j gets its rank-one update of the trailing columns
// k = j + 1 .. i and of the inverse's columns c = 0 .. j, i + 1 terms over eight threads per row.  The inverse shares
// the array: its entry (i, c) sits at [c][i + 1].  One SM's FP64 pipe takes 16 clocks per warp instruction, so
// nothing is computed twice: two warps form the square root and the reciprocal square root of the next pivot
// beside the update, and the column is scaled by a product.
constexpr int PF_L = 8, PF_U = NB * PF_L, PF_T = PF_U + 64;   // update threads, then the two pivot warps
__global__ void __launch_bounds__(PF_T) k_potrf(double* Ab, int64_t lda, int kb, double* Linv, unsigned* status) {
    if (*status) return;
    __shared__ double L[NB][NB + 3];
    __shared__ double s_piv[2], s_inv[2];
    __shared__ int bad;
    for (int e = threadIdx.x; e < NB * NB; e += PF_T) {
        const int i = e / NB, j = e % NB;
        if (j <= i) {
            L[i][j] = i < kb ? Ab[(int64_t)i * lda + j] : (i == j ? 1.0 : 0.0);
            L[j][i + 1] = 0.0;   // minus the sum over k of L_ik Linv_kj so far
        }
    }
    if (threadIdx.x == 0) bad = 0;
    __syncthreads();
    const int i = threadIdx.x / PF_L, q = threadIdx.x % PF_L;
    const bool root = threadIdx.x == PF_U, rroot = threadIdx.x == PF_U + 32;
    auto pivot = [&](int j, double pv) {
        if (root) {
            if (!(pv > 0.0) || !isfinite(pv)) bad = 1;
            s_piv[j & 1] = sqrt(pv);
        } else {
            s_inv[j & 1] = rsqrt(pv);
        }
    };
    if (root || rroot) pivot(0, L[0][0]);
    for (int j = 0; j < kb; ++j) {   // a last block of fewer rows ends there
        __syncthreads();
        if (bad) break;   // set before the barrier; nobody writes it until the next one
        const double piv = s_piv[j & 1], inv = s_inv[j & 1];
        if ((int)threadIdx.x < NB) {   // column j of the factor, row j of the inverse
            const int t = threadIdx.x;
            if (t > j) L[t][j] *= inv;
            else if (t == j) L[j][j] = piv;
        } else if ((int)threadIdx.x < 2 * NB) {
            const int t = threadIdx.x - NB;
            if (t < j) L[t][j + 1] *= inv;
            else if (t == j) L[j][j + 1] = inv;
        }
        __syncthreads();
        if ((int)threadIdx.x < PF_U) {
            if (i > j) {
                const double lij = L[i][j];
                for (int c = q; c <= i; c += PF_L) {
                    if (c <= j) L[c][i + 1] = fma(-lij, L[c][j + 1], L[c][i + 1]);
                    else if (c < i || i > j + 1) L[i][c] = fma(-lij, L[c][j], L[i][c]);   // the next pivot: below
                }
            }
        } else if ((root || rroot) && j + 1 < kb) {
            pivot(j + 1, fma(-L[j + 1][j], L[j + 1][j], L[j + 1][j + 1]));
        }
    }
    __syncthreads();
    if (bad) {
        if (threadIdx.x == 0) atomicOr(status, ST_NOT_SPD);
        return;
    }
    for (int e = threadIdx.x; e < kb * kb; e += PF_T) {
        const int r = e / kb, j = e % kb;
        Ab[(int64_t)r * lda + j] = j <= r ? L[r][j] : 0.0;
    }
    for (int e = threadIdx.x; e < NB * NB; e += PF_T) {
        const int r = e / NB, j = e % NB;
        Linv[e] = (j <= r && r < kb) ? L[j][r + 1] : 0.0;
    }
}

// Inverse of every NB x NB lower-triangular diagonal block of an n x n factor, in place (the factor is staged in
// shared memory; each thread writes one column of the inverse straight to the block); one CTA per block.
__global__ void __launch_bounds__(64) k_trtri(double* W, int64_t n, const unsigned* status) {
    if (*status) return;
    __shared__ double L[NB][NB + 1];
    const int64_t k0 = (int64_t)blockIdx.x * NB;
    const int kb = (int)min((int64_t)NB, n - k0);
    double* Ab = W + k0 * n + k0;
    for (int e = threadIdx.x; e < NB * NB; e += blockDim.x) {
        int i = e / NB, j = e % NB;
        L[i][j] = (i < kb && j <= i) ? Ab[(int64_t)i * n + j] : 0.0;
    }
    __syncthreads();
    const int col = threadIdx.x;
    if (col < kb) {
        for (int i = 0; i < kb; ++i) {
            double x = 0.0;
            if (i == col) x = 1.0 / L[i][i];
            else if (i > col) {
                double s = 0.0;
                for (int k = col; k < i; ++k) s += L[i][k] * Ab[(int64_t)k * n + col];
                x = -s / L[i][i];
            }
            Ab[(int64_t)i * n + col] = x;
        }
    }
}

// ----------------------------------------------------------------------------- projection
__global__ void k_mirror_lower(double* S, int64_t n) {
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t i = blockIdx.y; i < n; i += gridDim.y)
        if (j < i) S[j * n + i] = S[i * n + j];
}

// d_i = sum_j S_ij, one warp per row (fixed order).
__global__ void k_rowsum(const double* S, int64_t n, double* d) {
    int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
    int lane = threadIdx.x & 31;
    if (row >= n) return;
    double s = 0.0;
    for (int64_t j = lane; j < n; j += 32) s += S[row * n + j];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) d[row] = s;
}

// out[0] = sum_i v_i, single block, fixed order.
__global__ void k_sum1(const double* v, int64_t n, double* out) {
    __shared__ double sh[1024];
    double s = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) s += v[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = sh[0];
}

__global__ void k_project(double* S, float* S32, const double* d, const double* dsum, int64_t n, int symm,
                          double* u) {
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const double s = *dsum;
    for (int64_t i = blockIdx.y; i < n; i += gridDim.y) {
        double v = S[i * n + j];
        if (symm) v -= d[i] * d[j] / s;
        S[i * n + j] = v;
        S32[i * n + j] = (float)v;
        if (i == 0 && u) u[j] = symm ? d[j] / s : 0.0;
    }
}

// SG[i][g] = sum_{j in electrode g} S_ij, one warp per row; at most 16 electrodes.
__global__ void k_sg(const double* S, const int* group, int64_t n, int ng, double* SG) {
    int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
    int lane = threadIdx.x & 31;
    if (row >= n) return;
    double acc[16];
#pragma unroll
    for (int g = 0; g < 16; ++g) acc[g] = 0.0;
    for (int64_t j = lane; j < n; j += 32) {
        int g = group[j];
        double v = S[row * n + j];
#pragma unroll
        for (int h = 0; h < 16; ++h)
            if (h == g) acc[h] += v;
    }
    for (int g = 0; g < ng; ++g) {
        double s = acc[g < 16 ? g : 0];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) SG[row * ng + g] = s;
    }
}

cpm_status invert_and_project(cpm_ctx* c) {
    const int64_t n = c->n;
    cudaStream_t st = c->stream;
    double* W = c->W;
    double* Linv = c->red + 64;   // NB x NB scratch follows the scalars
    CPM_CUDA(c, cudaMemsetAsync(c->status, 0, sizeof(unsigned), st));
    CPM_CUDA(c, cudaMemcpyAsync(W, c->A, (size_t)n * n * sizeof(double), cudaMemcpyDeviceToDevice, st));
    // blocked right-looking Cholesky, lower triangle
    for (int64_t k0 = 0; k0 < n; k0 += NB) {
        const int kb = (int)std::min<int64_t>(NB, n - k0);
        k_potrf<<<1, PF_T, 0, st>>>(W + k0 * n + k0, n, kb, Linv, c->status);
        CPM_LAUNCH(c, "k_potrf");
        const int rows = (int)(n - k0 - kb);
        if (rows > 0) {
            double* P = W + (k0 + kb) * n + k0;
            // panel: P <- P L_kk^-T (in place; one 64-wide tile column, so every block owns its rows; 16 rows each,
            // for as many blocks as there are SMs)
            k_dgemm<false, true, 16, NB><<<dim3(1, (rows + 15) / 16), DG_T, 0, st>>>(rows, kb, kb, 1.0, P, n, Linv, NB, 0.0,
                                                                                    P, n, 0, 0, c->status);
            CPM_LAUNCH(c, "k_dgemm(panel)");
            // trailing update, lower triangle: A22 <- A22 - P P^T
            CPM_TRY(launch_dgemm(st, false, true, rows, rows, kb, -1.0, P, n, P, n, 1.0, W + (k0 + kb) * (n + 1), n, 1,
                                 0, c->status));
        }
    }
    unsigned hst = 0;
    CPM_CUDA(c, cudaMemcpyAsync(&hst, c->status, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
    CPM_CUDA(c, cudaStreamSynchronize(st));
    if (hst & ST_NOT_SPD) return set_err(c, CPM_E_NOT_SPD, "elastance matrix is not positive definite");
    // W <- L^-1: the diagonal blocks, then pairs of blocks of doubling size, with S as scratch
    k_trtri<<<(unsigned)((n + NB - 1) / NB), 64, 0, st>>>(W, n, c->status);
    CPM_LAUNCH(c, "k_trtri");
    for (int64_t s = NB; s < n; s *= 2) {
        const int64_t pairs = (n - s + 2 * s - 1) / (2 * s);
        for (int step = 1; step <= 2; ++step) {
            const unsigned large = (unsigned)(s / DG_LARGE), small = (unsigned)(s / DG_SMALL);
            if ((int64_t)large * large * pairs >= DG_MANY)
                k_trinv_level<DG_LARGE><<<dim3(large, large, (unsigned)pairs), DG_T, 0, st>>>(W, c->S, n, (int)s, step, c->status);
            else
                k_trinv_level<DG_SMALL><<<dim3(small, small, (unsigned)pairs), DG_T, 0, st>>>(W, c->S, n, (int)s, step, c->status);
        }
        CPM_LAUNCH(c, "k_trinv_level");
    }
    // A^-1 = W^T W, lower tiles, then mirrored
    CPM_TRY(launch_dgemm(st, true, false, (int)n, (int)n, (int)n, 1.0, W, n, W, n, 0.0, c->S, n, 1, 3, c->status));
    dim3 g2((unsigned)((n + 255) / 256), (unsigned)(n < 65535 ? n : 65535));
    k_mirror_lower<<<g2, 256, 0, st>>>(c->S, n);
    CPM_LAUNCH(c, "k_mirror_lower");
    return project_inverse(c);
}

// Row sums of the single-precision S in FP64 (one warp per row, a fixed order), into dvec.  The
// single-precision products centre b per output, sum_j S_ij (b_j - b_i); without the projection
// (symm = 0) the rows of A^-1 do not sum to zero, and the update adds b_i times these sums back.
__global__ void k_rowsum32(const float* S32, int64_t n, double* out) {
    const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
    const int lane = threadIdx.x & 31;
    if (row >= n) return;
    double s = 0.0;
    for (int64_t j = lane; j < n; j += 32) s += (double)S32[row * n + j];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) out[row] = s;
}

cpm_status fp32_rowsums(cpm_ctx* c) {
    if (c->p.symm) return CPM_OK;
    k_rowsum32<<<(unsigned)((c->n * 32 + 255) / 256), 256, 0, c->stream>>>(c->S32, c->n, c->dvec);
    CPM_LAUNCH(c, "k_rowsum32");
    return CPM_OK;
}

// With A^-1 in S: d = A^-1 e, e^T d, the projection of Eq. (S) (symm = 1), the FP32 copy of S, u and
// SG = S G; synchronises.
cpm_status project_inverse(cpm_ctx* c) {
    const int64_t n = c->n;
    cudaStream_t st = c->stream;
    dim3 g2((unsigned)((n + 255) / 256), (unsigned)(n < 65535 ? n : 65535));
    k_rowsum<<<(unsigned)((n * 32 + 255) / 256), 256, 0, st>>>(c->S, n, c->dvec);
    CPM_LAUNCH(c, "k_rowsum");
    k_sum1<<<1, 1024, 0, st>>>(c->dvec, n, c->red);
    CPM_LAUNCH(c, "k_sum1");
    k_project<<<g2, 256, 0, st>>>(c->S, c->S32, c->dvec, c->red, n, c->p.symm, c->u);
    CPM_LAUNCH(c, "k_project");
    k_sg<<<(unsigned)((n * 32 + 255) / 256), 256, 0, st>>>(c->S, c->group, n, c->ng, c->SG);
    CPM_LAUNCH(c, "k_sg");
    CPM_TRY(fp32_rowsums(c));
    CPM_CUDA(c, cudaMemcpyAsync(&c->etd, c->red, sizeof(double), cudaMemcpyDeviceToHost, st));
    CPM_CUDA(c, cudaStreamSynchronize(st));
    ccm_invalidate(c);
    return CPM_OK;
}

}  // namespace cpm
