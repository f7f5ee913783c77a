// P3M (particle-particle particle-mesh) reciprocal part of the electrolyte vector b: the k-space
// solver the paper's package offers beside the Ewald sum (Introduction; SI Sec. 1.A-B), written
// after the textbook method of Hockney and Eastwood:
//   1. every charge is assigned to the p^3 nearest mesh points with the order-p cardinal B-spline
//      W(s) = M_p(s + p/2) per axis,
//   2. the mesh is Fourier transformed, multiplied by the optimal influence function for potentials
//        G(k) = sum_m U^2(k_m) R(k_m) / (sum_m U^2(k_m))^2,  k_m = k + 2 pi m / h,  m in [-2, 2]^3,
//        U(k) = prod_d sinc(k_d h_d / 2)^p,  R(k) = 4 pi exp(-k^2 / 4 alpha^2) / k^2,  G(0) = 0,
//      and transformed back,
//   3. the mesh potential is interpolated at the electrode sites with the same weights:
//        phi_i = (1/V) sum_mesh W_i(x) IFFT[G FFT[rho]](x).
// The elastance matrix A keeps the Ewald sum; only the per-step b takes this path.
//
// GPU design (one GPU, m replicas per launch):
// * Two replicas share one complex mesh (real part, imaginary part).  G is real and even on the
//   mesh, so IFFT(G FFT(rho_a + i rho_b)) = phi_a + i phi_b exactly: one complex transform serves
//   two replicas.
// * Charge assignment: one CTA per (mesh brick, replica) owns the brick's points in shared
//   memory and takes every charge whose stencil reaches into the brick (listed beforehand), adding only
//   the points it owns.  Every mesh point is written by exactly one CTA, with a plain store: no halo exchange and
//   no global atomics.  Inside the brick the contributions are added as exact fixed-point integers
//   with 32-bit shared-memory atomics, so the mesh charge does not depend on the order of the
//   atomics and the whole path is deterministic.  Bricks that no charge reaches are not written, only marked,
//   and planes of such bricks are not transformed (an electrolyte fills a third of a slab cell).
// * Transforms: radix-2 decimation in time in shared memory with twiddles tabulated in FP64 on the
//   host.  The forward and inverse xy transforms take a whole plane per CTA; the z pass loads
//   16 z lines per CTA, transforms them forward, multiplies by G, transforms back and stores, so
//   the reciprocal-space product never leaves shared memory.
// * Interpolation: one warp per (site, replica pair); lanes take the p^2 (x, y) columns, each runs
//   over the p z points; the warp sum is a fixed butterfly.
//   Sites that share few heights (at most one per LAYER_MIN_SITES sites, as in the product basis): the z pass
//   applies each height's z weights while the line is in shared memory, the inverse xy transform runs on one plane
//   per height instead of on every plane a stencil reads, and a site sums p^2 points with weights kept since the
//   preparation.  Inverse xy transform and interpolation together: 4,320 sites x 8 replicas, 128 mesh planes,
//   29 -> 14 us; 16,384 sites x 16 replicas, 64 planes, 141 -> 43 us.
// Arithmetic in T = double (k_prec = FP64) or float (the single-precision paths); the influence
// function is computed in FP64 and stored in T.
#include <climits>

#include "common.cuh"

namespace cpm {

constexpr int P3M_THREADS = 256;
constexpr int P3M_ZTX = 16;                       // z lines per CTA of the z pass

__host__ __device__ inline int ilog2i(int v) { int l = 0; while ((1 << l) < v) ++l; return l; }

bool p3m_mesh_ok(const cpm_params* p) {
    if (p->p3m_order < 2 || p->p3m_order > 7) return false;
    for (int d = 0; d < 3; ++d) {
        const int K = p->p3m_mesh[d];
        if (K < 8 || K > P3M_MAX_MESH || (K & (K - 1))) return false;
    }
    const size_t cs = (p->k_prec == CPM_PREC_FP64 || p->p3m_matrix) ? 16 : 8;
    return (size_t)p->p3m_mesh[0] * p->p3m_mesh[1] * cs <= P3M_PLANE_BYTES;
}

// ----------------------------------------------------------------------------- influence function
// One thread per mesh point (x fastest); frequency index n_d = i_d for i_d < K_d / 2, else i_d - K_d
// (the ordering of a discrete Fourier transform).  Stores G / V in T.
template <typename T>
__global__ void k_p3m_green(int Kx, int Ky, int Kz, int P, double Lx, double Ly, double Lz, double alpha, double V,
                            T* __restrict__ G) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t N = (int64_t)Kx * Ky * Kz;
    if (t >= N) return;
    const int ix = (int)(t % Kx), iy = (int)((t / Kx) % Ky), iz = (int)(t / ((int64_t)Kx * Ky));
    const int K[3] = {Kx, Ky, Kz};
    const int I[3] = {ix, iy, iz};
    const double L[3] = {Lx, Ly, Lz};
    double u2[3][5], kk[3][5], den[3];
    for (int d = 0; d < 3; ++d) {
        const int nd = I[d] < K[d] / 2 ? I[d] : I[d] - K[d];
        den[d] = 0.0;
        for (int m = -2; m <= 2; ++m) {
            const double s = (double)nd / K[d] + m;
            const double sc = s == 0.0 ? 1.0 : sinpi(s) / (PI * s);
            double pw = 1.0;
            for (int e = 0; e < 2 * P; ++e) pw *= sc;
            u2[d][m + 2] = pw;
            den[d] += pw;
            kk[d][m + 2] = 2.0 * PI * (nd + (double)m * K[d]) / L[d];
        }
    }
    double num = 0.0;
    const double q = 1.0 / (4.0 * alpha * alpha);
    for (int a = 0; a < 5; ++a)
        for (int b = 0; b < 5; ++b)
            for (int c = 0; c < 5; ++c) {
                const double k2 = kk[0][a] * kk[0][a] + kk[1][b] * kk[1][b] + kk[2][c] * kk[2][c];
                if (k2 > 0.0) num += u2[0][a] * u2[1][b] * u2[2][c] * (4.0 * PI * exp(-k2 * q) / k2);
            }
    const double dd = den[0] * den[1] * den[2];
    const double g = (ix == 0 && iy == 0 && iz == 0) ? 0.0 : num / (dd * dd);
    G[t] = (T)(g / V);
}

// ----------------------------------------------------------------------------- charge preparation
// Per charge: the first mesh index of its stencil per axis, packed as bx | by << 10 | bz << 20 (-1 for
// Q = 0), and (fx, fy, fz, Q) with f the offset of the point from that stencil's assignment origin:
// u = x K / L (wrapped into the cell), t = u - p/2, base = floor(t) + 1, f = t - floor(t).  The weight of
// mesh point base + a is then M_p(f + p - 1 - a).
template <typename T> struct P3mV4;
template <> struct P3mV4<float> { using t = float4; };
template <> struct P3mV4<double> { using t = double4_32a; };

// The bricks of a mesh (x fastest) and those that the stencil of a charge reaches, each once.
constexpr int P3M_BZ = 4;            // planes per brick (lanes 8 z + y of the assignment)
struct P3mBricks {
    int BX, BY, nx, ny, nz;
    __host__ __device__ int n() const { return nx * ny * nz; }
    template <typename F> __device__ __forceinline__ void each(int kv, int P, F f) const {
        if (kv < 0) return;   // no charge
        const int x = kv & 1023, y = (kv >> 10) & 1023, z = kv >> 20;
        const int x0 = x / BX, y0 = y / BY, z0 = z / P3M_BZ;
        const int cx = min(nx, (x + P - 1) / BX - x0 + 1), cy = min(ny, (y + P - 1) / BY - y0 + 1),
                  cz = min(nz, (z + P - 1) / P3M_BZ - z0 + 1);
        for (int c = 0; c < cz; ++c)
            for (int b = 0; b < cy; ++b)
                for (int a = 0; a < cx; ++a) {
                    int bx = x0 + a, by = y0 + b, bz = z0 + c;
                    if (bx >= nx) bx -= nx;
                    if (by >= ny) by -= ny;
                    if (bz >= nz) bz -= nz;
                    f((bz * ny + by) * nx + bx);
                }
    }
    // at most this many bricks per charge
    int most(int P) const {
        return std::min(nx, (P + BX - 2) / BX + 1) * std::min(ny, (P + BY - 2) / BY + 1) * std::min(nz, (P + P3M_BZ - 2) / P3M_BZ + 1);
    }
};

template <typename T>
__global__ void k_p3m_prep(const double* __restrict__ xyz, const double* __restrict__ Q, int64_t ptot, Geometry g,
                           int Kx, int Ky, int Kz, int P, int* __restrict__ key, typename P3mV4<T>::t* __restrict__ fq,
                           int64_t ne, P3mBricks br, int nsplit, int64_t per, int* __restrict__ count) {
    grid_go();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ptot) return;
    const double q = Q[t];
    const int K[3] = {Kx, Ky, Kz};
    double f[3];
    int b[3];
    for (int d = 0; d < 3; ++d) {
        double s = xyz[3 * t + d] * g.inv[d];
        s -= floor(s);
        const double u = s * K[d] - 0.5 * P;
        const double fl = floor(u);
        f[d] = u - fl;
        int bi = ((int)fl + 1) % K[d];
        if (bi < 0) bi += K[d];
        b[d] = bi;
    }
    const int kv = q == 0.0 ? -1 : (b[0] | (b[1] << 10) | (b[2] << 20));
    key[t] = kv;
    const int64_t r = t / ne, row = r * nsplit + (t - r * ne) / per;
    br.each(kv, P, [&](int brick) { atomicAdd(&count[row * br.n() + brick], 1); });
    typename P3mV4<T>::t v;
    v.x = (T)f[0]; v.y = (T)f[1]; v.z = (T)f[2]; v.w = (T)q;
    fq[t] = v;
}

// The p weights M_p(f + p - 1 - a), a = 0..p-1, of offset f in [0, 1), by the B-spline recursion
// M_1 = 1 on [0, 1), M_n(x) = (x M_{n-1}(x) + (n - x) M_{n-1}(x - 1)) / (n - 1) evaluated at x = f + j.
template <typename T, int P>
__device__ __forceinline__ void bspline_weights(T f, T* w) {
    T m[P];   // m[j] = M_n(f + j), j = 0..n-1
    m[0] = (T)1;
#pragma unroll
    for (int j = 1; j < P; ++j) m[j] = (T)0;
#pragma unroll
    for (int n = 2; n <= P; ++n) {
        const T inv = (T)1 / (T)(n - 1);
#pragma unroll
        for (int j = n - 1; j >= 0; --j) {
            const T x = f + (T)j;
            const T lo = j > 0 ? m[j - 1] : (T)0;   // M_{n-1}(x - 1)
            m[j] = (x * m[j] + ((T)n - x) * lo) * inv;
        }
    }
#pragma unroll
    for (int a = 0; a < P; ++a) w[a] = m[P - 1 - a];
}

// ----------------------------------------------------------------------------- charge assignment
// grid (bricks, replicas, charge splits); a brick is BX x BY x BZ mesh points (x fastest), brick index bx fastest.
// The charges whose stencil reaches into a brick are listed beforehand (counted with the preparation, k_p3m_scan,
// k_p3m_fill; the order within a list varies, the sums do not): with each brick looking through all keys of its
// replica, that took half of the time (270 of 538 us for 16,384 sites x 16 replicas), and the weights of the few
// charges found were formed by warps with two lanes of work.  A split takes a fixed range of the replica's
// charges, so that its sum does not depend on the order either.  Their 3 p weights and the stencil origins
// relative to the brick go to shared memory, NT charges at a time; then a warp takes one charge at a time, lane =
// (plane of the brick, y offset), each lane adding its p x contributions.
// Every contribution is rounded to 2^-40 e (FP64: 2^-60 e) and added as exact integers split over
// 32-bit words, a = floor(v 2^20), then the next 20 bits (FP64: and 20 more), with native 32-bit
// shared-memory atomics; integer addition is associative, so the brick's charge does not depend on
// the order of the atomics.  The low words carry into the next at least every P3M_CARRY charges (each adds at
// most 2^20 to a low word), and a wraps modulo 2^32, exact while the final charge of a mesh
// point stays below 2,048 e.
// Layout: with the whole y period and four planes in a brick, 28 of 32 lanes have a row for order 7 (all of them
// in the brick but for its first and last planes); rows are padded to BX + 1 words and planes by 8, so the rows of
// one charge fall in distinct banks.  Bricks of half a y period and eight planes with the rows spread over
// threads left three of four lanes without work: 136 us for 8 EDL replicas.
// The split's brick goes to its own partial mesh (part, real and imaginary part for even and odd replicas) if a
// charge reached it (flag); the first transform sums the splits in split order.
template <typename T> struct P3mWords { static constexpr int n = std::is_same<T, double>::value ? 3 : 2; };
constexpr int P3M_NT = 512;          // threads and charges per chunk of the assignment
constexpr int P3M_CARRY = 1024;

// Every (replica, split) has a list of its own, at most `most` entries for each of its `per` charges, so that positions in
// it are ints: the plan takes enough splits for that.
constexpr int P3M_MOST = 12;   // stencils of seven points over bricks of 32 x 32 x 4 (and no wider ones): 2 x 2 x 3
static int64_t p3m_split_most(int most) { return (int64_t)INT_MAX / most / P3M_NT; }   // chunks of charges per split
static_assert(MAX_POINTS / P3M_NT / ((int64_t)INT_MAX / P3M_MOST / P3M_NT) + 1 <= 8, "splits of the largest call");

// start[r][split][brick]: exclusive sums of the nb counts of a (replica, split), one block each
constexpr int P3M_SCAN = 256;
__global__ void __launch_bounds__(P3M_SCAN) k_p3m_scan(const int* __restrict__ count, int nb, int* __restrict__ start) {
    grid_wait();
    grid_go();
    __shared__ int sw[P3M_SCAN / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t r0 = (int64_t)blockIdx.x * nb;
    int carry = 0;
    for (int i0 = 0; i0 < nb; i0 += P3M_SCAN) {
        const int i = i0 + threadIdx.x, c = i < nb ? count[r0 + i] : 0;
        int v = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += u;
        }
        if (lane == 31) sw[warp] = v;
        __syncthreads();
        int before = carry, all = 0;
#pragma unroll
        for (int w = 0; w < P3M_SCAN / 32; ++w) {
            before += w < warp ? sw[w] : 0;
            all += sw[w];
        }
        if (i < nb) start[r0 + i] = before + v - c;
        carry += all;
        __syncthreads();
    }
}

// list[(r nsplit + split) per most + start + ..]: the charges of every brick; the starts become ends
__global__ void __launch_bounds__(256) k_p3m_fill(const int* __restrict__ key, int64_t ptot, int64_t ne, int P, P3mBricks br,
                                                int nsplit, int64_t per, int most, int* __restrict__ start, int* __restrict__ list) {
    grid_wait();
    const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (t >= ptot) return;
    const int64_t r = t / ne, j = t - r * ne, row = r * nsplit + j / per;
    int* mine = list + row * per * most;
    br.each(key[t], P, [&](int brick) {
        mine[atomicAdd(&start[row * br.n() + brick], 1)] = (int)j;
    });
}

template <typename T, int P>
__global__ void __launch_bounds__(P3M_NT) k_p3m_spread(const int* __restrict__ key,
                                                       const typename P3mV4<T>::t* __restrict__ fq, int64_t ne, int m,
                                                       int Kx, int Ky, int Kz, int BX, int BY,
                                                       const int* __restrict__ count, const int* __restrict__ start,
                                                       const int* __restrict__ list, int64_t per, int most,
                                                       c2<T>* __restrict__ part, int* __restrict__ flag) {
    grid_wait();
    constexpr int NW = P3mWords<T>::n, BZ = P3M_BZ;
    extern __shared__ __align__(16) unsigned char p3m_smem[];
    const int RX = BX + 1, PS = BY * RX + 8;            // padded row and plane
    const int NB = PS * BZ;
    int* A = (int*)p3m_smem;                            // [NW words][NB]
    T* sw = (T*)(A + ((NW * NB + 3) & ~3));             // [NT][3 p + 1]: weights x | y | z, then Q
    int* so = (int*)(sw + P3M_NT * (3 * P + 1));        // [NT]: origin sx | sy << 10 | sz << 20
    const int nbx = Kx / BX, nby = Ky / BY;
    const int bi = blockIdx.x, rep = blockIdx.y;
    const int b0x = (bi % nbx) * BX, b0y = ((bi / nbx) % nby) * BY, b0z = (bi / (nbx * nby)) * BZ;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t base = (int64_t)rep * ne, at = ((int64_t)rep * gridDim.z + blockIdx.z) * gridDim.x + bi;
    const int total = count[at];
    if (threadIdx.x == 0) flag[((int64_t)blockIdx.z * m + rep) * gridDim.x + bi] = total > 0;
    if (total == 0) return;   // uniform
    const int* mine = list + ((int64_t)rep * gridDim.z + blockIdx.z) * per * most + start[at] - total;   // start holds the end
    auto carry = [&]() {   // every point's words belong to one thread here
        __syncthreads();
        for (int i = threadIdx.x; i < NB; i += P3M_NT) {
            int lo = A[NB + i];
            if (NW == 3) {
                const int c = A[2 * NB + i];
                lo += c >> 20;
                A[2 * NB + i] = c & 0xFFFFF;
            }
            A[i] += lo >> 20;
            A[NB + i] = lo & 0xFFFFF;
        }
        __syncthreads();
    };
    int added = 0;         // charges since the last carry
    for (int i = threadIdx.x; i < NW * NB; i += P3M_NT) A[i] = 0;
    for (int j0 = 0; j0 < total; j0 += P3M_NT) {
        const int L = min(P3M_NT, total - j0);
        if (added + L > P3M_CARRY) {
            carry();
            added = 0;
        }
        added += L;
        if ((int)threadIdx.x < L) {
            const int slot = threadIdx.x;
            const int64_t j = mine[j0 + slot];
            const int kv = key[base + j];
            const int sx = ((kv & 1023) - b0x + Kx) & (Kx - 1), sy = (((kv >> 10) & 1023) - b0y + Ky) & (Ky - 1),
                      sz = ((kv >> 20) - b0z + Kz) & (Kz - 1);
            const typename P3mV4<T>::t v = fq[base + j];
            T* w = sw + slot * (3 * P + 1);
            bspline_weights<T, P>(v.x, w);
            bspline_weights<T, P>(v.y, w + P);
            bspline_weights<T, P>(v.z, w + 2 * P);
            w[3 * P] = v.w;
            so[slot] = sx | (sy << 10) | (sz << 20);
        }
        __syncthreads();
        const int zz = lane >> 3, b = lane & 7;
        for (int sl = wid; sl < L; sl += P3M_NT / 32) {
            const int o = so[sl];
            const T* w = sw + sl * (3 * P + 1);
            const int c = (zz - (o >> 20)) & (Kz - 1);   // z offset whose plane is zz
            int gy = ((o >> 10) & 1023) + b;
            if (gy >= Ky) gy -= Ky;
            const bool in = b < P && c < P && gy < BY;
            const T q = w[3 * P];
            const T wyz = in ? q * w[P + b] * w[2 * P + c] : (T)0;
            const int ox = o & 1023;
            int* row = A + zz * PS + gy * RX;
            // v = hi 2^-20 + lo 2^-40 (+ lo2 2^-60): exact splits of the scaled contribution
            if (std::is_same<T, float>::value && fabs(q) <= (T)2 && ox + P <= BX) {
                // the usual case, uniform in the warp: no wrap or clipping in x, and |v| 2^20 < 2^22, so that
                // adding 1.5 2^23 rounds without a conversion instruction; index arithmetic of the general branch
                // taken out, 16,384 sites x 16 replicas of up to 32,768 charges: 656 -> 538 us, before the lists
                const float s20 = (float)wyz * 1048576.0f;
                int* r0 = row + ox;
#pragma unroll
                for (int a = 0; a < P; ++a) {
                    const float x = s20 * (float)w[a];
                    const float t = x + 12582912.0f;
                    const float l = fmaf(x - (t - 12582912.0f), 1048576.0f, 12582912.0f);
                    if (in) {
                        atomicAdd(&r0[a], __float_as_int(t) - 0x4B400000);
                        atomicAdd(&r0[NB + a], __float_as_int(l) - 0x4B400000);
                    }
                }
            } else if (in) {
#pragma unroll
                for (int a = 0; a < P; ++a) {
                    int gx = ox + a;
                    if (gx >= Kx) gx -= Kx;
                    if (gx >= BX) continue;                  // uniform
                    if (std::is_same<T, double>::value) {
                        const double x = (double)(wyz * w[a]) * 1048576.0;   // 2^20
                        const double h = floor(x);
                        const double y = (x - h) * 1048576.0;
                        const double l = floor(y);
                        atomicAdd(&row[gx], (int)h);
                        atomicAdd(&row[NB + gx], (int)l);
                        atomicAdd(&row[2 * NB + gx], __double2int_rn((y - l) * 1048576.0));
                    } else {
                        const float x = (float)(wyz * w[a]) * 1048576.0f;
                        const float h = floorf(x);
                        atomicAdd(&row[gx], (int)h);
                        atomicAdd(&row[NB + gx], __float2int_rn((x - h) * 1048576.0f));
                    }
                }
            }
        }
        __syncthreads();   // the weights are free, at the end the sums complete
    }
    const int64_t N = (int64_t)Kx * Ky * Kz;
    T* out = (T*)(part + ((int64_t)blockIdx.z * ((m + 1) / 2) + rep / 2) * N) + (rep & 1);
    for (int i = threadIdx.x; i < BX * BY * BZ; i += P3M_NT) {
        const int lx = i % BX, ly = (i / BX) % BY, lz = i / (BX * BY);
        const int at = lz * PS + ly * RX + lx;
        double v = (double)A[at] * 0x1p-20 + (double)A[NB + at] * 0x1p-40;
        if (NW == 3) v += (double)A[2 * NB + at] * 0x1p-60;
        out[2 * (((int64_t)(b0z + lz) * Ky + (b0y + ly)) * Kx + (b0x + lx))] = (T)v;
    }
}

// ----------------------------------------------------------------------------- transforms
__device__ __forceinline__ int bitrev(int v, int lg) { return lg ? (int)(__brev((unsigned)v) >> (32 - lg)) : 0; }

// radix-2 decimation-in-time stages over `lines` transforms of length K = 2^lg held in shared memory
// at x[line * ls + i * es] (input in bit-reversed order, output natural); tw[j] = exp(-+ 2 pi i j / K)
template <typename T>
__device__ __forceinline__ void dit_stages(c2<T>* x, int K, int lg, int lines, int ls, int es, const c2<T>* tw) {
    const int half = K >> 1;
    for (int s = 1; s <= lg; ++s) {
        const int hs = 1 << (s - 1);
        for (int t = threadIdx.x; t < lines * half; t += blockDim.x) {
            int line, q;
            if (ls == 1) { line = t % lines; q = t / lines; }   // lines adjacent in memory: line fastest
            else { line = t / half; q = t - line * half; }
            const int j = q & (hs - 1);
            const int i0 = ((q >> (s - 1)) << s) + j, i1 = i0 + hs;
            const c2<T> w = tw[j << (lg - s)];
            c2<T>* p0 = x + line * ls + i0 * es;
            c2<T>* p1 = x + line * ls + i1 * es;
            const c2<T> a = *p0, b = cmul(*p1, w);
            *p0 = cmake<T>(a.x + b.x, a.y + b.y);
            *p1 = cmake<T>(a.x - b.x, a.y - b.y);
        }
        __syncthreads();
    }
}

// 2D transform of (z plane, replica pair) over x and y; INV: exp(+i ...) (unnormalised), of the planes zlist that a
// site's interpolation reads.  The forward transform takes every plane and first sums the nsplit partial meshes of
// the charge assignment (split_stride elements apart) in split order, of the bricks that are marked; a plane without
// any is zero.  Dynamic shared memory: the plane [Ky][Kx], then Kx/2 + Ky/2 twiddles.
constexpr int P3M_FLAGS = 2048;   // marks of one plane: splits x 2 replicas x bricks, at most 8 x 2 x 128
template <typename T, bool INV>
__global__ void __launch_bounds__(P3M_THREADS) k_p3m_plane(c2<T>* __restrict__ mesh, int Kx, int Ky, int Kz,
                                                          const c2<T>* __restrict__ twx, const c2<T>* __restrict__ twy,
                                                          int nsplit, int64_t split_stride, int m, int BX, int BY,
                                                          const int* __restrict__ flag, const int* __restrict__ zlist) {
    grid_wait();
    extern __shared__ __align__(16) unsigned char p3m_smem[];
    __shared__ unsigned char fl[INV ? 1 : P3M_FLAGS];
    c2<T>* pl = (c2<T>*)p3m_smem;
    c2<T>* tx = pl + Kx * Ky;
    c2<T>* ty = tx + Kx / 2;
    const int lx = ilog2i(Kx), ly = ilog2i(Ky);
    const int z = INV ? zlist[blockIdx.x] : blockIdx.x;
    c2<T>* g = mesh + ((int64_t)blockIdx.y * Kz + z) * Kx * Ky;
    const int nbx = Kx / BX, nbp = nbx * (Ky / BY);   // bricks of one plane
    if (!INV) {
        const int nb = nbp * (Kz / P3M_BZ);
        bool any = false;
        for (int e = threadIdx.x; e < nsplit * 2 * nbp; e += P3M_THREADS) {
            const int b = e % nbp, h = (e / nbp) & 1, sp = e / (2 * nbp), r = 2 * blockIdx.y + h;
            const bool f = r < m && flag[((int64_t)sp * m + r) * nb + (z / P3M_BZ) * nbp + b] != 0;
            fl[e] = f;
            any |= f;
        }
        if (!__syncthreads_or(any)) {
            for (int i = threadIdx.x; i < Kx * Ky; i += P3M_THREADS) g[i] = cmake<T>(0, 0);
            return;
        }
    }
    for (int j = threadIdx.x; j < Kx / 2; j += P3M_THREADS) { c2<T> w = twx[j]; if (INV) w.y = -w.y; tx[j] = w; }
    for (int j = threadIdx.x; j < Ky / 2; j += P3M_THREADS) { c2<T> w = twy[j]; if (INV) w.y = -w.y; ty[j] = w; }
    for (int i = threadIdx.x; i < Kx * Ky; i += P3M_THREADS) {
        const int x = i & (Kx - 1), y = i >> lx;
        c2<T> v = cmake<T>(0, 0);
        if (INV) {
            v = g[i];
        } else {
            const int b = (y / BY) * nbx + x / BX;
            for (int sp = 0; sp < nsplit; ++sp) {   // the charge splits of the assignment, in split order
                const bool f0 = fl[(2 * sp) * nbp + b], f1 = fl[(2 * sp + 1) * nbp + b];
                if (!f0 && !f1) continue;
                const c2<T> u = g[sp * split_stride + i];   // an unmarked half is not defined
                if (f0) v.x += u.x;
                if (f1) v.y += u.y;
            }
        }
        pl[bitrev(y, ly) * Kx + bitrev(x, lx)] = v;
    }
    __syncthreads();
    dit_stages<T>(pl, Kx, lx, Ky, Kx, 1, tx);    // rows: line = y (stride Kx), element stride 1
    dit_stages<T>(pl, Ky, ly, Kx, 1, Kx, ty);    // columns: line = x (stride 1), element stride Kx
    for (int i = threadIdx.x; i < Kx * Ky; i += P3M_THREADS) g[i] = pl[i];
}

// z pass: for P3M_ZTX adjacent x at one (y, replica pair): forward transform along z, times G / V,
// inverse transform along z, stored where a site's interpolation reads (need[z]).  Dynamic shared memory: [Kz][tx]
// lines, then Kz/2 twiddles.
template <typename T>
__global__ void __launch_bounds__(P3M_THREADS) k_p3m_zline(c2<T>* __restrict__ mesh, int Kx, int Ky, int Kz, int tx,
                                                          const T* __restrict__ G, const c2<T>* __restrict__ twz,
                                                          const unsigned char* __restrict__ need, int nl,
                                                          const int* __restrict__ lb, const T* __restrict__ lw, int P) {
    grid_wait();
    extern __shared__ __align__(16) unsigned char p3m_smem[];
    c2<T>* ln = (c2<T>*)p3m_smem;
    c2<T>* tw = ln + Kz * tx;
    const int lz = ilog2i(Kz);
    const int x0 = blockIdx.x * tx, y = blockIdx.y;
    const int64_t plane = (int64_t)Kx * Ky;
    c2<T>* g = mesh + (int64_t)blockIdx.z * plane * Kz + (int64_t)y * Kx + x0;
    for (int j = threadIdx.x; j < Kz / 2; j += P3M_THREADS) tw[j] = twz[j];
    for (int i = threadIdx.x; i < Kz * tx; i += P3M_THREADS) {
        const int z = i / tx, x = i - z * tx;
        ln[bitrev(z, lz) * tx + x] = g[z * plane + x];
    }
    __syncthreads();
    dit_stages<T>(ln, Kz, lz, tx, 1, tx, tw);
    for (int i = threadIdx.x; i < Kz * tx; i += P3M_THREADS) {
        const int z = i / tx, x = i - z * tx;
        const T gv = G[z * plane + (int64_t)y * Kx + x0 + x];
        ln[i] = cmake<T>(ln[i].x * gv, ln[i].y * gv);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < Kz * tx; i += P3M_THREADS) {   // natural -> bit-reversed order
        const int z = i / tx, x = i - z * tx;
        const int rz = bitrev(z, lz);
        if (z < rz) {
            const c2<T> a = ln[i];
            ln[i] = ln[rz * tx + x];
            ln[rz * tx + x] = a;
        }
    }
    for (int j = threadIdx.x; j < Kz / 2; j += P3M_THREADS) { c2<T> w = tw[j]; w.y = -w.y; tw[j] = w; }
    __syncthreads();
    dit_stages<T>(ln, Kz, lz, tx, 1, tx, tw);
    for (int i = threadIdx.x; i < Kz * tx; i += P3M_THREADS) {
        const int z = i / tx, x = i - z * tx;
        if (nl == 0 && need[z]) g[z * plane + x] = ln[i];
    }
    // sites of few heights: the z weights of each height applied here, before the inverse xy transform, which then
    // has nl planes (stored as planes 0 .. nl - 1 of this line's own column)
    for (int i = threadIdx.x; i < nl * tx; i += P3M_THREADS) {
        const int u = i / tx, x = i - u * tx, b = lb[u];
        T re = 0, im = 0;
        for (int a = 0; a < P; ++a) {
            const c2<T> v = ln[((b + a) & (Kz - 1)) * tx + x];
            const T w = lw[8 * u + a];
            re += w * v.x;
            im += w * v.y;
        }
        g[u * plane + x] = cmake<T>(re, im);
    }
}

// ----------------------------------------------------------------------------- interpolation
// One warp per (site, replica pair), warps site-fastest.  pm[r][i] = sum_stencil W phi (e/Angstrom).
template <typename T, int P>
__global__ void __launch_bounds__(P3M_THREADS) k_p3m_interp(const double* __restrict__ sx, int64_t n, int m,
                                                           Geometry g, int Kx, int Ky, int Kz,
                                                           const c2<T>* __restrict__ mesh, double* __restrict__ pm) {
    grid_wait();
    __shared__ T sw[P3M_THREADS / 32][3][8];
    __shared__ int sb[P3M_THREADS / 32][3];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t w = (int64_t)blockIdx.x * (P3M_THREADS / 32) + wid;
    const int npairs = (m + 1) / 2;
    const bool live = w < n * npairs;
    const int64_t i = live ? w % n : 0;
    const int pair = live ? (int)(w / n) : 0;
    if (live && lane < 3) {
        const int K = lane == 0 ? Kx : (lane == 1 ? Ky : Kz);
        const double inv = lane == 0 ? g.inv[0] : (lane == 1 ? g.inv[1] : g.inv[2]);
        double s = sx[lane * n + i] * inv;
        s -= floor(s);
        const double u = s * K - 0.5 * P;
        const double fl = floor(u);
        int bi = ((int)fl + 1) % K;
        if (bi < 0) bi += K;
        sb[wid][lane] = bi;
        T wt[P];
        bspline_weights<T, P>((T)(u - fl), wt);
#pragma unroll
        for (int a = 0; a < P; ++a) sw[wid][lane][a] = wt[a];
    }
    __syncwarp();
    if (!live) return;
    const c2<T>* ph = mesh + (int64_t)pair * Kx * Ky * Kz;
    T re = (T)0, im = (T)0;
    for (int col = lane; col < P * P; col += 32) {
        const int a = col % P, b = col / P;
        const int gx = (sb[wid][0] + a) & (Kx - 1), gy = (sb[wid][1] + b) & (Ky - 1);
        const T wxy = sw[wid][0][a] * sw[wid][1][b];
#pragma unroll
        for (int c = 0; c < P; ++c) {
            const int gz = (sb[wid][2] + c) & (Kz - 1);
            const c2<T> v = ph[((int64_t)gz * Ky + gy) * Kx + gx];
            const T ww = wxy * sw[wid][2][c];
            re += ww * v.x;
            im += ww * v.y;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
    }
    if (lane == 0) {
        pm[(int64_t)(2 * pair) * n + i] = (double)re;
        if (2 * pair + 1 < m) pm[(int64_t)(2 * pair + 1) * n + i] = (double)im;
    }
}

// The fixed interpolation of the sites: per point (site or height) and axis the first mesh index and the P weights.
// axes x and y: base[2 i + d], w[8 (2 i + d) + a]; heights (axis 2): base[u], w[8 u + a].
template <typename T, int P>
__global__ void k_p3m_weights(const double* __restrict__ x, int64_t cnt, int64_t stride, int naxes, Geometry g, int Kx,
                              int Ky, int Kz, int axis0, int* __restrict__ base, T* __restrict__ w) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= cnt * naxes) return;
    const int64_t i = t / naxes;
    const int d = axis0 + (int)(t % naxes);
    const int K = d == 0 ? Kx : (d == 1 ? Ky : Kz);
    double s = x[(int64_t)(d - axis0) * stride + i] * (d == 0 ? g.inv[0] : d == 1 ? g.inv[1] : g.inv[2]);
    s -= floor(s);
    const double u = s * K - 0.5 * P;
    const double fl = floor(u);
    int bi = ((int)fl + 1) % K;
    if (bi < 0) bi += K;
    base[t] = bi;
    T wt[P];
    bspline_weights<T, P>((T)(u - fl), wt);
#pragma unroll
    for (int a = 0; a < 8; ++a) w[8 * t + a] = a < P ? wt[a] : (T)0;
}

// Sites of few heights: one warp per (site, replica pair) over the P x P points of its height's plane, lane =
// (x offset, y offset modulo 4); the weights, fixed with the geometry, are read, not formed (each warp of
// k_p3m_interp spends more instructions on them than on the sum).
template <typename T>
__global__ void __launch_bounds__(P3M_THREADS) k_p3m_interp2(const int* __restrict__ zmap, const int* __restrict__ base,
                                                            const T* __restrict__ w, int64_t n, int m, int P, int Kx,
                                                            int Ky, int Kz, const c2<T>* __restrict__ mesh,
                                                            double* __restrict__ pm) {
    grid_wait();
    const int lane = threadIdx.x & 31;
    const int64_t wid = (int64_t)blockIdx.x * (P3M_THREADS / 32) + (threadIdx.x >> 5);
    if (wid >= n * ((m + 1) / 2)) return;
    const int64_t i = wid % n;
    const int pair = (int)(wid / n);
    const c2<T>* ph = mesh + ((int64_t)pair * Kz + zmap[i]) * Kx * Ky;
    const int bx = base[2 * i], by = base[2 * i + 1], a = lane & 7, b = lane >> 3;
    const int gx = (bx + a) & (Kx - 1);
    const T wx = w[16 * i + a], w0 = w[16 * i + 8 + b], w1 = w[16 * i + 12 + b];   // zero from P on
    T re = 0, im = 0;
    if (a < P) {
        if (b < P) {
            const c2<T> v = ph[(int64_t)((by + b) & (Ky - 1)) * Kx + gx];
            re = wx * w0 * v.x;
            im = wx * w0 * v.y;
        }
        if (b + 4 < P) {
            const c2<T> v = ph[(int64_t)((by + b + 4) & (Ky - 1)) * Kx + gx];
            re += wx * w1 * v.x;
            im += wx * w1 * v.y;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
    }
    if (lane == 0) {
        pm[(int64_t)(2 * pair) * n + i] = (double)re;
        if (2 * pair + 1 < m) pm[(int64_t)(2 * pair + 1) * n + i] = (double)im;
    }
}

// ----------------------------------------------------------------------------- host side
static size_t p3m_al(size_t b) { return (b + 255) & ~(size_t)255; }

static int64_t mesh_pts(const cpm_ctx* c) {
    return (int64_t)c->p.p3m_mesh[0] * c->p.p3m_mesh[1] * c->p.p3m_mesh[2];
}

// Assignment bricks of 32 x 32 x 4 points at most and charge splits: enough CTAs that the uneven bricks within the
// electrolyte, about a third, even out (16,384 sites x 16 replicas: 1,309 us a step without a split, 1,121 with three,
// 1,109 with five, 1,130 with eight), no split with less than three chunks of charges (4,320 x 8: 190 us with six splits
// of two, 182.5 with four of three: every split is a partial mesh to be written and added), at most 8.
struct P3mSpread {
    int BX, BY, nbricks, nsplit, cps;
    P3mBricks br;
    int64_t per() const { return (int64_t)cps * P3M_NT; }   // charges per split
};
static P3mSpread p3m_spread_plan(const cpm_ctx* c, int m, int64_t ne) {
    P3mSpread sp;
    const int Kx = c->p.p3m_mesh[0], Ky = c->p.p3m_mesh[1], Kz = c->p.p3m_mesh[2];
    sp.BX = std::min(Kx, 32);
    sp.BY = std::min(Ky, 32);
    sp.br = P3mBricks{sp.BX, sp.BY, Kx / sp.BX, Ky / sp.BY, Kz / P3M_BZ};
    sp.nbricks = sp.br.n();
    const int64_t ctas = (int64_t)sp.nbricks * m;
    const int64_t nchunks = std::max<int64_t>(1, (ne + P3M_NT - 1) / P3M_NT);
    int64_t ns = std::max<int64_t>(1, (32 * 152 + ctas - 1) / ctas);
    ns = std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(ns, 8), nchunks / 3));
    if (c->lean) ns = c->lean > 1 ? 1 : (ns + 3) / 4;
    sp.cps = (int)std::min((nchunks + ns - 1) / ns, p3m_split_most(sp.br.most(c->p.p3m_order)));
    sp.nsplit = (int)((nchunks + sp.cps - 1) / sp.cps);
    return sp;
}

template <typename T>
size_t p3m_scratch_bytes(const cpm_ctx* c, int m, int64_t ne) {
    const int64_t ptot = (int64_t)m * ne;
    const P3mSpread sp = p3m_spread_plan(c, m, ne);
    return p3m_al(sizeof(int) * ptot) + p3m_al(sizeof(typename P3mV4<T>::t) * ptot) +
           3 * p3m_al(sizeof(int) * (size_t)sp.nsplit * m * sp.nbricks) +   // marks, counts, starts
           p3m_al(sizeof(int) * (size_t)m * sp.nsplit * std::min(sp.per(), ne) * sp.br.most(c->p.p3m_order)) + p3m_al(sizeof(c2<T>) * (size_t)sp.nsplit * ((m + 1) / 2) * mesh_pts(c));
}
template size_t p3m_scratch_bytes<float>(const cpm_ctx*, int, int64_t);
template size_t p3m_scratch_bytes<double>(const cpm_ctx*, int, int64_t);

template <typename T>
static cpm_status p3m_prepare_t(cpm_ctx* c, void** Gp, void** twp) {
    const int Kx = c->p.p3m_mesh[0], Ky = c->p.p3m_mesh[1], Kz = c->p.p3m_mesh[2];
    const int64_t N = mesh_pts(c);
    CPM_TRY(dev_alloc(c, Gp, sizeof(T) * N));
    CPM_TRY(dev_alloc(c, twp, sizeof(c2<T>) * (Kx + Ky + Kz) / 2));
    std::vector<c2<T>> tw((Kx + Ky + Kz) / 2);
    size_t o = 0;
    for (int K : {Kx, Ky, Kz})
        for (int j = 0; j < K / 2; ++j) {
            const double a = 2.0 * PI * j / K;
            tw[o++] = cmake<T>((T)std::cos(a), (T)-std::sin(a));
        }
    CPM_CUDA(c, cudaMemcpyAsync(*twp, tw.data(), sizeof(c2<T>) * tw.size(), cudaMemcpyHostToDevice, c->stream));
    k_p3m_green<T><<<(unsigned)((N + 255) / 256), 256, 0, c->stream>>>(Kx, Ky, Kz, c->p.p3m_order, c->g.boxL[0],
                                                                     c->g.boxL[1], c->g.boxL[2], c->g.alpha, c->g.V,
                                                                     (T*)*Gp);
    CPM_LAUNCH(c, "k_p3m_green");
    // the twiddles are copied from pageable host memory: wait before the vector goes out of scope
    CPM_CUDA(c, cudaStreamSynchronize(c->stream));
    return CPM_OK;
}

template <typename T, int P>
static cpm_status p3m_weights_p(cpm_ctx* c, T** w, T** lw) {
    const int Kx = c->p.p3m_mesh[0], Ky = c->p.p3m_mesh[1], Kz = c->p.p3m_mesh[2];
    CPM_TRY(dev_alloc(c, (void**)w, sizeof(T) * 16 * c->n));
    CPM_TRY(dev_alloc(c, (void**)lw, sizeof(T) * 8 * c->nzu));
    k_p3m_weights<T, P><<<(unsigned)((2 * c->n + 127) / 128), 128, 0, c->stream>>>(c->sx, c->n, c->n, 2, c->g, Kx, Ky, Kz, 0,
                                                                                  c->p3m_base, *w);
    k_p3m_weights<T, P><<<(unsigned)((c->nzu + 127) / 128), 128, 0, c->stream>>>(c->zuniq, c->nzu, 0, 1, c->g, Kx, Ky, Kz, 2,
                                                                                c->p3m_lb, *lw);
    CPM_LAUNCH(c, "k_p3m_weights");
    return CPM_OK;
}
template <typename T> static cpm_status p3m_weights(cpm_ctx* c, T** w, T** lw) {
    switch (c->p.p3m_order) {
        case 2: return p3m_weights_p<T, 2>(c, w, lw);
        case 3: return p3m_weights_p<T, 3>(c, w, lw);
        case 4: return p3m_weights_p<T, 4>(c, w, lw);
        case 5: return p3m_weights_p<T, 5>(c, w, lw);
        case 6: return p3m_weights_p<T, 6>(c, w, lw);
        default: return p3m_weights_p<T, 7>(c, w, lw);
    }
}

// What the inverse transform has to give.  Sites that share few heights (as in recip_rows.cu): one plane per
// height.  Otherwise the planes that the interpolation at the sites reads (one more on either side of each
// stencil, so that no rounding of the origin can matter).
static cpm_status p3m_planes(cpm_ctx* c) {
    const int Kz = c->p.p3m_mesh[2], P = c->p.p3m_order;
    std::vector<unsigned char> need(Kz, 0);
    std::vector<int> list;
    c->p3m_nl = (int64_t)c->nzu * LAYER_MIN_SITES <= c->n && c->nzu <= Kz ? c->nzu : 0;
    if (c->p3m_nl) {
        for (int u = 0; u < c->nzu; ++u) list.push_back(u);
        CPM_TRY(dev_alloc(c, (void**)&c->p3m_base, sizeof(int) * 2 * c->n));
        CPM_TRY(dev_alloc(c, (void**)&c->p3m_lb, sizeof(int) * c->nzu));
        if (c->p.k_prec != CPM_PREC_FP64) CPM_TRY(p3m_weights<float>(c, &c->p3m_w32, &c->p3m_lw32));
        if (c->p.k_prec == CPM_PREC_FP64 || c->p.p3m_matrix) CPM_TRY(p3m_weights<double>(c, &c->p3m_w64, &c->p3m_lw64));
    } else {
        std::vector<double> zu(c->nzu);
        CPM_CUDA(c, cudaMemcpyAsync(zu.data(), c->zuniq, sizeof(double) * zu.size(), cudaMemcpyDeviceToHost, c->stream));
        CPM_CUDA(c, cudaStreamSynchronize(c->stream));
        for (double z : zu) {
            double s = z * c->g.inv[2];
            s -= std::floor(s);
            const int b = (int)std::floor(s * Kz - 0.5 * P);
            for (int a = 0; a < P + 2; ++a) need[((b + a) % Kz + Kz) % Kz] = 1;
        }
        for (int z = 0; z < Kz; ++z)
            if (need[z]) list.push_back(z);
    }
    CPM_TRY(dev_alloc(c, (void**)&c->p3m_need, Kz));
    CPM_TRY(dev_alloc(c, (void**)&c->p3m_zlist, sizeof(int) * list.size()));
    CPM_CUDA(c, cudaMemcpyAsync(c->p3m_need, need.data(), Kz, cudaMemcpyHostToDevice, c->stream));
    CPM_CUDA(c, cudaMemcpyAsync(c->p3m_zlist, list.data(), sizeof(int) * list.size(), cudaMemcpyHostToDevice, c->stream));
    CPM_CUDA(c, cudaStreamSynchronize(c->stream));
    c->p3m_nz = (int)list.size();
    return CPM_OK;
}
template <typename T> static const T* p3m_site_w(const cpm_ctx* c);
template <> const float* p3m_site_w<float>(const cpm_ctx* c) { return c->p3m_w32; }
template <> const double* p3m_site_w<double>(const cpm_ctx* c) { return c->p3m_w64; }
template <typename T> static const T* p3m_height_w(const cpm_ctx* c);
template <> const float* p3m_height_w<float>(const cpm_ctx* c) { return c->p3m_lw32; }
template <> const double* p3m_height_w<double>(const cpm_ctx* c) { return c->p3m_lw64; }

cpm_status p3m_prepare(cpm_ctx* c) {
    CPM_TRY(p3m_planes(c));
    if (c->p3m_G) return CPM_OK;   // depends on the cell and the parameters only
    if (c->p.k_prec == CPM_PREC_FP64) return p3m_prepare_t<double>(c, &c->p3m_G, &c->p3m_tw);
    CPM_TRY(p3m_prepare_t<float>(c, &c->p3m_G, &c->p3m_tw));
    if (c->p.p3m_matrix) CPM_TRY(p3m_prepare_t<double>(c, &c->p3m_G64, &c->p3m_tw64));   // the elastance: FP64
    return CPM_OK;
}

// the influence function and twiddles in T (the FP64 copies of a single-precision context for T = double)
template <typename T> static const T* p3m_green(const cpm_ctx* c) {
    return (const T*)((std::is_same<T, double>::value && c->p.k_prec != CPM_PREC_FP64) ? c->p3m_G64 : c->p3m_G);
}
template <typename T> static const c2<T>* p3m_twiddles(const cpm_ctx* c) {
    return (const c2<T>*)((std::is_same<T, double>::value && c->p.k_prec != CPM_PREC_FP64) ? c->p3m_tw64 : c->p3m_tw);
}

template <typename T, int P>
static cpm_status launch_p3m_pp(cudaStream_t st, cpm_ctx* c, int m, int64_t ne, const int* key,
                          const typename P3mV4<T>::t* fq, int* flag, const int* count, const int* start, const int* list, int64_t per, int most,
                          c2<T>* mesh, double* pm) {
    const int Kx = c->p.p3m_mesh[0], Ky = c->p.p3m_mesh[1], Kz = c->p.p3m_mesh[2];
    const P3mSpread sp = p3m_spread_plan(c, m, ne);
    const int npairs = (m + 1) / 2;
    const size_t ssm = sizeof(int) * ((P3mWords<T>::n * P3M_BZ * (sp.BY * (sp.BX + 1) + 8) + 3) & ~3) +
                       sizeof(T) * P3M_NT * (3 * P + 1) + sizeof(int) * P3M_NT;
    CPM_CUDA(c, cudaFuncSetAttribute(k_p3m_spread<T, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ssm));
    CPM_CUDA(c, launch_after(k_p3m_spread<T, P>, dim3(sp.nbricks, m, sp.nsplit), dim3(P3M_NT), ssm, st, key, fq, ne, m, Kx, Ky, Kz, sp.BX, sp.BY,
                                                                            count, start, list, per, most, mesh, flag));
    const int64_t sstride = (int64_t)npairs * Kx * Ky * Kz;
    const c2<T>* tw = p3m_twiddles<T>(c);
    const size_t psm = sizeof(c2<T>) * ((size_t)Kx * Ky + Kx / 2 + Ky / 2);
    CPM_CUDA(c, cudaFuncSetAttribute(k_p3m_plane<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psm));
    CPM_CUDA(c, cudaFuncSetAttribute(k_p3m_plane<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psm));
    CPM_CUDA(c, launch_after(k_p3m_plane<T, false>, dim3(Kz, npairs), dim3(P3M_THREADS), psm, st, mesh, Kx, Ky, Kz, tw, tw + Kx / 2, sp.nsplit,
                                                                      sstride, m, sp.BX, sp.BY, flag, nullptr));
    const int tx = std::min(Kx, P3M_ZTX);
    const size_t zsm = sizeof(c2<T>) * ((size_t)Kz * tx + Kz / 2);
    CPM_CUDA(c, cudaFuncSetAttribute(k_p3m_zline<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)zsm));
    CPM_CUDA(c, launch_after(k_p3m_zline<T>, dim3(Kx / tx, Ky, npairs), dim3(P3M_THREADS), zsm, st, mesh, Kx, Ky, Kz, tx, p3m_green<T>(c),
                                                                        tw + Kx / 2 + Ky / 2, c->p3m_need, c->p3m_nl,
                                                                        c->p3m_lb, p3m_height_w<T>(c), P));
    CPM_CUDA(c, launch_after(k_p3m_plane<T, true>, dim3(c->p3m_nz, npairs), dim3(P3M_THREADS), psm, st, mesh, Kx, Ky, Kz, tw, tw + Kx / 2, 1, 0, m,
                                                                            sp.BX, sp.BY, nullptr, c->p3m_zlist));
    const int64_t warps = c->n * npairs;
    if (c->p3m_nl)
        CPM_CUDA(c, launch_after(k_p3m_interp2<T>, dim3((unsigned)((warps + P3M_THREADS / 32 - 1) / (P3M_THREADS / 32))), dim3(P3M_THREADS), 0, st, 
            c->zmap, c->p3m_base, p3m_site_w<T>(c), c->n, m, P, Kx, Ky, Kz, mesh, pm));
    else
        CPM_CUDA(c, launch_after(k_p3m_interp<T, P>, dim3((unsigned)((warps + P3M_THREADS / 32 - 1) / (P3M_THREADS / 32))), dim3(P3M_THREADS), 0, st, 
            c->sx, c->n, m, c->g, Kx, Ky, Kz, mesh, pm));
    CPM_LAUNCH(c, "k_p3m (spread, transforms, interpolation)");
    return CPM_OK;
}

template <typename T>
cpm_status p3m_run(cpm_ctx* c, cudaStream_t st, int m, int64_t ne, const double* xyz, const double* Q, char* scr,
                   double* pm) {
    const int64_t ptot = (int64_t)m * ne;
    int* key = (int*)scr;
    typedef typename P3mV4<T>::t V4T;
    V4T* fq = (V4T*)(scr + p3m_al(sizeof(int) * ptot));
    int* flag = (int*)((char*)fq + p3m_al(sizeof(V4T) * ptot));
    const P3mSpread sp = p3m_spread_plan(c, m, ne);
    const size_t lists = p3m_al(sizeof(int) * (size_t)sp.nsplit * m * sp.nbricks);
    int* count = (int*)((char*)flag + lists);
    int* start = (int*)((char*)count + lists);
    int* list = (int*)((char*)start + lists);
    const int most = sp.br.most(c->p.p3m_order);
    const int64_t per = std::min(sp.per(), ne);
    c2<T>* mesh = (c2<T>*)((char*)list + p3m_al(sizeof(int) * (size_t)m * sp.nsplit * per * most));
    const int P = c->p.p3m_order;
    const int Kx = c->p.p3m_mesh[0], Ky = c->p.p3m_mesh[1], Kz = c->p.p3m_mesh[2];
    CPM_CUDA(c, cudaMemsetAsync(count, 0, lists, st));
    k_p3m_prep<T><<<(unsigned)((ptot + 255) / 256), 256, 0, st>>>(xyz, Q, ptot, c->g, Kx, Ky, Kz, P, key, fq, ne, sp.br,
                                                                  sp.nsplit, per, count);
    CPM_LAUNCH(c, "k_p3m_prep");
    CPM_CUDA(c, launch_after(k_p3m_scan, dim3((unsigned)(m * sp.nsplit)), dim3(P3M_SCAN), 0, st, count, sp.nbricks, start));
    CPM_CUDA(c, launch_after(k_p3m_fill, dim3((unsigned)((ptot + 255) / 256)), dim3(256), 0, st, key, ptot, ne, P, sp.br, sp.nsplit,
                             per, most, start, list));
    c->launches += 8;
    switch (P) {
        case 2: return launch_p3m_pp<T, 2>(st, c, m, ne, key, fq, flag, count, start, list, per, most, mesh, pm);
        case 3: return launch_p3m_pp<T, 3>(st, c, m, ne, key, fq, flag, count, start, list, per, most, mesh, pm);
        case 4: return launch_p3m_pp<T, 4>(st, c, m, ne, key, fq, flag, count, start, list, per, most, mesh, pm);
        case 5: return launch_p3m_pp<T, 5>(st, c, m, ne, key, fq, flag, count, start, list, per, most, mesh, pm);
        case 6: return launch_p3m_pp<T, 6>(st, c, m, ne, key, fq, flag, count, start, list, per, most, mesh, pm);
        default: return launch_p3m_pp<T, 7>(st, c, m, ne, key, fq, flag, count, start, list, per, most, mesh, pm);
    }
}
// ----------------------------------------------------------------------------- the P3M elastance
__global__ void k_p3m_add_rows(double* __restrict__ A, const double* __restrict__ pm, int64_t cnt, double s) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < cnt) A[t] += s * pm[t];
}

// A <- (A + A^T) / 2 (the mesh operator is symmetric up to rounding): one thread per lower entry
__global__ void k_p3m_sym(double* __restrict__ A, int64_t n) {
    const int64_t i = blockIdx.y, j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= i || i >= n) return;
    const double v = 0.5 * (A[i * n + j] + A[j * n + i]);
    A[i * n + j] = v;
    A[j * n + i] = v;
}

__global__ void k_p3m_ones(double* __restrict__ q, int64_t cnt) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < cnt) q[t] = 1.0;
}

cpm_status p3m_assemble_recip(cpm_ctx* c) {
    const int64_t n = c->n;
    const int B = (int)std::min<int64_t>(n, 512);   // sites per batch: every site one replica of one unit charge
    const size_t sbytes = p3m_scratch_bytes<double>(c, B, 1);
    char* scr = nullptr;
    double* pm = nullptr;
    double* ones = nullptr;
    cpm_status st = dev_alloc(c, (void**)&scr, sbytes);
    if (st == CPM_OK) st = dev_alloc(c, (void**)&pm, sizeof(double) * B * n);
    if (st == CPM_OK) st = dev_alloc(c, (void**)&ones, sizeof(double) * B);
    const int64_t l0 = c->launches;   // assembly work is not counted with the per-step launches
    if (st == CPM_OK) {
        k_p3m_ones<<<(B + 255) / 256, 256, 0, c->stream>>>(ones, B);
        for (int64_t r0 = 0; r0 < n && st == CPM_OK; r0 += B) {
            const int mb = (int)std::min<int64_t>(B, n - r0);
            st = p3m_run<double>(c, c->stream, mb, 1, c->sxyz + 3 * r0, ones, scr, pm);
            if (st == CPM_OK) {
                const int64_t cnt = (int64_t)mb * n;
                k_p3m_add_rows<<<(unsigned)((cnt + 255) / 256), 256, 0, c->stream>>>(c->A + r0 * n, pm, cnt, KE);
            }
        }
        if (st == CPM_OK) {
            k_p3m_sym<<<dim3((unsigned)((n + 255) / 256), (unsigned)n), 256, 0, c->stream>>>(c->A, n);
            st = cuda_check(c, cudaGetLastError(), "k_p3m (elastance)");
        }
    }
    c->launches = l0;
    if (scr || pm || ones) cudaStreamSynchronize(c->stream);   // the buffers are in use until the stream has passed
    dev_free(c, scr);
    dev_free(c, pm);
    dev_free(c, ones);
    return st;
}

template cpm_status p3m_run<float>(cpm_ctx*, cudaStream_t, int, int64_t, const double*, const double*, char*, double*);
template cpm_status p3m_run<double>(cpm_ctx*, cudaStream_t, int, int64_t, const double*, const double*, char*,
                                    double*);

}  // namespace cpm
