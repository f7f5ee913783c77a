// Reciprocal-space part of b in the real product basis of an orthorhombic cell.
//
// The Ewald weights do not change when the sign of one component of k does, so the half-space sum over
// (+-nx, +-ny, +-nz) of one octant vector collapses to products of cosines,
//   sum_signs w cos(k.d) = W cos(kx dx) cos(ky dy) cos(kz dz),
//   W = w (2 if nx, ny > 0) (2 if nz > 0 and (nx, ny) != 0)   (w the half-space weight),
// and each cosine of a difference is cos cos + sin sin.  With pair p = (nx, ny), nx, ny >= 0, and
// part t = (x function) + 2 (y function), functions {cos, sin}:
//   stage 1  R_r[p][t][c]   = sum_j Q_j f_t(x_j, y_j) h_c(z_j),  c = 2 nz + {0: cos kz z, 1: sin kz z}
//   stage 2  T_r[u][p][t]   = sum_c W[p][nz_c] R_r[p][t][c] h_c(z_u)      for every distinct site height z_u
//   stage 3  b_r[i]        += sum_p sum_t f_t(x_i, y_i) T_r[u_i][p][t]
// Stage 1 takes two real multiply-adds per (charge, k) where complex products of columns and harmonics
// over both signs took four.  Electrodes are stacks of lattice planes, so few distinct heights u carry all
// sites: stage 2 sums the harmonics once per height instead of once per site, and stage 3 is left with
// one term per (site, pair, part) instead of one per (site, k).  Electrodes whose sites hardly share
// heights (rows_by_height) take the general site stage of bvec.cu or tc_recip.cu, whose operand w rho over signed columns k_rows_to_cols forms from R.
#include <cstring>
#include <vector>

#include "common.cuh"

namespace cpm {

// ----------------------------------------------------------------------------- tables
__device__ __forceinline__ uint64_t row_frac(double x, double invL) {
    double s = x * invL;
    s -= floor(s);
    const double t = s * 18446744073709551616.0;   // 2^64
    return t >= 18446744073709551616.0 ? 0ull : (uint64_t)t;
}

// exp(2 pi i h f) from the 64-bit fixed-point fraction f, h f reduced exactly (mod one turn)
template <typename T> __device__ __forceinline__ c2<T> row_phase(uint64_t u, int h);
template <> __device__ __forceinline__ double2 row_phase<double>(uint64_t u, int h) {
    double s, c;
    sincospi((double)(int64_t)(u * (uint64_t)(int64_t)h) * 0x1p-63, &s, &c);
    return make_double2(c, s);
}
template <> __device__ __forceinline__ float2 row_phase<float>(uint64_t u, int h) {
    float s, c;
    sincospif((float)(int32_t)(uint32_t)((u * (uint64_t)(int64_t)h) >> 32) * 0x1p-31f, &s, &c);
    return make_float2(c, s);
}

// W[p][nz], nz = 0..NZ, from the half-space weights of the column (nx, ny) (col = its index)
__global__ void k_pair_weights(const int4* __restrict__ pairs, const int* __restrict__ col, int np, int NZ,
                               const double* __restrict__ w, const float* __restrict__ w32, double* __restrict__ W,
                               float* __restrict__ W32) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= np * (NZ + 1)) return;
    const int p = t / (NZ + 1), nz = t % (NZ + 1);
    const int4 pr = pairs[p];
    const int64_t e = (int64_t)col[p] * (2 * NZ + 1) + NZ + nz;
    const double f = (pr.x > 0 && pr.y > 0 ? 2.0 : 1.0) * (nz > 0 && (pr.x > 0 || pr.y > 0) ? 2.0 : 1.0);
    W[t] = f * w[e];
    W32[t] = (float)f * w32[e];
}

// h_c of the distinct site heights: ZU[nz][u] = (cos, sin)(2 pi nz z_u / Lz)
template <typename T>
__global__ void k_layer_phases(const double* __restrict__ zu, int nzu, double iz, int NZ, c2<T>* __restrict__ ZU) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nzu * (NZ + 1)) return;
    ZU[t] = row_phase<T>(row_frac(zu[t % nzu], iz), t / nzu);
}

constexpr int FX_TAB = 1024;   // entries of each of the two tables of the fixed-point phases
static cpm_status charge_fixed_table(cpm_ctx* c);

// The tables of a geometry in one allocation, those formed on the host copied at once: with an allocation, a copy and a
// free each, some fifteen of them, a preparation took 50 to 100 us more (216 sites: FP64 936 us, now 859; FP32 822 and 773;
// F16X2 828 and 771).
class RowBlob {
    struct Part { void** ptr; size_t at; };
    std::vector<Part> parts;
    std::vector<char> host;
    size_t total = 0;
    static size_t al(size_t b) { return (b + 255) & ~(size_t)255; }

public:
    template <typename V> void put(V** d, const std::vector<V>& h) {   // before the first room()
        parts.push_back({(void**)d, total});
        host.resize(al(total + sizeof(V) * std::max<size_t>(1, h.size())));
        if (!h.empty()) memcpy(&host[total], h.data(), sizeof(V) * h.size());
        total = host.size();
    }
    template <typename V> void room(V** d, size_t count) {
        parts.push_back({(void**)d, total});
        total = al(total + sizeof(V) * std::max<size_t>(1, count));
    }
    // the copy is done when the stream is: the blob lives until then
    cpm_status place(cpm_ctx* c, char** base) {
        CPM_TRY(dev_alloc(c, (void**)base, total));
        for (const Part& p : parts) *p.ptr = *base + p.at;
        CPM_CUDA(c, cudaMemcpyAsync(*base, host.data(), host.size(), cudaMemcpyHostToDevice, c->stream));
        return CPM_OK;
    }
};

void free_rows(cpm_ctx* c) {
    RowTable& t = c->rows;
    dev_free(c, t.blob);
    t = RowTable{};
}

// After build_ktable and the site heights (zuniq, zmap): the pairs in the order of |k_perp| with their
// harmonic extents, their weights, the height tables and the site tiles of stage 3.
cpm_status build_rows(cpm_ctx* c) {
    free_rows(c);
    RowTable& t = c->rows;
    const KTable& k = c->kt;
    if (k.nk == 0) return CPM_OK;
    const int64_t n = c->n;
    RowBlob blob;
    std::vector<int2> cols(k.ncols);
    std::vector<int> ext(k.ncols), zm(n);
    CPM_CUDA(c, cudaMemcpyAsync(cols.data(), k.cols, sizeof(int2) * k.ncols, cudaMemcpyDeviceToHost, c->stream));
    CPM_CUDA(c, cudaMemcpyAsync(ext.data(), k.colext, sizeof(int) * k.ncols, cudaMemcpyDeviceToHost, c->stream));
    CPM_CUDA(c, cudaMemcpyAsync(zm.data(), c->zmap, sizeof(int) * n, cudaMemcpyDeviceToHost, c->stream));
    CPM_CUDA(c, cudaStreamSynchronize(c->stream));
    // (0, 0) alone can be without a harmonic; its weights are then zero
    std::vector<int> ymax(k.NX + 1, -1), off(k.NX + 2, 0);
    for (int q = 0; q < k.ncols; ++q)   // nx >= 0 in every column
        if (cols[q].y >= 0) ymax[cols[q].x] = std::max(ymax[cols[q].x], cols[q].y);
    for (int x = 0; x <= k.NX; ++x) off[x + 1] = off[x] + ymax[x] + 1;
    t.nslots = off[k.NX + 1];
    std::vector<int4> pairs;
    std::vector<int> col, list, slotpair(t.nslots, 0), order;
    for (int q = 0; q < k.ncols; ++q)
        if (cols[q].y >= 0) order.push_back(q);
    // The order of |k_perp| keeps pairs of like extents together.  The tensor-core stage takes 64 pairs per CTA
    // and stages every nx and ny between their smallest and largest: where that is more than it has room for,
    // the pairs go by nx or by ny instead (thin slices of the disc).
    std::vector<int4> titem, trange;
    auto plan_items = [&](const std::vector<int>& ord) {
        titem.clear();
        trange.clear();
        for (size_t f = 0; f < ord.size(); f += ROW_TC_PAIRS) {
            const size_t e = std::min(ord.size(), f + ROW_TC_PAIRS);
            int x0 = k.NX, x1 = 0, y0 = k.NY, y1 = 0, mx = 0;
            for (size_t q = f; q < e; ++q) {
                const int2 cc = cols[ord[q]];
                x0 = std::min(x0, cc.x); x1 = std::max(x1, cc.x);
                y0 = std::min(y0, cc.y); y1 = std::max(y1, cc.y);
                mx = std::max(mx, ext[ord[q]]);
            }
            if (x1 - x0 + 1 + y1 - y0 + 1 > ROW_TC_SLOTS) return false;
            for (int z = 0; z <= mx; z += 64) {
                titem.push_back(make_int4((int)f, (int)(e - f), z / 64, std::min(64, mx + 1 - z)));
                trange.push_back(make_int4(x0, x1 - x0 + 1, y0, y1 - y0 + 1));
            }
        }
        return true;
    };
    if (c->p.k_prec == CPM_PREC_F16X2) {
        std::vector<int> byx = order, byy = order;
        std::stable_sort(byx.begin(), byx.end(), [&](int a, int b) { return cols[a].x < cols[b].x; });
        std::stable_sort(byy.begin(), byy.end(), [&](int a, int b) { return cols[a].y < cols[b].y; });
        bool ok = plan_items(order);
        for (const auto* o : {&byx, &byy})
            if (!ok && (ok = plan_items(*o))) order = *o;
        if (ok) {
            t.tcitems = (int)titem.size();
            blob.put(&t.tcitem, titem);
            blob.put(&t.tcrange, trange);
        }
    }
    for (int q : order) {
        const int p = (int)pairs.size();
        pairs.push_back(make_int4(cols[q].x, cols[q].y, std::max(ext[q], 0), off[cols[q].x] + cols[q].y));
        col.push_back(q);
        slotpair[pairs[p].w] = p;
        for (int part = 0; part < 4; ++part)   // sin 0 = 0: no row
            if (!((part & 1) && cols[q].x == 0) && !((part & 2) && cols[q].y == 0)) list.push_back(4 * p + part);
    }
    std::vector<int2> pcols(pairs.size());   // the signed columns (nx, ny) and (nx, -ny) of every pair
    for (size_t p = 0; p < pairs.size(); ++p) pcols[p] = make_int2(col[p], -1);
    for (int q = 0; q < k.ncols; ++q)
        if (cols[q].y < 0) pcols[slotpair[off[cols[q].x] - cols[q].y]].y = q;
    if (c->p.k_prec == CPM_PREC_FP64) {
        std::vector<int4> i64;
        for (size_t f = 0; f < pairs.size(); f += ROW64_PAIRS) {
            const size_t e = std::min(pairs.size(), f + ROW64_PAIRS);
            int mx = 0;
            for (size_t q = f; q < e; ++q) mx = std::max(mx, pairs[q].z);
            for (int z = 0; z <= mx; z += ROW64_HARM)
                i64.push_back(make_int4((int)f, (int)(e - f), z, std::min(ROW64_HARM, mx + 1 - z)));
        }
        t.items64 = (int)i64.size();
        blob.put(&t.item64, i64);
    }
    t.np = (int)pairs.size();
    t.nrows = (int)list.size();
    t.hext.resize(t.np);
    for (int p = 0; p < t.np; ++p) t.hext[p] = pairs[p].z;
    t.hlist = list;
    // stage 3 splits the nx range into about equal numbers of pairs, 16 or more each: a thread waits for the
    // loads of one pair after the other (113 pairs in a row took 50 us on the co-axial tubes), and the
    // partial sums are added in FP64
    int last = 0;
    for (int x = 0; x <= k.NX; ++x)
        if (ymax[x] >= 0) last = x + 1;
    t.nchunk = std::max(1, std::min(std::min(last, 32), (t.nslots + 15) / 16));
    std::vector<int> cb(t.nchunk + 1, last);
    for (int q = 0, x = 0; q < t.nchunk; ++q) {
        cb[q] = x;
        while (x < last && off[x + 1] <= (int64_t)t.nslots * (q + 1) / t.nchunk) ++x;
    }
    cb[0] = 0;
    cb[t.nchunk] = last;
    t.chunkmax = 0;
    for (int q = 0; q < t.nchunk; ++q) t.chunkmax = std::max(t.chunkmax, off[cb[q + 1]] - off[cb[q]]);
    // the four weighted rows of a pair (stage 2) and the coefficients of a chunk (stage 3) must fit in shared memory
    t.layered = (int64_t)c->nzu * LAYER_MIN_SITES <= n && (size_t)(k.NZ + 1) * 64 <= 200 * 1024 &&
                (size_t)t.chunkmax * 128 <= 200 * 1024;
    if (t.layered) {
        std::vector<int> perm(n), cnt(c->nzu + 1, 0);
        for (int64_t i = 0; i < n; ++i) ++cnt[zm[i] + 1];
        for (int u = 0; u < c->nzu; ++u) cnt[u + 1] += cnt[u];
        std::vector<int> at(cnt.begin(), cnt.end() - 1);
        for (int64_t i = 0; i < n; ++i) perm[at[zm[i]]++] = (int)i;
        std::vector<int4> tiles;
        for (int u = 0; u < c->nzu; ++u)
            for (int f = cnt[u]; f < cnt[u + 1]; f += ROW_TILE)
                tiles.push_back(make_int4(u, f, std::min(ROW_TILE, cnt[u + 1] - f), 0));
        t.ntiles = (int)tiles.size();
        for (int u = 0; u < c->nzu; ++u)
            for (int f = cnt[u]; f < cnt[u + 1]; f += 64) t.hatiles.push_back(make_int4(u, f, std::min(64, cnt[u + 1] - f), 0));
        blob.put(&t.atiles, t.hatiles);
        blob.put(&t.lperm, perm);
        blob.put(&t.ltiles, tiles);
    }
    int* dcol = nullptr;
    blob.put(&t.pairs, pairs);
    blob.put(&t.list, list);
    blob.put(&t.nxoff, off);
    blob.put(&t.paircols, pcols);
    blob.put(&t.chunkb, cb);
    blob.put(&dcol, col);
    const size_t nw = (size_t)t.np * (k.NZ + 1), nu = (size_t)c->nzu * (k.NZ + 1);
    blob.room(&t.W, nw);
    blob.room(&t.W32, nw);
    if (t.layered) {
        blob.room(&t.zu64, nu);
        blob.room(&t.zu32, nu);
    }
    if (c->p.k_prec == CPM_PREC_FP64) blob.room(&t.fxtab, 2 * FX_TAB);
    CPM_TRY(blob.place(c, &t.blob));
    if (c->p.k_prec == CPM_PREC_FP64) CPM_TRY(charge_fixed_table(c));
    k_pair_weights<<<(unsigned)((nw + 255) / 256), 256, 0, c->stream>>>(t.pairs, dcol, t.np, k.NZ, k.w, k.w32, t.W, t.W32);
    CPM_LAUNCH(c, "k_pair_weights");
    if (t.layered) {
        k_layer_phases<double><<<(unsigned)((nu + 255) / 256), 256, 0, c->stream>>>(c->zuniq, c->nzu, c->g.inv[2], k.NZ, t.zu64);
        k_layer_phases<float><<<(unsigned)((nu + 255) / 256), 256, 0, c->stream>>>(c->zuniq, c->nzu, c->g.inv[2], k.NZ, t.zu32);
        CPM_LAUNCH(c, "k_layer_phases");
    }
    CPM_CUDA(c, cudaStreamSynchronize(c->stream));
    return CPM_OK;
}

// ----------------------------------------------------------------------------- charge phases
// X[h][j] = Q_j (cos, sin)(h theta_x), h = 0..NX; Y[h][j], Z[h][j] without the charge; j = r ne + charge.
// A warp holds 32 charges and one residue k of h modulo 8: it forms h = 8 a + k as the product of two directly
// evaluated phases, so that an axis of H harmonics needs about 8 + H / 8 sincospi and the rest are four
// multiply-adds (one rounding more than a direct evaluation).  The fractions, FP64 work, are made once per
// (charge, axis) by three warps: with one per thread the FP64 pipe took 9 us for 45,600 charges.
// CP_SPLIT (the tensor-core stage): the z phases stay two factors, k = 0..7 and 2^14 times the steps 8 a, which
// that kernel multiplies itself, and p runs over replicas padded to nep charges.
constexpr int CP_PTS = 32;
template <typename T, bool SPLIT>
__global__ void __launch_bounds__(8 * CP_PTS) k_charge_phases(const double* __restrict__ xyz,
                                                              const double* __restrict__ Q, int64_t P, int64_t ne,
                                                              int64_t nep, double ix, double iy, double iz, int NX,
                                                              int NY, int NZ, c2<T>* __restrict__ X,
                                                              c2<T>* __restrict__ Y, c2<T>* __restrict__ Z,
                                                              float* __restrict__ qmax, int* __restrict__ qlast) {
    __shared__ c2<T> sg[8][CP_PTS];
    __shared__ uint64_t sf[3][CP_PTS];
    __shared__ T sq[CP_PTS];
    const int pt = threadIdx.x % CP_PTS, k = threadIdx.x / CP_PTS;
    const int64_t p = (int64_t)blockIdx.x * CP_PTS + pt;
    const bool live = p < P;
    if (k < 3) {
        int64_t src = p;
        bool real = live;
        if (SPLIT) {
            const int64_t r = p / nep, j = p - r * nep;
            real = live && j < ne;
            src = r * ne + j;
        }
        const double q = real ? Q[src] : 0.0;
        // a zero charge (padding) contributes nothing wherever it sits
        sf[k][pt] = q != 0.0 ? row_frac(xyz[3 * src + k], k == 0 ? ix : k == 1 ? iy : iz) : 0ull;
        if (k == 0) {
            sq[pt] = (T)q;
            if (SPLIT) {   // the block's charges belong to one replica (nep is a multiple of 64)
                float mx = fabsf((float)q);
                const unsigned nz = __ballot_sync(0xffffffffu, q != 0.0);
                for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                if (pt == 0 && nz) {   // nonnegative floats are ordered as their bits
                    const int64_t r = p / nep;
                    atomicMax((int*)&qmax[r], __float_as_int(mx));
                    atomicMax(&qlast[r], (int)(p - r * nep) + 32 - __clz(nz));
                }
            }
        }
    }
    __syncthreads();
    for (int axis = 0; axis < 3; ++axis) {
        const int H = axis == 0 ? NX : axis == 1 ? NY : NZ, na = H / 8 + 1;
        c2<T>* out = axis == 0 ? X : axis == 1 ? Y : Z;
        const uint64_t f = sf[axis][pt];
        c2<T> base = cmake<T>(1, 0);
        if (k > 0 && (k <= H || SPLIT)) base = row_phase<T>(f, k);
        if (SPLIT && axis == 2) {
            if (!live) break;
            out[(int64_t)k * P + p] = base;
            for (int a = k; a < na; a += 8) {
                c2<T> v = a > 0 ? row_phase<T>(f, 8 * a) : cmake<T>(1, 0);
                v.x *= (T)TC_ZSCALE;
                v.y *= (T)TC_ZSCALE;
                out[(int64_t)(8 + a) * P + p] = v;
            }
            break;
        }
        if (axis == 0) { base.x *= sq[pt]; base.y *= sq[pt]; }
        for (int a0 = 0; a0 < na; a0 += 8) {   // eight steps 8 a at a time
            const int a = a0 + k;
            __syncthreads();
            if (a < na && a > 0) sg[k][pt] = row_phase<T>(f, 8 * a);
            __syncthreads();
            for (int b = 0; b < min(8, na - a0); ++b) {
                const int h = 8 * (a0 + b) + k;
                if (h <= H && live) out[(int64_t)h * P + p] = a0 + b == 0 ? base : cmul(sg[b][pt], base);
            }
        }
    }
}

// The same in fixed point, for FP64: cos and sin times 2^62 in 64-bit integers (tc_rows64.cu takes them as they are,
// X times the scaled charge, Z rounded to 2^55; k_rows_sf<double> converted at the end).  FP64 arithmetic took 34 us
// for 5,700 charges of 110 harmonics, the integers 9.5 us (100 charges in k_rows_sf<double>: 11 and 3 us): the 64-bit
// product of two phases is some 40 instructions of a pipe with thirty times the rate.  A phase is evaluated as T1[top
// ten bits] T2[next ten] (1 - d^2 / 2, d - d^3 / 6) with the angle d < 2 pi 2^-20 of the other 44 bits: the terms
// left out are below 2^-72, T1 is FP64's own cosine and sine, and T2's are kept as 1 - cos, exact to 2^-62.
__global__ void k_fixed_tab(longlong2* __restrict__ tab) {   // grid 2 x FX_TAB: T1 | T2
    const int t = threadIdx.x;
    double s, c;
    if (blockIdx.x == 0) {
        sincospi(2.0 * t / FX_TAB, &s, &c);
        tab[t] = make_longlong2(__double2ll_rn(c * 0x1p62), __double2ll_rn(s * 0x1p62));
    } else {
        const double a = t * (1.0 / (FX_TAB * (double)FX_TAB));   // half the angle, in half turns
        sincospi(a, &s, &c);
        tab[FX_TAB + t] = make_longlong2((1ll << 62) - __double2ll_rn(2.0 * s * s * 0x1p62), __double2ll_rn(2.0 * s * c * 0x1p62));
    }
}
__device__ __forceinline__ longlong2 fx_mul(longlong2 a, longlong2 b) {   // the floors of the two halves cancel, or cost one
    return make_longlong2((__mul64hi(a.x, b.x) - __mul64hi(a.y, b.y)) * 4,
                          (__mul64hi(a.x, b.y) + __mul64hi(a.y, b.x) + 1) * 4);
}
__device__ __forceinline__ longlong2 fx_phase(uint64_t f, const longlong2* __restrict__ tab) {
    const longlong2 b = fx_mul(__ldg(&tab[f >> 54]), __ldg(&tab[FX_TAB + ((f >> 44) & (FX_TAB - 1))]));
    const uint64_t D = __umul64hi(f << 20, 0x1921FB54442D1846ull);            // d 2^78 = (f mod 2^44) 2 pi 2^14
    const uint64_t d2 = __umul64hi(D, D);                                     // d^2 2^92
    const int64_t v4 = (int64_t)(d2 >> 31) * 4;                               // d^2 / 2 times 2^64
    const int64_t sn = (int64_t)(D - (uint32_t)(__umul64hi(D, d2) >> 28) / 6);   // (d - d^3 / 6) 2^78
    return make_longlong2(b.x - __mul64hi(b.x, v4) - (__mul64hi(b.y, sn) >> 14),
                          b.y - __mul64hi(b.y, v4) + (__mul64hi(b.x, sn) >> 14));
}
// v 2^-62, the exponent changed in integers
__device__ __forceinline__ double fx_double(int64_t v) {
    const double d = (double)v;
    return v ? __hiloint2double(__double2hiint(d) - (62 << 20), __double2loint(d)) : 0.0;
}
// grid (P / CP_PTS, axis).  FIXED: X, Y, Z in fixed point, replicas padded to nep, a multiple of CP_PTS, charges scaled
// with qexp.  Otherwise the phases in FP64 (k_rows_sf<double>): nep = ne, and X times the charge itself.
template <bool FIXED>
__global__ void __launch_bounds__(8 * CP_PTS) k_charge_fixed(const double* __restrict__ xyz, const double* __restrict__ Q,
                                                             int64_t P, int64_t ne, int64_t nep, double3 inv, int NX,
                                                             int NY, int NZ, const int* __restrict__ qexp,
                                                             const longlong2* __restrict__ tab, longlong2* __restrict__ X,
                                                             longlong2* __restrict__ Y, longlong2* __restrict__ Z) {
    grid_wait();
    __shared__ longlong2 sg[8][CP_PTS];
    __shared__ uint64_t sf[CP_PTS];
    __shared__ int64_t sq[CP_PTS];
    const int pt = threadIdx.x % CP_PTS, k = threadIdx.x / CP_PTS, axis = blockIdx.y;
    const int64_t p = (int64_t)blockIdx.x * CP_PTS + pt;
    if (k == 0) {
        const int64_t r = p / nep, j = p - r * nep, src = r * ne + j;
        const double q = p < P && j < ne ? Q[src] : 0.0;
        // a zero charge (padding) contributes nothing wherever it sits
        sf[pt] = q != 0.0 ? row_frac(xyz[3 * src + axis], axis == 0 ? inv.x : axis == 1 ? inv.y : inv.z) : 0ull;
        sq[pt] = FIXED ? __double2ll_rn(q * pow2_bits(2045 - min(max(qexp[r], 1), ROW64_EMAX)) * 0x1p62) : __double_as_longlong(q);
    }
    __syncthreads();
    const int H = axis == 0 ? NX : axis == 1 ? NY : NZ, na = H / 8 + 1;
    longlong2* out = axis == 0 ? X : axis == 1 ? Y : Z;
    const uint64_t f = sf[pt];
    longlong2 base = make_longlong2(1ll << 62, 0);
    if (k > 0 && k <= H) base = fx_phase(f * (uint64_t)k, tab);
    if (FIXED && axis == 0) base = make_longlong2(__mul64hi(base.x, sq[pt]) * 4 + 2, __mul64hi(base.y, sq[pt]) * 4 + 2);
    for (int a0 = 0; a0 < na; a0 += 8) {   // eight steps 8 a at a time
        const int a = a0 + k;
        __syncthreads();
        if (a < na && a > 0) sg[k][pt] = fx_phase(f * (uint64_t)(8 * a), tab);
        __syncthreads();
        for (int b = 0; b < min(8, na - a0); ++b) {
            const int h = 8 * (a0 + b) + k;
            if (h > H || p >= P) continue;
            longlong2 v = a0 + b == 0 ? base : fx_mul(sg[b][pt], base);
            if (FIXED) {
                if (axis == 2) v = make_longlong2((v.x + 64) >> 7, (v.y + 64) >> 7);
                out[(int64_t)h * P + p] = v;
            } else {
                const double q = axis == 0 ? __longlong_as_double(sq[pt]) : 1.0;
                double2 d = make_double2(fx_double(v.x), fx_double(v.y));
                if (axis == 0) { d.x *= q; d.y *= q; }
                ((double2*)out)[(int64_t)h * P + p] = d;
            }
        }
    }
}
static cpm_status charge_fixed_table(cpm_ctx* c) {
    k_fixed_tab<<<2, FX_TAB, 0, c->stream>>>(c->rows.fxtab);
    CPM_LAUNCH(c, "k_fixed_tab");
    return CPM_OK;
}

// ----------------------------------------------------------------------------- stage 1, CUDA cores
// part[s][r][4 p + t][c] over the s-th range of charges of replica r.  A block takes 16 TM rows x 8 TN
// harmonic functions with TM x TN accumulators per thread; the rows are those that are not identically
// zero, in the order of |k_perp|, so a tile's harmonics end at its largest extent.  FP64: the pipe retires
// two multiply-adds per clock and SM, so 4 x 4 accumulators are enough to keep it busy and small tiles
// waste less at the edge of the k ball; FP32: 8 x 8.
template <typename T> struct RowTileOf;
template <> struct RowTileOf<double> { static constexpr int TM = 4, TN = 4; };
template <> struct RowTileOf<float> { static constexpr int TM = 8, TN = 8; };
constexpr int RW_BK = 16, RW_THREADS = 128;

template <typename T>
__global__ void __launch_bounds__(RW_THREADS) k_rows_sf(const int4* __restrict__ pairs, const int* __restrict__ list,
                                                        int nrows, int np, int cw, const c2<T>* __restrict__ X,
                                                        const c2<T>* __restrict__ Y, const c2<T>* __restrict__ Z,
                                                        int64_t P, int64_t ne, int splits, int64_t chunk, int m,
                                                        T* __restrict__ part) {
    grid_wait();
    constexpr int TM = RowTileOf<T>::TM, TN = RowTileOf<T>::TN, BM = 16 * TM, BN = 8 * TN;
    __shared__ T Ps[RW_BK][BM + 1];
    __shared__ T Zs[RW_BK][BN + 1];
    __shared__ int s_row[BM];
    __shared__ int2 s_xy[BM];
    __shared__ int s_mx;
    const int r0 = blockIdx.x * BM, cb = blockIdx.y * BN;
    const int r = blockIdx.z / splits, sp = blockIdx.z % splits;
    if (threadIdx.x == 0) s_mx = -1;
    __syncthreads();
    for (int e = threadIdx.x; e < BM; e += RW_THREADS) {
        const int row = r0 + e < nrows ? list[r0 + e] : -1;
        s_row[e] = row;
        if (row >= 0) {
            const int4 pr = pairs[row >> 2];
            s_xy[e] = make_int2(pr.x, pr.y);
            atomicMax(&s_mx, pr.z);
        }
    }
    __syncthreads();
    if (cb > 2 * s_mx + 1) return;   // no row of the tile reaches these harmonics (block-uniform)
    const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
    const int qn = min(TN, (2 * (s_mx + 1) - cb + 7) / 8);   // groups of eight functions inside the ball
    T acc[TM][TN];
#pragma unroll
    for (int p = 0; p < TM; ++p)
#pragma unroll
        for (int q = 0; q < TN; ++q) acc[p][q] = 0;
    const int64_t jb = (int64_t)r * ne + (int64_t)sp * chunk;
    const int64_t je = min((int64_t)(r + 1) * ne, jb + chunk);
    const int kk = threadIdx.x % RW_BK, mm0 = threadIdx.x / RW_BK;   // staging: charge kk, rows mm0 + 8 i
    for (int64_t j0 = jb; j0 < je; j0 += RW_BK) {
        const int64_t j = j0 + kk;
        const bool in = j < je;
#pragma unroll
        for (int i = 0; i < BM / 8; ++i) {
            const int mm = mm0 + 8 * i, row = s_row[mm];
            T v = 0;
            if (in && row >= 0) {
                const int2 xy = s_xy[mm];
                const c2<T> x = X[(int64_t)xy.x * P + j], y = Y[(int64_t)xy.y * P + j];
                v = ((row & 1) ? x.y : x.x) * ((row & 2) ? y.y : y.x);
            }
            Ps[kk][mm] = v;
        }
#pragma unroll
        for (int i = 0; i < BN / 16; ++i) {
            const int h = mm0 + 8 * i, nz = cb / 2 + h;
            const c2<T> z = in && nz <= s_mx ? Z[(int64_t)nz * P + j] : cmake<T>(0, 0);
            Zs[kk][2 * h] = z.x;
            Zs[kk][2 * h + 1] = z.y;
        }
        __syncthreads();
#pragma unroll 4
        for (int q0 = 0; q0 < RW_BK; ++q0) {
            T a[TM], b[TN];
#pragma unroll
            for (int p = 0; p < TM; ++p) a[p] = Ps[q0][ty + 16 * p];
#pragma unroll
            for (int q = 0; q < TN; ++q) b[q] = Zs[q0][tx + 8 * q];
#pragma unroll
            for (int q = 0; q < TN; ++q) {
                // FP64: the eight functions past the tile's extent cost more than the test
                if (std::is_same<T, double>::value && q >= qn) break;
#pragma unroll
                for (int p = 0; p < TM; ++p) acc[p][q] = fma(a[p], b[q], acc[p][q]);
            }
        }
        __syncthreads();
    }
    T* out = part + ((int64_t)sp * m + r) * 4 * np * cw;
#pragma unroll
    for (int p = 0; p < TM; ++p) {
        const int row = s_row[ty + 16 * p];
        if (row < 0) continue;
#pragma unroll
        for (int q = 0; q < TN; ++q) {
            const int cc = cb + tx + 8 * q;
            if (cc < cw) out[(int64_t)row * cw + cc] = acc[p][q];
        }
    }
}

// ----------------------------------------------------------------------------- stage 2
// One block per (pair, replica): the split sums of the pair's four rows, weighted, in shared memory, then
// four lanes per (part, height) add the harmonics nz = lane, lane + 4, ... and combine by a fixed butterfly.
constexpr int RL_THREADS = 128;
// V[t][cc] = scale(cc) times the sum over the splits of the pair's row t; rows with sin 0 = 0 are not formed, and zero
template <typename T, typename F>
__device__ __forceinline__ void sum_pair_rows(int4 pr, const T* __restrict__ src, int cw, int ncc, int splits, int64_t sstride,
                                              T* __restrict__ V, F scale) {
    for (int e = threadIdx.x; e < 4 * ncc; e += RL_THREADS) {
        const int t = e / ncc, cc = e - t * ncc;
        T v = 0;
        if (!((t & 1) && pr.x == 0) && !((t & 2) && pr.y == 0)) {
            const T* q = src + (int64_t)t * cw + cc;
            int s = 0;
            for (; s + 8 <= splits; s += 8) {   // eight loads in flight, added in split order
                T x[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) x[u] = q[(s + u) * sstride];
#pragma unroll
                for (int u = 0; u < 8; ++u) v += x[u];
            }
            for (; s < splits; ++s) v += q[s * sstride];
        }
        V[e] = v * scale(cc);
    }
}
template <typename T>
__global__ void __launch_bounds__(RL_THREADS) k_rows_layers(const int4* __restrict__ pairs, int np, int cw, int NZ,
                                                            const T* __restrict__ part, int splits, int m,
                                                            const T* __restrict__ W, const c2<T>* __restrict__ ZU,
                                                            int nzu, int nslots, const float* __restrict__ qmax,
                                                            T* __restrict__ Tout) {
    grid_wait();
    grid_go();
    extern __shared__ __align__(16) unsigned char rl_smem[];
    const int p = blockIdx.x, r = blockIdx.y;
    const int4 pr = pairs[p];
    const int ncc = 2 * (pr.z + 1);
    T* V = (T*)rl_smem;   // [4][ncc]
    sum_pair_rows(pr, part + ((int64_t)r * np + p) * 4 * cw, cw, ncc, splits, (int64_t)m * 4 * np * cw, V,
                  [&](int cc) { return W[(int64_t)p * (NZ + 1) + (cc >> 1)]; });
    __syncthreads();
    const T f = qmax ? (T)(1.f / (TC_ZSCALE * pow2_below(qmax[r], 14))) : (T)1;   // a power of two
    const int l4 = threadIdx.x & 3;
    for (int o0 = 0; o0 < 4 * nzu; o0 += RL_THREADS / 4) {
        const int o = o0 + (threadIdx.x >> 2), t = o / nzu, u = o - t * nzu;
        T s = 0;
        if (o < 4 * nzu) {
            const T* v = V + t * ncc;
            for (int nz = l4; nz <= pr.z; nz += 4) {
                const c2<T> z = ZU[(int64_t)nz * nzu + u];
                s = fma(v[2 * nz], z.x, s);
                s = fma(v[2 * nz + 1], z.y, s);
            }
        }
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (l4 == 0 && o < 4 * nzu) Tout[(((int64_t)r * nzu + u) * nslots + pr.w) * 4 + t] = s * f;
    }
}

// ----------------------------------------------------------------------------- stage 3
// partial[r][chunk][i]: thread = site of one height, MR replicas at a time; nested sums over the chunk's nx
// and over ny, so that a (site, pair) costs four multiply-adds.  The chunk's coefficients T go through
// shared memory in one coalesced round trip; read from L2 where they are used, each pair waited for its own
// (10 against 16 us for 8 EDL replicas, caches cold).
template <typename T> struct T4of;
template <> struct T4of<float> { using t = float4; };
template <> struct T4of<double> { using t = double4_32a; };

template <typename T, int MR>
__global__ void __launch_bounds__(ROW_TILE) k_rows_sites(const int4* __restrict__ tiles, const int* __restrict__ perm,
                                                         const int* __restrict__ chunkb, const int* __restrict__ nxoff,
                                                         const typename T4of<T>::t* __restrict__ Tin, int nzu,
                                                         int nslots, const c2<T>* __restrict__ SX,
                                                         const c2<T>* __restrict__ SY, int64_t n, int m, int nchunk,
                                                         T* __restrict__ partial) {
    grid_wait();
    extern __shared__ __align__(32) unsigned char rs_smem[];
    typename T4of<T>::t* st = (typename T4of<T>::t*)rs_smem;   // [slot of the chunk][MR]
    const int4 tl = tiles[blockIdx.x];
    const int ch = blockIdx.y, rb = blockIdx.z * MR;
    const int x0 = chunkb[ch], x1 = chunkb[ch + 1];
    const int64_t i = perm[tl.y + min((int)threadIdx.x, tl.z - 1)];
    const int f0 = nxoff[x0], nsl = nxoff[x1] - f0;
    const typename T4of<T>::t* tb = Tin + ((int64_t)rb * nzu + tl.x) * nslots + f0;
    const int64_t rstride = (int64_t)nzu * nslots;
    for (int e = threadIdx.x; e < MR * nsl; e += ROW_TILE) {   // T has room for whole groups of MR
        const int k = e / nsl, sl = e - k * nsl;
        st[sl * MR + k] = tb[k * rstride + sl];
    }
    T acc[MR];
#pragma unroll
    for (int k = 0; k < MR; ++k) acc[k] = 0;
    __syncthreads();
    // ny from the high harmonics down: the large terms, of the long waves, come last and the sums stay small before
    // them.  An ascending counter, and nx and the heights' nz left as they were: with those reversed too the loads of
    // four replicas at 512 sites waited for one another (60 against 50 us a step)
    for (int x = x0; x < x1; ++x) {
        const int o0 = nxoff[x] - f0, cnt = nxoff[x + 1] - f0 - o0;
        if (cnt <= 0) continue;
        const c2<T> sx = SX[(int64_t)x * n + i];
        T ic[MR], is[MR];
#pragma unroll
        for (int k = 0; k < MR; ++k) ic[k] = is[k] = 0;
#pragma unroll 4
        for (int k0 = 0; k0 < cnt; ++k0) {
            const int y = cnt - 1 - k0;
            const c2<T> sy = SY[(int64_t)y * n + i];
#pragma unroll
            for (int k = 0; k < MR; ++k) {
                const typename T4of<T>::t v = st[(o0 + y) * MR + k];
                ic[k] = fma(sy.x, v.x, fma(sy.y, v.z, ic[k]));
                is[k] = fma(sy.x, v.y, fma(sy.y, v.w, is[k]));
            }
        }
#pragma unroll
        for (int k = 0; k < MR; ++k) acc[k] = fma(sx.x, ic[k], fma(sx.y, is[k], acc[k]));
    }
    if ((int)threadIdx.x >= tl.z) return;
    const int nrep = min(MR, m - rb);
#pragma unroll
    for (int k = 0; k < MR; ++k)
        if (k < nrep) partial[((int64_t)(rb + k) * nchunk + ch) * n + i] = acc[k];
}

// wrho[r][col][nz + NZ] = w rho of the signed columns, for the site stages that take every site by itself.  One block
// per (pair, replica): the split sums of the pair's four rows in shared memory, as in k_rows_layers, then the one or
// two columns that they make up, RC_HARM harmonics at a time.  With a thread per (column, harmonic) adding the splits of
// its eight values one after the other, b of one replica over 2,048 and 4,320 sites of distinct heights took 74.1 and
// 77.3 us, 61.9 and 65.8 now; FP32 on the CUDA cores 118.8 and 117.5, now 103.7 and 101.5.
constexpr int RC_HARM = 256;
template <typename T>
__global__ void __launch_bounds__(RL_THREADS) k_rows_to_cols(const int2* __restrict__ paircols, const int* __restrict__ colext,
                                                             int ncols, const int4* __restrict__ pairs, int np, int cw, int NZ,
                                                             const T* __restrict__ part, int splits, int m,
                                                             const T* __restrict__ w, const float* __restrict__ qmax,
                                                             c2<T>* __restrict__ wrho) {
    grid_wait();
    extern __shared__ __align__(16) unsigned char rl_smem[];
    const int p = blockIdx.x, r = blockIdx.y, nzw = 2 * NZ + 1;
    const int4 pr = pairs[p];
    const T f = qmax ? (T)(1.f / (TC_ZSCALE * pow2_below(qmax[r], 14))) : (T)1;   // a power of two
    const int2 pc = paircols[p];
    T* V = (T*)rl_smem;   // [4][ncc]
    for (int a0 = 0; a0 <= NZ; a0 += RC_HARM) {   // RC_HARM harmonics at a time
        const int nh = min(RC_HARM, NZ + 1 - a0), ncc = 2 * max(0, min(nh, pr.z + 1 - a0));
        __syncthreads();
        sum_pair_rows(pr, part + ((int64_t)r * np + p) * 4 * cw + 2 * a0, cw, ncc, splits, (int64_t)m * 4 * np * cw, V,
                      [](int) { return (T)1; });
        __syncthreads();
        for (int e = threadIdx.x; e < 4 * nh; e += RL_THREADS) {
            const int q = e / nh, az = a0 + e % nh, nz = q & 1 ? -az : az, col = q < 2 ? pc.x : pc.y;
            if (col < 0 || (q & 1 && az == 0)) continue;
            c2<T> v = cmake<T>(0, 0);
            const T wt = w[(int64_t)col * nzw + nz + NZ];
            if (az <= colext[col] && wt != (T)0) {
                const T* a = V + 2 * (az - a0);
                const T sy = q < 2 ? (T)1 : (T)-1, sz = q & 1 ? (T)-1 : (T)1, fw = wt * f;
                v.x = fw * ((a[0] - sy * a[3 * ncc]) - sz * (a[ncc + 1] + sy * a[2 * ncc + 1]));
                v.y = fw * (sz * (a[1] - sy * a[3 * ncc + 1]) + (a[ncc] + sy * a[2 * ncc]));
            }
            wrho[((int64_t)r * ncols + col) * nzw + nz + NZ] = v;
        }
    }
}

// ----------------------------------------------------------------------------- host side
template <typename T> RowDims row_dims(const cpm_ctx* c, int m, int64_t ne) {
    const RowTable& t = c->rows;
    RowDims d{};
    constexpr int BM = 16 * RowTileOf<T>::TM, BN = 8 * RowTileOf<T>::TN;
    d.cw = ((2 * (c->kt.NZ + 1) + 31) / 32) * 32;
    d.xt = (t.nrows + BM - 1) / BM;
    d.yt = (2 * (c->kt.NZ + 1) + BN - 1) / BN;
    int64_t work = 0;   // tiles inside the ball
    for (int b = 0; b < d.xt; ++b) {
        int mx = -1;
        for (int e = b * BM; e < std::min(t.nrows, (b + 1) * BM); ++e) mx = std::max(mx, t.hext[t.hlist[e] >> 2]);
        work += (2 * (mx + 1) + BN - 1) / BN;
    }
    // about six blocks per SM, so that the last ones to finish leave little of the GPU idle; no range
    // shorter than one K step
    const int64_t maxs = std::max<int64_t>(1, (ne + RW_BK - 1) / RW_BK);
    const int64_t want = c->lean > 1 ? 1 : ((6 * 152 + work * m - 1) / std::max<int64_t>(1, work * m)) >> (2 * c->lean);
    d.splits = (int)std::max<int64_t>(1, std::min<int64_t>(want, std::min<int64_t>(maxs, 64)));
    d.chunk = std::max<int64_t>(1, ((ne + d.splits - 1) / d.splits + RW_BK - 1) / RW_BK) * RW_BK;
    d.splits = (int)std::max<int64_t>(1, (ne + d.chunk - 1) / d.chunk);
    return d;
}
template RowDims row_dims<double>(const cpm_ctx*, int, int64_t);
template RowDims row_dims<float>(const cpm_ctx*, int, int64_t);

template <typename T> static const T* row_weights(const cpm_ctx* c);
template <> const double* row_weights<double>(const cpm_ctx* c) { return c->rows.W; }
template <> const float* row_weights<float>(const cpm_ctx* c) { return c->rows.W32; }
template <typename T> static const c2<T>* row_zu(const cpm_ctx* c);
template <> const double2* row_zu<double>(const cpm_ctx* c) { return c->rows.zu64; }
template <> const float2* row_zu<float>(const cpm_ctx* c) { return c->rows.zu32; }
template <typename T> static const Phases<T>& row_sites(const cpm_ctx* c);
template <> const Phases<double>& row_sites<double>(const cpm_ctx* c) { return c->site64; }
template <> const Phases<float>& row_sites<float>(const cpm_ctx* c) { return c->site32; }

template <>
cpm_status launch_charge_phases<float>(cpm_ctx* c, cudaStream_t st, int64_t P, const double* xyz, const double* Q, float2* X,
                                       float2* Y, float2* Z) {
    const KTable& k = c->kt;
    k_charge_phases<float, false><<<(unsigned)((P + CP_PTS - 1) / CP_PTS), 8 * CP_PTS, 0, st>>>(
        xyz, Q, P, P, P, c->g.inv[0], c->g.inv[1], c->g.inv[2], k.NX, k.NY, k.NZ, X, Y, Z, nullptr, nullptr);
    CPM_LAUNCH(c, "k_charge_phases");
    return CPM_OK;
}
template <>
cpm_status launch_charge_phases<double>(cpm_ctx* c, cudaStream_t st, int64_t P, const double* xyz, const double* Q, double2* X,
                                        double2* Y, double2* Z) {
    const KTable& k = c->kt;
    k_charge_fixed<false><<<dim3((unsigned)((P + CP_PTS - 1) / CP_PTS), 3), 8 * CP_PTS, 0, st>>>(
        xyz, Q, P, P, P, make_double3(c->g.inv[0], c->g.inv[1], c->g.inv[2]), k.NX, k.NY, k.NZ, nullptr, c->rows.fxtab,
        (longlong2*)X, (longlong2*)Y, (longlong2*)Z);
    CPM_LAUNCH(c, "k_charge_fixed");
    return CPM_OK;
}

int64_t charge_slots(const KTable& k) { return (k.NX + 1) + (k.NY + 1) + 8 + (k.NZ / 8 + 1); }

cpm_status launch_charge_slots(cpm_ctx* c, cudaStream_t st, int m, int64_t ne, int64_t nep, const double* xyz,
                               const double* Q, float2* tab, float* qmax, int* qlast) {
    const KTable& k = c->kt;
    const int64_t P = (int64_t)m * nep;
    float2* Y = tab + (int64_t)(k.NX + 1) * P;
    k_charge_phases<float, true><<<(unsigned)((P + CP_PTS - 1) / CP_PTS), 8 * CP_PTS, 0, st>>>(
        xyz, Q, P, ne, nep, c->g.inv[0], c->g.inv[1], c->g.inv[2], k.NX, k.NY, k.NZ, tab, Y, Y + (int64_t)(k.NY + 1) * P,
        qmax, qlast);
    CPM_LAUNCH(c, "k_charge_phases");
    return CPM_OK;
}

cpm_status launch_charge_fixed(cpm_ctx* c, cudaStream_t st, int m, int64_t ne, int64_t nep, const double* xyz,
                               const double* Q, const int* qexp, longlong2* X, longlong2* Y, longlong2* Z) {
    const KTable& k = c->kt;
    const int64_t P = (int64_t)m * nep;
    CPM_CUDA(c, launch_after(k_charge_fixed<true>, dim3((unsigned)(P / CP_PTS), 3), dim3(8 * CP_PTS), 0, st, 
        xyz, Q, P, ne, nep, make_double3(c->g.inv[0], c->g.inv[1], c->g.inv[2]), k.NX, k.NY, k.NZ, qexp, c->rows.fxtab, X, Y, Z));
    CPM_LAUNCH(c, "k_charge_fixed");
    return CPM_OK;
}

template <typename T>
cpm_status rows_sf(cpm_ctx* c, cudaStream_t st, const RowDims& d, int m, int64_t ne, const c2<T>* X, const c2<T>* Y,
                   const c2<T>* Z, T* part) {
    const RowTable& t = c->rows;
    CPM_CUDA(c, launch_after(k_rows_sf<T>, dim3(d.xt, d.yt, (unsigned)(m * d.splits)), dim3(RW_THREADS), 0, st, 
        t.pairs, t.list, t.nrows, t.np, d.cw, X, Y, Z, (int64_t)m * ne, ne, d.splits, d.chunk, m, part));
    CPM_LAUNCH(c, "k_rows_sf");
    return CPM_OK;
}
template cpm_status rows_sf<double>(cpm_ctx*, cudaStream_t, const RowDims&, int, int64_t, const double2*, const double2*, const double2*, double*);
template cpm_status rows_sf<float>(cpm_ctx*, cudaStream_t, const RowDims&, int, int64_t, const float2*, const float2*, const float2*, float*);

// Which site stage, both sides measured (b alone, us, by height / every site by itself; plates with their sites moved onto
// so many heights):
//   tensor cores (their general stage costs little per replica, more per site):
//     512 sites, 1 replica: 51 heights 39 / 43, 64 40 / 44;  8 replicas: 32 44 / 47, 51 47 / 46, 64 51 / 47
//     2,048 sites, 1 replica: 64 47 / 58, 97 51 / 57, 128 55 / 54, 204 65 / 58;  8 replicas: 32 81 / 86, 48 89 / 87, 64 96 / 86
//     4,320 sites, 1 replica: 130 60 / 70, 196 68 / 71, 270 87 / 68;  8 replicas: 48 108 / 112, 64 115 / 115, 96 131 / 111
//     16,384 sites, 1 replica: 364 147 / 210, 512 207 / 212;  8 replicas: 192 476 / 517, 256 531 / 519, 364 580 / 519
//   FP32 on the CUDA cores, one replica: 2,048 sites, 256 heights 90 / 103; 4,320: 270 116 / 128, 360 134 / 128, 540 167 /
//     128; 8,192: 512 200 / 244; four: 4,320, 540 275 / 311
//   FP64: 4,320 sites, 540 heights 1,038 / 1,720
bool rows_by_height(const cpm_ctx* c, int m) {
    const int64_t nu = c->nzu, n = c->n;
    if (!c->rows.layered) return false;
    if (c->rows.tcitems) return nu <= std::max<int64_t>(std::max(48, 128 / m), n / (m == 1 ? 32 : 64));
    return c->p.k_prec == CPM_PREC_FP64 || m > 1 || nu <= std::max<int64_t>(256, n / 16);
}

template <typename T>
cpm_status rows_layers(cpm_ctx* c, cudaStream_t st, int cw, int splits, int m, const T* part, const float* qmax, T* Tbuf) {
    const RowTable& t = c->rows;
    const size_t sm = sizeof(T) * 4 * 2 * (c->kt.NZ + 1);
    if (sm > 48 * 1024) CPM_CUDA(c, cudaFuncSetAttribute(k_rows_layers<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    CPM_CUDA(c, launch_after(k_rows_layers<T>, dim3(t.np, m), dim3(RL_THREADS), sm, st, t.pairs, t.np, cw, c->kt.NZ, part, splits, m,
                                                            row_weights<T>(c), row_zu<T>(c), c->nzu, t.nslots, qmax, Tbuf));
    CPM_LAUNCH(c, "k_rows_layers");
    return CPM_OK;
}
template cpm_status rows_layers<double>(cpm_ctx*, cudaStream_t, int, int, int, const double*, const float*, double*);
template cpm_status rows_layers<float>(cpm_ctx*, cudaStream_t, int, int, int, const float*, const float*, float*);

template <typename T, int MR>
static cpm_status rows_sites_mr(cpm_ctx* c, cudaStream_t st, int m, const T* Tbuf, T* partial) {
    const RowTable& t = c->rows;
    const Phases<T>& s = row_sites<T>(c);
    const size_t sm = sizeof(T) * 4 * MR * t.chunkmax;
    if (sm > 48 * 1024) cudaFuncSetAttribute(k_rows_sites<T, MR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    CPM_CUDA(c, launch_after(k_rows_sites<T, MR>, dim3(t.ntiles, t.nchunk, (m + MR - 1) / MR), dim3(ROW_TILE), sm, st, 
        t.ltiles, t.lperm, t.chunkb, t.nxoff, (const typename T4of<T>::t*)Tbuf, c->nzu, t.nslots, s.X,
        s.Y + (int64_t)c->kt.NY * c->n, c->n, m, t.nchunk, partial));
    return CPM_OK;
}
// replicas per thread: the site phases are read once for all of them; one replica alone keeps the
// registers of one
template <typename T> static int rows_mr(int m) { return m == 1 ? 1 : m <= 4 || std::is_same<T, double>::value ? 4 : 8; }
template <typename T> int64_t rows_T_elems(const cpm_ctx* c, int m) {
    const int mr = rows_mr<T>(m);
    return (int64_t)((m + mr - 1) / mr) * mr * c->nzu * c->rows.nslots * 4;
}
template int64_t rows_T_elems<double>(const cpm_ctx*, int);
template int64_t rows_T_elems<float>(const cpm_ctx*, int);

template <typename T>
cpm_status rows_sites(cpm_ctx* c, cudaStream_t st, int m, const T* Tbuf, T* partial) {
    if (rows_mr<T>(m) == 1) CPM_TRY((rows_sites_mr<T, 1>(c, st, m, Tbuf, partial)));
    else if (rows_mr<T>(m) == 4) CPM_TRY((rows_sites_mr<T, 4>(c, st, m, Tbuf, partial)));
    else CPM_TRY((rows_sites_mr<T, 8>(c, st, m, Tbuf, partial)));
    CPM_LAUNCH(c, "k_rows_sites");
    return CPM_OK;
}
template cpm_status rows_sites<double>(cpm_ctx*, cudaStream_t, int, const double*, double*);
template cpm_status rows_sites<float>(cpm_ctx*, cudaStream_t, int, const float*, float*);

template <typename T>
cpm_status rows_to_cols(cpm_ctx* c, cudaStream_t st, int cw, int splits, int m, const T* part, const float* qmax, c2<T>* wrho) {
    const RowTable& t = c->rows;
    const KTable& k = c->kt;
    const T* w = std::is_same<T, float>::value ? (const T*)k.w32 : (const T*)k.w;
    const size_t sm = sizeof(T) * 4 * 2 * std::min(k.NZ + 1, RC_HARM);
    CPM_CUDA(c, launch_after(k_rows_to_cols<T>, dim3(t.np, m), dim3(RL_THREADS), sm, st, t.paircols, k.colext, k.ncols, t.pairs,
                             t.np, cw, k.NZ, part, splits, m, w, qmax, wrho));
    CPM_LAUNCH(c, "k_rows_to_cols");
    return CPM_OK;
}
template cpm_status rows_to_cols<double>(cpm_ctx*, cudaStream_t, int, int, int, const double*, const float*, double2*);
template cpm_status rows_to_cols<float>(cpm_ctx*, cudaStream_t, int, int, int, const float*, const float*, float2*);

}  // namespace cpm
