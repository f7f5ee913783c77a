// Real-space part of b in FP64 (k_prec = FP64): b_i(real) = sum_j Q_j f(r_ij) over the pairs within r_c,
// f(r) = (erfc(alpha r) - erfc(eta_i r)) / r.
//
// The FP64 pipe retires two multiply-adds per clock and SM here, so what counts is the number of FP64
// instructions per pair and how many lanes each serves.  A direct evaluation takes a square root, a division
// and two erfc, about 150 instructions, in the lanes of one cell at a time (1 in 4 useful).  Instead:
//   * f is an entire function of s = r^2, tabulated per Gaussian width as polynomials of degree R6_DEG on
//     intervals of relative width 1/16 (16 per octave of s, one interval below r6_smin): interpolation error
//     below 1e-16 of f(0), so a pair is a difference, s, and R6_DEG + 2 multiply-adds;
//   * a warp takes one site and streams the charges of its stencil rows, 32 at a time across the ends of
//     rows, testing the distance in FP32 (with a margin that covers its rounding); those that can be in range
//     wait in a queue, and FP64 work runs on 32 of them at once.
// 4,320 sites x 5,700 charges (EDL capacitor, r_c = 18): 94 us against 2,750 us; 216 sites x 100 charges: 14 against 186.
#include <cmath>
#include <vector>

#include "common.cuh"

namespace cpm {

constexpr int R6_DEG = 8;
constexpr int R6_ROW = R6_DEG + 2;     // coefficients, then the interval's centre
constexpr int R6_SUB = 16;             // intervals per octave
constexpr int R6_WARPS = 4;
constexpr int R6_F = 15;               // image shifts of at most R6_F periods per axis

// ----------------------------------------------------------------------------- table (host, FP64)
static double pair_f(double r, double alpha, double eta) {
    if (eta * r < 0.5) return (std::erf(eta * r) - std::erf(alpha * r)) / r;   // no difference of two values near 1
    return (std::erfc(alpha * r) - std::erfc(eta * r)) / r;
}

cpm_status build_real64(cpm_ctx* c, const std::vector<double>& etas) {
    dev_free(c, c->r64tab);
    c->r64tab = nullptr;
    c->r64n = 0;
    if (c->p.k_prec != CPM_PREC_FP64 || !c->rtab_id || etas.empty()) return CPM_OK;
    const CellGrid cg = make_grid(c->g);
    for (int d = 0; d < 3; ++d)
        if ((cg.S[d] + cg.nc[d] - 1) / cg.nc[d] > R6_F) return CPM_OK;   // a cut-off of many periods: k_real_b
    double emax = c->g.alpha;
    for (double e : etas) emax = std::max(emax, e);
    // below smin = 2^e0 the variation of f is a fraction of one Gaussian width
    const int e0 = (int)std::floor(std::log2(0.25 / (emax * emax)));
    const double rc2 = c->g.rcut * c->g.rcut;
    const int oct = std::max(1, (int)std::floor(std::log2(rc2 * 1.000001)) - e0 + 1);
    const int nint = 1 + oct * R6_SUB;
    if (oct > 60) return CPM_OK;
    std::vector<double> tab((size_t)etas.size() * nint * R6_ROW);
    constexpr int N = R6_DEG + 1;
    double node[N], cosine[N][N];   // Chebyshev nodes, cos(j acos(node i)): 0.3 ms of a set-up when formed per interval
    for (int i = 0; i < N; ++i) {
        node[i] = std::cos(PI * (i + 0.5) / N);
        for (int j = 0; j < N; ++j) cosine[j][i] = std::cos(PI * j * (i + 0.5) / N);
    }
    for (size_t t = 0; t < etas.size(); ++t)
        for (int k = 0; k < nint; ++k) {
            double lo = 0.0, hi = std::ldexp(1.0, e0);
            if (k > 0) {
                const int o = (k - 1) / R6_SUB, j = (k - 1) % R6_SUB;
                lo = std::ldexp(1.0 + (double)j / R6_SUB, e0 + o);
                hi = std::ldexp(1.0 + (double)(j + 1) / R6_SUB, e0 + o);
            }
            const double mid = 0.5 * (lo + hi), half = 0.5 * (hi - lo);
            double gk[N], ch[N], mono[N] = {}, t0[N] = {}, t1[N] = {}, tn[N] = {};
            for (int i = 0; i < N; ++i) gk[i] = pair_f(std::sqrt(mid + half * node[i]), c->g.alpha, etas[t]);
            for (int j = 0; j < N; ++j) {
                double s = 0.0;
                for (int i = 0; i < N; ++i) s += gk[i] * cosine[j][i];
                ch[j] = (j == 0 ? 1.0 : 2.0) * s / N;
            }
            t0[0] = 1.0;
            t1[1] = 1.0;
            mono[0] = ch[0];
            mono[1] = ch[1];
            for (int j = 2; j < N; ++j) {   // T_{j+1} = 2 v T_j - T_{j-1}
                for (int i = 0; i < N; ++i) tn[i] = (i > 0 ? 2.0 * t1[i - 1] : 0.0) - t0[i];
                for (int i = 0; i < N; ++i) { mono[i] += ch[j] * tn[i]; t0[i] = t1[i]; t1[i] = tn[i]; }
            }
            double* row = &tab[(t * nint + k) * R6_ROW];
            double f = 1.0;
            for (int i = 0; i < N; ++i, f /= half) row[i] = mono[i] * f;
            row[N] = mid;
        }
    CPM_TRY(dev_alloc(c, (void**)&c->r64tab, sizeof(double) * tab.size()));
    CPM_CUDA(c, cudaMemcpyAsync(c->r64tab, tab.data(), sizeof(double) * tab.size(), cudaMemcpyHostToDevice, c->stream));
    CPM_CUDA(c, cudaStreamSynchronize(c->stream));
    c->r64n = nint;
    c->r64e0 = e0;
    return CPM_OK;
}

// ----------------------------------------------------------------------------- the kernel
struct R6Row { int beg, pre; };

// One warp per (site, replica).  The rows (dy, dz) of the site's stencil are taken 32 at a time, lane = row: each
// row, trimmed to the sphere, is one contiguous run of the cell-sorted charges per image shift along x.
// sorted32: the same charges in single precision.  slack covers the rounding of the FP32 test.
__global__ void __launch_bounds__(32 * R6_WARPS)
    k_real64(const double* __restrict__ sx, int64_t n, int m, Geometry g, CellGrid cg, const int* __restrict__ start,
             const double4_32a* __restrict__ sorted, const float4* __restrict__ sorted32, const double* __restrict__ tab,
             int nint, int e0, const int* __restrict__ tabid, float slack, double* __restrict__ out) {
    grid_wait();
    __shared__ R6Row s_row[R6_WARPS][33];
    __shared__ float4 s_sh[R6_WARPS][32];            // image shift of a run, w: the shift counts packed
    __shared__ int2 s_q[R6_WARPS][64];               // queue: (charge, shift counts)
    __shared__ double s_per[3][2 * R6_F + 1];        // whole numbers of periods
    for (int e = threadIdx.x; e < 3 * (2 * R6_F + 1); e += 32 * R6_WARPS) {
        const int d = e / (2 * R6_F + 1), f = e % (2 * R6_F + 1) - R6_F;
        s_per[d][f + R6_F] = f * g.boxL[d];
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t wid = (int64_t)blockIdx.x * R6_WARPS + warp;
    if (wid >= (int64_t)m * n) return;
    const int r = (int)(wid / n);
    const int64_t i = wid - (int64_t)r * n;
    double sw[3];
    int ci[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double x = sx[d * n + i];
        sw[d] = x - g.boxL[d] * floor(x * g.inv[d]);
        if (sw[d] >= g.boxL[d]) sw[d] -= g.boxL[d];
        if (sw[d] < 0) sw[d] = 0;
        ci[d] = min(cg.nc[d] - 1, (int)(sw[d] / cg.h[d]));
    }
    const double* tb = tab + (int64_t)tabid[i] * nint * R6_ROW;
    const double rc2 = g.rcut * g.rcut;
    const float px = (float)sw[0], py = (float)sw[1], pz = (float)sw[2];
    const float hx = (float)cg.h[0], hy = (float)cg.h[1], hz = (float)cg.h[2];
    const float lx = (float)g.boxL[0], ly = (float)g.boxL[1], lz = (float)g.boxL[2];
    const float rt2 = (float)rc2 + slack;            // FP32 test: nothing in range is beyond it
    const int shift_bits = (127 + e0) << 4;          // interval 1 starts at 2^e0
    double acc = 0.0;
    auto eval = [&](int2 q) {
        const double4_32a v = sorted[q.x];
        const double ddx = sw[0] - (v.x + s_per[0][q.y & 31]), ddy = sw[1] - (v.y + s_per[1][(q.y >> 5) & 31]),
                     ddz = sw[2] - (v.z + s_per[2][q.y >> 10]);
        const double s = ddx * ddx + ddy * ddy + ddz * ddz;
        if (s < rc2) {
            const int k = min(max((__float_as_int((float)s) >> 19) - shift_bits + 1, 0), nint - 1);
            const double* row = tb + k * R6_ROW;
            const double t = s - row[R6_DEG + 1];
            double p = row[R6_DEG];
#pragma unroll
            for (int a = R6_DEG - 1; a >= 0; --a) p = fma(p, t, row[a]);
            acc = fma(v.w, p, acc);
        }
    };
    int nq = 0;   // queued charges, warp-uniform
    R6Row* row_ = s_row[warp];
    float4* sh_ = s_sh[warp];
    int2* q_ = s_q[warp];
    const int wy = 2 * cg.S[1] + 1, nrows = wy * (2 * cg.S[2] + 1);
    for (int g0 = 0; g0 < nrows; g0 += 32) {
        const int row = g0 + lane;
        int ux = 0, uxe = -1, fx = 0, fy = 0, fz = 0, base = 0;
        if (row < nrows) {
            const int uy = ci[1] + row % wy - cg.S[1], uz = ci[2] + row / wy - cg.S[2];
            const float dy = fmaxf(0.f, fmaxf((float)uy * hy - py, py - (float)(uy + 1) * hy));
            const float dz = fmaxf(0.f, fmaxf((float)uz * hz - pz, pz - (float)(uz + 1) * hz));
            const float rx2 = rt2 * 1.0001f - dy * dy - dz * dz;
            if (rx2 > 0.f) {
                const float rx = sqrtf(rx2) * 1.0001f + 1e-3f;
                ux = max(ci[0] - cg.S[0], (int)floorf((px - rx) / hx));
                uxe = min(ci[0] + cg.S[0], (int)floorf((px + rx) / hx));
                fx = floordiv(ux, cg.nc[0]);
                fy = floordiv(uy, cg.nc[1]);
                fz = floordiv(uz, cg.nc[2]);
                base = r * cg.ncells + ((uz - fz * cg.nc[2]) * cg.nc[1] + (uy - fy * cg.nc[1])) * cg.nc[0];
            }
        }
        // one image shift along x at a time: lane's run of it, if it has one
        while (__any_sync(0xffffffffu, ux <= uxe)) {
            int b = 0, len = 0;
            if (ux <= uxe) {
                const int last = min(uxe, fx * cg.nc[0] + cg.nc[0] - 1);
                b = start[base + ux - fx * cg.nc[0]];
                len = start[base + last - fx * cg.nc[0] + 1] - b;
                sh_[lane] = make_float4((float)fx * lx, (float)fy * ly, (float)fz * lz,
                                        __int_as_float((fx + R6_F) | (fy + R6_F) << 5 | (fz + R6_F) << 10));
                ux = last + 1;
                ++fx;
            }
            int inc = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += v;
            }
            const int total = __shfl_sync(0xffffffffu, inc, 31);
            row_[lane] = {b, inc - len};
            if (lane == 0) row_[32] = {0, total};
            __syncwarp();
            // charge v of the concatenated runs belongs to run ec: found once, then moved forward
            int ec = 0;
            {
                int hi = 31;
                while (ec < hi) {
                    const int mid = (ec + hi + 1) >> 1;
                    if (row_[mid].pre <= lane) ec = mid; else hi = mid - 1;
                }
            }
            for (int v0 = 0; v0 < total; v0 += 32) {
                const int v = v0 + lane;
                bool keep = false;
                int2 q = make_int2(0, 0);
                if (v < total) {
                    while (row_[ec + 1].pre <= v) ++ec;
                    q.x = row_[ec].beg + (v - row_[ec].pre);
                    const float4 c = sorted32[q.x], sh = sh_[ec];
                    const float ex = px - (c.x + sh.x), ey = py - (c.y + sh.y), ez = pz - (c.z + sh.z);
                    keep = ex * ex + ey * ey + ez * ez < rt2;
                    q.y = __float_as_int(sh.w);
                }
                const unsigned bal = __ballot_sync(0xffffffffu, keep);
                if (keep) q_[nq + __popc(bal & ((1u << lane) - 1u))] = q;
                nq += __popc(bal);
                __syncwarp();
                if (nq >= 32) {   // the last 32 of the queue
                    nq -= 32;
                    const int2 e = q_[nq + lane];
                    __syncwarp();
                    eval(e);
                }
            }
            __syncwarp();
        }
    }
    if (lane < nq) eval(q_[lane]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) out[(int64_t)r * n + i] = acc;
}

cpm_status real64_run(cpm_ctx* c, cudaStream_t st, int m, const CellGrid& cg, const int* start, const void* sorted,
                      const float4* sorted32, double* out, bool chained) {
    // a coordinate and an image shift round to 2^-24 of at most a few box lengths each
    const double lmax = std::max(c->g.boxL[0], std::max(c->g.boxL[1], c->g.boxL[2])) + c->g.rcut;
    const float slack = (float)(4e-6 * c->g.rcut * lmax);
    const unsigned grid = (unsigned)(((int64_t)m * c->n + R6_WARPS - 1) / R6_WARPS);
    auto launch = [&](auto... a) {   // chained: the kernel in front of this one in the stream is all it waits for
        if (chained) return launch_after(k_real64, dim3(grid), dim3(32 * R6_WARPS), 0, st, a...);
        k_real64<<<grid, 32 * R6_WARPS, 0, st>>>(a...);
        return cudaSuccess;
    };
    CPM_CUDA(c, launch(c->sx, c->n, m, c->g, cg, start, (const double4_32a*)sorted, sorted32, c->r64tab, c->r64n, c->r64e0, c->rtab_id,
        slack, out));
    CPM_LAUNCH(c, "k_real64");
    return CPM_OK;
}

}  // namespace cpm
