// Reciprocal-space part of the electrolyte vector b on the 5th-generation tensor cores.
//
// Stage 1 (every geometry) is the structure factor in the real product basis of recip_rows.cu,
//   R_r[p][t][c] = sum_j Q_j f_t(x_j, y_j) h_c(z_j),
// a real matrix product over the charges: A = Q f_t (rows 4 pair + part, K = charges), B = h_c (rows c, K =
// charges).  Heights shared by many sites then take the height-wise stages of recip_rows.cu.  For electrodes
// whose sites hardly share heights stage 2 here is a complex product over the harmonics,
//   T_r[c][i] = sum_nz conj(Z_i[nz]) W_r[c][nz],  W_r = w rho_r,
//   b_r[i]   += sum_c Re[ conj(X_i[nx_c] Y_i[ny_c]) T_r[c][i] ]
// over the signed columns c = (nx, ny), with (re, im) interleaved along K and N: A = site phases (rows i, K =
// (nz, re/im)), B rows (c, r, re) = (Wr, Wi), (c, r, im) = (Wi, -Wr); the epilogue contracts over c.
//
// Operand precision: every operand x is scaled by a power of two s (|s x| < 2^14) and split as
// x0 = fp16(s x), x1 = fp16(s x - x0) (22 significant bits); the products x0 y0 + x0 y1 + x1 y0
// are accumulated in FP32 in tensor memory and the scales are removed exactly afterwards.  The
// k_perp = 0 column keeps its double-float treatment (its single-precision weight is zero here).
//
// One thread issues the tcgen05.mma instructions; every mbarrier wait is bounded by wall time and on expiry
// the CTA records ST_TIMEOUT, frees its tensor memory and returns.
#include <cuda_fp16.h>

#include <algorithm>

#include "common.cuh"
#include "tc_common.cuh"

namespace cpm {

constexpr uint64_t RT_WAIT_NS = 2000000000ull;   // bound on any single mbarrier wait: 2 s

// stage 1 (structure factor)
constexpr int RF_PAIRS = ROW_TC_PAIRS;         // pairs per CTA: two row tiles (MMA M = 128) of 32 pairs x 4 parts
constexpr int RF_KC = ROW_TC_STEP;             // charges per K step (64 fp16 = 128 bytes per operand row)
constexpr int RF_GEN = 512;                    // operand-building threads (warps 0-15)
constexpr int RF_THREADS = RF_GEN + 32;        // + the MMA warp
constexpr int RF_TERM = 128 * 128;             // one fp16 term of a 128-row operand tile (16 KB)
constexpr int RF_STAGE = 6 * RF_TERM;          // A: two tiles x two terms, B: two terms (96 KB)
constexpr int RF_STAGES = 2;
constexpr int RF_RANGE = 16;                   // K steps of one accumulation at most
constexpr int RF_SLOTS = ROW_TC_SLOTS + 16;    // staged table rows of a step: x and y harmonics, 8 + 8 z phases
constexpr int RF_PX = (RF_SLOTS + 15) / 16;    // staging entries (16 bytes) per builder
constexpr int RF_SMEM = 1024 + RF_STAGES * RF_STAGE + 1024 + RF_SLOTS * RF_KC * 8;
static_assert(RF_SMEM <= 232448, "shared memory of one CTA");

// stage 2 (site potentials)
constexpr int RS_BM = 128;                     // sites per tile (MMA M)
constexpr int RS_EPI = 8;                      // epilogue warps (two per TMEM lane quarter)
constexpr int RS_THREADS = 32 * (RS_EPI + 2);   // warps 0-7 epilogue, warp 8 TMA, warp 9 MMA
constexpr int RS_TMA_WARP = RS_EPI, RS_MMA_WARP = RS_EPI + 1;
constexpr int RS_A = RS_BM * 128;              // one fp16 term of the site-phase tile (16 KB)
constexpr int RS_BMAX = 256 * 128;             // one fp16 term of the W tile, N <= 256 (32 KB)
constexpr int RS_STAGE = 2 * RS_A + 2 * RS_BMAX;
constexpr int RS_STAGES = 2;
constexpr int RS_SMEM = 1024 + RS_STAGES * RS_STAGE + 256;
constexpr int RS_ZEXP = 14;                    // site phases scaled by 2^14
constexpr int RS_CT = 16;                      // columns per group (N = 2 x 16 x replicas of the group)
constexpr int RS_MR = 8;                       // replicas per group

// (re, im) -> two packed fp16 pairs: hi = fp16(v), lo = fp16(v - hi); low half = re
__device__ __forceinline__ void split2(float2 v, uint32_t& hi, uint32_t& lo) {
    const __half2 h = __floats2half2_rn(v.x, v.y);
    const float2 f = __half22float2(h);
    const __half2 l = __floats2half2_rn(v.x - f.x, v.y - f.y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}
// the same for a packed pair of FP32 values (the pair of charges of one operand word)
__device__ __forceinline__ void split2p(uint64_t v, uint32_t& hi, uint32_t& lo) {
    const float2 x = up2(v);
    const __half2 h = __floats2half2_rn(x.x, x.y);
    const float2 f = __half22float2(h);
    const float2 d = up2(sub2(v, pk2(f.x, f.y)));
    const __half2 l = __floats2half2_rn(d.x, d.y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}
__device__ __forceinline__ uint32_t neg_hi(uint32_t h) { return h ^ 0x80000000u; }            // (a, b) -> (a, -b)
__device__ __forceinline__ uint32_t swap_h(uint32_t h) { return __byte_perm(h, 0u, 0x1032); }  // (a, b) -> (b, a)

// barrier 1 over the RF_GEN operand-building threads; returns the AND of every thread's flag
__device__ __forceinline__ bool gen_bar_and(bool flag) {
    uint32_t out;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "bar.red.and.pred q, 1, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}\n"
        : "=r"(out)
        : "r"((uint32_t)flag), "n"(RF_GEN)
        : "memory");
    return out != 0;
}
__device__ __forceinline__ void gen_bar() { asm volatile("bar.sync 1, %0;" ::"n"(RF_GEN) : "memory"); }

__device__ __forceinline__ void sts128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void sts32(uint32_t addr, uint32_t a) {
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(a) : "memory");
}
// byte offset of 16-byte chunk ch of row r in a K-major tile of 128-byte rows, 128-byte swizzle
__device__ __forceinline__ uint32_t sw128(int r, int ch) { return (uint32_t)(r * 128 + ((ch ^ (r & 7)) << 4)); }

// ----------------------------------------------------------------------------- stage 1
// part[s][r][4 p + t][c] = 2^14 sA_r sum over the K steps of range s of replica r; sA_r = 2^e, |Q| sA_r < 2^14.
// grid items x (m splits), items fastest; an item is (first pair, pairs, harmonic tile, harmonics) and its range of staged
// harmonics (x0, nx, y0, ny).  Per K step of 64 charges the 512 builders stage the x and y harmonics and the z
// phases of the step in shared memory (loads issued one step ahead), then each forms the four rows
// (cos, sin) x (cos, sin) of one pair for eight charges, and eight z functions for two charges (h = 8 a + k as
// a product of two phases), both split into two fp16 terms in 128-byte-swizzled operand tiles.
// The leading products have an accumulator of their own, the cross products another: the tensor core truncates
// the sum at each of its additions, so the error of a long range grows with their number (one accumulator for
// all three and 86 steps: b of a 16-replica 8,192-site batch 9.7e-6 off; RF_RANGE bounds the steps).
// What bounds it: shared memory.  A step moves about 64 KB of operand reads and 96 KB of operand writes by
// the builders and 160 KB of operand reads by the 16 MMAs, at 128 B per clock; real products of pairs need
// half the MMAs and a quarter of the z operand of complex columns over both signs of nz.
__global__ void __launch_bounds__(RF_THREADS, 1)
    k_tc_rows(const int4* __restrict__ items, const int4* __restrict__ ranges, const int4* __restrict__ pairs,
              const float2* __restrict__ tab, int64_t P, int64_t nep, int NX, int NY, int NZ,
              const float* __restrict__ qmax, const int* __restrict__ qlast, int nitems, int splits, int spc, int m, int np,
              int cw, float* __restrict__ part, unsigned* __restrict__ status, uint64_t wait_ns) {
    grid_wait();
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    uint8_t* aux = smem + RF_STAGES * RF_STAGE;
    uint64_t* full = (uint64_t*)aux;
    uint64_t* empty = full + RF_STAGES;
    uint64_t* done = empty + RF_STAGES;
    uint32_t* tmem_slot = (uint32_t*)(done + 1);
    volatile int* abort = (volatile int*)(tmem_slot + 1);
    float4* stg = (float4*)(aux + 1024);           // [slot][32 units of two charges]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int bi = blockIdx.x % nitems, br = blockIdx.x / nitems;
    const int4 it = items[bi];                     // (first pair, pairs, harmonic tile, harmonics)
    const int4 rg = ranges[bi];                    // (x0, nx, y0, ny)
    const int r = br / splits, sp = br % splits;
    const int ntile = it.y > RF_PAIRS / 2 ? 2 : 1;
    const int nused = ((2 * it.w + 15) / 16) * 16;
    const int s0 = sp * spc, nsteps = max(0, min((qlast[r] + RF_KC - 1) / RF_KC, s0 + spc) - s0);

    const int g = threadIdx.x, nxy = rg.y + rg.w;
    // staging: 16-byte unit uu of slots g / 32 + 16 k; sources advance by one step (64 charges) at a time
    const int uu = g & 31;
    const float4* src[RF_PX];
    int dst[RF_PX];
    float4 px[RF_PX];
    float sA = 1.f;
    auto prefetch = [&](int t) {
#pragma unroll
        for (int k = 0; k < RF_PX; ++k)
            if (dst[k] >= 0) px[k] = src[k][t * (RF_KC / 2)];
    };
    if (warp < RF_GEN / 32) {
        sA = pow2_below(qmax[r], 14);
        const int64_t p0 = (int64_t)r * nep + (int64_t)s0 * RF_KC + 2 * uu;
#pragma unroll
        for (int k = 0; k < RF_PX; ++k) {
            const int slot = (g >> 5) + 16 * k;
            int row = 0;
            dst[k] = -1;
            if (slot < rg.y) row = rg.x + slot;
            else if (slot < nxy) row = NX + 1 + rg.z + (slot - rg.y);
            else if (slot < nxy + 8) row = NX + NY + 2 + (slot - nxy);
            else row = NX + NY + 10 + min(8 * it.z + (slot - nxy - 8), NZ / 8);
            // x and y units are permuted so that eight threads of eight charges each read 128 contiguous bytes
            if (slot < nxy) dst[k] = slot * 32 + (uu & 3) * 8 + (uu >> 2);
            else if (slot < nxy + 16) dst[k] = slot * 32 + uu;
            src[k] = reinterpret_cast<const float4*>(tab + (int64_t)row * P + p0);
        }
        if (nsteps > 0) prefetch(0);   // in flight during the set-up below
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < RF_STAGES; ++s) { mbar_init(&full[s], RF_GEN); mbar_init(&empty[s], 1); }
        mbar_init(done, 1);
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == RF_GEN / 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp < RF_GEN / 32) {
        const int ch = g & 7, pl = g >> 3;             // A: charges 8 ch .. 8 ch + 7 of pair pl
        const bool live = pl < it.y;                   // rows past the last pair are never read back
        const int4 pr = live ? pairs[it.x + pl] : make_int4(rg.x, rg.z, 0, 0);
        const float4* xr = stg + (pr.x - rg.x) * 32 + ch;
        const float4* yr = stg + (rg.y + pr.y - rg.z) * 32 + ch;
        const int hq = g >> 5, h0 = 4 * hq;            // B: harmonics h0 .. h0 + 3 of the tile, charges 2 uu, 2 uu + 1
        const float4* zb = stg + (nxy + (h0 & 4)) * 32 + uu;
        const float4* zg = stg + (nxy + 8 + (h0 >> 3)) * 32 + uu;
        for (int t = 0; t < nsteps; ++t) {
            const int s = t % RF_STAGES;
            bool ok = true;
            if (t >= RF_STAGES) ok = mbar_wait(&empty[s], ((t / RF_STAGES) - 1) & 1, abort, wait_ns);
            if (!gen_bar_and(ok)) break;   // uniform; also: everyone is done reading the staged step t - 1
#pragma unroll
            for (int k = 0; k < RF_PX; ++k) {
                if (dst[k] < 0) continue;
                // (cos, cos, sin, sin) of the two charges: operands of packed arithmetic
                const float f = (g >> 5) + 16 * k < rg.y ? sA : 1.f;
                stg[dst[k]] = make_float4(px[k].x * f, px[k].z * f, px[k].y * f, px[k].w * f);
            }
            gen_bar();   // the staged rows of step t are complete
            if (t + 1 < nsteps) prefetch(t + 1);
            const uint32_t sa = su32(smem + s * RF_STAGE);
            if (h0 < it.w) {
                const uint32_t sb = sa + 4 * RF_TERM + 4 * (uu & 3), sl = sb + nused * 128;
                const float4 gz = *zg;
                const uint64_t gc = pk2(gz.x, gz.y), gs = pk2(gz.z, gz.w), ngs = pk2(-gz.z, -gz.w);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float4 bz = zb[k * 32];
                    const uint64_t bc = pk2(bz.x, bz.y), bs = pk2(bz.z, bz.w);
                    uint32_t h, l;
                    const int row = 2 * (h0 + k);
                    if (row >= nused) break;   // the rows above belong to the second term
                    split2p(fma2(ngs, bs, mul2(gc, bc)), h, l);
                    const uint32_t o0 = sw128(row, uu >> 2);
                    sts32(sb + o0, h);
                    sts32(sl + o0, l);
                    split2p(fma2(gs, bc, mul2(gc, bs)), h, l);
                    const uint32_t o1 = sw128(row + 1, uu >> 2);
                    sts32(sb + o1, h);
                    sts32(sl + o1, l);
                }
            }
            if (live) {
                const uint32_t at = sa + (pl >> 5) * 2 * RF_TERM;
                const int row = (pl & 31) * 4;
                uint32_t h[4][4], l[4][4];   // [part][unit of two charges]
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float4 x = xr[u * 8], y = yr[u * 8];
                    const uint64_t xc = pk2(x.x, x.y), xs = pk2(x.z, x.w), yc = pk2(y.x, y.y), ys = pk2(y.z, y.w);
                    split2p(mul2(xc, yc), h[0][u], l[0][u]);
                    split2p(mul2(xs, yc), h[1][u], l[1][u]);
                    split2p(mul2(xc, ys), h[2][u], l[2][u]);
                    split2p(mul2(xs, ys), h[3][u], l[3][u]);
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t o = sw128(row + q, ch);
                    sts128(at + o, h[q][0], h[q][1], h[q][2], h[q][3]);
                    sts128(at + RF_TERM + o, l[q][0], l[q][1], l[q][2], l[q][3]);
                }
            }
            fence_async_smem();
            mbar_arrive(&full[s]);
        }
    } else if (lane == 0) {
        // MMA issuer: per 16-wide K slice and row tile A0 [B0 B1] (the terms of B one after the other: columns
        // 0 .. nused - 1 the leading products, nused .. 2 nused - 1 the cross ones) and A1 B0 on the latter
        const uint32_t id1 = idesc_f16(128, nused), id2 = idesc_f16(128, 2 * nused);
        for (int t = 0; t < nsteps; ++t) {
            const int s = t % RF_STAGES;
            if (!mbar_wait(&full[s], (t / RF_STAGES) & 1, abort, wait_ns)) break;
            tc_fence_after();
            const uint32_t sa = su32(smem + s * RF_STAGE), sb = sa + 4 * RF_TERM;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                const uint64_t b0 = sdesc_sw128(sb + kk * 32);
                for (int q = 0; q < ntile; ++q) {
                    const uint32_t at = sa + q * 2 * RF_TERM + kk * 32, acc = tmem + 256 * q;
                    umma_f16(acc, sdesc_sw128(at), b0, id2, (t > 0 || kk > 0) ? 1u : 0u);
                    umma_f16(acc + nused, sdesc_sw128(at + RF_TERM), b0, id1, 1u);
                }
            }
            umma_commit(&empty[s]);
        }
        umma_commit(done);   // also after an abort: the epilogue then waits for the MMAs in flight
    }
    if (warp < RF_GEN / 32) {
        // epilogue: warp w reads accumulator lanes 32 (w % 4) .. + 31 of row tile (w / 4) % 2, columns
        // 16 (w / 8) + 32 i: sixteen harmonic functions of one row per thread
        const bool ok = mbar_wait(done, 0, abort, wait_ns);
        tc_fence_after();
        const bool good = __all_sync(0xffffffffu, ok && !*abort) != 0;
        const int lq = warp & 3, tile = (warp >> 2) & 1;
        if (!good) {
            if (lane == 0) atomicOr(status, ST_TIMEOUT);
        } else if (tile < ntile) {
            const int row = tile * 128 + lq * 32 + lane;
            const uint32_t trow = tmem + 256 * tile + ((uint32_t)(lq * 32) << 16);
            float* out = part + (((int64_t)sp * m + r) * np + it.x) * 4 * cw + (int64_t)row * cw + it.z * 128;
            for (int q0 = 16 * (warp >> 3); q0 < nused; q0 += 32) {
                float v[16];
                if (nsteps > 0) {
                    float lo[16];
                    tmem_ld16(trow + q0, v);
                    tmem_ld16(trow + nused + q0, lo);
#pragma unroll
                    for (int k = 0; k < 16; ++k) v[k] += lo[k];
                } else {
#pragma unroll
                    for (int k = 0; k < 16; ++k) v[k] = 0.f;
                }
                if ((row >> 2) < it.y) {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        *reinterpret_cast<float4*>(out + q0 + 4 * k) = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == RF_GEN / 32) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// qsum[r] = sum |Q| of replica r, the scale of the site stage: one block each, a fixed order
__global__ void __launch_bounds__(1024) k_qsum_abs(const double* __restrict__ Q, int64_t ne, float* __restrict__ qsum) {
    __shared__ float ss[32];
    const int r = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float sum = 0.f;
    for (int64_t j0 = threadIdx.x; j0 < ne; j0 += 8 * 1024) {   // eight loads in flight
        float q[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) q[k] = j0 + 1024 * k < ne ? (float)Q[(int64_t)r * ne + j0 + 1024 * k] : 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) sum += fabsf(q[k]);
    }
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) ss[warp] = sum;
    __syncthreads();
    if (warp == 0) {
        sum = ss[lane];
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) qsum[r] = sum;
    }
}

// ----------------------------------------------------------------------------- between the stages
// W planes (two fp16 terms) of the site stage from the weighted structure factor w rho of the signed columns:
// row (group g, pair p, re) = (Wr, Wi) and row (.., im) = (Wi, -Wr) at K = 2 zi, 2 zi + 1, scaled by
// sW_r = 2^e with wmax (sum |Q|) sW_r < 2^14.
// Groups hold CT columns x mr replicas: g = (r / mr) ncb + c / CT, p = (r % mr) CT + c % CT.
// One block transposes a 32-harmonic x 32-column tile of one replica slot.
__global__ void __launch_bounds__(1024)
    k_tc_wsplit(const float2* __restrict__ wrho, int m, int nzw, int ncols, const float* __restrict__ qsum, float wmax,
                int CT, int mr, int ncb, int NB, int KZ, uint32_t* __restrict__ w16, int64_t plane_words) {
    grid_wait();
    __shared__ float2 tile[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int zb = blockIdx.x * 32, cb0 = blockIdx.y * 32, rp = blockIdx.z;
    {
        const int zi = zb + tx, c = cb0 + ty;
        float2 W = make_float2(0.f, 0.f);
        if (rp < m && c < ncols && zi < nzw) {
            const float f = pow2_below(wmax * qsum[rp], 14);
            const float2 v = wrho[((int64_t)rp * ncols + c) * nzw + zi];
            W = make_float2(v.x * f, v.y * f);
        }
        tile[tx][ty] = W;
    }
    __syncthreads();
    const int rb = rp / mr, rr = rp % mr;
    const int kw = KZ / 2;
    const int c = cb0 + ty, zi = zb + tx;
    if (c >= ncb * CT || zi >= kw) return;
    const int64_t row = (int64_t)(rb * ncb + c / CT) * NB + 2 * (rr * CT + c % CT);
    uint32_t h, l;
    split2(tile[tx][ty], h, l);
    const int64_t w0 = row * kw + zi;
    w16[w0] = h;
    w16[w0 + kw] = neg_hi(swap_h(h));
    w16[plane_words + w0] = l;
    w16[plane_words + w0 + kw] = neg_hi(swap_h(l));
}

// ----------------------------------------------------------------------------- stage 2
struct SiteMaps {
    CUtensorMap a[2];
    CUtensorMap b[2];
};

// K steps (64 wide) covering the harmonics zi in [NZ - mx, NZ + mx] of column group g (two K entries
// per harmonic), mx = the largest harmonic extent of the group's columns; nsteps = 0 for no column
__device__ __forceinline__ void site_group_steps(const int* __restrict__ colext, int ncols, int NZ, int g, int ncb,
                                                 int& t0, int& nsteps) {
    const int cb = g % ncb;
    const int cfirst = cb * RS_CT, clast = min(ncols, cfirst + RS_CT);
    int mx = -1;
    for (int c = cfirst; c < clast; ++c) mx = max(mx, colext[c]);
    t0 = mx >= 0 ? (2 * (NZ - mx)) / 64 : 0;
    nsteps = mx >= 0 ? (2 * (NZ + mx + 1) + 63) / 64 - t0 : 0;
}

// partial[r][cb][i] = sum over the 16 columns of block cb of Re[conj(X_i Y_i) T_r[c][i]]
// Persistent: CTA b takes the tiles tau = b, b + gridDim.x, ... of the (site tile, group) grid, in
// group-major order (groups of low |k_perp| have the most harmonics and come first); group g holds
// mr <= 8 replicas x 16 columns.  Two accumulators in tensor memory (columns 256 buf + 32 rr + 2 cc
// + {re, im}): the epilogue warps read tile k from one while the MMA thread fills the other with
// tile k + 1; tfull[buf] / tempty[buf] hand the buffers over.
__global__ void __launch_bounds__(RS_THREADS, 1)
    k_tc_site(const __grid_constant__ SiteMaps maps, const int* __restrict__ colext, int ncols, int NZ,
              int mr, int ncb, int NB, int m, int ntx, int ntiles, const float2* __restrict__ XY, int64_t n,
              const float* __restrict__ qsum, float wmax, float* __restrict__ partial,
              unsigned* __restrict__ status, uint64_t wait_ns) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    uint64_t* full = (uint64_t*)(smem + RS_STAGES * RS_STAGE);
    uint64_t* empty = full + RS_STAGES;
    uint64_t* tfull = empty + RS_STAGES;
    uint64_t* tempty = tfull + 2;
    uint64_t* done = tempty + 2;
    uint32_t* tmem_slot = (uint32_t*)(done + 1);
    volatile int* abort = (volatile int*)(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < RS_STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&tfull[b], 1); mbar_init(&tempty[b], RS_EPI); }
        mbar_init(done, 1);
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == RS_MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    grid_wait();   // what is above touches nothing that another kernel writes
    const uint32_t stage_bytes = 2 * RS_A + 2 * NB * 128;

    if (warp == RS_TMA_WARP && lane == 0) {
        // TMA producer: one ring over the K steps of all this CTA's tiles
        int it = 0;
        for (int tau = blockIdx.x; tau < ntiles && !*abort; tau += gridDim.x) {
            const int g = tau / ntx, tx = tau % ntx;
            int t0, nsteps;
            site_group_steps(colext, ncols, NZ, g, ncb, t0, nsteps);
            for (int t = 0; t < nsteps; ++t, ++it) {
                const int s = it % RS_STAGES;
                if (it >= RS_STAGES && !mbar_wait(&empty[s], ((it / RS_STAGES) - 1) & 1, abort, wait_ns)) break;
                uint8_t* st = smem + s * RS_STAGE;
                mbar_expect_tx(&full[s], stage_bytes);
                const int kx = (t0 + t) * 64;
                tma_load_2d(st, &maps.a[0], kx, tx * RS_BM, &full[s]);
                tma_load_2d(st + RS_A, &maps.a[1], kx, tx * RS_BM, &full[s]);
                tma_load_2d(st + 2 * RS_A, &maps.b[0], kx, g * NB, &full[s]);
                tma_load_2d(st + 2 * RS_A + RS_BMAX, &maps.b[1], kx, g * NB, &full[s]);
            }
        }
        if (*abort) {
            // let the copies still in flight land (bounded): only the last RS_STAGES issued steps can be
            for (int t = max(0, it - RS_STAGES); t < it; ++t) {
                const int s = t % RS_STAGES;
                const uint64_t ts = gtimer_ns();
                while (!mbar_try(&full[s], (t / RS_STAGES) & 1) && gtimer_ns() - ts < wait_ns) {}
            }
        }
    } else if (warp == RS_MMA_WARP && lane == 0) {
        // MMA issuer
        const uint32_t idesc = idesc_f16(RS_BM, NB);
        int it = 0, k = 0;
        for (int tau = blockIdx.x; tau < ntiles; tau += gridDim.x, ++k) {
            const int g = tau / ntx;
            int t0, nsteps;
            site_group_steps(colext, ncols, NZ, g, ncb, t0, nsteps);
            const int buf = k & 1;
            if (k >= 2 && !mbar_wait(&tempty[buf], ((k >> 1) - 1) & 1, abort, wait_ns)) break;
            tc_fence_after();
            const uint32_t acc = tmem + (uint32_t)(256 * buf);
            bool ok = true;
            for (int t = 0; t < nsteps; ++t, ++it) {
                const int s = it % RS_STAGES;
                if (!mbar_wait(&full[s], (it / RS_STAGES) & 1, abort, wait_ns)) { ok = false; break; }
                tc_fence_after();
                const uint32_t sa = su32(smem + s * RS_STAGE), sb = sa + 2 * RS_A;
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const uint64_t a0 = sdesc_sw128(sa + kk * 32), a1 = sdesc_sw128(sa + RS_A + kk * 32);
                    const uint64_t b0 = sdesc_sw128(sb + kk * 32), b1 = sdesc_sw128(sb + RS_BMAX + kk * 32);
                    umma_f16(acc, a0, b0, idesc, (t > 0 || kk > 0) ? 1u : 0u);
                    umma_f16(acc, a0, b1, idesc, 1u);
                    umma_f16(acc, a1, b0, idesc, 1u);
                }
                umma_commit(&empty[s]);
            }
            if (!ok) break;
            umma_commit(&tfull[buf]);
        }
        umma_commit(done);   // also after an abort: the MMAs in flight complete before the dealloc
        const uint64_t ts = gtimer_ns();
        while (!mbar_try(done, 0) && gtimer_ns() - ts < wait_ns) {}
    } else if (warp < RS_EPI) {
        // epilogue: thread = site i of the tile, accumulator lane (warp % 4) * 32 + lane; warp w takes
        // the replicas of parity w / 4 of the group
        const int lq = warp & 3, rpar = warp >> 2;
        const uint32_t trow = (uint32_t)(lq * 32) << 16;
        const float zinv = ldexpf(1.f, -RS_ZEXP);
        int k = 0;
        for (int tau = blockIdx.x; tau < ntiles; tau += gridDim.x, ++k) {
            const int g = tau / ntx, tx = tau % ntx;
            const int rb = g / ncb, cb = g % ncb;
            const int cfirst = cb * RS_CT, clast = min(ncols, cfirst + RS_CT);
            int t0, nsteps;
            site_group_steps(colext, ncols, NZ, g, ncb, t0, nsteps);
            const int64_t i = (int64_t)tx * RS_BM + lq * 32 + lane;
            float2 xy[RS_CT];   // the column factors of this thread's site, loaded while the products run
#pragma unroll
            for (int u = 0; u < RS_CT; ++u) {
                const int c = cfirst + u;
                xy[u] = (c < clast && i < n) ? XY[(int64_t)c * n + i] : make_float2(0.f, 0.f);
            }
            const int buf = k & 1;
            const bool ok = mbar_wait(&tfull[buf], (k >> 1) & 1, abort, wait_ns);
            tc_fence_after();
            if (__any_sync(0xffffffffu, !ok || *abort)) break;
            for (int rr = rpar; rr < mr; rr += RS_EPI / 4) {
                float v[2 * RS_CT];
                if (nsteps > 0) {
                    tmem_ld32(tmem + trow + (uint32_t)(256 * buf + 2 * RS_CT * rr), v);
                } else {
#pragma unroll
                    for (int q = 0; q < 2 * RS_CT; ++q) v[q] = 0.f;
                }
                float sacc = 0.f;
#pragma unroll
                for (int u = 0; u < RS_CT; ++u) {
                    sacc = fmaf(xy[u].x, v[2 * u], sacc);
                    sacc = fmaf(xy[u].y, v[2 * u + 1], sacc);
                }
                const int r = rb * mr + rr;
                if (r < m && i < n)
                    partial[((int64_t)r * ncb + cb) * n + i] = sacc * (zinv / pow2_below(wmax * qsum[r], 14));
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[buf]);
        }
        if (*abort && threadIdx.x == 0) atomicOr(status, ST_TIMEOUT);
    }
    tc_fence_before();
    __syncthreads();
    if (*abort && threadIdx.x == 0) atomicOr(status, ST_TIMEOUT);
    if (warp == RS_MMA_WARP) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// ----------------------------------------------------------------------------- fixed site operands
// a[q][i][2 zi + {0,1}] = term q of 2^14 (Re, Im) Z_i[zi], split in FP64; zero padding rows/columns
__global__ void k_tc_site_a(const double2* __restrict__ Zs, int64_t n, int64_t npad, int nzw, int KZ,
                            uint32_t* __restrict__ a) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int kw = KZ / 2;
    if (t >= npad * kw) return;
    const int64_t i = t / kw;
    const int zi = (int)(t % kw);
    const double2 z = (i < n && zi < nzw) ? Zs[(int64_t)zi * n + i] : make_double2(0.0, 0.0);
    const double zr = ldexp(z.x, RS_ZEXP), zm = ldexp(z.y, RS_ZEXP);
    const __half hr = __double2half(zr), hm = __double2half(zm);
    const __half lr = __double2half(zr - (double)__half2float(hr)), lm = __double2half(zm - (double)__half2float(hm));
    const __half2 h = __halves2half2(hr, hm), l = __halves2half2(lr, lm);
    a[t] = *reinterpret_cast<const uint32_t*>(&h);
    a[npad * kw + t] = *reinterpret_cast<const uint32_t*>(&l);
}

// xy[c][i] = X_i[nx_c] Y_i[ny_c] (FP64 product, rounded once)
__global__ void k_tc_site_xy(const double2* __restrict__ SX, const double2* __restrict__ SY,
                             const int2* __restrict__ cols, int ncols, int NY, int64_t n, float2* __restrict__ xy) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)ncols * n) return;
    const int c = (int)(t / n);
    const int64_t i = t % n;
    const int2 cn = cols[c];
    const double2 x = SX[(int64_t)cn.x * n + i], y = SY[(int64_t)(cn.y + NY) * n + i];
    xy[t] = make_float2((float)(x.x * y.x - x.y * y.y), (float)(x.x * y.y + x.y * y.x));
}

// ----------------------------------------------------------------------------- host side
TcRecipDims tc_recip_dims(const cpm_ctx* c, int m, int64_t ne) {
    const KTable& k = c->kt;
    TcRecipDims d;
    d.nep = ((ne + RF_KC - 1) / RF_KC) * RF_KC;
    d.cw = ((2 * (k.NZ + 1) + 31) / 32) * 32;
    // charge ranges: the fewest K steps one after the other (whole waves of CTAs, one per SM, times the
    // steps of a range and about three more for its set-up and epilogue); every extra range is written and
    // read back, so it has to gain 3 %
    const int64_t steps = std::max<int64_t>(1, d.nep / RF_KC), base = (int64_t)std::max(1, c->rows.tcitems) * m;
    d.splits = (int)((steps + RF_RANGE - 1) / RF_RANGE);
    d.spc = RF_RANGE;
    double best = 1e300;
    for (int s = (int)((steps + RF_RANGE - 1) / RF_RANGE); s <= steps && s <= (int)((steps + RF_RANGE - 1) / RF_RANGE) + 64; ++s) {
        const int64_t spc = (steps + s - 1) / s, used = (steps + spc - 1) / spc;
        if (used != s) continue;
        if (c->lean && best < 1e300) break;
        const double t = (double)((base * s + 151) / 152) * (double)(spc + 3);
        if (t < 0.97 * best) {
            best = t;
            d.splits = s;
            d.spc = (int)spc;
        }
    }
    d.mr = std::min(m, RS_MR);
    d.nrb = (m + d.mr - 1) / d.mr;
    d.CT = RS_CT;
    d.ncb = (k.ncols + d.CT - 1) / d.CT;
    d.NB = 2 * d.CT * d.mr;
    d.ngroups = d.nrb * d.ncb;
    d.KZ = ((2 * k.nzw + 63) / 64) * 64;
    d.npad = ((c->n + RS_BM - 1) / RS_BM) * RS_BM;
    return d;
}

size_t tc_recip_w16_bytes(const TcRecipDims& d) { return 2 * sizeof(uint16_t) * (size_t)d.ngroups * d.NB * d.KZ; }

// site operands that stay fixed with the geometry: phase planes and column factors X_i Y_i
cpm_status tc_recip_prepare(cpm_ctx* c) {
    const KTable& k = c->kt;
    dev_free(c, c->tcz);
    dev_free(c, c->tcxy);
    c->tcz = nullptr;
    c->tcxy = nullptr;
    const TcRecipDims d = tc_recip_dims(c, 1, 0);
    const int64_t n = c->n;
    CPM_TRY(dev_alloc(c, &c->tcz, sizeof(uint16_t) * 2 * (size_t)d.npad * d.KZ));
    CPM_TRY(dev_alloc(c, (void**)&c->tcxy, sizeof(float2) * (size_t)k.ncols * n));
    const int64_t ta = d.npad * (d.KZ / 2);
    k_tc_site_a<<<(unsigned)((ta + 255) / 256), 256, 0, c->stream>>>(c->site64.Z, n, d.npad, k.nzw, d.KZ,
                                                                    (uint32_t*)c->tcz);
    CPM_LAUNCH(c, "k_tc_site_a");
    const int64_t tx = (int64_t)k.ncols * n;
    k_tc_site_xy<<<(unsigned)((tx + 255) / 256), 256, 0, c->stream>>>(c->site64.X, c->site64.Y, k.cols, k.ncols, k.NY,
                                                                     n, c->tcxy);
    CPM_LAUNCH(c, "k_tc_site_xy");
    // bound on the weights: w_k <= (8 pi / V) / |k|^2 <= (8 pi / V) / k_min^2
    double kmin2 = 1e300;
    for (int a = 0; a < 3; ++a) {
        const double kk = 2.0 * PI * c->g.inv[a];
        kmin2 = std::min(kmin2, kk * kk);
    }
    c->tc_wmax = (float)(1.01 * 8.0 * PI / c->g.V / kmin2);
    return CPM_OK;
}

cpm_status tc_recip_scales(cpm_ctx* c, cudaStream_t st, int m, int64_t ne, const double* Q, float* qsum) {
    k_qsum_abs<<<m, 1024, 0, st>>>(Q, ne, qsum);
    CPM_LAUNCH(c, "k_qsum_abs");
    return CPM_OK;
}

cpm_status tc_recip_sf(cpm_ctx* c, cudaStream_t st, const TcRecipDims& d, int m, const float2* tab, const float* qmax,
                       const int* qlast, float* part, bool chained) {
    const KTable& k = c->kt;
    const RowTable& t = c->rows;
    CPM_CUDA(c, cudaFuncSetAttribute(k_tc_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, RF_SMEM));
    const dim3 grid((unsigned)(t.tcitems * (int64_t)m * d.splits));
    auto launch = [&](auto... a) {   // chained: the kernel in front of this one in the stream is all it waits for
        if (chained) return launch_after(k_tc_rows, grid, dim3(RF_THREADS), RF_SMEM, st, a...);
        k_tc_rows<<<grid, RF_THREADS, RF_SMEM, st>>>(a...);
        return cudaSuccess;
    };
    CPM_CUDA(c, launch(t.tcitem, t.tcrange, t.pairs, tab, (int64_t)m * d.nep, d.nep, k.NX, k.NY, k.NZ, qmax, qlast, t.tcitems,
                       d.splits, d.spc, m, t.np, d.cw, part, c->status, RT_WAIT_NS));
    CPM_LAUNCH(c, "k_tc_rows");
    return CPM_OK;
}

cpm_status tc_recip_sites(cpm_ctx* c, cudaStream_t st, const TcRecipDims& d, int m, const float2* wrho,
                          const float* qsum, void* w16, float* site_partial) {
    const KTable& k = c->kt;
    const int64_t n = c->n;
    if (!c->tcz || !c->tcxy) return set_err(c, CPM_E_STATE, "tensor-core reciprocal operands not prepared");
    const int64_t plane_words = (int64_t)d.ngroups * d.NB * (d.KZ / 2);
    dim3 gw((unsigned)((d.KZ / 2 + 31) / 32), (unsigned)((d.ncb * d.CT + 31) / 32), (unsigned)(d.nrb * d.mr));
    CPM_CUDA(c, launch_after(k_tc_wsplit, gw, dim3(1024), 0, st, wrho, m, k.nzw, k.ncols, qsum, c->tc_wmax, d.CT, d.mr, d.ncb,
                             d.NB, d.KZ, (uint32_t*)w16, plane_words));
    CPM_LAUNCH(c, "k_tc_wsplit");
    SiteMaps maps;
    const uint16_t* za = (const uint16_t*)c->tcz;
    const uint16_t* wb = (const uint16_t*)w16;
    for (int q = 0; q < 2; ++q) {
        if (!make_map(&maps.a[q], za + (size_t)q * d.npad * d.KZ, d.npad, d.KZ, RS_BM, CU_TENSOR_MAP_DATA_TYPE_FLOAT16) ||
            !make_map(&maps.b[q], wb + (size_t)q * d.ngroups * d.NB * d.KZ, (int64_t)d.ngroups * d.NB, d.KZ, d.NB,
                      CU_TENSOR_MAP_DATA_TYPE_FLOAT16))
            return set_err(c, CPM_E_CUDA, "cuTensorMapEncodeTiled failed");
    }
    CPM_CUDA(c, cudaFuncSetAttribute(k_tc_site, cudaFuncAttributeMaxDynamicSharedMemorySize, RS_SMEM));
    const int ntx = (int)(d.npad / RS_BM), ntiles = ntx * d.ngroups;
    CPM_CUDA(c, launch_after(k_tc_site, dim3((unsigned)std::min(ntiles, 152)), dim3(RS_THREADS), RS_SMEM, st,
        maps, k.colext, k.ncols, k.NZ, d.mr, d.ncb, d.NB, m, ntx, ntiles, c->tcxy, n, qsum, c->tc_wmax, site_partial,
        c->status, RT_WAIT_NS));
    CPM_LAUNCH(c, "k_tc_site");
    return CPM_OK;
}

}  // namespace cpm
