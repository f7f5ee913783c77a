// FP64 structure factor (stage 1 of recip_rows.cu) by exact integer products on the 5th-generation tensor cores.
//
//   R_r[p][t][c] = sum_j P_tj h_cj,   P_tj = Q_j f_t(x_j, y_j),  |P| < 1 after scaling by a power of two, |h| <= 1.
//
// The FP64 pipe retires two multiply-adds per clock and SM, the tensor cores 4,096 fp16 ones.  Both operands are
// taken in fixed point to 2^-55 and written as eight balanced digits of base 128 (after Ozaki, Ogita, Oishi and
// Rump, Numer. Algorithms 59, 2012: error-free splitting of a matrix product),
//   P = sum_i a_i 128^(7-i) 2^-55,  h = sum_j b_j 128^(7-j) 2^-55,   a_i, b_j integers in [-64, 64],
// exact in fp16.  The 36 products of digits with i + j = w <= 7 are added per w: every product is at most 2^12
// and a sum of at most 8 x 480 of them below 2^24, so the FP32 accumulation in tensor memory is exact, whatever
// its order.  The sums S_w are combined as 64-bit integers, over the charge ranges too, and become FP64 once:
//   R = sum_w S_w 2^(-12 - 7 w).
// What is left out, i + j >= 8, is at most 7 x 2^-56 per product P h, about 2^-53.2 (the seven digit products of order 8;
// random operands 2^-56.2 in the mean square, 2^-53.9 at most), and the fixed-point operands are rounded at 2^-56: errors
// in units of the replica's largest |Q|, where an FP64 multiply-add rounds relative to its own product and to the sum
// so far.  A charge of 10^-6 of the largest keeps 35 bits; next to what the sums over all charges hold, b
// is as far from 80-bit values as with the FP64 pipe (3e-13 on the EDL capacitor).
//
// One CTA: 32 pairs (128 rows) x 32 harmonics (64 functions) x one range of charges in steps of 32.  512 builders form
// the digits: the products Q f_x f_y as the high half of a 64 x 64-bit integer product, two charges at a time
// (fields of 7 bits of both in one register, (1024 + field) - 1088 in packed fp16 gives the digit); digit tiles
// with 64-byte rows (64-byte swizzle).  B digits lie one after the other, so digit i of A meets digits 0 .. 7 - i of B
// in one MMA of up to 256 columns, column block i + j.  One thread issues; two stages of 96 KB; every wait is
// bounded as in tc_recip.cu.
// EDL capacitor, one replica of 5,700 charges: this kernel 31 us and its sum 9, where the FP64 pipe took 571 us for two
// multiply-adds per (charge, k).  What bounds it: forming the digits (96 registers, one CTA per SM by shared memory).
#include <cuda_fp16.h>

#include <algorithm>

#include "common.cuh"
#include "tc_common.cuh"

namespace cpm {

constexpr int R4_DIG = 8;                      // digits
constexpr int R4_PAIRS = ROW64_PAIRS;          // pairs per CTA (4 rows each: MMA M = 128)
constexpr int R4_H = ROW64_HARM;               // harmonics per CTA (64 functions)
constexpr int R4_KC = ROW64_STEP;              // charges per step (64 bytes of fp16 per operand row)
constexpr int R4_RANGE = 15;                   // steps of one range: 480 charges, sums below 2^24
constexpr int R4_GEN = 512, R4_THREADS = R4_GEN + 32;
constexpr int R4_A = 128 * 64;                 // one digit of the A tile
constexpr int R4_B = 64 * 64;                  // one digit of the B tile
constexpr int R4_STAGE = R4_DIG * (R4_A + R4_B);
constexpr int R4_STAGES = 2;
constexpr int R4_SMEM = 1024 + R4_STAGES * R4_STAGE + 256;
constexpr int R4_EMAX = ROW64_EMAX;
constexpr uint64_t R4_WAIT_NS = 2000000000ull;

// byte offset of 16-byte chunk ch of row r in a K-major tile of 64-byte rows, 64-byte swizzle
__device__ __forceinline__ uint32_t sw64(int r, int ch) { return (uint32_t)(r * 64 + ((ch ^ ((r >> 1) & 3)) << 4)); }
// its operand descriptor: 8-row atoms 512 B apart
__device__ __forceinline__ uint64_t sdesc_sw64(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(512 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)4 << 61;
    return d;
}

// (1024 + field) - 1088 for two 7 or 8 bit fields
__device__ __forceinline__ uint32_t digit2(uint32_t fields) {
    const uint32_t u = fields | 0x64006400u, c = 0x64406440u;   // fp16 1024 + field, 1088
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&u), *reinterpret_cast<const __half2*>(&c));
    return *reinterpret_cast<const uint32_t*>(&h);
}

// eight digits (most significant first) of two fixed-point values |v| <= 2^55, packed in pairs
__device__ __forceinline__ void digits8(int64_t v0, int64_t v1, uint32_t (&d)[R4_DIG]) {
    constexpr uint64_t BIAS = 64ull * 0x0002040810204081ull;   // 64 in every base-128 digit, 64 (128^8 - 1) / 127
    const uint64_t u0 = (uint64_t)v0 + BIAS, u1 = (uint64_t)v1 + BIAS;
    const uint32_t l0 = (uint32_t)u0, h0 = (uint32_t)(u0 >> 32), l1 = (uint32_t)u1, h1 = (uint32_t)(u1 >> 32);
    uint32_t w[4];   // 14 bits of each value, the upper ones 15
    w[0] = (l0 & 0x3FFFu) | ((l1 & 0x3FFFu) << 16);
    w[1] = ((l0 >> 14) & 0x3FFFu) | (((l1 >> 14) & 0x3FFFu) << 16);
    w[2] = (__funnelshift_r(l0, h0, 28) & 0x3FFFu) | ((__funnelshift_r(l1, h1, 28) & 0x3FFFu) << 16);
    w[3] = (h0 >> 10) | ((h1 >> 10) << 16);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        d[7 - 2 * p] = digit2(w[p] & 0x007F007Fu);
        d[6 - 2 * p] = digit2((w[p] >> 7) & (p == 3 ? 0x00FF00FFu : 0x007F007Fu));
    }
}

__device__ __forceinline__ void sts32r(uint32_t addr, uint32_t a) {
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(a) : "memory");
}

// part[s][r][4 p + t][c] = (sum_{w < 4} S_w 128^(3 - w), sum_{w >= 4} S_w 128^(7 - w)); R = (2^28 first + second) 2^-61.
// grid items x (m splits), items fastest; an item is (first pair, pairs, first harmonic, harmonics).
// X, Y: slot h of charge j at [h P + j], (cos, sin) times 2^62 (x also times Q and the replica's scale); Z: times 2^55.
__global__ void __launch_bounds__(R4_THREADS, 1)
    k_tc_rows64(const int4* __restrict__ items, const int4* __restrict__ pairs, const longlong2* __restrict__ X,
                const longlong2* __restrict__ Y, const longlong2* __restrict__ Z, int64_t P, int64_t nep, int NZ,
                int nitems, int splits, int spc, int steps, int m, int np, int cw, longlong2* __restrict__ part,
                unsigned* __restrict__ status, uint64_t wait_ns) {
    grid_wait();
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    uint64_t* full = (uint64_t*)(smem + R4_STAGES * R4_STAGE);
    uint64_t* empty = full + R4_STAGES;
    uint64_t* done = empty + R4_STAGES;
    uint32_t* tmem_slot = (uint32_t*)(done + 1);
    volatile int* abort = (volatile int*)(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int bi = blockIdx.x % nitems, br = blockIdx.x / nitems;
    const int4 it = items[bi];
    const int r = br / splits, sp = br % splits;
    const int s0 = sp * spc, nsteps = max(0, min(steps, s0 + spc) - s0);

    if (threadIdx.x == 0) {
        for (int s = 0; s < R4_STAGES; ++s) { mbar_init(&full[s], R4_GEN); mbar_init(&empty[s], 1); }
        mbar_init(done, 1);
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == R4_GEN / 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp < R4_GEN / 32) {
        // builder g: charges 2 cp, 2 cp + 1 of pair pl (A rows t 32 + pl) and of harmonic pl (B rows t 32 + pl)
        const int g = threadIdx.x, cp = g & 15, pl = g >> 4;
        const bool alive = pl < it.y, blive = pl < it.w;   // rows past the last are never read back
        const int4 pr = pairs[it.x + (alive ? pl : 0)];
        const int64_t p0 = (int64_t)r * nep + (int64_t)s0 * R4_KC + 2 * cp;
        const longlong2* xs = X + (int64_t)pr.x * P + p0;
        const longlong2* ys = Y + (int64_t)pr.y * P + p0;
        const longlong2* zs = Z + (int64_t)min(it.z + pl, NZ) * P + p0;
        longlong2 x[2], y[2], z[2], xn[2], yn[2], zn[2];   // of this step and the next
        auto fetch = [&](int t) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                xn[k] = xs[t * R4_KC + k];
                yn[k] = ys[t * R4_KC + k];
                zn[k] = zs[t * R4_KC + k];
            }
        };
        if (nsteps > 0) fetch(0);
        const int ch = cp >> 2, in16 = (cp & 3) * 4;
        bool ok = true;
        for (int t = 0; t < nsteps && ok; ++t) {
            const int s = t % R4_STAGES;
            if (t >= R4_STAGES) ok = mbar_wait(&empty[s], ((t / R4_STAGES) - 1) & 1, abort, wait_ns);
            if (!ok) break;
#pragma unroll
            for (int k = 0; k < 2; ++k) { x[k] = xn[k]; y[k] = yn[k]; z[k] = zn[k]; }
            if (t + 1 < nsteps) fetch(t + 1);
            const uint32_t sa = su32(smem + s * R4_STAGE), sb = sa + R4_DIG * R4_A;
            uint32_t d[R4_DIG];
            if (blive) {
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    digits8(q ? z[0].y : z[0].x, q ? z[1].y : z[1].x, d);
                    const uint32_t o = sb + sw64(q * R4_H + pl, ch) + in16;
#pragma unroll
                    for (int k = 0; k < R4_DIG; ++k) sts32r(o + k * R4_B, d[k]);
                }
            }
            if (alive) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {   // products at 2^60, rounded to 2^55
                    const int64_t a0 = (q & 1) ? x[0].y : x[0].x, b0 = (q & 2) ? y[0].y : y[0].x;
                    const int64_t a1 = (q & 1) ? x[1].y : x[1].x, b1 = (q & 2) ? y[1].y : y[1].x;
                    digits8((__mul64hi(a0, b0) + 16) >> 5, (__mul64hi(a1, b1) + 16) >> 5, d);
                    const uint32_t o = sa + sw64(q * R4_PAIRS + pl, ch) + in16;
#pragma unroll
                    for (int k = 0; k < R4_DIG; ++k) sts32r(o + k * R4_A, d[k]);
                }
            }
            fence_async_smem();
            mbar_arrive(&full[s]);
        }
    } else if (lane == 0) {
        // MMA issuer: per 16-wide K slice digit i of A against digits 0 .. 7 - i of B, four at a time
        for (int t = 0; t < nsteps; ++t) {
            const int s = t % R4_STAGES;
            if (!mbar_wait(&full[s], (t / R4_STAGES) & 1, abort, wait_ns)) break;
            tc_fence_after();
            const uint32_t sa = su32(smem + s * R4_STAGE), sb = sa + R4_DIG * R4_A;
            for (int kk = 0; kk < R4_KC / 16; ++kk)
#pragma unroll
                for (int i = 0; i < R4_DIG; ++i) {
                    const uint64_t a = sdesc_sw64(sa + i * R4_A + kk * 32);
#pragma unroll
                    for (int j = 0; j < R4_DIG - i; j += 4) {
                        const int nd = R4_DIG - i - j < 4 ? R4_DIG - i - j : 4;
                        umma_f16(tmem + 64 * (i + j), a, sdesc_sw64(sb + j * R4_B + kk * 32), idesc_f16(128, 64 * nd),
                                 (t > 0 || kk > 0 || i > 0) ? 1u : 0u);
                    }
                }
            umma_commit(&empty[s]);
        }
        umma_commit(done);   // also after an abort: the epilogue then waits for the MMAs in flight
    }
    if (warp < R4_GEN / 32) {
        // epilogue: warp w reads accumulator lanes 32 (w % 4) .. + 31 (rows t = w % 4 of the pairs), columns 16 (w / 4)
        // .. + 15 of every column block
        const bool ok = mbar_wait(done, 0, abort, wait_ns);
        tc_fence_after();
        const bool good = __all_sync(0xffffffffu, ok && !*abort) != 0;
        if (!good) {
            if (lane == 0) atomicOr(status, ST_TIMEOUT);
        } else {
            const int lq = warp & 3, c16 = 16 * (warp >> 2);
            const uint32_t trow = tmem + ((uint32_t)(lq * 32) << 16) + c16;
            int64_t hi[16], lo[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) hi[k] = lo[k] = 0;
            if (nsteps > 0) {
#pragma unroll
                for (int w = 0; w < R4_DIG; ++w) {
                    float v[16];
                    tmem_ld16(trow + 64 * w, v);
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        const int64_t sv = (int64_t)(int)v[k];   // an integer below 2^24
                        if (w < 4) hi[k] += sv << (7 * (3 - w));
                        else lo[k] += sv << (7 * (7 - w));
                    }
                }
            }
            // row t = lq of pair lane; column n = q 32 + h is function 2 (first harmonic + h) + q
            const int q = c16 >> 5, h0 = c16 & 31;
            if (lane < it.y) {
                longlong2* out = part + ((((int64_t)sp * m + r) * np + it.x + lane) * 4 + lq) * cw;
#pragma unroll
                for (int k = 0; k < 16; ++k)
                    if (h0 + k < it.w) out[2 * (it.z + h0 + k) + q] = make_longlong2(hi[k], lo[k]);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == R4_GEN / 32) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// out[r][4 p + t][c]: the ranges added as integers, then FP64; the replica's scale removed.  A charge that is no
// finite number makes the replica's sums not a number.  grid (pairs, m, 4 rows t); one function per thread
__global__ void __launch_bounds__(128) k_rows64_sum(const int4* __restrict__ pairs, int np, int cw,
                                                    const longlong2* __restrict__ part, int splits, int m,
                                                    const int* __restrict__ qexp, double* __restrict__ out) {
    grid_wait();
    grid_go();
    const int p = blockIdx.x, r = blockIdx.y;
    const int nc = 2 * (pairs[p].z + 1);
    const int64_t stride = (int64_t)m * np * 4 * cw;
    const int qe = qexp[r];
    const double f = qe > R4_EMAX ? nan("") : pow2_bits(max(qe, 1) + 1);
    const int t = blockIdx.z;
    for (int c = threadIdx.x; c < nc; c += 128) {
        const int64_t at = (((int64_t)r * np + p) * 4 + t) * cw + c;
        long long hi = 0, lo = 0;
        for (int s0 = 0; s0 < splits; s0 += 8) {   // eight loads in flight
            longlong2 v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = s0 + k < splits ? part[at + (s0 + k) * stride] : make_longlong2(0, 0);
#pragma unroll
            for (int k = 0; k < 8; ++k) { hi += v[k].x; lo += v[k].y; }
        }
        out[at] = fma((double)hi, 0x1p28, (double)lo) * 0x1p-61 * f;
    }
}

// largest biased exponent of Q per replica (zero before)
__global__ void __launch_bounds__(256) k_qexp(const double* __restrict__ Q, int64_t ne, int* __restrict__ qexp) {
    grid_go();
    const int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x;
    int v = j < ne ? exp_bits(Q[(int64_t)blockIdx.y * ne + j]) : 0;
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0 && v > 0) atomicMax(&qexp[blockIdx.y], v);
}

// ----------------------------------------------------------------------------- host side
Rows64Dims rows64_dims(const cpm_ctx* c, int m, int64_t ne) {
    const RowTable& t = c->rows;
    Rows64Dims d{};
    d.nep = ((ne + R4_KC - 1) / R4_KC) * R4_KC;
    d.cw = ((2 * (c->kt.NZ + 1) + 31) / 32) * 32;
    d.steps = (int)(d.nep / R4_KC);
    // whole waves of CTAs (one per SM) times the steps of a range and about six more for its set-up and epilogue;
    // at most R4_RANGE steps, beyond which the sums would not be exact
    const int64_t base = (int64_t)std::max(1, t.items64) * m;
    const int least = std::max(1, (d.steps + R4_RANGE - 1) / R4_RANGE);
    d.splits = least;
    d.spc = std::max(1, (d.steps + least - 1) / least);
    double best = 1e300;
    for (int s = least; s <= d.steps && s < least + 64; ++s) {
        const int spc = (d.steps + s - 1) / s;
        if ((d.steps + spc - 1) / spc != s) continue;
        if (c->lean && best < 1e300) break;
        const double tt = (double)((base * s + 151) / 152) * (spc + 6);
        if (tt < 0.97 * best) {
            best = tt;
            d.splits = s;
            d.spc = spc;
        }
    }
    // 2 FP64 multiply-adds per (charge, k) at 304 per clock against about 15 us of fixed cost here: 2e7 is 35 us
    // (its partial sums, 16 bytes each, are kept below 128 MiB: beyond that the CUDA cores take the call)
    d.use = c->lean < 2 && t.items64 > 0 && 2.0 * (double)c->kt.nk * (double)ne * m >= 2e7 &&
            sizeof(longlong2) * (size_t)d.splits * m * 4 * t.np * d.cw <= ((size_t)128 << 20);
    return d;
}

cpm_status rows64_sf(cpm_ctx* c, cudaStream_t st, const Rows64Dims& d, int m, const longlong2* X, const longlong2* Y,
                     const longlong2* Z, const int* qexp, longlong2* ipart, double* part) {
    const RowTable& t = c->rows;
    CPM_CUDA(c, cudaFuncSetAttribute(k_tc_rows64, cudaFuncAttributeMaxDynamicSharedMemorySize, R4_SMEM));
    CPM_CUDA(c, launch_after(k_tc_rows64, dim3((unsigned)(t.items64 * (int64_t)m * d.splits)), dim3(R4_THREADS), R4_SMEM, st, 
        t.item64, t.pairs, X, Y, Z, (int64_t)m * d.nep, d.nep, c->kt.NZ, t.items64, d.splits, d.spc, d.steps, m, t.np,
        d.cw, ipart, c->status, R4_WAIT_NS));
    CPM_LAUNCH(c, "k_tc_rows64");
    CPM_CUDA(c, launch_after(k_rows64_sum, dim3(t.np, m, 4), dim3(128), 0, st, t.pairs, t.np, d.cw, ipart, d.splits, m, qexp, part));
    CPM_LAUNCH(c, "k_rows64_sum");
    return CPM_OK;
}

cpm_status launch_qexp(cpm_ctx* c, cudaStream_t st, int m, int64_t ne, const double* Q, int* qexp) {
    k_qexp<<<dim3((unsigned)((ne + 255) / 256), (unsigned)m), 256, 0, st>>>(Q, ne, qexp);
    CPM_LAUNCH(c, "k_qexp");
    return CPM_OK;
}

}  // namespace cpm
