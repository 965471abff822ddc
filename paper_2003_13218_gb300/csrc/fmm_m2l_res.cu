// fmm_m2l_res.cu -- the FP64 path's M2L (Eq. Lcoeffdef) as exact residue products on the tensor cores.
//
// GB300 issues 2 FP64 operations per SM and clock, so the CUDA-core M2L (2 (p+1)^4 flop per source and target)
// is bound by that pipe: 1.29 s per evaluation of 100,000 charges at p = 12, and far more than its flops at small
// sizes, whose levels fill a few SMs.  The 16-bit tensor pipe is ~1,500 times as fast.  The products are therefore
// taken in whole numbers, exactly, modulo 11 to 15 small coprime numbers (the Chinese remainder theorem; its use
// for matrix products on low-precision units is the "Ozaki scheme II" of Ozaki, Uchino & Imamura, 2025):
//   * moments and operators are balanced as in the mixed path, M~ = M^ s(n,m), T~ = T / (s s), |T~| <= 1/2, and
//     rounded to whole numbers, M_int = round(M~ 2^g) with |M_int| < 2^B (g from the level's largest |M~|) and
//     T_int = round(T~ 2^C): B = 56 to 58, as the moduli allow, C = 56, or 58 at ws = 2 and up to order 3;
//   * a whole number has the level's exponent, a double its own.  A target whose sources are all more than 2^(B - K)
//     below the level's largest (far from a dominant charge) therefore takes the FP64 sum instead (k_res_low).  K = 54,
//     53 from order 3, 52 from 5 and 51 from 12 on, where the FP64 sum rounds more: with one source in a list right at that
//     line, the worst case, the gradients of the potential err by 0.5 to 0.95 times as much as with the FP64 sum and the
//     potentials by 0.1 to 1.0 times (p = 0 to 12, against 64-bit mantissas); with 40 sources of the same size by 0.1;
//   * sum_delta sum_k |T_int| <= 137 2^C (ws = 1) or 277 2^C (ws = 2), whatever the order, so |L_int| < 2^(B + C + 7.2)
//     or 2^(B + C + 8.2), and it follows from its residues modulo p_1 .. p_n with prod p_i above twice that;
//   * residues are centred, |r| <= p/2, exact in fp16; a product of two is a whole number, and a chain of G = 2
//     offsets sums 2 (p+1)^2 of them: with 2 (p+1)^2 (p/2)^2 <= 2^24 the FP32 accumulator is exact.  The drained
//     accumulators are added up as 32-bit integers (fmm_tc.cuh);
//   * the operator residues carry the factor (P / p_i)^-1 mod p_i, so the results y_i give
//     L_int / P = sum_i y_i / p_i mod 1 directly: a 96-bit fixed-point sum, good to 2^-83 P.
// Orders above 15 (more than 256 coefficients) stay on the CUDA cores.
//
// Measured (energy, forces and solute-solvent energy, FP64 CUDA cores -> residues): 100,000 charges at depth 5,
// p = 12 1,290 -> 12.4 ms (M2L kernels 1,283 -> 6.0 ms; now 4.7 of a call's 7.0); 2,998 charges at depth 3, p = 8 581 ->
// 1.6 ms, now 0.51; the lists of targets that take the FP64 sum cost 5 to 40 us of these calls.  Forces
// against the same sums in 80-bit arithmetic: 3.7e-16 relative (FP64 sums 7.2e-16) at 1,000 charges, p = 8;
// 4.9e-16 (5.4e-16) at 2,998, p = 4; 7.4e-15 (7.5e-15, the operator tables' own rounding) at p = 12.  The field at each
// charge against the whole method in 80-bit arithmetic, median of the relative errors, twelve boxes of 30 to 6,000
// charges, p = 1 to 12, ws = 1 and 2: 2.3e-16 to 8.1e-16 (FP64 sums 6.4e-16 to 1.1e-14); of these with one charge 1e6
// times the others, d = 5, p = 3: 5.9e-16 (FP64 sums 2.8e-15, whole numbers without k_res_low 3.7e-15).
#include <math.h>
#include <string.h>

#include <new>

#include "fmm_tc.cuh"

namespace fmm {

namespace {

constexpr int RES_MAX = 16;        // moduli
constexpr int RES_CHAIN = 2;       // offsets per accumulator (G)
constexpr int RES_M_BITS = 56, RES_M_BITS_MAX = 58;  // |M_int| < 2^B, B as the moduli allow
static_assert(RES_M_BITS_MAX < 63 && RES_M_BITS_MAX >= RES_M_BITS, "whole numbers of 64 bits");
constexpr int JOIN_THREADS = 256;

struct ResConsts {
    int n;
    int p[RES_MAX], c18[RES_MAX], c36[RES_MAX];  // modulus, 2^18 and 2^36 modulo it (centred)
    int inv[RES_MAX];                            // (P / p_i)^-1 mod p_i, centred
    float rp[RES_MAX];
    uint32_t w[RES_MAX][3];                      // floor(2^96 / p_i), low word first
    double pscale;                               // P / 2^(96 + C)
    int mbits, tbits, keep;                      // B, C, K
};

struct ResState {
    ResConsts c;
    int npad = 0, kp = 0, noff = 0;
    uint16_t *ops = nullptr;      // [modulus][chunk][slot][npad][64]
    size_t ops_elems = 0;         // per modulus
    bool ops_borrowed = false;
    uint16_t *planes = nullptr;   // [modulus of the launch][chunk][class][hz][hy][hx][64], one level at a time
    int16_t *resid = nullptr;     // [group][modulus of the launch][cell][nc]
    uint32_t *frac = nullptr;     // [3][cells nc] 96-bit sums between the launches of a level
    TcMaps maps[9];
    CUtensorMap mapB2[2];         // S, C of half operator tiles (CTA pairs)
    int batch[9];                 // moduli per launch of a level
    int bx[9], by[9], bz[9], groups[9], per_group[9];
    double *s64 = nullptr;        // [nc] s(n,m); amax, cmax, low and mods are in its allocation
    unsigned long long *amax = nullptr;  // [9] bits of the largest |M^ s| per level
    uint32_t *cmax = nullptr;            // the same per cell, upper words, levels 1 .. d behind one another
    uint32_t *low = nullptr;             // targets that take the FP64 sum (numbered as in cmax)
    int *low_count = nullptr;            // behind amax: their count, then [LOW_CELLS] blocks done
    int low_cells = 0;                   // targets whose offsets can be split ([LOW_GROUPS][nc] sums each, in planes)
    int *mods = nullptr;
};

// x mod p, centred: 18-bit limbs (the highest signed) against 2^18 and 2^36 mod p, then one approximate quotient and
// a correction (limbs_fit: how large x may be)
__device__ __forceinline__ int residue(int x0, int x1, int x2, int p, int c18, int c36, float rp)
{
    int r = mod_near(x0 + x1 * c18 + x2 * c36, p, rp);
    const int h = p >> 1;
    if (r > h) r -= p;
    if (r < -h) r += p;
    return r;
}

__device__ __forceinline__ void limbs(long long x, int &x0, int &x1, int &x2)
{
    x0 = (int)(x & 0x3FFFF);
    x1 = (int)((x >> 18) & 0x3FFFF);
    x2 = (int)(x >> 36);
}

constexpr int GAIN_MAX = 800;

// g of a level from the bits of its largest |M~|: |M~ 2^g| < 2^mbits
__device__ __forceinline__ int res_gain_raw(unsigned long long bits, int mbits)
{
    return bits == 0ull ? 0 : mbits - 1 - ((int)(bits >> 52) - 1023);
}

// whether the whole numbers hold a level: its largest moment is finite, and 2^g and its products with the scales and
// with P are normal doubles; else all its targets take the FP64 sum
__device__ __forceinline__ bool res_holds(unsigned long long bits, int mbits)
{
    const int g = res_gain_raw(bits, mbits);
    return (bits >> 52) != 2047 && g <= GAIN_MAX && g >= -GAIN_MAX;
}

__device__ __forceinline__ double pow2d(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }

// 2^(sign g), 1 where the level is not held
__device__ __forceinline__ double res_gain(unsigned long long bits, int mbits, int sign)
{
    return res_holds(bits, mbits) ? pow2d(sign * res_gain_raw(bits, mbits)) : 1.0;
}

// s(n,m) = sqrt((n+m)! (n-m)!) per real coefficient, and the moduli (by a kernel: the host would have to wait for the
// stream to stage a copy)
__global__ void k_res_setup(int p, double *__restrict__ s, int *__restrict__ mods, const __grid_constant__ ResConsts c)
{
    for (int e = threadIdx.x; e < (p + 1) * (p + 1); e += blockDim.x) {
        const int n = e / (p + 1), m = e % (p + 1);
        if (m > n) continue;
        double f = 1.0;
        for (int i = 2; i <= n + m; ++i) f *= i;
        for (int i = 2; i <= n - m; ++i) f *= i;
        s[cre(n, m)] = sqrt(f);
        if (m > 0) s[cim(n, m)] = sqrt(f);
    }
    for (int i = threadIdx.x; i < RES_MAX; i += blockDim.x) mods[i] = c.p[i];
}

// T~ of every slot -> residues times (P / p_i)^-1, [modulus][chunk][slot][j][k] with zero padding
__global__ void k_res_ops(int noff, const double *__restrict__ T, int nc, int npad, int kp, const double *__restrict__ s,
                          uint16_t *__restrict__ ops, size_t elems, const __grid_constant__ ResConsts c)
{
    const int64_t total = (int64_t)noff * npad * kp;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int k = (int)(e % kp);
        const int j = (int)((e / kp) % npad);
        const int slot = (int)(e / ((int64_t)kp * npad));
        long long x = 0;
        if (j < nc && k < nc)
            x = llrint(T[((int64_t)slot * nc + k) * nc + j] / (s[k] * s[j]) * (double)(1ll << c.tbits));
        int x0, x1, x2;
        limbs(x, x0, x1, x2);
        const int64_t at = chunk_at((int64_t)slot * npad + j, (int64_t)noff * npad, k, 64);
#pragma unroll
        for (int i = 0; i < RES_MAX; ++i) {
            if (i >= c.n) break;
            const int t2 = mod_near(x2, c.p[i], c.rp[i]);  // |x2| up to 2^21
            const int r = residue(x0, x1, t2, c.p[i], c.c18[i], c.c36[i], c.rp[i]);
            const int y = residue(r * c.inv[i], 0, 0, c.p[i], 0, 0, c.rp[i]);
            ops[at + i * elems] = __half_as_ushort(__int2half_rn(y));
        }
    }
}

// FP64 class-layout moments -> residue planes of moduli m0 .. m0 + nb - 1 with a periodic halo, 8 coefficients per
// thread (16-byte stores per plane), zero beyond nc.  Bound by the integer arithmetic of the residues (~15
// instructions each) and the planes' bytes.
__global__ void k_res_split(const double *__restrict__ M, int np, int hw, int nc, int kp, const double *__restrict__ s,
                            const unsigned long long *__restrict__ amax, int m0, int nb, uint16_t *__restrict__ planes,
                            const __grid_constant__ ResConsts c)
{
    const int np2 = np + 2 * hw;
    const int G = kp / 8;
    const int64_t ncell = 8 * (int64_t)np2 * np2 * np2, total = ncell * G;
    const double g = res_gain(*amax, c.mbits, 1);
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t cell = t / G;
        const int k0 = (int)(t - cell * G) * 8;
        const int hx = (int)(cell % np2);
        const int hy = (int)((cell / np2) % np2);
        const int hzc = (int)(cell / ((int64_t)np2 * np2));
        const int cl = hzc / np2, hz = hzc % np2;
        const int px = ((hx - hw) % np + np) % np, py = ((hy - hw) % np + np) % np, pz = ((hz - hw) % np + np) % np;
        const double *row = M + ((int64_t)cl * np * np * np + px + (int64_t)np * (py + (int64_t)np * pz)) * nc;
        int x0[8], x1[8], x2[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int k = k0 + u;
            const long long x = k < nc ? __double2ll_rn(row[k] * __ldg(s + k) * g) : 0;
            limbs(x, x0[u], x1[u], x2[u]);
        }
        uint16_t *out = planes + chunk_at(cell, ncell, k0, 64);
        for (int m = 0; m < nb; ++m) {
            const int p = c.p[m0 + m], a = c.c18[m0 + m], b = c.c36[m0 + m];
            const float rp = c.rp[m0 + m];
            uint32_t w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const __half2 h = __halves2half2(__int2half_rn(residue(x0[2 * u], x1[2 * u], x2[2 * u], p, a, b, rp)),
                                                 __int2half_rn(residue(x0[2 * u + 1], x1[2 * u + 1], x2[2 * u + 1], p, a,
                                                                       b, rp)));
                w[u] = *reinterpret_cast<const uint32_t *>(&h);
            }
            *reinterpret_cast<uint4 *>(out + (size_t)m * ncell * kp) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

// cell of the o-th source of target `cell` of a level with class side 2^lg, and its operator slot
__device__ __forceinline__ int64_t res_source(const int *__restrict__ il, int n_il, int lg, int ws, int64_t cell, int o,
                                              int &slot)
{
    const int c = (int)(cell >> (3 * lg)), mask = (1 << lg) - 1;
    int dx, dy, dz;
    il_unpack(__ldg(il + c * n_il + o), dx, dy, dz);
    slot = off_slot(dx, dy, dz, ws);
    const int sx = (c & 1) + dx, sy = ((c >> 1) & 1) + dy, sz = (c >> 2) + dz;
    const int x = ((int)cell + (sx >> 1)) & mask, y = ((int)(cell >> lg) + (sy >> 1)) & mask,
              z = ((int)(cell >> (2 * lg)) + (sz >> 1)) & mask;
    return ((int64_t)((sx & 1) | ((sy & 1) << 1) | ((sz & 1) << 2)) << (3 * lg)) + x + (((int64_t)z << lg) + y << lg);
}

// Where the targets that take the FP64 sum are listed, and what tells them
struct ResLow {
    const uint32_t *cmax;  // the level's
    const int *il;
    int n_il, lg, ws;
    uint32_t base;         // of the level in the list's numbers
    uint32_t *list;
    int *count;
};

// whether every source of a target is below the upper word `lim` and one is not zero (a whole warp; mostly the first
// 32 sources settle it)
__device__ __forceinline__ bool res_low_list(const ResLow &d, int64_t cell, uint32_t lim, int lane)
{
    bool any = false;
    for (int o0 = 0; o0 < d.n_il; o0 += 32) {
        int slot;
        const uint32_t v = o0 + lane < d.n_il ? d.cmax[res_source(d.il, d.n_il, d.lg, d.ws, cell, o0 + lane, slot)] : 0u;
        if (__any_sync(0xffffffffu, v >= lim)) return false;
        any |= v > 0u;
    }
    return __any_sync(0xffffffffu, any) != 0;
}

// Residues y_i of nb moduli (and of the offset groups) -> the 96-bit fraction sum y_i / p_i mod 1, and on the last
// launch of the level L^ = P (fraction) 2^-(g + C) s(j).  Two neighbouring elements per thread (their
// residues are one 32-bit load); frac carries the sums between the launches of a level.  The last launch also lists the
// targets whose sources are too far below the level's largest, all of them where the whole numbers do not hold that.
__global__ void __launch_bounds__(JOIN_THREADS) k_res_join(int64_t n, int nc, int groups, int m0, int nb,
                                                           const int16_t *__restrict__ resid, uint32_t *__restrict__ frac,
                                                           bool first, bool last, const double *__restrict__ s,
                                                           const unsigned long long *__restrict__ amax,
                                                           double *__restrict__ L, const ResLow d,
                                                           const __grid_constant__ ResConsts c)
{
    const int64_t e0 = 2 * (blockIdx.x * (int64_t)JOIN_THREADS), e = e0 + 2 * threadIdx.x;
    const unsigned long long bits = *amax;
    if (last) {  // a warp per cell that begins in the block
        const int64_t e1 = e0 + 2 * JOIN_THREADS < n ? e0 + 2 * JOIN_THREADS : n;
        const uint32_t hi = (uint32_t)(bits >> 32), down = (uint32_t)(c.mbits - c.keep) << 20;
        for (int64_t cell = (e0 + nc - 1) / nc + (threadIdx.x >> 5); cell * nc < e1; cell += JOIN_THREADS / 32)
            if (!res_holds(bits, c.mbits) || (hi > down && res_low_list(d, cell, hi - down, threadIdx.x & 31)))
                if ((threadIdx.x & 31) == 0) d.list[atomicAdd(d.count, 1)] = d.base + (uint32_t)cell;
    }
    if (e >= n) return;  // n is even (8 parity classes)
    const double f = c.pscale * res_gain(bits, c.mbits, -1);
    long long a0[2] = {0, 0}, a1[2] = {0, 0}, a2[2] = {0, 0};
    for (int g = 0; g < groups; ++g)
#pragma unroll 8
        for (int m = 0; m < nb; ++m) {
            const int v = *reinterpret_cast<const int *>(resid + ((int64_t)g * nb + m) * n + e);
            const int y[2] = {(int)(short)(v & 0xFFFF), v >> 16};
            const uint32_t w0 = c.w[m0 + m][0], w1 = c.w[m0 + m][1], w2 = c.w[m0 + m][2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                a0[u] += (long long)y[u] * w0;
                a1[u] += (long long)y[u] * w1;
                a2[u] += (long long)y[u] * w2;
            }
        }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        if (!first) {
            a0[u] += frac[e + u];
            a1[u] += frac[n + e + u];
            a2[u] += frac[2 * n + e + u];
        }
        // carries: limbs of 32 bits, the top one modulo 2^32 (the fraction is taken modulo 1)
        a1[u] += a0[u] >> 32;
        a2[u] += a1[u] >> 32;
        const uint32_t lo = (uint32_t)a0[u], mid = (uint32_t)a1[u], hi = (uint32_t)a2[u];
        if (!last) {
            frac[e + u] = lo;
            frac[n + e + u] = mid;
            frac[2 * n + e + u] = hi;
            continue;
        }
        const long long top = (long long)(((uint64_t)hi << 32) | mid);  // signed: |L_int| < P / 2
        double v = (double)top * 4294967296.0 + (double)lo;
        L[e + u] = v * f * s[(int)((e + u) % nc)];
    }
}

// place of level l in the list's numbers and in cmax
__host__ __device__ inline uint32_t cmax_at(int l) { return (uint32_t)((((int64_t)1 << (3 * l)) - 8) / 7); }

struct ResLevels {
    const double *M[9];
    double *L[9];
};

// The FP64 sums of the listed targets, over the results of k_res_join.  A few targets: their offsets are split over
// LOW_GROUPS blocks each, and the block that finishes last adds their sums in order (a thread per output took 9.6 ms for
// 8 targets at p = 12).  Many targets take a block each, which is bound by the FP64 pipe.  Empty sources are left out.
constexpr int LOW_THREADS = 128, LOW_CELLS = 128, LOW_GROUPS = 63;

__global__ void __launch_bounds__(LOW_THREADS) k_res_low(int nc, int d, int ws, int n_il, const __grid_constant__ ResLevels lv,
                                                         const uint32_t *__restrict__ cmax, const double *__restrict__ Top,
                                                         const int *__restrict__ il, const uint32_t *__restrict__ list,
                                                         const int *__restrict__ count, int split_max,
                                                         double *__restrict__ part, int *__restrict__ done)
{
    constexpr int Q = 256 / LOW_THREADS;  // coefficients per thread
    __shared__ double sM[256];
    __shared__ int last;
    const int n = *count;
    const int ng = n <= split_max ? LOW_GROUPS : 1, per = (n_il + ng - 1) / ng;
    for (int64_t it = blockIdx.x; it < (int64_t)n * ng; it += gridDim.x) {
        const int i = (int)(it / ng), g = (int)(it - (int64_t)i * ng);
        const uint32_t code = list[i];
        int l = 2;
        while (l < d && code >= cmax_at(l + 1)) ++l;
        const int64_t cell = code - cmax_at(l);
        double acc[Q] = {};
        for (int o = g * per; o < n_il && o < (g + 1) * per; ++o) {
            int slot;
            const int64_t src = res_source(il, n_il, l - 1, ws, cell, o, slot);
            if (cmax[cmax_at(l) + src] == 0u) continue;  // the same for the whole block
            __syncthreads();
            for (int k = threadIdx.x; k < nc; k += LOW_THREADS) sM[k] = lv.M[l][src * nc + k];
            __syncthreads();
            const double *T = Top + (size_t)slot * nc * nc;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int j = threadIdx.x + q * LOW_THREADS;
                if (j >= nc) break;
#pragma unroll 8
                for (int k = 0; k < nc; ++k) acc[q] += T[(size_t)k * nc + j] * sM[k];
            }
        }
        double *out = ng == 1 ? lv.L[l] + cell * nc : part + (size_t)(i * LOW_GROUPS + g) * nc;
#pragma unroll
        for (int q = 0; q < Q; ++q)
            if (threadIdx.x + q * LOW_THREADS < nc) out[threadIdx.x + q * LOW_THREADS] = acc[q];
        if (ng == 1) continue;
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(done + i, 1) == ng - 1;
        __syncthreads();
        if (last) {
            __threadfence();
            for (int j = threadIdx.x; j < nc; j += LOW_THREADS) {
                double v = 0;
                for (int k = 0; k < ng; ++k) v += __ldcg(part + (size_t)(i * LOW_GROUPS + k) * nc + j);
                lv.L[l][cell * nc + j] = v;
            }
        }
        __syncthreads();
    }
}

// whether residue() takes whole numbers below 2^bits: the limbs' products fit 31 bits, and the approximate quotient
// (three roundings of 2^-24) is off by less than 1/2
bool limbs_fit(const ResConsts &c, int bits)
{
    for (int i = 0; i < c.n; ++i) {
        const double v = ldexp(fabs((double)c.c36[i]), bits - 36) + ldexp(fabs((double)c.c18[i]), 18) + ldexp(1.0, 18);
        if (v >= ldexp(1.0, 31) || 3.0 * v >= ldexp(0.45 * c.p[i], 24)) return false;
    }
    return true;
}

// the largest pairwise coprime numbers below the exactness bound until their product exceeds 2^(B + C + sum_bits), the
// bits of the largest sum with its sign; B then takes what they have left
bool choose_moduli(int nc, int tbits, double sum_bits, ResConsts &c)
{
    c.tbits = tbits;
    const double bits = RES_M_BITS + tbits + sum_bits;
    int h = 1;
    while ((int64_t)RES_CHAIN * nc * (h + 1) * (h + 1) <= (1 << 24)) ++h;
    int top = 2 * h + 1;
    if (top > 2047) top = 2047;  // whole numbers of fp16; residues stay below 2^11
    double have = 0;
    c.n = 0;
    for (int p = top; p > 2 && have < bits; --p) {
        bool ok = true;
        for (int i = 0; i < c.n && ok; ++i) {
            int a = p, b = c.p[i];
            while (b) {
                const int t = a % b;
                a = b;
                b = t;
            }
            ok = a == 1;
        }
        if (!ok) continue;
        if (c.n == RES_MAX) return false;
        c.p[c.n++] = p;
        have += log2((double)p);
    }
    if (have < bits) return false;
    double pscale = 1.0;
    for (int i = 0; i < c.n; ++i) pscale *= (double)c.p[i] * ldexp(1.0, -6);
    c.pscale = ldexp(pscale, 6 * c.n - 96 - tbits);
    for (int i = 0; i < c.n; ++i) {
        const int p = c.p[i];
        auto centred = [p](int64_t v) {
            int r = (int)(((v % p) + p) % p);
            return r > p / 2 ? r - p : r;
        };
        c.rp[i] = 1.f / (float)p;
        c.c18[i] = centred((int64_t)1 << 18);
        c.c36[i] = centred((int64_t)1 << 36);
        int64_t q = 1;  // P / p_i mod p_i
        for (int j = 0; j < c.n; ++j)
            if (j != i) q = q * c.p[j] % p;
        int64_t inv = 1;
        while (q * inv % p != 1) ++inv;
        c.inv[i] = centred(inv);
        // floor(2^96 / p), base 2^32 long division
        uint64_t rem = 1;
        for (int w = 2; w >= 0; --w) {
            rem <<= 32;
            c.w[i][w] = (uint32_t)(rem / p);
            rem %= p;
        }
    }
    if (!limbs_fit(c, RES_M_BITS)) return false;
    c.mbits = RES_M_BITS;
    while (c.mbits < RES_M_BITS_MAX && have >= c.mbits + 1 + tbits + sum_bits && limbs_fit(c, c.mbits + 1)) ++c.mbits;
    return true;
}

#define FMM_RES_CASES(X) \
    X(1) X(2) X(3) X(4) X(6) X(7) X(8) X(9) X(11) X(13) X(15) X(16)

TcKernel res_kernel(int nch)
{
    switch (nch) {
#define X(n) \
    case n: return (TcKernel)k_m2l_tc<2, 2, n, 128, true>;
        FMM_RES_CASES(X)
#undef X
    default: return nullptr;
    }
}

TcKernel res_pair_kernel(int nch)
{
    switch (nch) {
#define X(n) \
    case n: return (TcKernel)k_m2l_tc_pair<n, true>;
        FMM_RES_CASES(X)
#undef X
    default: return nullptr;
    }
}

constexpr size_t RES_CLEAR = sizeof(unsigned long long) * 9 + sizeof(int) * (1 + LOW_CELLS);  // amax and behind it

bool pairs_at(const ResState *S, int l)
{
    const int np = 1 << (l - 1);
    const int tiles = (np / S->bx[l]) * (np / S->by[l]) * (np / S->bz[l]);
    return S->bx[l] * S->by[l] * S->bz[l] == TC_ROWS && tiles % 2 == 0;
}

unsigned blocks_upto(int64_t n, int t, int64_t most)
{
    const int64_t b = (n + t - 1) / t;
    return (unsigned)(b < most ? b : most);
}

fmm_status prepare(Plan &P, ResState *S, const ResState *src, size_t plane_budget)
{
    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
    if (!enc) return FMM_ERR_UNSUPPORTED;
    // |L_int| < 2^B 2^C 137 (ws = 1: log2 137 = 7.10) or 277 (ws = 2: 8.12), and its sign
    S->c.keep = P.p < 3 ? 54 : P.p < 5 ? 53 : P.p < 12 ? 52 : 51;
    if (!choose_moduli(P.nc, P.ws == 2 || P.p <= 3 ? 58 : 56, (P.ws == 1 ? 7.2 : 8.2) + 1.0, S->c)) return FMM_ERR_UNSUPPORTED;
    S->npad = (P.nc + 15) / 16 * 16;
    S->kp = (P.nc + 63) / 64 * 64;
    S->noff = noff(P.ws);
    const int kc = S->kp / 64, n = S->c.n;
    const size_t cells_all = cmax_at(P.d + 1);
    // s64, amax and what is cleared with it, mods, cmax, low in one allocation
    FMM_CUDA_TRY(cudaMalloc(&S->s64, sizeof(double) * P.nc + RES_CLEAR + sizeof(int) * RES_MAX +
                                         2 * sizeof(uint32_t) * cells_all));
    S->amax = (unsigned long long *)(S->s64 + P.nc);
    S->low_count = (int *)(S->amax + 9);
    S->mods = (int *)((char *)S->amax + RES_CLEAR);
    S->cmax = (uint32_t *)(S->mods + RES_MAX);
    S->low = S->cmax + cells_all;
    k_res_setup<<<1, 256, 0, P.stream>>>(P.p, S->s64, S->mods, S->c);
    FMM_LAUNCH_CHECK(P);
    S->ops_elems = (size_t)S->noff * S->npad * S->kp;
    S->ops_borrowed = src != nullptr;
    if (src) S->ops = src->ops;
    else {
        FMM_CUDA_TRY(cudaMalloc(&S->ops, sizeof(uint16_t) * S->ops_elems * n));
        k_res_ops<<<1216, 256, 0, P.stream>>>(S->noff, P.tab.Top64, P.nc, S->npad, S->kp, S->s64, S->ops, S->ops_elems,
                                              S->c);
        FMM_LAUNCH_CHECK(P);
    }
    int sms = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
        sms = 152;
    size_t planes = 0, resid = 0, frac = 0;
    for (int l = 2; l <= P.d; ++l) {  // level 1 is part of the top operator
        const int np = 1 << (l - 1);
        const size_t np2 = (size_t)np + 2 * P.ws, cells = (size_t)8 * np * np * np;
        S->bx[l] = tile_dim(np, TC_ROWS);
        S->by[l] = tile_dim(np, TC_ROWS / S->bx[l]);
        S->bz[l] = tile_dim(np, TC_ROWS / (S->bx[l] * S->by[l]));
        const size_t plane = 8 * np2 * np2 * np2 * S->kp * sizeof(uint16_t);
        int b = (int)(plane_budget / plane);
        b = b < 1 ? 1 : (b > n ? n : b);
        b = (n + (n + b - 1) / b - 1) / ((n + b - 1) / b);  // even launches
        S->batch[l] = b;
        const int tiles = 8 * (np / S->bx[l]) * (np / S->by[l]) * (np / S->bz[l]);
        split_offsets(n_il(P.ws), tiles * b, 27, sms, S->groups[l], S->per_group[l]);
        if (plane * b > planes) planes = plane * b;
        const size_t r = (size_t)S->groups[l] * b * cells * P.nc * sizeof(int16_t);
        if (r > resid) resid = r;
        if (b < n && cells * P.nc > frac) frac = cells * P.nc;
    }
    // the launch of the FP64 sums follows the last level's and takes its place in the planes (at least 16 targets)
    const size_t low_cell = sizeof(double) * LOW_GROUPS * P.nc;
    if (planes < 16 * low_cell) planes = 16 * low_cell;
    S->low_cells = planes / low_cell < LOW_CELLS ? (int)(planes / low_cell) : LOW_CELLS;
    FMM_CUDA_TRY(cudaMalloc(&S->planes, planes));
    FMM_CUDA_TRY(cudaMalloc(&S->resid, resid));
    if (frac) FMM_CUDA_TRY(cudaMalloc(&S->frac, frac * 3 * sizeof(uint32_t)));
    const CUtensorMapDataType dt = CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
    fmm_status st = encode_operators(enc, &S->maps[0].bS, nullptr, &S->maps[0].bC, dt, S->ops, kc, n, S->npad, S->noff,
                                     S->npad, 128);
    if (st == FMM_OK)
        st = encode_operators(enc, &S->mapB2[0], nullptr, &S->mapB2[1], dt, S->ops, kc, n, S->npad, S->noff, S->npad / 2,
                              128);
    for (int l = 2; l <= P.d && st == FMM_OK; ++l) {
        const int np = 1 << (l - 1);
        const int64_t np2 = np + 2 * P.ws;
        TcMaps &m = S->maps[l];
        m = S->maps[0];
        st = encode_planes(enc, &m.aS, nullptr, &m.aC, dt, S->planes, kc, S->batch[l], np2, np2, 8 * np2, S->bx[l],
                           S->by[l], S->bz[l], 128);
        m.aP = m.lS = m.lP = m.aS;  // unused kernel parameters
        m.bP = m.bS;
    }
    if (st != FMM_OK) return st;
    const TcKernel k1 = res_kernel(S->npad / 16), k2 = res_pair_kernel(S->npad / 16);
    if (!k1 || !k2) return FMM_ERR_INTERNAL;
    FMM_CUDA_TRY(cudaFuncSetAttribute((const void *)k1, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)tc_smem_bytes(2, 2, S->npad, 128)));
    FMM_CUDA_TRY(cudaFuncSetAttribute((const void *)k2, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)tc_pair_smem_bytes(S->npad)));
    return FMM_OK;
}

}  // namespace

bool res_available(const Plan &P, int level) { return P.res != nullptr && level >= 1 && level <= P.d; }

// The residue state of an FP64 plan; without the memory for it the plan keeps the CUDA-core M2L.  Nothing here waits for
// the plan's stream: a call that only enqueues does so the first time as well.  With `src`, a plan of the same p and ws
// that has the state, the operators are src's (which must outlive P; its stream may still be filling them).
fmm_status res_ensure(Plan &P, const Plan *src, size_t plane_budget)
{
    if (P.res || P.res_tried || P.precision != FMM_PREC_FP64 || P.p > TC_PMAX) return FMM_OK;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    FMM_CUDA_TRY(cudaStreamIsCapturing(P.stream, &cap));
    if (cap != cudaStreamCaptureStatusNone) return FMM_OK;
    P.res_tried = true;
    ResState *S = new (std::nothrow) ResState();
    if (!S) return FMM_ERR_OOM;
    P.res = S;
    // allocations of this thread leave a capture in another one alone
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    const bool relaxed = cudaThreadExchangeStreamCaptureMode(&mode) == cudaSuccess;
    const bool borrow = src && src->res && src->p == P.p && src->ws == P.ws;
    const fmm_status st = prepare(P, S, borrow ? (const ResState *)src->res : nullptr, plane_budget);
    if (relaxed) cudaThreadExchangeStreamCaptureMode(&mode);
    if (st == FMM_OK) return FMM_OK;
    cudaStreamSynchronize(P.stream);
    res_free(P);
    P.res_tried = true;
    if (st == FMM_ERR_OOM || st == FMM_ERR_UNSUPPORTED) {
        cudaGetLastError();
        return FMM_OK;
    }
    return st;
}

fmm_status res_clear_amax(Plan &P)
{
    ResState *S = (ResState *)P.res;
    if (S) FMM_CUDA_TRY(cudaMemsetAsync(S->amax, 0, RES_CLEAR, P.stream));
    return FMM_OK;
}

unsigned long long *res_amax(Plan &P, int l, const double **s, uint32_t **cmax)
{
    ResState *S = (ResState *)P.res;
    *s = S ? S->s64 : nullptr;
    *cmax = S ? S->cmax + cmax_at(l) : nullptr;
    return S ? S->amax + l : nullptr;
}

// L[l] = M2L of level l (the L2L from level l - 1 is added by launch_l2l), but for the targets that it lists
fmm_status launch_m2l_res(Plan &P, int l)
{
    ResState *S = (ResState *)P.res;
    if (!S) return FMM_ERR_INTERNAL;
    const int np = 1 << (l - 1), nc = P.nc, n = S->c.n;
    const int64_t np2 = np + 2 * P.ws, cells = (int64_t)8 * np * np * np;
    TcArgs a;
    memset(&a, 0, sizeof(a));
    a.np = np;
    a.bx = S->bx[l];
    a.by = S->by[l];
    a.bz = S->bz[l];
    a.rows = a.bx * a.by * a.bz;
    a.tiles_x = np / a.bx;
    a.tiles_y = np / a.by;
    a.tiles_per_class = a.tiles_x * a.tiles_y * (np / a.bz);
    a.nc = nc;
    a.npad = S->npad;
    a.nslots = a.noff = S->noff;
    a.groups = S->groups[l];
    a.per_group = S->per_group[l];
    a.n_off = a.n_il = n_il(P.ws);
    a.ws = P.ws;
    for (int k = 0; k < S->kp / 64; ++k) a.gchunks |= 1u << (2 * k);  // one product per chunk, two chunks a stage
    a.acc_group = RES_CHAIN;
    a.wait_ns = P.wait_ns;
    a.inject_stall = P.inject_stall ? 1 : 0;
    a.err = P.d_err;
    a.mods = S->mods;
    a.il = P.tab.il;
    a.resid = S->resid;
    const bool pair = pairs_allowed(P) && pairs_at(S, l);
    TcMaps maps = S->maps[l];
    if (pair) {
        maps.bS = S->mapB2[0];
        maps.bC = S->mapB2[1];
    }
    a.stages = pair ? tc_pair_stages(S->npad) : tc_stages(2, 2, S->npad, 128);
    a.idesc = (1u << 4) | ((uint32_t)(S->npad >> 3) << 17) | ((uint32_t)((pair ? 2 * TC_ROWS : TC_ROWS) >> 4) << 24);
    const TcKernel k = pair ? res_pair_kernel(S->npad / 16) : res_kernel(S->npad / 16);
    const size_t smem = pair ? tc_pair_smem_bytes(S->npad) : tc_smem_bytes(2, 2, S->npad, 128);
    const ResLow low{S->cmax + cmax_at(l), P.tab.il, n_il(P.ws), l - 1, P.ws, cmax_at(l), S->low, S->low_count};
    const int64_t halo = 8 * np2 * np2 * np2 * (S->kp / 8), elems = cells * nc;
    for (int m0 = 0; m0 < n; m0 += S->batch[l]) {
        const int nb = n - m0 < S->batch[l] ? n - m0 : S->batch[l];
        k_res_split<<<blocks_upto(halo, 256, 8 * 1216), 256, 0, P.stream>>>((const double *)P.M[l], np, P.ws, nc, S->kp,
                                                                            S->s64, S->amax + l, m0, nb, S->planes, S->c);
        FMM_LAUNCH_CHECK(P);
        a.mod0 = m0;
        a.nmods = nb;
        k<<<8u * (unsigned)a.tiles_per_class * (unsigned)a.groups * (unsigned)nb, TC_THREADS, smem, P.stream>>>(maps, a);
        FMM_LAUNCH_CHECK(P);
        k_res_join<<<(unsigned)((elems / 2 + JOIN_THREADS - 1) / JOIN_THREADS), JOIN_THREADS, 0, P.stream>>>(
            elems, nc, a.groups, m0, nb, S->resid, S->frac, m0 == 0, m0 + nb == n, S->s64, S->amax + l, (double *)P.L[l],
            low, S->c);
        FMM_LAUNCH_CHECK(P);
    }
    return FMM_OK;
}

// the listed targets of all levels
fmm_status launch_m2l_res_low(Plan &P)
{
    ResState *S = (ResState *)P.res;
    if (!S) return FMM_ERR_INTERNAL;
    ResLevels lv = {};
    for (int l = 2; l <= P.d; ++l) {
        lv.M[l] = (const double *)P.M[l];
        lv.L[l] = (double *)P.L[l];
    }
    k_res_low<<<4 * 152, LOW_THREADS, 0, P.stream>>>(P.nc, P.d, P.ws, n_il(P.ws), lv, S->cmax, P.tab.Top64, P.tab.il, S->low,
                                                     S->low_count, S->low_cells, (double *)S->planes, S->low_count + 1);
    FMM_LAUNCH_CHECK(P);
    return FMM_OK;
}

void res_free(Plan &P)
{
    ResState *S = (ResState *)P.res;
    P.res_tried = false;
    if (!S) return;
    if (!S->ops_borrowed) cudaFree(S->ops);
    cudaFree(S->planes);
    cudaFree(S->resid);
    cudaFree(S->frac);
    cudaFree(S->s64);  // and what shares its allocation
    delete S;
    P.res = nullptr;
}

}  // namespace fmm
