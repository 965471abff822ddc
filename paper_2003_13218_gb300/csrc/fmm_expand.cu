// fmm_expand.cu -- the expansion operators of Appendix B on the GPU:
// P2M (Eq. P2M), the level-0 lattice operator (Eq. 12), M2L over the
// interaction lists (Eq. Lcoeffdef, CUDA-core version) and L2P with its
// gradient (Eq. EqFF); plus the per-plan operator tables.
//
// Solid harmonics (normalisation that makes the printed equations hold with
// no conjugates): R_n^m = r^n P_n^m e^{im phi}/(n+m)!,
// I_n^m = (-1)^(n+m) (n-m)! P_n^m e^{im phi} / r^(n+1); both obey
// C_n^{-m} = (-1)^m conj C_n^m, so only m >= 0 is stored.
#include <math.h>

#include <stdlib.h>

#include <type_traits>
#include <vector>

#include "fmm_internal.cuh"

namespace fmm {

namespace {

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// ------------------------------------------------------------------ tables
// R_n^m at the eight child-centre offsets w_c = ((c_x - 1/2)/2, ...) (in
// units of the parent side): the M2M and L2L shift vectors.
__global__ void k_octant_table(int p, double *__restrict__ R64)
{
    int c = threadIdx.x;
    if (c >= 8) return;
    int nc = ncoef(p);
    double w[3] = {((c & 1) - 0.5) * 0.5, (((c >> 1) & 1) - 0.5) * 0.5, (((c >> 2) & 1) - 0.5) * 0.5};
    double tmp[NC_MAX];
    regular_real<double>(p, w[0], w[1], w[2], tmp);
    for (int i = 0; i < nc; ++i) R64[c * nc + i] = tmp[i];
}

// complex I_j^k for any sign of k from the m >= 0 triangle
__device__ inline Cx<double> tri_get(const Cx<double> *t, int j, int k)
{
    int ak = k < 0 ? -k : k;
    Cx<double> v = t[tri(j, ak)];
    if (k < 0) {
        v.im = -v.im;
        if (ak & 1) {
            v.re = -v.re;
            v.im = -v.im;
        }
    }
    return v;
}

// Real form of Eq. Lcoeffdef: L_n^m = sum_{lambda, eta} M_lambda^eta O_{n+lambda}^{-(m+eta)}.
// With M_lambda^{-eta} = (-1)^eta conj M_lambda^eta and M_lambda^eta = x + i y:
//   eta = 0: L += x O(lambda, 0)
//   eta > 0: L += x A + i y B,  A = O(lambda, eta) + (-1)^eta O(lambda, -eta),
//                                B = O(lambda, eta) - (-1)^eta O(lambda, -eta),
// where O(lambda, e) = O_{n+lambda}^{-(m+e)}.  Entry [k][j] maps input real k
// to output real j.
__device__ void build_real_operator(int p, const Cx<double> *O, double *__restrict__ Tout)
{
    int nc = ncoef(p);
    for (int e = threadIdx.x; e < nc * nc; e += blockDim.x) {
        int k = e / nc, j = e % nc;
        // output (n, m, part)
        int n = (int)sqrt((double)j);
        while (n * n > j) --n;
        while ((n + 1) * (n + 1) <= j) ++n;
        int r = j - n * n;
        int m = (r + 1) / 2;
        bool out_im = (m > 0) && (r == 2 * m);
        // input (lambda, eta, part)
        int lam = (int)sqrt((double)k);
        while (lam * lam > k) --lam;
        while ((lam + 1) * (lam + 1) <= k) ++lam;
        int ri = k - lam * lam;
        int eta = (ri + 1) / 2;
        bool in_im = (eta > 0) && (ri == 2 * eta);
        double val;
        Cx<double> o1 = tri_get(O, n + lam, -(m + eta));
        if (eta == 0) {
            val = out_im ? o1.im : o1.re;
        } else {
            Cx<double> o2 = tri_get(O, n + lam, eta - m);
            double sg = (eta & 1) ? -1.0 : 1.0;
            if (!in_im) {
                Cx<double> A = {o1.re + sg * o2.re, o1.im + sg * o2.im};
                val = out_im ? A.im : A.re;
            } else {
                Cx<double> B = {o1.re - sg * o2.re, o1.im - sg * o2.im};
                val = out_im ? B.re : -B.im;
            }
        }
        Tout[(size_t)k * nc + j] = val;
    }
}

// one block per offset slot delta in [-(2 ws + 1), 2 ws + 1]^3 (the (2 ws + 1)^3 near slots stay zero)
__global__ void k_m2l_operators(int p, int ws, double *__restrict__ T64, float *__restrict__ T32)
{
    extern __shared__ Cx<double> Ish[];
    int slot = blockIdx.x;
    const int side = off_side(ws), h = 2 * ws + 1;
    int dx = slot % side - h, dy = (slot / side) % side - h, dz = slot / (side * side) - h;
    int nc = ncoef(p);
    double *T = T64 + (size_t)slot * nc * nc;
    if (abs(dx) <= ws && abs(dy) <= ws && abs(dz) <= ws) {
        for (int e = threadIdx.x; e < nc * nc; e += blockDim.x) {
            T[e] = 0.0;
            T32[(size_t)slot * nc * nc + e] = 0.0f;
        }
        return;
    }
    // I at r_L - r_M = -(delta) in cell units: target t, source t + delta
    if (threadIdx.x == 0) irregular_tri<double>(2 * p, -(double)dx, -(double)dy, -(double)dz, Ish);
    __syncthreads();
    build_real_operator(p, Ish, T);
    __syncthreads();
    for (int e = threadIdx.x; e < nc * nc; e += blockDim.x) T32[(size_t)slot * nc * nc + e] = (float)T[e];
}

// single irregular harmonic I_j^k (k >= 0) by the column recurrence
__device__ Cx<double> irregular_one(int j, int k, double x, double y, double z)
{
    double r2 = x * x + y * y + z * z, ir2 = 1.0 / r2;
    Cx<double> dg = {1.0 / sqrt(r2), 0.0};
    for (int m = 1; m <= k; ++m) {
        double s = -(2.0 * m - 1.0) * ir2;
        dg = {s * (x * dg.re - y * dg.im), s * (x * dg.im + y * dg.re)};
    }
    Cx<double> p2 = {0, 0}, p1 = dg;
    for (int n = k + 1; n <= j; ++n) {
        double a = -(2.0 * n - 1.0) * z, b = (double)((n + k - 1) * (n - k - 1));
        Cx<double> c = {(a * p1.re - b * p2.re) * ir2, (a * p1.im - b * p2.im) * ir2};
        p2 = p1;
        p1 = c;
    }
    return p1;
}

struct KS {
    double s = 0, c = 0;
    __device__ void add(double x)
    {
        double t = s + x;
        if (fabs(s) >= fabs(x)) c += (s - t) + x;
        else c += (x - t) + s;
        s = t;
    }
    __device__ double val() const { return s + c; }
};

// Eq. 12 on a unit box with splitting parameter kb = kappa * b:
//   S_j^k = sum_{nu != 0} I_j^k(nu) Q(j + 1/2, kb^2 nu^2)                         (12a)
//         + pi^{3/2} i^j / (2^{j-2} Gamma(j + 1/2)) sum_{k != 0} I_j^k(k) k^{2j-1} e^{-k^2/4kb^2}  (12b)
//         - 2 kb / sqrt(pi) delta_{j0}                                           (12c)
//         - sum_{nu in {-1,0,1}^3, nu != 0} I_j^k(nu)      (images covered by levels 1..l_max)
// Q(a, x) = Gamma(a, x)/Gamma(a) by Q(1/2, x) = erfc(sqrt x) and
// Q(a + 1, x) = Q(a, x) + x^a e^{-x} / Gamma(a + 1).  One block per (j, k):
// threads stride over the lattice vectors, then a fixed-order reduction.
constexpr int LAT_THREADS = 256;

__device__ void block_merge(KS &v, double (*sh)[2])
{
    sh[threadIdx.x][0] = v.s;
    sh[threadIdx.x][1] = v.c;
    __syncthreads();
    for (int o = LAT_THREADS / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) {
            KS a;
            a.s = sh[threadIdx.x][0];
            a.c = sh[threadIdx.x][1];
            a.add(sh[threadIdx.x + o][0]);
            a.add(sh[threadIdx.x + o][1]);
            sh[threadIdx.x][0] = a.s;
            sh[threadIdx.x][1] = a.c;
        }
        __syncthreads();
    }
    v.s = sh[0][0];
    v.c = sh[0][1];
    __syncthreads();
}

__global__ void __launch_bounds__(LAT_THREADS) k_lattice_sum(int jmax, double kb, int ws, int nu_max, int nk_max,
                                                              double *__restrict__ S)
{
    __shared__ double sh[LAT_THREADS][2];
    int t = blockIdx.x;
    int j = 0;
    while (tri(j + 1, 0) <= t) ++j;
    int k = t - tri(j, 0);
    const double PI = 3.14159265358979323846;
    KS re, im;
    // real space (12a) and the near block
    const int side = 2 * nu_max + 1;
    const int nvec = side * side * side;
    for (int v = threadIdx.x; v < nvec; v += LAT_THREADS) {
        int nx = v % side - nu_max, ny = (v / side) % side - nu_max, nz = v / (side * side) - nu_max;
        if (nx == 0 && ny == 0 && nz == 0) continue;
        double r2 = (double)(nx * nx + ny * ny + nz * nz);
        double x = kb * kb * r2;
        double Q = erfc(sqrt(x));
        double g = sqrt(PI);  // Gamma(1/2)
        for (int i = 0; i < j; ++i) {
            double a = i + 0.5;
            g *= a;  // Gamma(i + 3/2)
            Q += exp(a * log(x) - x) / g;
        }
        bool near = abs(nx) <= ws && abs(ny) <= ws && abs(nz) <= ws;
        double w = near ? Q - 1.0 : Q;
        Cx<double> I = irregular_one(j, k, nx, ny, nz);
        re.add(w * I.re);
        im.add(w * I.im);
    }
    // reciprocal space (12b), k = 2 pi n
    double gh = sqrt(PI);
    for (int i = 0; i < j; ++i) gh *= (i + 0.5);  // Gamma(j + 1/2)
    double pref = pow(PI, 1.5) / (ldexp(1.0, j - 2) * gh);
    // i^j: j even -> (-1)^(j/2); odd degrees vanish by symmetry (kept exact)
    KS rre, rim;
    const int kside = 2 * nk_max + 1;
    const int nk = kside * kside * kside;
    for (int v = threadIdx.x; v < nk; v += LAT_THREADS) {
        int nx = v % kside - nk_max, ny = (v / kside) % kside - nk_max, nz = v / (kside * kside) - nk_max;
        if (nx == 0 && ny == 0 && nz == 0) continue;
        double kx = 2 * PI * nx, ky = 2 * PI * ny, kz = 2 * PI * nz;
        double k2 = kx * kx + ky * ky + kz * kz;
        double kk = sqrt(k2);
        double w = pow(kk, 2 * j - 1) * exp(-k2 / (4 * kb * kb));
        Cx<double> I = irregular_one(j, k, kx, ky, kz);
        rre.add(w * I.re);
        rim.add(w * I.im);
    }
    block_merge(re, sh);
    block_merge(im, sh);
    block_merge(rre, sh);
    block_merge(rim, sh);
    if (threadIdx.x != 0) return;
    double cr = rre.val() * pref, ci = rim.val() * pref;
    // multiply by i^j
    double ore, oim;
    switch (j & 3) {
    case 0: ore = cr; oim = ci; break;
    case 1: ore = -ci; oim = cr; break;
    case 2: ore = -cr; oim = -ci; break;
    default: ore = ci; oim = -cr; break;
    }
    re.add(ore);
    im.add(oim);
    if (j == 0) re.add(-2.0 * kb / sqrt(PI));
    S[2 * t] = re.val();
    S[2 * t + 1] = im.val();
}

__global__ void k_lattice_operator(int p, const double *__restrict__ S, double *__restrict__ T0)
{
    extern __shared__ Cx<double> Ssh[];
    int ntri = (2 * p + 1) * (2 * p + 2) / 2;
    for (int i = threadIdx.x; i < ntri; i += blockDim.x) Ssh[i] = {S[2 * i], S[2 * i + 1]};
    __syncthreads();
    build_real_operator(p, Ssh, T0);
}

// ------------------------------------------------------------------ P2M
// Eq. P2M in level-scaled form: Mhat_n^m = sum_j q_j R_n^m((r_M - r_j)/h).
// factors of the recurrences R_n^m = (a_nm z R_{n-1}^m - b_nm r^2 R_{n-2}^m) and R_m^m = c_m (x + iy) R_{m-1}^{m-1}
template <typename T>
struct ExpandFactors {
    T a[(P_MAX + 1) * (P_MAX + 1)], b[(P_MAX + 1) * (P_MAX + 1)], c[P_MAX + 1];
    constexpr ExpandFactors() : a{}, b{}, c{}
    {
        for (int m = 0; m <= P_MAX; ++m) {
            c[m] = m > 0 ? T(-0.5) / T(m) : T(0);
            for (int n = m + 1; n <= P_MAX; ++n) {
                a[m * (P_MAX + 1) + n] = T(2 * n - 1) / T((n + m) * (n - m));
                b[m * (P_MAX + 1) + n] = T(1) / T((n + m) * (n - m));
            }
        }
    }
};
__constant__ ExpandFactors<double> expand_factors64 = ExpandFactors<double>();
__constant__ ExpandFactors<float> expand_factors32 = ExpandFactors<float>();
template <typename T>
__device__ __forceinline__ const ExpandFactors<T> &expand_factors();
template <>
__device__ __forceinline__ const ExpandFactors<double> &expand_factors<double>() { return expand_factors64; }
template <>
__device__ __forceinline__ const ExpandFactors<float> &expand_factors<float>() { return expand_factors32; }

__device__ __forceinline__ unsigned p2m_bits(float x) { return __float_as_uint(fmaxf(0.f, fabsf(x))); }  // a NaN drops
__device__ __forceinline__ unsigned long long p2m_bits(double x)  // a NaN is larger than all
{
    return (unsigned long long)__double_as_longlong(x) & ~(1ull << 63);
}

// Any order, FP64 or FP32: a warp takes `lb` consecutive leaves, whose charges are contiguous, and runs the recurrences
// with one charge per lane, 32 at a time; the columns m of the 32 charges go through shared memory, where the lanes
// take one coefficient each and add up every leaf's charges in order.  GB300's FP64 pipe takes 16 cycles per warp
// instruction however many lanes are active, so what counts is that no lane idles: with one thread per (leaf, m), whose
// loops run to the longest column and fullest leaf of the warp, 100,000 charges at p = 12 took 776 us and 2,998 at
// p = 8 109 us; here 302 us and, shared, 22 us.  The warps of a block share the same charges and take the columns m in
// turn (small systems: one warp, on one of an SM's four FP64 pipes, took 46 us for the latter).  sx, amax (or null): the
// level's largest |M sx| is folded in; cmax (FP64, with amax): that of each leaf, the double's upper word.
constexpr int P2M_SHARE = 4;  // warps that share 32 charges in small systems

template <typename T, typename U>
__global__ void __launch_bounds__(32 * P2M_SHARE) k_p2m(int p, int d, int lb, const int *__restrict__ start,
                                            const Particle<T> *__restrict__ sp, T inv_h, T *__restrict__ M,
                                            const T *__restrict__ sx, U *__restrict__ amax,
                                            uint32_t *__restrict__ cmax)
{
    extern __shared__ __align__(16) unsigned char p2m_smem[];
    const ExpandFactors<T> &F = expand_factors<T>();
    const int nc = ncoef(p), lane = threadIdx.x & 31, warp = threadIdx.x >> 5, share = blockDim.x >> 5, nside = 1 << d;
    const int64_t nleaf = (int64_t)1 << (3 * d), leaf0 = (int64_t)blockIdx.x * lb;
    const int nl = (int)(nleaf - leaf0 < lb ? nleaf - leaf0 : lb);
    T *rows = reinterpret_cast<T *>(p2m_smem);  // [lb][nc]
    T *col = rows + lb * nc + warp * 2 * (p + 1) * 33;  // [2 (p + 1)][33]: the column's (n, Re | Im) of the 32 charges
    int *st = reinterpret_cast<int *>(rows + lb * nc + share * 2 * (p + 1) * 33);
    for (int i = threadIdx.x; i <= nl; i += blockDim.x) st[i] = start[leaf0 + i];
    for (int e = threadIdx.x; e < nl * nc; e += blockDim.x) rows[e] = 0;
    __syncthreads();
    const int s1 = st[nl];
    for (int c0 = st[0]; c0 < s1; c0 += 32) {
        Particle<T> pt = {};
        if (c0 + lane < s1) pt = sp[c0 + lane];
        const T vx = -pt.x * inv_h, vy = -pt.y * inv_h, vz = -pt.z * inv_h;
        const T r2 = vx * vx + vy * vy + vz * vz;
        T dre = pt.q, dim = 0;  // q R_m^m
        for (int m = 0; m <= p; ++m) {
            if (m > 0) {
                const T cx = F.c[m] * vx, cy = F.c[m] * vy;
                const T nre = cx * dre - cy * dim;
                dim = cx * dim + cy * dre;
                dre = nre;
            }
            if (m % share != warp) continue;  // another warp's column
            T p2re = 0, p2im = 0, p1re = dre, p1im = dim;
            col[lane] = dre;
            col[33 + lane] = dim;
            for (int n = m + 1; n <= p; ++n) {
                const T a = F.a[m * (P_MAX + 1) + n] * vz, b = F.b[m * (P_MAX + 1) + n] * r2;
                const T cr = a * p1re - b * p2re, ci = a * p1im - b * p2im;
                col[(2 * (n - m)) * 33 + lane] = cr;
                col[(2 * (n - m) + 1) * 33 + lane] = ci;
                p2re = p1re;
                p2im = p1im;
                p1re = cr;
                p1im = ci;
            }
            __syncwarp();
            for (int v = lane; v < 2 * (p - m + 1); v += 32) {
                const int n = m + (v >> 1);
                if (m == 0 && (v & 1)) continue;
                const int idx = v & 1 ? cim(n, m) : cre(n, m);
                for (int i = 0; i < nl; ++i) {
                    const int b = st[i] > c0 ? st[i] - c0 : 0, e = st[i + 1] < c0 + 32 ? st[i + 1] - c0 : 32;
                    if (b >= e) continue;
                    T acc = rows[i * nc + idx];
                    for (int j = b; j < e; ++j) acc += col[v * 33 + j];
                    rows[i * nc + idx] = acc;
                }
            }
            __syncwarp();
        }
    }
    __syncthreads();
    U mx = 0;
    for (int i = warp; i < nl; i += share) {
        const int leaf = (int)(leaf0 + i);
        const int64_t cell = cell_index(d, leaf & (nside - 1), (leaf >> d) & (nside - 1), leaf >> (2 * d));
        T *out = M + cell * nc;
        U mc = 0;
        for (int k = lane; k < nc; k += 32) {
            const T v = rows[i * nc + k];
            out[k] = v;
            if (amax) {
                const U b = p2m_bits(v * sx[k]);
                mc = b > mc ? b : mc;
            }
        }
        mx = mc > mx ? mc : mx;
        if constexpr (sizeof(U) == 8) {
            if (cmax) {
                const uint32_t h = __reduce_max_sync(0xffffffffu, (uint32_t)(mc >> 32));
                if (lane == 0) cmax[cell] = h;
            }
        }
    }
    if (amax) {
        for (int o = 16; o > 0; o >>= 1) {
            const U v = __shfl_xor_sync(0xffffffffu, mx, o);
            mx = v > mx ? v : mx;
        }
        if (lane == 0 && mx > 0) atomicMax(amax, mx);
    }
}

// The same P2M at a compile-time order PP in FP32, LPL lanes per leaf: a warp takes 32 / LPL leaves of one
// parity class with consecutive parent coordinates (consecutive rows of the level's class layout),
// each lane runs the recurrences of Eq. P2M for its share of its leaf's charges with all (PP+1)^2 coefficients in
// registers (indices fold into immediates); the LPL lanes' sums are added in a fixed tree.  One lane per leaf is
// best where the leaves fill the GPU (262,144 leaves of 4 charges: 85 us); small trees and dense leaves leave it
// idle or serial, and take up to 8 (launch_p2m_fixed).  The rows go through shared memory (row stride (PP+1)^2, odd,
// so the 32 lanes hit 32 banks) and leave as 32 contiguous rows.  When `amax` is set (fp16x2 split) the
// warp also folds max_k |Mhat_k s(k)| into *amax (positive floats order as their bit patterns), which
// the tensor-core operand split needs for the level gain.
constexpr int P2M_WARPS = 4;

template <int PP, int LPL>
__global__ void __launch_bounds__(32 * P2M_WARPS) k_p2m_fixed(int d, const int *__restrict__ start,
                                                              const Particle<float> *__restrict__ sp, float inv_h,
                                                              float *__restrict__ M, const float *__restrict__ s,
                                                              unsigned *__restrict__ amax)
{
    constexpr int NC = (PP + 1) * (PP + 1);
    constexpr int ROWS = 32 / LPL;
    extern __shared__ float p2m_tile[];  // [P2M_WARPS][ROWS][NC]
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float *tile = p2m_tile + w * ROWS * NC;
    const int np = 1 << (d - 1);
    const int64_t ncls = (int64_t)np * np * np;
    const int64_t row0 = ((int64_t)blockIdx.x * P2M_WARPS + w) * ROWS;
    if (row0 >= 8 * ncls) return;
    const int64_t row = row0 + lane / LPL;
    const bool valid = row < 8 * ncls;
    float acc[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) acc[k] = 0.f;
    if (valid) {
        const int c = (int)(row / ncls);
        const int64_t P = row - c * ncls;
        const int x = 2 * (int)(P % np) + (c & 1), y = 2 * (int)((P / np) % np) + ((c >> 1) & 1),
                  z = 2 * (int)(P / ((int64_t)np * np)) + ((c >> 2) & 1);
        const int nside = 2 * np;
        const int leaf = x + nside * (y + nside * z);
        const int b = start[leaf], e = start[leaf + 1];
        for (int j = b + lane % LPL; j < e; j += LPL) {
            const Particle<float> pt = sp[j];
            const float vx = -pt.x * inv_h, vy = -pt.y * inv_h, vz = -pt.z * inv_h;
            const float r2 = vx * vx + vy * vy + vz * vz;
            float dre = pt.q, dim = 0.f;  // q R_m^m
#pragma unroll
            for (int m = 0; m <= PP; ++m) {
                if (m > 0) {
                    const float sc = -0.5f / (float)m;
                    const float nre = sc * (vx * dre - vy * dim);
                    const float nim = sc * (vx * dim + vy * dre);
                    dre = nre;
                    dim = nim;
                }
                acc[cre(m, m)] += dre;
                if (m > 0) acc[cim(m, m)] += dim;
                float p2re = 0.f, p2im = 0.f, p1re = dre, p1im = dim;
                // a trip count fixed at compile time (n = m + 1 + i, dead steps folded away) so that both
                // loops unroll completely and acc[] stays in registers
#pragma unroll
                for (int i = 0; i < PP; ++i) {
                    const int n = m + 1 + i;
                    if (n > PP) break;
                    const float a = (float)(2 * n - 1) * vz;
                    const float inv = 1.f / (float)((n + m) * (n - m));
                    const float cr = (a * p1re - r2 * p2re) * inv;
                    const float ci = (a * p1im - r2 * p2im) * inv;
                    acc[cre(n, m)] += cr;
                    if (m > 0) acc[cim(n, m)] += ci;
                    p2re = p1re;
                    p2im = p1im;
                    p1re = cr;
                    p1im = ci;
                }
            }
        }
    }
#pragma unroll
    for (int o = LPL / 2; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < NC; ++k) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
    float mx = 0.f;
    if (lane % LPL == 0) {
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            tile[(lane / LPL) * NC + k] = acc[k];
            if (amax) mx = fmaxf(mx, fabsf(acc[k] * __ldg(s + k)));
        }
    }
    __syncwarp();
    const int64_t nrows = 8 * ncls - row0 < ROWS ? 8 * ncls - row0 : ROWS;
    float *dst = M + row0 * NC;
    for (int64_t e = lane; e < nrows * NC; e += 32) dst[e] = tile[e];
    if (amax) {
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0 && mx > 0.f) atomicMax(amax, __float_as_uint(mx));
    }
}

template <int PP, int LPL>
fmm_status run_p2m_fixed(Plan &P, const Particle<float> *sp, float inv_h, unsigned *amax, const float *s)
{
    constexpr int NC = (PP + 1) * (PP + 1), ROWS = 32 / LPL;
    const size_t sh = sizeof(float) * P2M_WARPS * ROWS * NC;
    static bool attr = false;
    if (!attr) {
        FMM_CUDA_TRY(cudaFuncSetAttribute(k_p2m_fixed<PP, LPL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh));
        attr = true;
    }
    const unsigned blocks = (unsigned)((P.nleaf + ROWS * P2M_WARPS - 1) / (ROWS * P2M_WARPS));
    k_p2m_fixed<PP, LPL><<<blocks, 32 * P2M_WARPS, sh, P.stream>>>(P.d, P.cell_start, sp, inv_h, (float *)P.M[P.d], s, amax);
    FMM_LAUNCH_CHECK(P);
    return FMM_OK;
}

// lanes per leaf: the fewest that give every SM 8 warps and no lane more than about 6 charges (beyond 8 the
// shuffles of the (p+1)^2 sums cost more than the charges)
template <int PP>
fmm_status launch_p2m_fixed(Plan &P, const Particle<float> *sp, float inv_h, unsigned *amax, const float *s)
{
    int lpl = 1;
    while (lpl < 8 && (P.nleaf * lpl < 32 * 1216 || (double)P.N > 6.0 * lpl * (double)P.nleaf)) lpl *= 2;
    switch (lpl) {
    case 1: return run_p2m_fixed<PP, 1>(P, sp, inv_h, amax, s);
    case 2: return run_p2m_fixed<PP, 2>(P, sp, inv_h, amax, s);
    case 4: return run_p2m_fixed<PP, 4>(P, sp, inv_h, amax, s);
    default: return run_p2m_fixed<PP, 8>(P, sp, inv_h, amax, s);
    }
}

// leaves per warp: about 28 charges, so that mostly one round of 32 does, within 24 KB of rows and 32 leaves
template <typename T, typename U>
fmm_status launch_p2m(Plan &P, const Particle<T> *sp, T inv_h, const T *sx, U *amax, uint32_t *cmax)
{
    const double occ = (double)P.N / (double)P.nleaf;
    const int fit = (int)(24576 / (sizeof(T) * P.nc)), most = fit < 32 ? fit : 32;
    int lb = (int)(28.0 / occ < most ? 28.0 / occ : most);
    if (lb < 1) lb = 1;
    // a warp per charge group where those groups fill the SMs' pipes; a column buffer per warp, 48 KB in all
    int share = P.N < 152 * 32 * 4 ? P2M_SHARE : 1;
    if (sizeof(T) * 2 * (P.p + 1) * 33 * share > 23000) share = 2;
    const size_t sh = sizeof(T) * ((size_t)lb * P.nc + 2 * (P.p + 1) * 33 * share) + sizeof(int) * (lb + 1);
    k_p2m<T, U><<<(unsigned)((P.nleaf + lb - 1) / lb), 32 * share, sh, P.stream>>>(P.p, P.d, lb, P.cell_start, sp, inv_h,
                                                                            (T *)P.M[P.d], sx, amax, cmax);
    FMM_LAUNCH_CHECK(P);
    return FMM_OK;
}

// ------------------------------------------------------------------ M2L (CUDA cores)
// Eq. Lcoeffdef over the 189-cell interaction list of each target, as dense
// real operators per offset.  Block: TT targets of one parity class, one
// thread per output coefficient.  Sources are read with periodic wrap.
template <typename T, int TT>
__global__ void k_m2l_simt(int p, int l, int cls, int ws, const T *__restrict__ Top, const T *__restrict__ M,
                           T *__restrict__ L)
{
    extern __shared__ unsigned char smem_raw[];
    T *S = reinterpret_cast<T *>(smem_raw);  // [TT][nc]
    int nc = ncoef(p);
    int np = 1 << (l - 1);
    int64_t ncls = (int64_t)np * np * np;
    int64_t t0 = (int64_t)blockIdx.x * TT;
    int cx = cls & 1, cy = (cls >> 1) & 1, cz = (cls >> 2) & 1;
    int j = threadIdx.x;
    T acc[TT];
#pragma unroll
    for (int t = 0; t < TT; ++t) acc[t] = 0;
    // delta per axis in [-2 ws - c, 2 ws + 1 - c]: the children of the parent's
    // (2 ws + 1)^3 neighbours that are not the target's own neighbours
    for (int dz = -2 * ws - cz; dz <= 2 * ws + 1 - cz; ++dz)
        for (int dy = -2 * ws - cy; dy <= 2 * ws + 1 - cy; ++dy)
            for (int dx = -2 * ws - cx; dx <= 2 * ws + 1 - cx; ++dx) {
                if (abs(dx) <= ws && abs(dy) <= ws && abs(dz) <= ws) continue;
                int sx = cx + dx, sy = cy + dy, sz = cz + dz;  // in [-2 ws, 2 ws + 1]
                int scls = (sx & 1) | ((sy & 1) << 1) | ((sz & 1) << 2);
                int Dx = sx >> 1, Dy = sy >> 1, Dz = sz >> 1;  // floor division
                __syncthreads();
                for (int e = threadIdx.x; e < TT * nc; e += blockDim.x) {
                    int t = e / nc, k = e % nc;
                    int64_t tg = t0 + t;
                    T v = 0;
                    if (tg < ncls) {
                        int Px = (int)(tg % np), Py = (int)((tg / np) % np), Pz = (int)(tg / ((int64_t)np * np));
                        int Qx = ((Px + Dx) % np + np) % np, Qy = ((Py + Dy) % np + np) % np,
                            Qz = ((Pz + Dz) % np + np) % np;
                        int64_t src = scls * ncls + Qx + (int64_t)np * (Qy + (int64_t)np * Qz);
                        v = M[src * nc + k];
                    }
                    S[t * nc + k] = v;
                }
                __syncthreads();
                if (j < nc) {
                    const T *Tp = Top + (size_t)off_slot(dx, dy, dz, ws) * nc * nc + j;
                    for (int k = 0; k < nc; ++k) {
                        T w = Tp[(size_t)k * nc];
#pragma unroll
                        for (int t = 0; t < TT; ++t) acc[t] += w * S[t * nc + k];
                    }
                }
            }
    if (j < nc) {
        for (int t = 0; t < TT; ++t) {
            int64_t tg = t0 + t;
            if (tg < ncls) L[(cls * ncls + tg) * nc + j] = acc[t];
        }
    }
}

// ------------------------------------------------------------------ L2P
// Phi(r) = (1/h) sum L_n^m R_n^m(v), v = (r - r_L')/h, and
// grad Phi = (1/h^2) sum_{n',m'} G_{n'}^{m'} R_{n'}^{m'}(v) with
//   G^z = L_{n'+1}^{m'},  G^x = (L_{n'+1}^{m'-1} - L_{n'+1}^{m'+1})/2,
//   G^y = -i (L_{n'+1}^{m'-1} + L_{n'+1}^{m'+1})/2.
// Any order, `split` neighbouring lanes per charge, which take the columns m in turn: in small FP64 systems a charge's
// whole sum by one thread is a long chain on few warps (an FP64 warp instruction holds one of an SM's four pipes for 64
// cycles; 2,998 charges at p = 8: 44 us, here 29 us).  The sums over n of a column are formed without its weight (1 for m = 0, else
// 2) and without the halves of G^x and G^y.
template <typename T>
__global__ void __launch_bounds__(128) k_l2p(int p, int split, int d, int64_t N, const int *__restrict__ sleaf,
                                             const Particle<T> *__restrict__ sp, T inv_h, const T *__restrict__ L,
                                             T *__restrict__ phi, T *__restrict__ grad)
{
    const ExpandFactors<T> &F = expand_factors<T>();
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const bool on = t < N * split;
    const int64_t s = on ? t / split : N - 1;  // the spare lanes of the last warp take part in the shuffles
    const int sub = (int)(t % split);
    const int mask = (1 << d) - 1, leaf = sleaf[s];
    const T *Lc = L + cell_index(d, leaf & mask, (leaf >> d) & mask, leaf >> (2 * d)) * ncoef(p);
    const Particle<T> pt = sp[s];
    const T vx = pt.x * inv_h, vy = pt.y * inv_h, vz = pt.z * inv_h;
    const T r2 = vx * vx + vy * vy + vz * vz;
    T pot = 0, gx = 0, gy = 0, gz = 0;
    T dre = 1, dim = 0;
    int at = 0;  // (dre, dim) = R_at^at
    for (int m = sub; m <= p; m += split) {
        for (; at < m; ++at) {
            const T cx = F.c[at + 1] * vx, cy = F.c[at + 1] * vy;
            const T nre = cx * dre - cy * dim;
            dim = cx * dim + cy * dre;
            dre = nre;
        }
        T p2re = 0, p2im = 0, rre = dre, rim = dim;
        T spot = 0, sx = 0, sy = 0, sz = 0;
        for (int n = m; n <= p; ++n) {
            if (n > m) {
                const T a = F.a[m * (P_MAX + 1) + n] * vz, b = F.b[m * (P_MAX + 1) + n] * r2;
                const T cr = a * rre - b * p2re, ci = a * rim - b * p2im;
                p2re = rre;
                p2im = rim;
                rre = cr;
                rim = ci;
            }
            const Cx<T> Lnm = coef(Lc, n, m);
            spot += Lnm.re * rre - Lnm.im * rim;
            if (grad && n < p) {
                const Cx<T> a = coef(Lc, n + 1, m - 1), b = coef(Lc, n + 1, m + 1), c = coef(Lc, n + 1, m);
                sx += (a.re - b.re) * rre - (a.im - b.im) * rim;
                sy += (a.im + b.im) * rre + (a.re + b.re) * rim;
                sz += c.re * rre - c.im * rim;
            }
        }
        const T w = m == 0 ? T(1) : T(2);
        pot += w * spot;
        gx += w * sx;
        gy += w * sy;
        gz += w * sz;
    }
    for (int o = 1; o < split; o <<= 1) {
        pot += __shfl_xor_sync(0xffffffffu, pot, o);
        gx += __shfl_xor_sync(0xffffffffu, gx, o);
        gy += __shfl_xor_sync(0xffffffffu, gy, o);
        gz += __shfl_xor_sync(0xffffffffu, gz, o);
    }
    if (!on || sub != 0) return;
    phi[s] = pot * inv_h;
    if (grad) {
        const T s2 = inv_h * inv_h;
        grad[3 * s] = T(0.5) * gx * s2;
        grad[3 * s + 1] = T(0.5) * gy * s2;
        grad[3 * s + 2] = gz * s2;
    }
}

// L2P at a compile-time order PP, one thread per charge: the loops unroll, the recurrences' reciprocals fold into
// constants and the coefficient indices into immediates.  The expansions of the block's leaves
// (consecutive in the sorted order) are staged in shared memory when at most L2P_LEAVES of them span
// the block: a warp's particles sit in several leaves, and each of its coefficient loads would touch
// as many L1 lines.
constexpr int L2P_LEAVES = 48;
constexpr int L2P_THREADS = 128;

template <typename T, int PP>
__global__ void __launch_bounds__(L2P_THREADS) k_l2p_fixed(int d, int64_t N, const int *__restrict__ sleaf,
                                                           const Particle<T> *__restrict__ sp, T inv_h,
                                                           const T *__restrict__ L, T *__restrict__ phi,
                                                           T *__restrict__ grad)
{
    constexpr int NC = (PP + 1) * (PP + 1);
    extern __shared__ __align__(16) unsigned char l2p_smem[];
    T *sL = reinterpret_cast<T *>(l2p_smem);
    const int64_t s0 = (int64_t)blockIdx.x * L2P_THREADS;
    const int64_t slast = (s0 + L2P_THREADS < N ? s0 + L2P_THREADS : N) - 1;
    const int nside = 1 << d, mask = nside - 1;
    const int leaf0 = sleaf[s0];
    const int nl = sleaf[slast] - leaf0 + 1;
    const bool staged = nl <= L2P_LEAVES;
    if (staged) {
        for (int e = threadIdx.x; e < nl * NC; e += L2P_THREADS) {
            const int li = e / NC, c = e - li * NC;
            const int leaf = leaf0 + li;
            sL[e] = L[cell_index(d, leaf & mask, (leaf >> d) & mask, leaf >> (2 * d)) * NC + c];
        }
    }
    __syncthreads();
    const int64_t s = s0 + threadIdx.x;
    if (s >= N) return;
    const int leaf = sleaf[s];
    const T *Lc = staged ? sL + (leaf - leaf0) * NC : L + cell_index(d, leaf & mask, (leaf >> d) & mask, leaf >> (2 * d)) * NC;
    const Particle<T> pt = sp[s];
    const T vx = pt.x * inv_h, vy = pt.y * inv_h, vz = pt.z * inv_h;
    const T r2 = vx * vx + vy * vy + vz * vz;
    T pot = 0, gx = 0, gy = 0, gz = 0;
    T dre = 1, dim = 0;
#pragma unroll
    for (int m = 0; m <= PP; ++m) {
        if (m > 0) {
            const T sc = T(-0.5) / T(m);
            const T nre = sc * (vx * dre - vy * dim);
            const T nim = sc * (vx * dim + vy * dre);
            dre = nre;
            dim = nim;
        }
        const T w = m == 0 ? T(1) : T(2);
        T p2re = 0, p2im = 0, rre = dre, rim = dim;
#pragma unroll
        for (int n = m; n <= PP; ++n) {
            if (n > m) {
                const T a = T(2 * n - 1) * vz;
                const T inv = T(1) / T((n + m) * (n - m));
                const T cr = (a * rre - r2 * p2re) * inv;
                const T ci = (a * rim - r2 * p2im) * inv;
                p2re = rre;
                p2im = rim;
                rre = cr;
                rim = ci;
            }
            const Cx<T> Lnm = coef(Lc, n, m);
            pot += w * (Lnm.re * rre - Lnm.im * rim);
            if (grad && n < PP) {
                const Cx<T> a = coef(Lc, n + 1, m - 1), b = coef(Lc, n + 1, m + 1), c = coef(Lc, n + 1, m);
                const Cx<T> Gx = {T(0.5) * (a.re - b.re), T(0.5) * (a.im - b.im)};
                const Cx<T> Gy = {T(0.5) * (a.im + b.im), -T(0.5) * (a.re + b.re)};
                gx += w * (Gx.re * rre - Gx.im * rim);
                gy += w * (Gy.re * rre - Gy.im * rim);
                gz += w * (c.re * rre - c.im * rim);
            }
        }
    }
    phi[s] = pot * inv_h;
    if (grad) {
        const T s2 = inv_h * inv_h;
        grad[3 * s] = gx * s2;
        grad[3 * s + 1] = gy * s2;
        grad[3 * s + 2] = gz * s2;
    }
}

template <typename T, int PP>
fmm_status launch_l2p_fixed(Plan &P, T inv_h, const T *L, T *phi, T *grad)
{
    const size_t sh = sizeof(T) * L2P_LEAVES * (PP + 1) * (PP + 1);
    static bool attr = false;
    if (!attr) {
        FMM_CUDA_TRY(cudaFuncSetAttribute(k_l2p_fixed<T, PP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh));
        attr = true;
    }
    k_l2p_fixed<T, PP><<<blocks_for(P.N, L2P_THREADS), L2P_THREADS, sh, P.stream>>>(
        P.d, P.N, P.sleaf, (const Particle<T> *)(P.sorted), inv_h, L, phi, grad);
    return FMM_OK;
}

// L2P of the plan at its order: the fixed-order kernel for the usual orders, else the generic one, and that with four
// lanes per charge in FP64 where one lane each would leave a pipe without a warp
template <typename T>
fmm_status l2p_t(Plan &P, T inv_h, const T *L, T *phi, T *grad)
{
    const int split = std::is_same<T, double>::value && P.N < 152 * 32 * 4 ? 4 : 1;
    switch (split > 1 ? -1 : P.p) {
    case 4: return launch_l2p_fixed<T, 4>(P, inv_h, L, phi, grad);
    case 6: return launch_l2p_fixed<T, 6>(P, inv_h, L, phi, grad);
    case 8: return launch_l2p_fixed<T, 8>(P, inv_h, L, phi, grad);
    case 10: return launch_l2p_fixed<T, 10>(P, inv_h, L, phi, grad);
    case 12: return launch_l2p_fixed<T, 12>(P, inv_h, L, phi, grad);
    default:
        k_l2p<T><<<blocks_for(P.N * split, 128), 128, 0, P.stream>>>(P.p, split, P.d, P.N, P.sleaf,
                                                                     (const Particle<T> *)P.sorted, inv_h, L, phi, grad);
        return FMM_OK;
    }
}

template <typename T>
fmm_status upward_t(Plan &P, bool solute_only)
{
    const int nside = 1 << P.d;
    const Particle<T> *sp = (const Particle<T> *)(solute_only ? P.sorted_u : P.sorted);
    T inv_h = (T)((double)nside / P.box);
    const bool tc = tc_translations(P);
    {
        fmm_status st = tc ? tc_clear_amax(P) : res_clear_amax(P);
        if (st != FMM_OK) return st;
    }
    // where the M2L runs on the tensor cores, the P2M folds the level maximum of |Mhat s| in as it writes.  FP32 at the
    // usual orders keeps its coefficients in registers, unless leaves are so full that 8 lanes each would run long
    fmm_status st;
    if constexpr (std::is_same<T, float>::value) {
        unsigned *amax = tc ? tc_amax(P, P.d) : nullptr;
        const float *sc = tc ? tc_scale(P) : nullptr;
        const bool sparse = (double)P.N <= 128.0 * (double)P.nleaf;
        st = sparse && P.p == 4    ? launch_p2m_fixed<4>(P, sp, inv_h, amax, sc)
             : sparse && P.p == 6  ? launch_p2m_fixed<6>(P, sp, inv_h, amax, sc)
             : sparse && P.p == 8  ? launch_p2m_fixed<8>(P, sp, inv_h, amax, sc)
             : sparse && P.p == 10 ? launch_p2m_fixed<10>(P, sp, inv_h, amax, sc)
             : sparse && P.p == 12 ? launch_p2m_fixed<12>(P, sp, inv_h, amax, sc)
                                   : launch_p2m<float, unsigned>(P, sp, inv_h, sc, amax, nullptr);
    } else {
        const double *sc = nullptr;
        uint32_t *cmax = nullptr;
        unsigned long long *amax = res_amax(P, P.d, &sc, &cmax);
        st = launch_p2m<double, unsigned long long>(P, sp, inv_h, sc, amax, cmax);
    }
    if (st != FMM_OK) return st;
    for (int l = P.d - 1; l >= 1; --l) {  // the top operator starts from level 1
        fmm_status st = launch_m2m(P, l);
        if (st != FMM_OK) return st;
    }
    return tc ? tc_split_moments(P) : FMM_OK;
}

}  // namespace

// ------------------------------------------------------------------ host side
fmm_status build_tables(Plan &P)
{
    free_tables(P);
    int p = P.p, nc = P.nc;
    FMM_CUDA_TRY(cudaMalloc(&P.tab.Rw64, sizeof(double) * 8 * nc));
    int ntri2 = (2 * p + 1) * (2 * p + 2) / 2;
    FMM_CUDA_TRY(cudaMalloc(&P.tab.S, sizeof(double) * 2 * ntri2));
    FMM_CUDA_TRY(cudaMalloc(&P.tab.T0, sizeof(double) * nc * nc));
    FMM_CUDA_TRY(cudaMalloc(&P.tab.Top64, sizeof(double) * (size_t)noff(P.ws) * nc * nc));
    FMM_CUDA_TRY(cudaMalloc(&P.tab.Top32, sizeof(float) * (size_t)noff(P.ws) * nc * nc));
    {
        const int n = n_il(P.ws), ws = P.ws;
        std::vector<int> h;
        h.reserve((size_t)8 * n);
        for (int c = 0; c < 8; ++c)
            for (int dz = -2 * ws - (c >> 2); dz <= 2 * ws + 1 - (c >> 2); ++dz)
                for (int dy = -2 * ws - ((c >> 1) & 1); dy <= 2 * ws + 1 - ((c >> 1) & 1); ++dy)
                    for (int dx = -2 * ws - (c & 1); dx <= 2 * ws + 1 - (c & 1); ++dx)
                        if (!(abs(dx) <= ws && abs(dy) <= ws && abs(dz) <= ws)) h.push_back(il_pack(dx, dy, dz));
        if (h.size() != (size_t)8 * n) return FMM_ERR_INTERNAL;
        FMM_CUDA_TRY(cudaMalloc(&P.tab.il, sizeof(int) * h.size()));
        FMM_CUDA_TRY(cudaMemcpyAsync(P.tab.il, h.data(), sizeof(int) * h.size(), cudaMemcpyHostToDevice, P.stream));
        FMM_CUDA_TRY(cudaStreamSynchronize(P.stream));
    }
    k_octant_table<<<1, 32, 0, P.stream>>>(p, P.tab.Rw64);
    FMM_LAUNCH_CHECK(P);
    {
        fmm_status st = build_translation_ops(P);
        if (st != FMM_OK) return st;
    }
    size_t shI = sizeof(Cx<double>) * ntri2;
    k_m2l_operators<<<noff(P.ws), 256, shI, P.stream>>>(p, P.ws, P.tab.Top64, P.tab.Top32);
    FMM_LAUNCH_CHECK(P);
    double kappa = P.kappa > 0 ? P.kappa : 2.0 / P.box;
    double kb = kappa * P.box;
    int nu_max = (int)ceil(8.0 / kb) + 3 + P.ws;
    int nk_max = (int)ceil(2.2 * kb) + 3;
    k_lattice_sum<<<ntri2, LAT_THREADS, 0, P.stream>>>(2 * p, kb, P.ws, nu_max, nk_max, P.tab.S);
    FMM_LAUNCH_CHECK(P);
    k_lattice_operator<<<1, 256, shI, P.stream>>>(p, P.tab.S, P.tab.T0);
    FMM_LAUNCH_CHECK(P);
    return build_top(P);
}

fmm_status build_lattice(Plan &P)
{
    if (!P.tab.S || !P.tab.T0) return build_tables(P);
    int p = P.p;
    int ntri2 = (2 * p + 1) * (2 * p + 2) / 2;
    double kappa = P.kappa > 0 ? P.kappa : 2.0 / P.box;
    double kb = kappa * P.box;
    int nu_max = (int)ceil(8.0 / kb) + 3 + P.ws;
    int nk_max = (int)ceil(2.2 * kb) + 3;
    k_lattice_sum<<<ntri2, LAT_THREADS, 0, P.stream>>>(2 * p, kb, P.ws, nu_max, nk_max, P.tab.S);
    FMM_LAUNCH_CHECK(P);
    k_lattice_operator<<<1, 256, sizeof(Cx<double>) * ntri2, P.stream>>>(p, P.tab.S, P.tab.T0);
    FMM_LAUNCH_CHECK(P);
    return build_top(P);
}

void free_tables(Plan &P)
{
    cudaFree(P.tab.Rw64);
    cudaFree(P.tab.S);
    cudaFree(P.tab.T0);
    cudaFree(P.tab.Top64);
    cudaFree(P.tab.Top32);
    cudaFree(P.tab.l2l64);
    cudaFree(P.tab.l2l32);
    cudaFree(P.tab.m2m64);
    cudaFree(P.tab.m2m_fold64);  // and the other folded tables behind it
    cudaFree(P.tab.il);
    cudaFree(P.tab.G64);
    cudaFree(P.tab.G32);
    P.tab = Tables{};
}

fmm_status launch_upward(Plan &P, bool solute_only)
{
    return P.precision == FMM_PREC_FP64 ? upward_t<double>(P, solute_only) : upward_t<float>(P, solute_only);
}

fmm_status launch_m2l_simt(Plan &P, int l)
{
    int nc = P.nc;
    int threads = ((nc + 31) / 32) * 32;
    int64_t np = (int64_t)1 << (l - 1);
    int64_t ncls = np * np * np;
    static bool attr_set = false;
    if (!attr_set) {
        FMM_CUDA_TRY(cudaFuncSetAttribute(k_m2l_simt<double, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)(sizeof(double) * 16 * NC_MAX)));
        FMM_CUDA_TRY(cudaFuncSetAttribute(k_m2l_simt<float, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)(sizeof(float) * 32 * NC_MAX)));
        attr_set = true;
    }
    for (int cls = 0; cls < 8; ++cls) {
        if (P.precision == FMM_PREC_FP64) {
            constexpr int TT = 16;
            size_t sh = sizeof(double) * TT * nc;
            k_m2l_simt<double, TT><<<blocks_for(ncls, TT), threads, sh, P.stream>>>(
                P.p, l, cls, P.ws, P.tab.Top64, (const double *)P.M[l], (double *)P.L[l]);
        } else {
            constexpr int TT = 32;
            size_t sh = sizeof(float) * TT * nc;
            k_m2l_simt<float, TT><<<blocks_for(ncls, TT), threads, sh, P.stream>>>(
                P.p, l, cls, P.ws, P.tab.Top32, (const float *)P.M[l], (float *)P.L[l]);
        }
        FMM_LAUNCH_CHECK(P);
    }
    return FMM_OK;
}

fmm_status launch_l2p(Plan &P, bool gradient, bool solute_only)
{
    int nside = 1 << P.d;
    double inv_h = (double)nside / P.box;
    fmm_status st;
    if (P.precision == FMM_PREC_FP64)
        st = l2p_t<double>(P, inv_h, (const double *)P.L[P.d], (double *)(solute_only ? P.phi_u : P.phi_ff),
                           gradient ? (double *)P.g_ff : nullptr);
    else
        st = l2p_t<float>(P, (float)inv_h, (const float *)P.L[P.d], (float *)(solute_only ? P.phi_u : P.phi_ff),
                          gradient ? (float *)P.g_ff : nullptr);
    if (st != FMM_OK) return st;
    FMM_LAUNCH_CHECK(P);
    return FMM_OK;
}

}  // namespace fmm
