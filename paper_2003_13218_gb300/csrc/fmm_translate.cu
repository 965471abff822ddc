// fmm_translate.cu -- M2M and L2L (Appendix B), folded over the eight child octants.
//
// In level-scaled coefficients both translations are fixed linear maps per
// child octant s (w_s = child-centre offset / parent side = (+-1/4)^3):
//   L2L: Lhat_k^l(child) = sum_{n >= k, m} Lhat_n^m(parent) R_{n-k}^{m-l}(w_s) 2^{-(k+1)}
//   M2M: Mhat_n^m(parent) = sum_s sum_{k <= n, l} R_{n-k}^{m-l}(-w_s) Mhat_k^l(child_s) 2^{-k}
// The octants are mirror images of octant 0, and a reflection only changes signs of the real coefficients
// (x: (-1)^m for Re, -(-1)^m for Im; y: Im; z: (-1)^(n+m)).  With chi_j the three sign bits of coefficient j
// and A the operator of octant 0, A_s[j][k] = (-1)^((chi_j ^ chi_k) . s) A[j][k], so
//   M2M: M[j]   = sum_k A[j][k] W_{chi_j ^ chi_k}[k],          W_c[k] = sum_s (-1)^(c . s) m_s[k]
//   L2L: L_s[j] = sum_c (-1)^(c . s) V_c[j],                   V_c[j] = sum_{k: chi_j ^ chi_k = c} A[j][k] l[k]
// with butterflies over the eight children: one operator instead of eight.  A is sparse as well (|m - l| <= |n - k|,
// and half of the rest vanishes on the diagonal x = y): a quarter of the entries at p = 6, less above.  Together
// 1/30 of the dense products, which leaves loads as the bound: shared memory on wide levels, the latency of a row's
// chain on the top ones.
//
// Measured: FP64, 100,000 charges at depth 5, p = 12: 0.51 ms for all M2M and L2L launches, the call 11.7 -> 8.05 ms
// (dense FP64 products, 1.2 TFLOP/s at most).  Mixed path: the M2M ran on the tensor cores on operands rounded to two
// fp16 terms and waited for the level's split; in FP32 here, with one split launch for all levels, 2,998 charges take
// 300 us (316), 61,000 with 210 solute charges 559 us (602); 1M and 10M within 1 % of before.
#include <math.h>

#include <algorithm>
#include <vector>

#include "fmm_internal.cuh"

namespace fmm {

namespace {

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

__host__ __device__ inline void split_index(int j, int &n, int &m, bool &im)
{
    n = (int)sqrt((double)j);
    while (n * n > j) --n;
    while ((n + 1) * (n + 1) <= j) ++n;
    int r = j - n * n;
    m = (r + 1) / 2;
    im = (m > 0) && (r == 2 * m);
}

// unit input coefficient: C_n^m = u (u = 1 or i), C_n^{-m} = (-1)^m conj(u)
__device__ inline Cx<double> unit_pos(bool im) { return im ? Cx<double>{0, 1} : Cx<double>{1, 0}; }
__device__ inline Cx<double> unit_neg(bool im, int m)
{
    Cx<double> u = unit_pos(im);
    u.im = -u.im;
    if (m & 1) {
        u.re = -u.re;
        u.im = -u.im;
    }
    return u;
}

// L2L operators, row-major [8 nc][nc]: row c nc + j (child output j), column e (parent input)
__global__ void k_l2l_ops(int p, const double *__restrict__ Rw, double *__restrict__ A64, float *__restrict__ A32)
{
    int nc = ncoef(p);
    int64_t total = (int64_t)8 * nc * nc;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        int e = (int)(t % nc);
        int row = (int)(t / nc);
        int c = row / nc, j = row % nc;
        int k, l, n, m;
        bool oim, iim;
        split_index(j, k, l, oim);
        split_index(e, n, m, iim);
        double v = 0;
        if (n >= k) {
            const double *R = Rw + c * nc;
            Cx<double> acc = {0, 0};
            int dn = n - k;
            if (m - l >= -dn && m - l <= dn) acc = cmul(unit_pos(iim), coef(R, dn, m - l));
            if (m > 0 && -m - l >= -dn && -m - l <= dn) {
                Cx<double> t2 = cmul(unit_neg(iim, m), coef(R, dn, -m - l));
                acc.re += t2.re;
                acc.im += t2.im;
            }
            double s = ldexp(1.0, -(k + 1));
            v = s * (oim ? acc.im : acc.re);
        }
        A64[t] = v;
        A32[t] = (float)v;
        const size_t tt = (size_t)total + (size_t)e * (8 * nc) + row;  // transposed copy [nc][8 nc]
        A64[tt] = v;
        A32[tt] = (float)v;
    }
}

// M2M operators, row-major [nc][8 nc]: row j (parent output), column c nc + e (child input)
__global__ void k_m2m_ops(int p, const double *__restrict__ Rw, double *__restrict__ B64)
{
    int nc = ncoef(p);
    int64_t total = (int64_t)8 * nc * nc;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        int col = (int)(t % (8 * nc));
        int j = (int)(t / (8 * nc));
        int c = col / nc, e = col % nc;
        int n, m, k, l;
        bool oim, iim;
        split_index(j, n, m, oim);
        split_index(e, k, l, iim);
        double v = 0;
        if (k <= n) {
            const double *R = Rw + c * nc;
            int dn = n - k;
            double sg = (dn & 1) ? -1.0 : 1.0;  // R(-w) = (-1)^deg R(w)
            Cx<double> acc = {0, 0};
            if (m - l >= -dn && m - l <= dn) acc = cmul(coef(R, dn, m - l), unit_pos(iim));
            if (l > 0 && m + l >= -dn && m + l <= dn) {
                Cx<double> t2 = cmul(coef(R, dn, m + l), unit_neg(iim, l));
                acc.re += t2.re;
                acc.im += t2.im;
            }
            double s = sg * ldexp(1.0, -k);
            v = s * (oim ? acc.im : acc.re);
        }
        B64[t] = v;
    }
}

// ------------------------------------------------------------------ folded products
template <typename T>
struct alignas(2 * sizeof(T)) FoldEntry {  // a nonzero of a row of A: its value and the operand's index
    T v;
    int at;
};

// sign bits of coefficient j under the reflections of x (1), y (2) and z (4)
__host__ __device__ inline int mirror_signs(int j)
{
    int n, m;
    bool im;
    split_index(j, n, m, im);
    return ((m + im) & 1) | ((int)im << 1) | (((n + m) & 1) << 2);
}

// L2L: the nonzeros of row j of A, one warp per row, [entry][row] so that neighbouring rows' entries are contiguous; by
// c = chi_j ^ chi_k, at = k, those of c from beg[c nc + j] to beg[(c + 1) nc + j]
__global__ void k_l2l_entries(int nc, const double *__restrict__ A, FoldEntry<double> *__restrict__ e64,
                              FoldEntry<float> *__restrict__ e32, int *__restrict__ beg)
{
    const int j = blockIdx.x, lane = threadIdx.x;
    const int sj = mirror_signs(j);
    int at = 0;
    for (int c = 0; c < 8; ++c) {
        if (lane == 0) beg[c * nc + j] = at;
        for (int k0 = 0; k0 < nc; k0 += 32) {
            const int k = k0 + lane;
            const double v = k < nc ? A[(size_t)j * nc + k] : 0.0;
            const bool take = v != 0.0 && (sj ^ mirror_signs(k)) == c;
            const unsigned b = __ballot_sync(0xffffffffu, take);
            if (take) {
                const size_t o = (size_t)(at + __popc(b & ((1u << lane) - 1u))) * nc + j;
                e64[o] = {v, k};
                e32[o] = {(float)v, k};
            }
            at += __popc(b);
        }
    }
    if (lane == 0) beg[8 * nc + j] = at;
}

// M2M: the nonzeros of A's rows (A [nc][nc] on the host), at = (chi_j ^ chi_k) nc + k, cnt[j] of them, [entry][row].
// Eight neighbouring rows are read by a quarter warp, whose 16-byte loads of shared memory take one cycle if the
// operands' indices differ modulo 8 (in order of k they met 2 to 3 at a time, and the wide kernel is bound by those
// loads): each row in turn takes, of the residues that the step has left free, the one it has most entries of.
void m2m_entries(int nc, const std::vector<double> &A, std::vector<FoldEntry<double>> &ent, std::vector<int> &cnt)
{
    ent.assign((size_t)nc * nc, FoldEntry<double>{0.0, 0});
    cnt.assign(nc, 0);
    std::vector<int> sign(nc);
    for (int k = 0; k < nc; ++k) sign[k] = mirror_signs(k);
    for (int j0 = 0; j0 < nc; j0 += 8) {
        std::vector<int> left[8][8];  // [row][residue]: the k still to take, the lowest last
        for (int r = 0; r < 8 && j0 + r < nc; ++r)
            for (int k = nc - 1; k >= 0; --k)
                if (A[(size_t)(j0 + r) * nc + k] != 0.0)
                    left[r][((sign[j0 + r] ^ sign[k]) * nc + k) & 7].push_back(k);
        for (bool more = true; more;) {
            more = false;
            bool used[8] = {};
            for (int r = 0; r < 8 && j0 + r < nc; ++r) {
                int best = -1;
                size_t score = 0;
                for (int q = 0; q < 8; ++q) {
                    const size_t w = left[r][q].empty() ? 0 : left[r][q].size() + (used[q] ? 0 : (size_t)nc);
                    if (w > score) {
                        score = w;
                        best = q;
                    }
                }
                if (best < 0) continue;
                const int j = j0 + r, k = left[r][best].back();
                left[r][best].pop_back();
                used[best] = more = true;
                ent[(size_t)cnt[j]++ * nc + j] = {A[(size_t)j * nc + k], (sign[j] ^ sign[k]) * nc + k};
            }
        }
    }
}

template <typename T, int PB>
__device__ __forceinline__ void get_vec(const T *p, T (&v)[PB])
{
    if constexpr (PB * sizeof(T) >= 16) {
#pragma unroll
        for (int i = 0; i < (int)(PB * sizeof(T) / 16); ++i)
            reinterpret_cast<uint4 *>(v)[i] = reinterpret_cast<const uint4 *>(p)[i];
    } else {
#pragma unroll
        for (int i = 0; i < PB; ++i) v[i] = p[i];
    }
}

template <typename T, int PB>
__device__ __forceinline__ void put_vec(T *p, const T (&v)[PB])
{
    if constexpr (PB * sizeof(T) >= 16) {
#pragma unroll
        for (int i = 0; i < (int)(PB * sizeof(T) / 16); ++i)
            reinterpret_cast<uint4 *>(p)[i] = reinterpret_cast<const uint4 *>(v)[i];
    } else {
#pragma unroll
        for (int i = 0; i < PB; ++i) p[i] = v[i];
    }
}

// w_c = sum_s (-1)^(c . s) w_s in place (its own inverse up to 8)
template <typename T, int PB>
__device__ __forceinline__ void butterflies(T (&w)[8][PB])
{
#pragma unroll
    for (int bit = 1; bit < 8; bit <<= 1)
#pragma unroll
        for (int s = 0; s < 8; ++s)
            if (!(s & bit))
#pragma unroll
                for (int b = 0; b < PB; ++b) {
                    const T u = w[s][b], v = w[s | bit][b];
                    w[s][b] = u + v;
                    w[s | bit][b] = u - v;
                }
}

__device__ __forceinline__ unsigned mag_bits(float x) { return __float_as_uint(fmaxf(0.f, fabsf(x))); }  // a NaN drops
__device__ __forceinline__ unsigned long long mag_bits(double x)  // a NaN is larger than all
{
    return (unsigned long long)__double_as_longlong(x) & ~(1ull << 63);
}

constexpr int FOLD_PB = 4;     // parents per block where there are many
constexpr int FOLD_SPLIT = 2;  // threads per row of A where there are few (2 x 448 threads at p = 20)

// M2M into level l (natural parent order n, 8^l of them): a block takes PB parents, a thread one coefficient.  The
// children's rows of one octant are contiguous in n, so every load is a run of PB nc values; W sits in shared memory
// with the PB parents side by side, which one entry of A then serves in one vector load.  A lone parent's rows (PB = 1, levels
// whose blocks leave most of the GPU idle) are read by FOLD_SPLIT threads each, whose sums are added in order: the loop
// over a row is a chain of loads.  sx, amax (or null): the level's largest |M sx| is folded in for the gain of the
// M2L's operands; cmax (FP64, with amax): that of each parent, the double's upper word.
template <typename T, int PB, typename U>
__global__ void k_m2m_fold(int nc, int l, const FoldEntry<T> *__restrict__ ent, const int *__restrict__ cnt,
                           const T *__restrict__ child, T *__restrict__ parent, const T *__restrict__ sx,
                           U *__restrict__ amax, uint32_t *__restrict__ cmax)
{
    constexpr int SPLIT = PB == 1 ? FOLD_SPLIT : 1;
    constexpr int NM = sizeof(U) == 8 ? PB : 1;  // maxima kept apart: per parent in FP64
    extern __shared__ __align__(16) unsigned char fold_smem[];
    __shared__ U mx_sh[NM];
    T *W = reinterpret_cast<T *>(fold_smem);  // [8][nc][PB], then [SPLIT - 1][nc] partial sums
    const int64_t np3 = (int64_t)1 << (3 * l), n0 = (int64_t)blockIdx.x * PB;  // PB divides 8^l
    const int width = blockDim.x / SPLIT;
    const int part = SPLIT > 1 ? threadIdx.x / width : 0, k = threadIdx.x - part * width;
    if (threadIdx.x < NM) mx_sh[threadIdx.x] = 0;
    if (k < nc && part == 0) {
        alignas(16) T w[8][PB];
#pragma unroll
        for (int s = 0; s < 8; ++s)
#pragma unroll
            for (int b = 0; b < PB; ++b) w[s][b] = child[(s * np3 + n0 + b) * nc + k];
        butterflies<T, PB>(w);
#pragma unroll
        for (int c = 0; c < 8; ++c) put_vec<T, PB>(W + (c * nc + k) * PB, w[c]);
    }
    __syncthreads();
    U mx[NM] = {};
    alignas(16) T acc[PB] = {};
    if (k < nc) {
        const int n = cnt[k];
#pragma unroll 4
        for (int i = part; i < n; i += SPLIT) {
            const FoldEntry<T> e = ent[(size_t)i * nc + k];
            alignas(16) T w[PB];
            get_vec<T, PB>(W + e.at * PB, w);
#pragma unroll
            for (int b = 0; b < PB; ++b) acc[b] += e.v * w[b];
        }
        if (part > 0) W[(7 + part) * nc + k] = acc[0];
    }
    if (SPLIT > 1) __syncthreads();
    if (k < nc && part == 0) {
#pragma unroll
        for (int g = 1; g < SPLIT; ++g) acc[0] += W[(7 + g) * nc + k];
        const int side = 1 << l;
#pragma unroll
        for (int b = 0; b < PB; ++b) {
            const int p = (int)(n0 + b);
            parent[cell_index(l, p & (side - 1), (p >> l) & (side - 1), p >> (2 * l)) * nc + k] = acc[b];
            if (amax) {
                const U v = mag_bits(acc[b] * sx[k]);
                mx[b % NM] = v > mx[b % NM] ? v : mx[b % NM];
            }
        }
    }
    if (amax) {
#pragma unroll
        for (int b = 0; b < NM; ++b) {
            for (int o = 16; o > 0; o >>= 1) {
                const U v = __shfl_xor_sync(0xffffffffu, mx[b], o);
                mx[b] = v > mx[b] ? v : mx[b];
            }
            if ((threadIdx.x & 31) == 0 && mx[b] > 0) atomicMax(&mx_sh[b], mx[b]);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            U m = mx_sh[0];
#pragma unroll
            for (int b = 1; b < NM; ++b) m = mx_sh[b] > m ? mx_sh[b] : m;
            if (m > 0) atomicMax(amax, m);
        }
        if constexpr (sizeof(U) == 8) {
            if (cmax && threadIdx.x < PB) {
                const int p = (int)n0 + threadIdx.x, side = 1 << l;
                cmax[cell_index(l, p & (side - 1), (p >> l) & (side - 1), p >> (2 * l))] = (uint32_t)(mx_sh[threadIdx.x] >> 32);
            }
        }
    }
}

// L2L from level l - 1 into level l, added to the children: PB parents per block (in the children's parent order), a
// thread one coefficient of their eight children, V in registers.  PB = 1 (few parents): the eight V_c of a coefficient
// are as many items spread over the block, through shared memory.
template <typename T, int PB>
__global__ void k_l2l_fold(int nc, int l, const FoldEntry<T> *__restrict__ ent, const int *__restrict__ beg,
                           const T *__restrict__ parent, T *__restrict__ child)
{
    extern __shared__ __align__(16) unsigned char fold_smem[];
    T *X = reinterpret_cast<T *>(fold_smem);  // [nc][PB]
    const int64_t np3 = (int64_t)1 << (3 * (l - 1)), n0 = (int64_t)blockIdx.x * PB;  // PB divides 8^(l - 1)
    const int k = threadIdx.x, side = 1 << (l - 1);
    if (k < nc) {
        alignas(16) T x[PB];
#pragma unroll
        for (int b = 0; b < PB; ++b) {
            const int p = (int)(n0 + b);
            x[b] = parent[cell_index(l - 1, p & (side - 1), (p >> (l - 1)) & (side - 1), p >> (2 * (l - 1))) * nc + k];
        }
        put_vec<T, PB>(X + k * PB, x);
    }
    __syncthreads();
    if constexpr (PB == 1) {
        T *Vs = X + nc;  // [8][nc]
        for (int e = k; e < 8 * nc; e += blockDim.x) {
            const int j = e % nc, end = beg[e + nc];  // e = c nc + j
            T v = 0;
#pragma unroll 4
            for (int i = beg[e]; i < end; ++i) {
                const FoldEntry<T> t = ent[(size_t)i * nc + j];
                v += t.v * X[t.at];
            }
            Vs[e] = v;
        }
        __syncthreads();
        for (int e = k; e < 8 * nc; e += blockDim.x) {
            const int s = e / nc, j = e - s * nc;
            T v = Vs[j];
#pragma unroll
            for (int c = 1; c < 8; ++c) v += __popc(c & s) & 1 ? -Vs[c * nc + j] : Vs[c * nc + j];
            child[(s * np3 + n0) * nc + j] += v;
        }
        return;
    }
    if (k >= nc) return;
    alignas(16) T V[8][PB];
    int i = beg[k];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
#pragma unroll
        for (int b = 0; b < PB; ++b) V[c][b] = 0;
        const int end = beg[(c + 1) * nc + k];
#pragma unroll 2
        for (; i < end; ++i) {
            const FoldEntry<T> e = ent[(size_t)i * nc + k];
            alignas(16) T x[PB];
            get_vec<T, PB>(X + e.at * PB, x);
#pragma unroll
            for (int b = 0; b < PB; ++b) V[c][b] += e.v * x[b];
        }
    }
    butterflies<T, PB>(V);
#pragma unroll
    for (int s = 0; s < 8; ++s)
#pragma unroll
        for (int b = 0; b < PB; ++b) child[(s * np3 + n0 + b) * nc + k] += V[s][b];
}

// four parents share each entry of A where that still leaves several blocks per SM, else one parent a block with its work
// spread over more threads (L2L at 8 and 64 parents, FP64, p = 8: 37 us with a thread per coefficient, 11 us spread)
inline bool fold_wide(int64_t parents) { return parents >= 8 * 152 * FOLD_PB / 2; }

template <typename T, typename U>
fmm_status m2m_t(Plan &P, int l, const void *ent, const T *sx, U *amax, uint32_t *cmax)
{
    const int64_t n = (int64_t)1 << (3 * l);
    const int threads = (P.nc + 31) / 32 * 32;  // at most 448
    const FoldEntry<T> *e = (const FoldEntry<T> *)ent;
    const T *child = (const T *)P.M[l + 1];
    T *parent = (T *)P.M[l];
    if (fold_wide(n))
        k_m2m_fold<T, FOLD_PB, U><<<(unsigned)(n / FOLD_PB), threads, sizeof(T) * 8 * P.nc * FOLD_PB, P.stream>>>(
            P.nc, l, e, P.tab.fold_cnt, child, parent, sx, amax, cmax);
    else
        k_m2m_fold<T, 1, U><<<(unsigned)n, FOLD_SPLIT * threads, sizeof(T) * (7 + FOLD_SPLIT) * P.nc, P.stream>>>(
            P.nc, l, e, P.tab.fold_cnt, child, parent, sx, amax, cmax);
    FMM_LAUNCH_CHECK(P);
    return FMM_OK;
}

template <typename T>
fmm_status l2l_t(Plan &P, int l, const void *ent)
{
    const int64_t n = (int64_t)1 << (3 * (l - 1));
    const int threads = (P.nc + 31) / 32 * 32;
    const FoldEntry<T> *e = (const FoldEntry<T> *)ent;
    if (fold_wide(n))
        k_l2l_fold<T, FOLD_PB><<<(unsigned)(n / FOLD_PB), threads, sizeof(T) * P.nc * FOLD_PB, P.stream>>>(
            P.nc, l, e, P.tab.fold_beg, (const T *)P.L[l - 1], (T *)P.L[l]);
    else
        k_l2l_fold<T, 1><<<(unsigned)n, 4 * threads < 1024 ? 4 * threads : 1024, sizeof(T) * 9 * P.nc, P.stream>>>(
            P.nc, l, e, P.tab.fold_beg, (const T *)P.L[l - 1], (T *)P.L[l]);
    FMM_LAUNCH_CHECK(P);
    return FMM_OK;
}

}  // namespace

fmm_status build_translation_ops(Plan &P)
{
    const int nc = P.nc;
    const size_t n = (size_t)8 * nc * nc;
    if (!P.tab.l2l64) {  // the L2L tables are followed by their transposes
        FMM_CUDA_TRY(cudaMalloc(&P.tab.l2l64, sizeof(double) * 2 * n));
        FMM_CUDA_TRY(cudaMalloc(&P.tab.l2l32, sizeof(float) * 2 * n));
        FMM_CUDA_TRY(cudaMalloc(&P.tab.m2m64, sizeof(double) * n));
        const size_t n64 = sizeof(FoldEntry<double>) * nc * nc, n32 = sizeof(FoldEntry<float>) * nc * nc;
        char *fold = nullptr;  // one allocation, m2m_fold64's
        FMM_CUDA_TRY(cudaMalloc(&fold, 2 * n64 + 2 * n32 + sizeof(int) * 10 * nc));
        P.tab.m2m_fold64 = fold;
        P.tab.l2l_fold64 = fold + n64;
        P.tab.m2m_fold32 = fold + 2 * n64;
        P.tab.l2l_fold32 = fold + 2 * n64 + n32;
        P.tab.fold_cnt = (int *)(fold + 2 * n64 + 2 * n32);
        P.tab.fold_beg = P.tab.fold_cnt + nc;
    }
    k_l2l_ops<<<blocks_for(n, 256), 256, 0, P.stream>>>(P.p, P.tab.Rw64, P.tab.l2l64, P.tab.l2l32);
    FMM_LAUNCH_CHECK(P);
    k_m2m_ops<<<blocks_for(n, 256), 256, 0, P.stream>>>(P.p, P.tab.Rw64, P.tab.m2m64);
    FMM_LAUNCH_CHECK(P);
    k_l2l_entries<<<nc, 32, 0, P.stream>>>(nc, P.tab.l2l64, (FoldEntry<double> *)P.tab.l2l_fold64,
                                           (FoldEntry<float> *)P.tab.l2l_fold32, P.tab.fold_beg);
    FMM_LAUNCH_CHECK(P);
    {
        std::vector<double> A((size_t)nc * nc);  // octant 0's columns of the M2M
        FMM_CUDA_TRY(cudaMemcpy2DAsync(A.data(), sizeof(double) * nc, P.tab.m2m64, sizeof(double) * 8 * nc,
                                       sizeof(double) * nc, nc, cudaMemcpyDeviceToHost, P.stream));
        FMM_CUDA_TRY(cudaStreamSynchronize(P.stream));
        std::vector<FoldEntry<double>> e64;
        std::vector<int> cnt;
        m2m_entries(nc, A, e64, cnt);
        const size_t used = (size_t)nc * *std::max_element(cnt.begin(), cnt.end());  // entries of the longest row
        e64.resize(used);
        std::vector<FoldEntry<float>> e32(used);
        for (size_t i = 0; i < e64.size(); ++i) e32[i] = {(float)e64[i].v, e64[i].at};
        FMM_CUDA_TRY(cudaMemcpyAsync(P.tab.m2m_fold64, e64.data(), sizeof(e64[0]) * e64.size(), cudaMemcpyHostToDevice,
                                     P.stream));
        FMM_CUDA_TRY(cudaMemcpyAsync(P.tab.m2m_fold32, e32.data(), sizeof(e32[0]) * e32.size(), cudaMemcpyHostToDevice,
                                     P.stream));
        FMM_CUDA_TRY(cudaMemcpyAsync(P.tab.fold_cnt, cnt.data(), sizeof(int) * nc, cudaMemcpyHostToDevice, P.stream));
    }
    // four parents at p = 20 take 113 KB (FP64)
    FMM_CUDA_TRY(cudaFuncSetAttribute(k_m2m_fold<double, FOLD_PB, unsigned long long>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)(sizeof(double) * 8 * NC_MAX * FOLD_PB)));
    FMM_CUDA_TRY(cudaFuncSetAttribute(k_m2m_fold<float, FOLD_PB, unsigned>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)(sizeof(float) * 8 * NC_MAX * FOLD_PB)));
    return FMM_OK;
}

// M2M into level l (parents) from level l + 1; where the M2L runs on the tensor cores, level l's largest balanced
// moment is folded in
fmm_status launch_m2m(Plan &P, int l)
{
    if (P.precision == FMM_PREC_FP64) {
        const double *sx = nullptr;
        uint32_t *cmax = nullptr;
        unsigned long long *amax = res_amax(P, l, &sx, &cmax);
        return m2m_t<double, unsigned long long>(P, l, P.tab.m2m_fold64, sx, amax, cmax);
    }
    return m2m_t<float, unsigned>(P, l, P.tab.m2m_fold32, tc_scale(P), tc_amax(P, l), nullptr);
}

// L2L from level l - 1 into level l (added to the M2L result)
fmm_status launch_l2l(Plan &P, int l)
{
    if (P.precision == FMM_PREC_FP64) return l2l_t<double>(P, l, P.tab.l2l_fold64);
    return l2l_t<float>(P, l, P.tab.l2l_fold32);
}

}  // namespace fmm
