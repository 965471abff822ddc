// fmm_top.cu -- the top of the tree as one dense operator: from the moments of the 8 cells of level 1 to their
// local expansions,
//   L(1) = [ M2L over level 1's interaction lists  +  L2L(0 -> 1) . lattice operator (Eq. 12) . M2M(1 -> 0) ] M(1).
// Every part is linear and fixed for a plan (it changes with kappa only), so M2M into the root, the lattice
// operator, the root's L2L and level 1's M2L -- a chain of a dozen launches on a handful of cells, ~120 us of
// latency per far-field pass -- become one (8 nc) x (8 nc) product.  At level 1 the 189 (875) offsets of a target
// reach only 8 source cells, so summing their operators first also leaves 1/24 (1/109) of the M2L's products.
// The operator is composed in FP64; the mixed path reads it in FP32.  One launch of 4-16 us (2,998 charges, p = 8:
// 533 -> 420 us a call together with the solute pass's regrouping; 100,000 charges, p = 12, energy and forces: 906 ->
// 840 us).
#include "fmm_internal.cuh"

namespace fmm {

namespace {

// G[s nc + k][t nc + j] = sum of T_delta[k][j] over the interaction list of target t (class t) whose source is s
__global__ void k_top_m2l(int nc, int ws, int n_il, const int *__restrict__ il, const double *__restrict__ T,
                          double *__restrict__ G)
{
    const int s = blockIdx.y >> 3, t = blockIdx.y & 7, k = blockIdx.x;
    for (int j = threadIdx.x; j < nc; j += blockDim.x) {
        double v = 0;
        for (int o = 0; o < n_il; ++o) {
            int dx, dy, dz;
            il_unpack(il[t * n_il + o], dx, dy, dz);
            const int src = (((t & 1) + dx) & 1) | ((((t >> 1) + dy) & 1) << 1) | ((((t >> 2) + dz) & 1) << 2);
            if (src == s) v += T[((size_t)off_slot(dx, dy, dz, ws) * nc + k) * nc + j];
        }
        G[(size_t)(s * nc + k) * (8 * nc) + t * nc + j] = v;
    }
}

// C (rows x cols, ldc) (+)= A^T B for A [n][rows] and B [n][cols]: 32 x 32 outputs per block, 2 x 2 per thread
template <bool ADD>
__global__ void __launch_bounds__(256) k_atb(int n, int rows, int cols, const double *__restrict__ A, int lda,
                                             const double *__restrict__ B, int ldb, double *__restrict__ C, int ldc)
{
    __shared__ double sa[16][33], sb[16][33];
    const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32, tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    double acc[2][2] = {{0, 0}, {0, 0}};
    for (int k0 = 0; k0 < n; k0 += 16) {
        for (int e = threadIdx.x; e < 512; e += 256) {
            const int k = e >> 5, c = e & 31;
            sa[k][c] = (k0 + k < n && r0 + c < rows) ? A[(size_t)(k0 + k) * lda + r0 + c] : 0.0;
            sb[k][c] = (k0 + k < n && c0 + c < cols) ? B[(size_t)(k0 + k) * ldb + c0 + c] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 16; ++k)
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) acc[i][j] += sa[k][ty + 16 * i] * sb[k][tx + 16 * j];
        __syncthreads();
    }
    for (int i = 0; i < 2; ++i)
        for (int j = 0; j < 2; ++j) {
            const int r = r0 + ty + 16 * i, c = c0 + tx + 16 * j;
            if (r < rows && c < cols) C[(size_t)r * ldc + c] = ADD ? C[(size_t)r * ldc + c] + acc[i][j] : acc[i][j];
        }
}

__global__ void k_to_f32(size_t n, const double *__restrict__ a, float *__restrict__ b)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        b[i] = (float)a[i];
}

// L(1) = G M(1): OUT outputs per block, the 8 nc inputs split over 1024 / OUT threads each, partial sums added in
// a fixed tree.  Inputs: M (all 8 cells, or none) plus sgn times the moments MU of the active cells of a solute
// pass (list `cells`, count *ncells).  Outputs: L, all 8 cells, folding max |L sx| into *amax when given; or Lt,
// the active cells' rows.  Bound by the operator's bytes (7.3 MB in FP32 at p = 12), in FP64 by the 2 operations
// per SM and clock: 8 outputs per block then, so that every SM takes a share.
template <typename TA, typename TM, int OUT>
__global__ void __launch_bounds__(1024) k_top(int nc, const TA *__restrict__ G, const TM *__restrict__ M,
                                              const TM *__restrict__ MU, const int *__restrict__ cells,
                                              const int *__restrict__ ncells, int sgn, TA *__restrict__ L,
                                              double *__restrict__ Lt, const float *__restrict__ sx,
                                              unsigned *__restrict__ amax)
{
    constexpr int KS = 1024 / OUT;
    extern __shared__ __align__(16) unsigned char top_smem[];
    TA *in = reinterpret_cast<TA *>(top_smem);  // [8 nc]
    TA *part = in + 8 * nc;                     // [OUT][KS + 1]
    const int n = 8 * nc;
    const int na = ncells ? *ncells : 0;
    if (Lt && na == 0) return;
    for (int e = threadIdx.x; e < n; e += 1024) in[e] = M ? (TA)M[e] : TA(0);
    __syncthreads();
    for (int e = threadIdx.x; e < na * nc; e += 1024) {
        const int i = e / nc, k = e - i * nc;
        in[cells[i] * nc + k] += TA(sgn) * (TA)MU[e];
    }
    __syncthreads();
    const int o = threadIdx.x % OUT, ks = threadIdx.x / OUT;
    const int out = blockIdx.x * OUT + o;
    TA a0 = 0, a1 = 0;
    if (out < n) {
        int k = ks;
#pragma unroll 4
        for (; k + KS < n; k += 2 * KS) {
            a0 += G[(size_t)k * n + out] * in[k];
            a1 += G[(size_t)(k + KS) * n + out] * in[k + KS];
        }
        if (k < n) a0 += G[(size_t)k * n + out] * in[k];
    }
    part[o * (KS + 1) + ks] = a0 + a1;
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (w >= OUT) return;
    TA v = 0;
    for (int k = lane; k < KS; k += 32) v += part[w * (KS + 1) + k];
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    const int oo = blockIdx.x * OUT + w;
    if (lane != 0 || oo >= n) return;
    if (L) {
        L[oo] = v;
        if (amax) {
            const float m = fabsf((float)v * sx[oo % nc]);
            if (m > 0.f) atomicMax(amax, __float_as_uint(m));
        }
    } else {
        const int c = oo / nc;
        for (int i = 0; i < na; ++i)
            if (cells[i] == c) Lt[(size_t)i * nc + oo % nc] = (double)v;
    }
}

template <typename TA, typename TM, int OUT>
fmm_status run_top(Plan &P, cudaStream_t st, const TA *G, const TM *M, const TM *MU, const int *cells, const int *ncells,
                   int sgn, TA *L, double *Lt, const float *sx, unsigned *amax)
{
    const int n = 8 * P.nc;
    const size_t sh = sizeof(TA) * (n + OUT * (1024 / OUT + 1));
    k_top<TA, TM, OUT><<<(n + OUT - 1) / OUT, 1024, sh, st>>>(P.nc, G, M, MU, cells, ncells, sgn, L, Lt, sx, amax);
    FMM_LAUNCH_CHECK(P);
    return FMM_OK;
}

}  // namespace

// composes the operator from the plan's M2L, M2M, L2L and lattice tables (plan creation, a change of kappa or ws)
fmm_status build_top(Plan &P)
{
    const int nc = P.nc, n = 8 * nc;
    if (!P.tab.G64) {
        FMM_CUDA_TRY(cudaMalloc(&P.tab.G64, sizeof(double) * (size_t)n * n));
        FMM_CUDA_TRY(cudaMalloc(&P.tab.G32, sizeof(float) * (size_t)n * n));
    }
    double *A = nullptr;  // [nc][8 nc]: the root's local expansion per moment of level 1
    FMM_CUDA_TRY(cudaMalloc(&A, sizeof(double) * (size_t)nc * n));
    k_top_m2l<<<dim3(nc, 64), 128, 0, P.stream>>>(nc, P.ws, n_il(P.ws), P.tab.il, P.tab.Top64, P.tab.G64);
    P.launches++;
    // A[j][col] = sum_i T0[i][j] M2M[i][col]
    k_atb<false><<<dim3((n + 31) / 32, (nc + 31) / 32), 256, 0, P.stream>>>(nc, nc, n, P.tab.T0, nc, P.tab.m2m64, n, A, n);
    P.launches++;
    // G[col][out] += sum_j A[j][col] L2L^T[j][out] (the transposed L2L table follows the table)
    k_atb<true><<<dim3((n + 31) / 32, (n + 31) / 32), 256, 0, P.stream>>>(nc, n, n, A, n, P.tab.l2l64 + (size_t)n * nc, n,
                                                                         P.tab.G64, n);
    P.launches++;
    k_to_f32<<<608, 256, 0, P.stream>>>((size_t)n * n, P.tab.G64, P.tab.G32);
    P.launches++;
    const cudaError_t e = cudaStreamSynchronize(P.stream);
    cudaFree(A);
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}

fmm_status launch_top(Plan &P)
{
    if (P.precision == FMM_PREC_FP64)
        return run_top<double, double, 8>(P, P.stream, P.tab.G64, (const double *)P.M[1], nullptr, nullptr, nullptr, 0,
                                          (double *)P.L[1], nullptr, nullptr, nullptr);
    const float *sx = nullptr;
    unsigned *amax = tc_amaxL(P, 1, &sx);
    return run_top<float, float, 32>(P, P.stream, P.tab.G32, (const float *)P.M[1], nullptr, nullptr, nullptr, 0,
                                     (float *)P.L[1], nullptr, sx, amax);
}

// solute-only pass: Lu(1) of the active cells' moments alone
fmm_status launch_top_solute(Plan &P, cudaStream_t st, const void *MU1, const int *cells, const int *ncells, void *Lu1)
{
    if (P.precision == FMM_PREC_FP64)
        return run_top<double, double, 8>(P, st, P.tab.G64, nullptr, (const double *)MU1, cells, ncells, 1, (double *)Lu1,
                                          nullptr, nullptr, nullptr);
    return run_top<float, float, 32>(P, st, P.tab.G32, nullptr, (const float *)MU1, cells, ncells, 1, (float *)Lu1, nullptr,
                                     nullptr, nullptr);
}

// the solvent's field at the active cells of level 1, FP64: Lt = G (M - MU)
fmm_status launch_top_active(Plan &P, cudaStream_t st, const void *MU1, const int *cells, const int *ncells, double *Lt1)
{
    if (P.precision == FMM_PREC_FP64)
        return run_top<double, double, 8>(P, st, P.tab.G64, (const double *)P.M[1], (const double *)MU1, cells, ncells, -1,
                                          nullptr, Lt1, nullptr, nullptr);
    return run_top<double, float, 8>(P, st, P.tab.G64, (const float *)P.M[1], (const float *)MU1, cells, ncells, -1,
                                     nullptr, Lt1, nullptr, nullptr);
}

}  // namespace fmm
