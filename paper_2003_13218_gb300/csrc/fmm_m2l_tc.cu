// fmm_m2l_tc.cu -- M2L of Eq. Lcoeffdef on the 5th-generation tensor cores
// (tcgen05) for the mixed-precision path.
//
// For one level and one parity class c, the local coefficients of 128 target
// cells (a brick of parent coordinates) are
//     L[t][j] = sum_{delta in IL(c)} sum_k M[t + delta][k] T_delta[k][j]
// i.e. 189 dense products (128 x K) . (K x N):
//   M dimension = 128 targets, N = (p+1)^2 output coefficients padded to 16,
//   K = (p+1)^2 input coefficients padded to 16 (rows stored padded to a whole copy box).
// The A operand of offset delta is the same brick shifted to class
// (c + delta) & 1 and parent offset (c + delta) >> 1 in {-1, 0, 1}^3; the
// source planes carry a one-cell periodic halo so that every TMA box lies
// inside the array.  Operands are split into bf16 terms, x = x0 + x1 (+ x2),
// and the products x_i y_j with i + j below the split order are summed
// (bf16x3: 6 products, ~2^-24 relative; bf16x2: 3 products, ~2^-16).
//
// fp16x2 split.  fp16 keeps 11 significant bits, so two terms give ~2^-22
// with 3 products, but its range is narrow.  The moments and operators are
// therefore balanced first: with s(n,m) = sqrt((n+m)! (n-m)!),
//     M~ = M^ s(n,m) gM,   T~[k][j] = T[k][j] / (s(k) s(j)) gT,   L^ = L~ s(j) / (gM gT).
// Because |P_n^m| <= sqrt((n+m)!/(n-m)!) and binomial coefficients are at
// most 2^N, |T~| <= 2^N / |delta|^(N+1) <= 1/2 for well-separated cells
// (|delta| >= 2 cells), and |M~| is bounded by the absolute charge of the
// cell.  gT = 2^14 and gM = 2^(14 - E), E the binary exponent of the level's
// largest |M^ s|, put both operands' largest entries at 2^13..2^15, far below
// fp16's 65504 and far above its subnormal range.
//
// The operand rows are stored padded to whole copy boxes (32 K elements = 64
// bytes for the bf16 splits, 64 = 128 bytes for the fp16 split, whose 2-term
// stages still fit twice in shared memory and move in half as many requests),
// but the MMAs stop at K = (p+1)^2 padded to 16.
//
// Degree grading (fp16 split, FMM_OPT_M2L_GRADE = D2 | D1 << 8).  The smaller
// product terms matter less for the higher input degrees: a K chunk whose
// lowest degree is >= D1 takes the one product x0 y0 (two such chunks share a
// pipeline stage), and in a 3-product chunk the K16 steps whose lowest degree
// reaches D2 drop x1 y0 (one compile-time MMA sequence per split point).  The
// defaults D2 = 4, D1 = 8 give 16 K16 MMA steps per offset at p = 12 instead
// of 33.
//
// Accumulation.  The tensor core's FP32 accumulation rounds with a bias, which
// over thousands of MMAs into one accumulator shows up at the 1e-5 level.  So
// the products of a short run of offsets (FMM_OPT_M2L_ACC_GROUP, default 2) go
// into a fresh TMEM accumulator (two, alternating), and the epilogue warps
// drain it and add it to the row held in FP32 registers (round to nearest)
// while the tensor core works on the next run.
//
// The kernels are in fmm_tc.cuh.
#include <math.h>
#include <string.h>

#include <new>
#include <vector>

#include "fmm_tc.cuh"

namespace fmm {

namespace {

// operator slots of the B tables: the noff(ws) M2L offsets, then the L2L per child octant

struct TcState {
    bool f16 = false;               // fp16x2 split with balanced scaling (and fused L2L)
    int pa = 0, pb = 0;             // terms of the plan's split
    int parts = 0;                  // terms stored (3 for the bf16 splits: the solute pass uses 3 x 3)
    int npad = 0, kp = 0;
    int noff = 0;                   // M2L operator slots (the slot cube of the plan's ws)
    int sw = 64;                    // bytes per swizzled operand row in shared memory
    uint16_t *planes[9] = {};       // bf16 or fp16 bit patterns
    size_t part_elems[9] = {};
    uint16_t *ops = nullptr;
    size_t ops_part_elems = 0;
    bool ops_borrowed = false;      // ops belongs to another plan's state (tc_share_operators)
    TcMaps maps[9];                 // per level; the B maps box whole operator tiles
    CUtensorMap mapB2[3];           // S, P, C of operator tiles boxed N/2 rows (one half per CTA of a pair)
    uint16_t *planesL = nullptr;    // natural order [term][chunk][z][y][x][KCH], sized for level d - 1
    size_t partL_elems = 0;
    int bx[9], by[9], bz[9];
    int groups[9], per_group[9];    // offset groups per tile (small levels run more CTAs)
    float *Lpart = nullptr;         // partial sums of the offset groups
    float *s32 = nullptr;           // [nc] s(n,m) per real coefficient (fp16 split)
    float *s32inv = nullptr;        // [nc] 1 / s(n,m)
    double *s64 = nullptr;
    unsigned *amax = nullptr;       // [9] bits of the largest |M^ s| per level (fp16 split)
    unsigned *amaxL = nullptr;      // [9] bits of the largest |L^ / s| per level (behind amax: one clear per pass)
};

// ------------------------------------------------------------------ operand preparation
// x = x0 + x1 (+ x2) in bf16 or fp16 terms, each term the rounding of the
// remaining residual; stored as bit patterns `stride` elements apart
template <bool F16>
__device__ __forceinline__ void split_terms(float v, int parts, uint16_t *o, size_t stride)
{
    float r = v;
    for (int i = 0; i < parts; ++i) {
        if (F16) {
            const __half t = __float2half_rn(r);
            o[i * stride] = __half_as_ushort(t);
            r -= __half2float(t);
        } else {
            const __nv_bfloat16 t = __float2bfloat16_rn(r);
            o[i * stride] = __bfloat16_as_ushort(t);
            r -= __bfloat162float(t);
        }
    }
}

// FP32 class-layout moments -> bf16 split planes [part][chunk][class][hz][hy][hx][k] with a
// periodic halo; rows kp wide (zero beyond nc).  One warp per halo cell, lanes over the coefficients.
__global__ void k_split_halo(const float *__restrict__ M, int np, int hw, int nc, int kp, int parts,
                             int kch, uint16_t *__restrict__ planes, size_t part_elems)
{
    const int np2 = np + 2 * hw;
    const int64_t ncell = 8 * (int64_t)np2 * np2 * np2;
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t cell = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); cell < ncell; cell += warps) {
        const int hx = (int)(cell % np2);
        const int hy = (int)((cell / np2) % np2);
        const int hzc = (int)(cell / ((int64_t)np2 * np2));
        const int c = hzc / np2, hz = hzc % np2;
        const int px = ((hx - hw) % np + np) % np, py = ((hy - hw) % np + np) % np, pz = ((hz - hw) % np + np) % np;
        const float *row = M + ((int64_t)c * np * np * np + px + (int64_t)np * (py + (int64_t)np * pz)) * nc;
        for (int k = lane; k < kp; k += 32)
            split_terms<false>(k < nc ? row[k] : 0.f, parts, planes + chunk_at(cell, ncell, k, kch), part_elems);
    }
}

// FP32 class-layout local expansion of level `lev` >= 1 (side n = 2^lev) -> fp16
// split planes in natural order [part][chunk][z][y][x][k], balanced L~ = L^ / s(k) gL
// (the A operand of the fused L2L): natural cell `cell`, lanes over the coefficients.
__device__ __forceinline__ void split_L_cell(const float *__restrict__ L, int lev, int nc, int kp,
                                             const float *__restrict__ sinv, float g, uint16_t *__restrict__ planes,
                                             size_t part_elems, int64_t cell, int lane)
{
    const int n = 1 << lev, h = n >> 1;
    const int x = (int)(cell % n), y = (int)((cell / n) % n), z = (int)(cell / ((int64_t)n * n));
    const int64_t src = (int64_t)((x & 1) | ((y & 1) << 1) | ((z & 1) << 2)) * h * h * h + (x >> 1) +
                        (int64_t)h * ((y >> 1) + (int64_t)h * (z >> 1));
    const float *row = L + src * nc;
    const int64_t ncell = (int64_t)n * n * n;
    for (int k = lane; k < kp; k += 32) {
        const float v = k < nc ? __ldcg(row + k) * (__ldg(sinv + k) * g) : 0.f;
        split_terms<true>(v, 2, planes + chunk_at(cell, ncell, k, kchunk_of(128)), part_elems);
    }
}

// all cells of level `lev`, one warp per cell
__global__ void k_split_L(const float *__restrict__ L, int lev, int nc, int kp, const float *__restrict__ sinv,
                          const unsigned *__restrict__ amaxL, uint16_t *__restrict__ planes, size_t part_elems)
{
    const int n = 1 << lev;
    const int64_t ncell = (int64_t)n * n * n;
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const float g = pow2f(gain_m_exp(*amaxL));
    for (int64_t cell = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); cell < ncell; cell += warps)
        split_L_cell(L, lev, nc, kp, sinv, g, planes, part_elems, cell, lane);
}

// FP64 operators -> split B tables [part][chunk][slot][j][k] (K-major, rows kp wide in chunks of kch):
// slots < noff the M2L operators T[slot][k][j] (input-major), then per child
// octant o the L2L operator (L2L[o nc + j][k], child output j).  fp16: balanced with gT,
//   M2L  T~ = T / (s(k) s(j)),  L2L  U~ = U s(k) / s(j);
// bf16: the L2L slots stay zero (unused).
template <bool F16>
__global__ void k_split_ops(int noff, const double *__restrict__ T, const double *__restrict__ l2l, int nc, int npad, int kp, int kch, int parts,
                            const double *__restrict__ s, uint16_t *__restrict__ ops, size_t part_elems)
{
    const int64_t total = (int64_t)(noff + 8) * npad * kp;
    const double gT = (double)pow2f(GAIN_T_EXP);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int k = (int)(e % kp);
        const int j = (int)((e / kp) % npad);
        const int slot = (int)(e / ((int64_t)kp * npad));
        double r = 0.0;
        if (j < nc && k < nc) {
            if (slot < noff) {
                r = T[((int64_t)slot * nc + k) * nc + j];
                if (F16) r = r / (s[k] * s[j]) * gT;
            } else if (F16) {
                const int o = slot - noff;
                r = l2l[((int64_t)o * nc + j) * nc + k] * s[k] / s[j] * gT;
            }
        }
        const int64_t at = chunk_at((int64_t)slot * npad + j, (int64_t)(noff + 8) * npad, k, kch);
        for (int i = 0; i < parts; ++i) {
            if (F16) {
                const __half t = __float2half_rn((float)r);
                ops[at + i * part_elems] = __half_as_ushort(t);
                r -= (double)__half2float(t);
            } else {
                const __nv_bfloat16 t = __float2bfloat16_rn((float)r);
                ops[at + i * part_elems] = __bfloat16_as_ushort(t);
                r -= (double)__bfloat162float(t);
            }
        }
    }
}

// L = sum over the offset groups, in group order; with amax (fp16 split) the largest |L_e sx(e mod nc)|
// is folded into *amax.  Elements [e0, e1) by threads t = 0 .. nt - 1, four at a time (16-byte loads and
// stores) when n is a multiple of 4 (the partial arrays then stay 16-byte aligned); each element is the
// same ordered sum either way.  Returns this thread's share of the maximum.
__device__ __forceinline__ float group_sum_range(int64_t n, int groups, const float *__restrict__ part,
                                                 float *__restrict__ L, int nc, const float *__restrict__ sx,
                                                 bool fold, int64_t e0, int64_t e1, int64_t t, int64_t nt)
{
    float mx = 0.f;
    if ((n & 3) == 0 && (e0 & 3) == 0) {
        for (int64_t e = e0 + 4 * t; e < e1; e += 4 * nt) {
            if (e + 4 > e1) {  // a ragged end of the range
                for (int64_t k = e; k < e1; ++k) {
                    float s = 0.f;
                    for (int g = 0; g < groups; ++g) s += __ldcg(part + (int64_t)g * n + k);
                    L[k] = s;
                    if (fold) mx = fmaxf(mx, fabsf(s * __ldg(sx + (int)(k % nc))));
                }
                break;
            }
            float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int g = 0; g < groups; ++g) {
                const float4 v = __ldcg(reinterpret_cast<const float4 *>(part + (int64_t)g * n + e));
                s.x += v.x;
                s.y += v.y;
                s.z += v.z;
                s.w += v.w;
            }
            *reinterpret_cast<float4 *>(L + e) = s;
            if (fold) {
                const int c = (int)(e % nc);
                mx = fmaxf(mx, fabsf(s.x * __ldg(sx + c)));
                mx = fmaxf(mx, fabsf(s.y * __ldg(sx + (c + 1 < nc ? c + 1 : c + 1 - nc))));
                mx = fmaxf(mx, fabsf(s.z * __ldg(sx + (c + 2 < nc ? c + 2 : c + 2 - nc))));
                mx = fmaxf(mx, fabsf(s.w * __ldg(sx + (c + 3 < nc ? c + 3 : c + 3 - nc))));
            }
        }
    } else {
        for (int64_t e = e0 + t; e < e1; e += nt) {
            float s = 0.f;
            for (int g = 0; g < groups; ++g) s += __ldcg(part + (int64_t)g * n + e);
            L[e] = s;
            if (fold) mx = fmaxf(mx, fabsf(s * __ldg(sx + (int)(e % nc))));
        }
    }
    return mx;
}

__global__ void k_group_sum(int64_t n, int groups, const float *__restrict__ part, float *__restrict__ L, int nc,
                            const float *__restrict__ sx, unsigned *__restrict__ amax)
{
    float mx = group_sum_range(n, groups, part, L, nc, sx, amax != nullptr, 0, n,
                               blockIdx.x * (int64_t)blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x);
    if (amax) {
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if ((threadIdx.x & 31) == 0 && mx > 0.f) atomicMax(amax, __float_as_uint(mx));
    }
}

// fp16 split: FP32 class-layout moments -> the two balanced fp16 halo planes, 8 coefficients per thread
// (16-byte stores per plane); rows kp wide, zero beyond nc.  One launch for all levels, the deepest first.
struct SplitLevel {
    const float *M;
    const unsigned *amax;
    uint16_t *planes;
    size_t part_elems;
    int64_t end;  // threads of this level and those before it
    int np;
};
struct SplitLevels {
    SplitLevel l[8];
    int64_t total;
};

__global__ void k_split_halo16(const __grid_constant__ SplitLevels lv, int hw, int nc, int kp, const float *__restrict__ s)
{
    const int G = kp / 8;
    for (int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t0 < lv.total;
         t0 += (int64_t)gridDim.x * blockDim.x) {
        int i = 0;
        int64_t t = t0, total = lv.l[0].end;
        while (t0 >= lv.l[i].end) {
            t = t0 - lv.l[i].end;
            total = lv.l[i + 1].end - lv.l[i].end;
            ++i;
        }
        const int np = lv.l[i].np, np2 = np + 2 * hw;
        const float g = pow2f(gain_m_exp(__ldg(lv.l[i].amax)));
        const int64_t cell = t / G;
        const int k0 = (int)(t - cell * G) * 8;
        const int hx = (int)(cell % np2);
        const int hy = (int)((cell / np2) % np2);
        const int hzc = (int)(cell / ((int64_t)np2 * np2));
        const int c = hzc / np2, hz = hzc % np2;
        const int px = ((hx - hw) % np + np) % np, py = ((hy - hw) % np + np) % np, pz = ((hz - hw) % np + np) % np;
        const float *row = lv.l[i].M + ((int64_t)c * np * np * np + px + (int64_t)np * (py + (int64_t)np * pz)) * nc;
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            uint16_t h2[2], l2[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int k = k0 + 2 * w + u;
                const float v = k < nc ? row[k] * (__ldg(s + k) * g) : 0.f;
                const __half t0h = __float2half_rn(v);
                const __half t1h = __float2half_rn(v - __half2float(t0h));
                h2[u] = __half_as_ushort(t0h);
                l2[u] = __half_as_ushort(t1h);
            }
            hi[w] = (uint32_t)h2[0] | ((uint32_t)h2[1] << 16);
            lo[w] = (uint32_t)l2[0] | ((uint32_t)l2[1] << 16);
        }
        uint16_t *out = lv.l[i].planes + chunk_at(cell, total / G, k0, kchunk_of(128));
        *reinterpret_cast<uint4 *>(out) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        *reinterpret_cast<uint4 *>(out + lv.l[i].part_elems) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
}

// ------------------------------------------------------------------ persistent sweep of a batch
// The tensor-core levels of many boxes (the lambda windows or frames of a batch) in one launch of
// persistent CTA pairs.  Per (box, level) three stages, each a run of work items:
//   P  the parent level's local expansion split into the fused L2L's fp16 planes (k_split_L), and the
//      reset of the level's largest |L^ / s|;
//   M  the tile pairs of the level's M2L + fused L2L (the k_m2l_tc_pair work, same offset groups): one
//      item per tile pair running its groups in turn, or per offset group where the level is small;
//   G  with offset groups > 1, the group sum into L (k_group_sum), folding the level's maximum.
// The items of all boxes sit in one device queue in level order, and P, M, G within a level, so every
// item depends only on items before it.  A pair claims the next item with an atomic add, waits (bounded,
// globaltimer) until the stage it depends on has counted all its items done, runs it, and adds one to
// its own stage's counter (release after the pair's writes).  Because items are claimed in queue order
// and the oldest unfinished item is always held by a running pair with its inputs complete, the sweep
// makes progress whatever number of pairs is resident.  A wait that runs out sets the queue's abort
// word: every pair stops claiming and the launch ends with FMM_ERR_TIMEOUT recorded.
constexpr int SWEEP_P_CELLS = 512;         // parent cells per P item
constexpr int64_t SWEEP_G_ELEMS = 1 << 16;  // L elements per G item

struct SweepLevel {
    TcMaps maps;                      // the level's pair-kernel tensor maps
    TcArgs a;                         // the level's pair-kernel arguments
    const float *Lprev;               // P: L of level l - 1 (class layout)
    const float *sinv;                // P: 1 / s(k)
    const unsigned *amaxL_prev;       // P: largest |L^ / s| of level l - 1 (final when P runs)
    uint16_t *planesL;                // P: the fused L2L planes
    size_t partL;                     // P: elements per term of planesL
    unsigned *amaxL;                  // this level's largest |L^ / s|, reset by P, folded by M or G
    int64_t gs_n;                     // G: elements of the level's L
    int lev, nc, kp;
    int gpi;                          // M: offset groups per item (all of a tile pair's, or one)
    int n_items[3];                   // items of stages P, M, G (G: 0 with one offset group)
    int prev;                         // the same box's previous sweep level (-1: done before the launch)
};

__device__ __forceinline__ int ld_acquire(const int *p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ int ld_relaxed(const int *p)
{
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// counter of stage `st` of level entry `e`: q[2 + 3 e + st]; q[0] is the queue head, q[1] the abort word
__device__ __forceinline__ int *sweep_counter(int *q, int e, int st) { return q + 2 + 3 * e + st; }

// bounded wait for the dependency of item `it` (stage, level entry, index); false after limit_ns or abort
__device__ bool sweep_wait(const SweepLevel *__restrict__ lv, int4 it, int *q, uint64_t limit_ns, int stall)
{
    const int *c;
    int target;
    if (it.x == 0) {
        const int pe = lv[it.y].prev;
        if (pe < 0) return true;
        const int st = lv[pe].n_items[2] > 0 ? 2 : 1;
        c = sweep_counter(q, pe, st);
        target = lv[pe].n_items[st];
    } else {
        c = sweep_counter(q, it.y, it.x - 1);
        target = lv[it.y].n_items[it.x - 1];
    }
    target += stall;  // test hook: a count that is never reached
    if (ld_acquire(c) >= target) return true;
    const uint64_t t0 = global_ns();
    for (uint32_t i = 0;; ++i) {
        __nanosleep(100);
        if (ld_acquire(c) >= target) return true;
        if ((i & 15) == 15) {
            if (ld_relaxed(q + 1)) return false;
            if (global_ns() - t0 > limit_ns) return false;
        }
    }
}

template <int NCH>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TC_THREADS, 1)
    k_m2l_sweep(const SweepLevel *__restrict__ lv, const int4 *__restrict__ items, int n_items, int stages,
                int *__restrict__ q, uint64_t wait_ns, int stall_item)
{
    extern __shared__ uint8_t smem_dyn[];
    __shared__ __align__(8) PairBars bars;
    __shared__ uint32_t tmem_sh;
    __shared__ int abort_sh;
    __shared__ int item_sh;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = warp_uniform(cluster_rank());
    const bool leader = rank == 0;
    const uint32_t smem0 = warp_uniform((smem_u32(smem_dyn) + 1023u) & ~1023u);
    if (threadIdx.x == 0) {
        pair_bars_init(bars, stages);
        abort_sh = 0;
        item_sh = n_items;
    }
    cluster_sync_all();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_sh)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = warp_uniform(tmem_sh);
    const uint32_t el = elect_one();
    float *stage = reinterpret_cast<float *>(smem_dyn + (smem0 - smem_u32(smem_dyn)));
    PairPipe pp;
    int done_entry = -1, done_stage = 0;  // the item the pair finished last (leader thread 0)
    for (;;) {
        // ---- the leader's thread 0 publishes the finished item, claims the next and waits for its inputs
        if (leader && threadIdx.x == 0) {
            if (done_entry >= 0) {
                __threadfence();
                atomicAdd(sweep_counter(q, done_entry, done_stage), 1);
            }
            int j = n_items;
            if (!ld_relaxed(q + 1)) {
                j = atomicAdd(q, 1);
                if (j < n_items && !sweep_wait(lv, items[j], q, wait_ns, j == stall_item ? 1 : 0)) {
                    atomicOr(lv[items[j].y].a.err, ERRF_TIMEOUT);
                    atomicExch(q + 1, 1);
                    j = n_items;
                }
                if (j > n_items) j = n_items;
            }
            item_sh = j;
            asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(map_shared(smem_u32(&item_sh), 1)), "r"(j)
                         : "memory");
        }
        __syncwarp();
        cluster_sync_all();
        const int j = item_sh;
        if (j >= n_items) break;
        const int4 it = items[j];
        const SweepLevel &e = lv[it.y];
        if (it.x == 1) {
            // stage M: one tile pair; the maps live in global memory, and the planes it copies were written
            // by other pairs through the generic proxy
            if (warp == 0 && el) {
#pragma unroll
                for (int m = 0; m < (int)(sizeof(TcMaps) / sizeof(CUtensorMap)); ++m)
                    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(&e.maps.aS + m) : "memory");
                asm volatile("fence.proxy.async.global;" ::: "memory");
            }
            __syncwarp();
            // the item's offset groups of one tile pair in turn (the ring runs on from group to group); only
            // the last group's epilogue stages its rows in the ring
            for (int g = 0; g < e.gpi; ++g) {
                if (*(volatile int *)&abort_sh) break;  // a wait ran out: the remaining groups are skipped
                pair_tile<NCH>(e.maps, e.a, it.z * e.gpi + g,
                               rank, smem0, stage, g == e.gpi - 1, bars, tmem, &abort_sh, pp, el);
            }
        } else if (it.x == 0) {
            // stage P: parent cells [SWEEP_P_CELLS it.z, ...) of level l - 1, one warp per cell over the pair
            const int64_t ncell = (int64_t)1 << (3 * (e.lev - 1));
            const int64_t c0 = (int64_t)it.z * SWEEP_P_CELLS;
            const int64_t c1 = c0 + SWEEP_P_CELLS < ncell ? c0 + SWEEP_P_CELLS : ncell;
            const float g = pow2f(gain_m_exp(__ldcg(e.amaxL_prev)));
            const int gw = (int)rank * (TC_THREADS / 32) + warp;
            for (int64_t cell = c0 + gw; cell < c1; cell += 2 * (TC_THREADS / 32))
                split_L_cell(e.Lprev, e.lev - 1, e.nc, e.kp, e.sinv, g, e.planesL, e.partL, cell, lane);
            if (it.z == 0 && leader && threadIdx.x == 0) atomicExch(e.amaxL, 0u);
            asm volatile("fence.proxy.async.global;" ::: "memory");  // the planes are read by TMA next
        } else {
            // stage G: L elements [SWEEP_G_ELEMS it.z, ...), thread per element over the pair
            const int64_t e0 = (int64_t)it.z * SWEEP_G_ELEMS;
            const int64_t e1 = e0 + SWEEP_G_ELEMS < e.gs_n ? e0 + SWEEP_G_ELEMS : e.gs_n;
            float mx = group_sum_range(e.gs_n, e.a.groups, e.a.Lpart, e.a.L, e.nc, e.sinv, true, e0, e1,
                                       (int64_t)rank * TC_THREADS + threadIdx.x, 2 * TC_THREADS);
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            if (lane == 0 && mx > 0.f) atomicMax(e.amaxL, __float_as_uint(mx));
        }
        __syncthreads();
        if (threadIdx.x == 0 && abort_sh) atomicExch(q + 1, 1);
        __syncwarp();
        cluster_sync_all();  // both CTAs are done with the item
        if (leader && threadIdx.x == 0) {
            done_entry = it.y;
            done_stage = it.x;
        }
    }

    // ---------------- teardown: every MMA done (bounded wait), pair barrier, collective TMEM release
    if (warp == 1 && el && leader) mma_commit_pair(smem_u32(&bars.done));
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile int no_abort = 0;
        if (!mbar_wait_cluster(smem_u32(&bars.done), 0, &no_abort)) atomicExch(q + 1, 1);
    }
    fence_before();
    __syncthreads();
    cluster_sync_all();
    fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    cluster_sync_all();
}

// every box of the sweep reports a launch that stopped early
__global__ void k_sweep_status(const int *__restrict__ q, int *const *__restrict__ errs, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && q[1]) atomicOr(errs[i], ERRF_TIMEOUT);
}

TcKernel pick_pair_kernel(int nch)
{
    switch (nch) {
#define FMM_TC_CASE(n) \
    case n: return (TcKernel)k_m2l_tc_pair<n>;
        FMM_TC_CASE(1) FMM_TC_CASE(2) FMM_TC_CASE(3) FMM_TC_CASE(4) FMM_TC_CASE(6) FMM_TC_CASE(7) FMM_TC_CASE(8)
        FMM_TC_CASE(9) FMM_TC_CASE(11) FMM_TC_CASE(13) FMM_TC_CASE(15) FMM_TC_CASE(16)
#undef FMM_TC_CASE
    default: return nullptr;
    }
}

typedef void (*SweepKernel)(const SweepLevel *, const int4 *, int, int, int *, uint64_t, int);

// the sweep is built for the orders p = 6, 8, 10 and 12 (NCH 4, 6, 8, 11)
SweepKernel pick_sweep_kernel(int nch)
{
    switch (nch) {
    case 4: return k_m2l_sweep<4>;
    case 6: return k_m2l_sweep<6>;
    case 8: return k_m2l_sweep<8>;
    case 11: return k_m2l_sweep<11>;
    default: return nullptr;
    }
}

// NCH = ((p+1)^2 rounded to 16) / 16 takes the values below for p <= 15
template <int PA, int PB, int SW>
TcKernel pick_kernel_n(int nch)
{
    switch (nch) {
#define FMM_TC_CASE(n) \
    case n: return (TcKernel)k_m2l_tc<PA, PB, n, SW>;
        FMM_TC_CASE(1) FMM_TC_CASE(2) FMM_TC_CASE(3) FMM_TC_CASE(4) FMM_TC_CASE(6) FMM_TC_CASE(7) FMM_TC_CASE(8)
        FMM_TC_CASE(9) FMM_TC_CASE(11) FMM_TC_CASE(13) FMM_TC_CASE(15) FMM_TC_CASE(16)
#undef FMM_TC_CASE
    default: return nullptr;
    }
}

TcKernel pick_kernel(int pa, int pb, int nch, int sw)
{
    if (sw == 128) return pa == 2 && pb == 2 ? pick_kernel_n<2, 2, 128>(nch) : nullptr;
    if (pa == 3 && pb == 3) return pick_kernel_n<3, 3, 64>(nch);
    if (pa == 2 && pb == 3) return pick_kernel_n<2, 3, 64>(nch);
    if (pa == 2 && pb == 2) return pick_kernel_n<2, 2, 64>(nch);
    return nullptr;
}

#define TRY_TC(x)                          \
    do {                                   \
        fmm_status st_ = (x);              \
        if (st_ != FMM_OK) return st_;     \
    } while (0)

int chunks_of(const TcState *S) { return S->kp / kchunk_of(S->sw); }

CUtensorMapDataType type_of(const TcState *S)
{
    return S->f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
}

// level l's A and L maps for tiles of bx x by x bz cells (np a class side, hw the halo width)
fmm_status encode_level(PFN_cuTensorMapEncodeTiled_v12000 enc, const TcState *S, int l, int np, int hw, int bx, int by,
                        int bz, TcMaps *m)
{
    const int64_t np2 = np + 2 * hw;
    const int kc = chunks_of(S);
    fmm_status st = encode_planes(enc, &m->aS, S->f16 ? &m->aP : nullptr, S->f16 ? &m->aC : nullptr, type_of(S),
                                  S->planes[l], kc, S->parts, np2, np2, 8 * np2, bx, by, bz, S->sw);
    // L of level l - 1 (side np) in natural order, boxed like the level-l bricks; all levels share one buffer,
    // used one level at a time
    if (st == FMM_OK && S->f16)
        st = encode_planes(enc, &m->lS, &m->lP, nullptr, type_of(S), S->planesL, kc, 2, np, np, np, bx, by, bz, S->sw);
    if (!S->f16) m->aP = m->aC = m->lS = m->lP = m->aS;  // unused kernel parameters
    return st;
}

// level l's maps for the CTA-pair kernel: half operator tiles
TcMaps pair_maps(const TcState *S, int l)
{
    TcMaps m = S->maps[l];
    m.bS = S->mapB2[0];
    m.bP = S->mapB2[1];
    m.bC = S->mapB2[2];
    return m;
}

void fill_common(const Plan &P, const TcState *S, int pa, int pb, TcArgs &a)
{
    a.nc = P.nc;
    a.npad = S->npad;
    a.nslots = S->noff + 8;
    a.stages = tc_stages(pa, pb, S->npad, S->sw);
    // instruction descriptor: FP32 accumulator, A and B both bf16 (format 1) or both fp16 (format 0),
    // K-major, N >> 3 at bit 17, M >> 4 at bit 24
    const uint32_t ab = S->f16 ? 0u : 1u;
    a.idesc = (1u << 4) | (ab << 7) | (ab << 10) | ((uint32_t)(S->npad >> 3) << 17) | ((uint32_t)(TC_ROWS >> 4) << 24);
    a.Lpart = S->Lpart;
    a.il = P.tab.il;
    a.mod0 = a.nmods = 0;
    a.mods = nullptr;
    a.resid = nullptr;
    a.err = P.d_err;
    a.amax_out = nullptr;
    a.sx = nullptr;
    a.acc_group = P.acc_group;
    a.wait_ns = P.wait_ns;
    a.inject_stall = P.inject_stall ? 1 : 0;
    a.amaxL = nullptr;
    a.ws = P.ws;
    a.n_il = n_il(P.ws);
    a.noff = noff(P.ws);
    // degree grading of the fp16x2 M2L (FMM_OPT_M2L_GRADE), per K chunk: chunk kc holds input
    // coefficients KCH kc .. KCH kc + KCH - 1, whose lowest degree is floor(sqrt(KCH kc))
    a.gchunks = 0;
    a.gsteps = 0;
    const int d2 = P.grade & 0xFF, d1 = (P.grade >> 8) & 0xFF;
    auto lowest_degree = [](int k) {  // of input coefficient k: floor(sqrt(k))
        int lam = 0;
        while ((lam + 1) * (lam + 1) <= k) ++lam;
        return lam;
    };
    if (S->f16 && pa == 2 && pb == 2 && (d2 > 0 || d1 > 0)) {
        const int kch = kchunk_of(S->sw);
        for (int kc = 0; kc < chunks_of(S) && kc < 10; ++kc) {
            const int lam = lowest_degree(kch * kc);
            const int np = (d1 > 0 && lam >= d1) ? 1 : (d2 > 0 && lam >= d2) ? 2 : 3;
            if (np < 3) a.gchunks |= (uint32_t)np << (2 * kc);
            // a 3-product chunk whose later K16 steps reach D2 drops x1 y0 there
            if (np == 3 && d2 > 0)
                for (int st = 1; st * 16 < kch; ++st)
                    if (lowest_degree(kch * kc + 16 * st) >= d2) {
                        a.gsteps |= (uint32_t)st << (3 * kc);
                        break;
                    }
        }
    }
}

}  // namespace

bool tc_available(const Plan &P, int level)
{
    return P.tc != nullptr && level >= 1 && level <= P.d;
}

bool tc_translations(const Plan &P)
{
    return P.tc != nullptr && ((const TcState *)P.tc)->f16;
}

fmm_status tc_prepare(Plan &P)
{
    tc_free(P);
    if (P.precision != FMM_PREC_MIXED || P.p > TC_PMAX) return FMM_OK;  // CUDA-core M2L
    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
    if (!enc) return FMM_OK;
    TcState *S = new (std::nothrow) TcState();
    if (!S) return FMM_ERR_OOM;
    P.tc = S;
    S->f16 = P.split == FMM_SPLIT_FP16X2;
    S->pa = P.split == FMM_SPLIT_BF16X3 ? 3 : 2;
    S->pb = (P.split == FMM_SPLIT_BF16X2 || S->f16) ? 2 : 3;
    S->parts = S->f16 ? 2 : 3;  // bf16: three terms always, the solute-only pass uses the 3 x 3 split
    S->npad = (P.nc + 15) / 16 * 16;
    S->noff = noff(P.ws);
    // 128-byte swizzled rows for the fp16 split (two 2-term stages fit), 64 bytes for the bf16 splits;
    // rows padded to whole copy boxes (aligned pieces); the MMAs stop at (p+1)^2 padded to 16
    S->sw = S->f16 ? 128 : 64;
    S->kp = (P.nc + kchunk_of(S->sw) - 1) / kchunk_of(S->sw) * kchunk_of(S->sw);
    if (S->f16) {
        // s(n,m) = sqrt((n+m)! (n-m)!) per real coefficient
        double h_s[(TC_PMAX + 1) * (TC_PMAX + 1)];
        float h_s32[(TC_PMAX + 1) * (TC_PMAX + 1)], h_inv[(TC_PMAX + 1) * (TC_PMAX + 1)];
        for (int n = 0; n <= P.p; ++n)
            for (int m = 0; m <= n; ++m) {
                double f = 1.0;
                for (int i = 2; i <= n + m; ++i) f *= i;
                for (int i = 2; i <= n - m; ++i) f *= i;
                const double v = sqrt(f);
                const int re = m == 0 ? n * n : n * n + 2 * m - 1;
                h_s[re] = v;
                if (m > 0) h_s[re + 1] = v;
            }
        for (int k = 0; k < P.nc; ++k) {
            h_s32[k] = (float)h_s[k];
            h_inv[k] = (float)(1.0 / h_s[k]);
        }
        FMM_CUDA_TRY(cudaMalloc(&S->s64, sizeof(double) * P.nc));
        FMM_CUDA_TRY(cudaMalloc(&S->s32, sizeof(float) * P.nc));
        FMM_CUDA_TRY(cudaMalloc(&S->s32inv, sizeof(float) * P.nc));
        FMM_CUDA_TRY(cudaMalloc(&S->amax, sizeof(unsigned) * 18));
        S->amaxL = S->amax + 9;
        FMM_CUDA_TRY(cudaMemcpyAsync(S->s64, h_s, sizeof(double) * P.nc, cudaMemcpyHostToDevice, P.stream));
        FMM_CUDA_TRY(cudaMemcpyAsync(S->s32, h_s32, sizeof(float) * P.nc, cudaMemcpyHostToDevice, P.stream));
        FMM_CUDA_TRY(cudaMemcpyAsync(S->s32inv, h_inv, sizeof(float) * P.nc, cudaMemcpyHostToDevice, P.stream));
    }
    // operator tables
    S->ops_part_elems = (size_t)(S->noff + 8) * S->npad * S->kp;
    FMM_CUDA_TRY(cudaMalloc(&S->ops, sizeof(uint16_t) * S->ops_part_elems * S->parts));
    if (S->f16)
        k_split_ops<true><<<1216, 256, 0, P.stream>>>(S->noff, P.tab.Top64, P.tab.l2l64, P.nc, S->npad, S->kp,
                                                      kchunk_of(S->sw), S->parts, S->s64, S->ops, S->ops_part_elems);
    else
        k_split_ops<false><<<1216, 256, 0, P.stream>>>(S->noff, P.tab.Top64, nullptr, P.nc, S->npad, S->kp,
                                                       kchunk_of(S->sw), S->parts, nullptr, S->ops, S->ops_part_elems);
    FMM_LAUNCH_CHECK(P);
    {
        TcMaps &m = S->maps[0];  // the operator maps, the same on every level
        TRY_TC(encode_operators(enc, &m.bS, S->f16 ? &m.bP : nullptr, S->f16 ? &m.bC : nullptr, type_of(S), S->ops,
                                chunks_of(S), S->parts, S->npad, S->noff + 8, S->npad, S->sw));
        if (!S->f16) m.bP = m.bC = m.bS;  // unused kernel parameters
    }
    if (S->f16) {
        TRY_TC(encode_operators(enc, &S->mapB2[0], &S->mapB2[1], &S->mapB2[2], type_of(S), S->ops, chunks_of(S), S->parts,
                                S->npad, S->noff + 8, S->npad / 2, S->sw));
        TcKernel kp2 = pick_pair_kernel(S->npad / 16);
        if (!kp2) return FMM_ERR_INTERNAL;
        FMM_CUDA_TRY(cudaFuncSetAttribute((const void *)kp2, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)tc_pair_smem_bytes(S->npad)));
    }
    // natural-order planes of the parent-level local expansions (fused L2L), sized for level d - 1
    if (S->f16) {
        const int64_t n = (int64_t)1 << (P.d - 1);
        S->partL_elems = (size_t)n * n * n * S->kp;
        FMM_CUDA_TRY(cudaMalloc(&S->planesL, sizeof(uint16_t) * S->partL_elems * 2));
    }
    // source planes per level
    size_t lpart_elems = 0;
    int sms = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                 cudaSuccess || sms < 1)
        sms = 152;
    for (int l = 2; l <= P.d; ++l) {  // level 1 is part of the top operator
        int np = 1 << (l - 1);
        int64_t np2 = np + 2 * P.ws;  // periodic halo of ws cells
        S->bx[l] = tile_dim(np, TC_ROWS);
        S->by[l] = tile_dim(np, TC_ROWS / S->bx[l]);
        S->bz[l] = tile_dim(np, TC_ROWS / (S->bx[l] * S->by[l]));
        S->part_elems[l] = (size_t)8 * np2 * np2 * np2 * S->kp;
        FMM_CUDA_TRY(cudaMalloc(&S->planes[l], sizeof(uint16_t) * S->part_elems[l] * S->parts));
        S->maps[l] = S->maps[0];
        TRY_TC(encode_level(enc, S, l, np, P.ws, S->bx[l], S->by[l], S->bz[l], &S->maps[l]));
        const int tiles = 8 * (np / S->bx[l]) * (np / S->by[l]) * (np / S->bz[l]);
        split_offsets(n_il(P.ws) + (S->f16 ? 1 : 0), tiles, 27, sms, S->groups[l], S->per_group[l]);
        if (S->groups[l] > 1) {
            size_t need = (size_t)S->groups[l] * 8 * np * np * np * P.nc;
            if (need > lpart_elems) lpart_elems = need;
        }
    }
    if (lpart_elems) FMM_CUDA_TRY(cudaMalloc(&S->Lpart, sizeof(float) * lpart_elems));
    TcKernel k = pick_kernel(S->pa, S->pb, S->npad / 16, S->sw);
    if (!k) return FMM_ERR_INTERNAL;
    FMM_CUDA_TRY(cudaFuncSetAttribute((const void *)k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)tc_smem_bytes(S->pa, S->pb, S->npad, S->sw)));
    if (!S->f16) {
        TcKernel kp = pick_kernel(3, 3, S->npad / 16, S->sw);  // the solute-only pass
        if (!kp) return FMM_ERR_INTERNAL;
        FMM_CUDA_TRY(cudaFuncSetAttribute((const void *)kp, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)tc_smem_bytes(3, 3, S->npad, S->sw)));
    }
    FMM_CUDA_TRY(cudaStreamSynchronize(P.stream));
    return FMM_OK;
}

unsigned *tc_amax(Plan &P, int l)
{
    TcState *S = (TcState *)P.tc;
    return S && S->f16 && l >= 0 && l <= P.d ? S->amax + l : nullptr;
}

fmm_status tc_clear_amax(Plan &P)
{
    TcState *S = (TcState *)P.tc;
    if (S && S->f16) FMM_CUDA_TRY(cudaMemsetAsync(S->amax, 0, sizeof(unsigned) * 18, P.stream));
    return FMM_OK;
}

unsigned *tc_amaxL(Plan &P, int l, const float **sx)
{
    TcState *S = (TcState *)P.tc;
    if (!S || !S->f16) return nullptr;
    *sx = S->s32inv;
    return S->amaxL + l;
}

const float *tc_scale(const Plan &P)
{
    const TcState *S = (const TcState *)P.tc;
    return S && S->f16 ? S->s32 : nullptr;
}

// fp16 split: the balanced halo planes of every level, whose largest |M^ s| the P2M and M2M have folded in
fmm_status tc_split_moments(Plan &P)
{
    TcState *S = (TcState *)P.tc;
    if (!S || !S->f16) return FMM_ERR_INTERNAL;
    SplitLevels lv;
    memset(&lv, 0, sizeof(lv));
    int i = 0;
    for (int l = P.d; l >= 2; --l, ++i) {
        const int np = 1 << (l - 1);
        const int64_t np2 = np + 2 * P.ws;
        lv.total += 8 * np2 * np2 * np2 * (S->kp / 8);
        lv.l[i] = {(const float *)P.M[l], S->amax + l, S->planes[l], S->part_elems[l], lv.total, np};
    }
    const int64_t nb = (lv.total + 255) / 256;
    k_split_halo16<<<(unsigned)(nb < 8 * 1216 ? nb : 8 * 1216), 256, 0, P.stream>>>(lv, P.ws, P.nc, S->kp, S->s32);
    FMM_LAUNCH_CHECK(P);
    return FMM_OK;
}

// Arguments of the level-l M2L (+ fused L2L with the fp16 split); returns whether the level runs on CTA
// pairs (an even number of full 128-row tiles per class), whose stage ring and M = 256 descriptor it sets
static bool m2l_args(const Plan &P, const TcState *S, int l, bool precise, int pa, int pb, TcArgs &a)
{
    const int np = 1 << (l - 1);
    fill_common(P, S, pa, pb, a);
    if (precise) a.gchunks = a.gsteps = 0;  // the solute-only pass keeps every product
    a.np = np;
    a.bx = S->bx[l];
    a.by = S->by[l];
    a.bz = S->bz[l];
    a.rows = a.bx * a.by * a.bz;
    a.tiles_x = np / a.bx;
    a.tiles_y = np / a.by;
    a.tiles_per_class = a.tiles_x * a.tiles_y * (np / a.bz);
    a.groups = S->groups[l];
    a.per_group = S->per_group[l];
    a.n_off = a.n_il + (S->f16 ? 1 : 0);
    a.L = (float *)P.L[l];
    a.post = S->f16 ? S->s32 : nullptr;
    a.amax = S->f16 ? S->amax + l : nullptr;
    a.amaxL = S->f16 ? S->amaxL + l - 1 : nullptr;
    if (S->f16) {
        a.amax_out = a.groups == 1 ? S->amaxL + l : nullptr;
        a.sx = S->s32inv;
    }
    const bool pair = S->f16 && pairs_allowed(P) && a.rows == TC_ROWS && a.tiles_per_class % 2 == 0;
    if (pair) {
        a.stages = tc_pair_stages(S->npad);
        a.idesc = (1u << 4) | ((uint32_t)(S->npad >> 3) << 17) | ((uint32_t)((2 * TC_ROWS) >> 4) << 24);  // M = 256
    }
    return pair;
}

fmm_status launch_m2l_tc(Plan &P, int l, bool precise)
{
    TcState *S = (TcState *)P.tc;
    if (!S) return FMM_ERR_INTERNAL;
    // the fp16 split is already as accurate as the 3 x 3 bf16 one
    const int pa = precise && !S->f16 ? 3 : S->pa;
    const int pb = precise && !S->f16 ? 3 : S->pb;
    int np = 1 << (l - 1);
    int64_t np2 = np + 2 * P.ws;
    if (S->f16) {
        // parent-level local expansion for the fused L2L; its largest |L^ / s| was folded in by the level
        // l - 1 launch (levels run in order)
        const int64_t ncl = (int64_t)np * np * np;
        k_split_L<<<(unsigned)((ncl + 7) / 8 < 1216 ? (ncl + 7) / 8 : 1216), 256, 0, P.stream>>>(
            (const float *)P.L[l - 1], l - 1, P.nc, S->kp, S->s32inv, S->amaxL + l - 1, S->planesL,
            (size_t)ncl * S->kp);
        FMM_LAUNCH_CHECK(P);
    } else {
        const int64_t nhalo = 8 * np2 * np2 * np2;
        k_split_halo<<<(unsigned)((nhalo + 7) / 8 < 4864 ? (nhalo + 7) / 8 : 4864), 256, 0, P.stream>>>(
            (const float *)P.M[l], np, P.ws, P.nc, S->kp, pa, kchunk_of(S->sw), S->planes[l], S->part_elems[l]);
        FMM_LAUNCH_CHECK(P);
    }
    TcArgs a;
    const bool pair = m2l_args(P, S, l, precise, pa, pb, a);
    unsigned grid = 8u * (unsigned)a.tiles_per_class * (unsigned)a.groups;
    const bool time_it = P.timings_on && l == P.d && P.ev_top[0] && !precise;
    if (time_it) cudaEventRecord(P.ev_top[0], P.stream);
    if (pair) {
        TcKernel k2 = pick_pair_kernel(S->npad / 16);
        if (!k2) return FMM_ERR_INTERNAL;
        k2<<<grid, TC_THREADS, tc_pair_smem_bytes(S->npad), P.stream>>>(pair_maps(S, l), a);
    } else {
        TcKernel k = pick_kernel(pa, pb, S->npad / 16, S->sw);
        if (!k) return FMM_ERR_INTERNAL;
        k<<<grid, TC_THREADS, tc_smem_bytes(pa, pb, S->npad, S->sw), P.stream>>>(S->maps[l], a);
    }
    FMM_LAUNCH_CHECK(P);
    if (time_it) {
        cudaEventRecord(P.ev_top[1], P.stream);
        P.top_recorded = true;
    }
    if (a.groups > 1) {
        int64_t n = (int64_t)8 * np * np * np * P.nc;
        k_group_sum<<<(unsigned)((n + 255) / 256 < 2048 ? (n + 255) / 256 : 2048), 256, 0, P.stream>>>(
            n, a.groups, S->Lpart, a.L, P.nc, S->f16 ? S->s32inv : nullptr, S->f16 ? S->amaxL + l : nullptr);
        FMM_LAUNCH_CHECK(P);
    }
    return FMM_OK;
}

// ------------------------------------------------------------------ persistent sweep (host)
int tc_sweep_first_level(const Plan &P)
{
    const TcState *S = (const TcState *)P.tc;
    if (!S || !S->f16 || !pairs_allowed(P) || P.precision != FMM_PREC_MIXED) return 0;
    for (int l = 2; l <= P.d; ++l) {
        const int np = 1 << (l - 1);
        const int tpc = (np / S->bx[l]) * (np / S->by[l]) * (np / S->bz[l]);
        if (S->bx[l] * S->by[l] * S->bz[l] == TC_ROWS && tpc % 2 == 0) return l;  // and every deeper level
    }
    return 0;
}

struct Sweep {
    std::vector<Plan *> plans;  // the plans taking part
    std::vector<int> first;     // their first sweep level
    int nch = 0, stages = 0, pairs = 0, n_items = 0, n_lv = 0, stall_item = -1;
    size_t smem = 0;
    SweepLevel *d_lv = nullptr;
    int4 *d_items = nullptr;
    int *d_q = nullptr;
    int **d_errs = nullptr;
};

void sweep_destroy(Sweep *sw)
{
    if (!sw) return;
    for (Plan *P : sw->plans) P->sweep_from = 0;
    cudaFree(sw->d_lv);
    cudaFree(sw->d_items);
    cudaFree(sw->d_q);
    cudaFree(sw->d_errs);
    delete sw;
}

void sweep_enable(Sweep *sw, bool on)
{
    if (!sw) return;
    for (size_t k = 0; k < sw->plans.size(); ++k) sw->plans[k]->sweep_from = on ? sw->first[k] : 0;
}

int sweep_plans(const Sweep *sw) { return sw ? (int)sw->plans.size() : 0; }

fmm_status sweep_create(Plan *const *plans, int n, Sweep **out)
{
    *out = nullptr;
    Sweep *sw = new (std::nothrow) Sweep();
    if (!sw) return FMM_ERR_OOM;
    for (int i = 0; i < n; ++i) {
        Plan &P = *plans[i];
        const int l0 = tc_sweep_first_level(P);
        if (l0 <= 0) continue;
        const int c = ((const TcState *)P.tc)->npad / 16;
        if (!pick_sweep_kernel(c) || (sw->nch && c != sw->nch)) continue;  // stays on its per-level launches
        sw->nch = c;
        sw->plans.push_back(&P);
        sw->first.push_back(l0);
    }
    if (sw->plans.empty()) {
        delete sw;
        return FMM_OK;
    }
    // one entry per (plan, level), each pointing at the same plan's previous level
    std::vector<SweepLevel> lv;
    int lmin = 1 << 30, lmax = 0;
    for (size_t k = 0; k < sw->plans.size(); ++k) {
        Plan &P = *sw->plans[k];
        const TcState *S = (const TcState *)P.tc;
        int prev = -1;
        for (int l = sw->first[k]; l <= P.d; ++l) {
            SweepLevel e;
            memset((void *)&e, 0, sizeof(e));
            if (!m2l_args(P, S, l, false, S->pa, S->pb, e.a) || (sw->stages && e.a.stages != sw->stages)) {
                sweep_destroy(sw);
                return FMM_ERR_INTERNAL;
            }
            sw->stages = e.a.stages;
            e.maps = pair_maps(S, l);
            const int64_t ncl = (int64_t)1 << (3 * (l - 1));  // cells of level l - 1
            e.Lprev = (const float *)P.L[l - 1];
            e.sinv = S->s32inv;
            e.amaxL_prev = S->amaxL + l - 1;
            e.planesL = S->planesL;
            e.partL = (size_t)ncl * S->kp;
            e.amaxL = S->amaxL + l;
            e.gs_n = 8 * ncl * P.nc;
            e.lev = l;
            e.nc = P.nc;
            e.kp = S->kp;
            e.n_items[0] = (int)((ncl + SWEEP_P_CELLS - 1) / SWEEP_P_CELLS);
            e.gpi = e.a.groups;  // set per level below
            e.n_items[1] = 4 * e.a.tiles_per_class;  // tile pairs: 8 classes x tiles / 2
            e.n_items[2] = e.a.groups > 1 ? (int)((e.gs_n + SWEEP_G_ELEMS - 1) / SWEEP_G_ELEMS) : 0;
            e.prev = prev;
            prev = (int)lv.size();
            lv.push_back(e);
            lmin = l < lmin ? l : lmin;
            lmax = l > lmax ? l : lmax;
        }
    }
    // item grain per level: whole tile pairs (all their offset groups in turn: one ramp and one exposed
    // epilogue per tile pair) when the level's tile pairs over all entries fill the resident pairs twice;
    // otherwise one offset group per item, so that a lone deep box's small levels spread over the GPU
    {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        for (int l = lmin; l <= lmax; ++l) {
            long long tp = 0;
            for (const SweepLevel &e : lv)
                if (e.lev == l) tp += e.n_items[1];
            for (SweepLevel &e : lv)
                if (e.lev == l && tp < (long long)sms) {  // 2 x (sms / 2) pairs
                    e.gpi = 1;
                    e.n_items[1] *= e.a.groups;
                }
        }
    }
    // the queue: level by level, within a level stage P of every entry, then M, then G
    std::vector<int4> items;
    int m_items = 0;
    for (int l = lmin; l <= lmax; ++l)
        for (int st = 0; st < 3; ++st)
            for (size_t e = 0; e < lv.size(); ++e) {
                if (lv[e].lev != l) continue;
                for (int i = 0; i < lv[e].n_items[st]; ++i) {
                    if (st == 1 && sw->stall_item < 0) sw->stall_item = (int)items.size();
                    if (st == 1) ++m_items;
                    items.push_back(make_int4(st, (int)e, i, 0));
                }
            }
    sw->n_lv = (int)lv.size();
    sw->n_items = (int)items.size();
    std::vector<int *> errs;
    for (Plan *P : sw->plans) errs.push_back(P->d_err);
    fmm_status s = FMM_OK;
    if (cudaMalloc(&sw->d_lv, sizeof(SweepLevel) * lv.size()) != cudaSuccess ||
        cudaMalloc(&sw->d_items, sizeof(int4) * items.size()) != cudaSuccess ||
        cudaMalloc(&sw->d_q, sizeof(int) * (2 + 3 * lv.size())) != cudaSuccess ||
        cudaMalloc(&sw->d_errs, sizeof(int *) * errs.size()) != cudaSuccess)
        s = FMM_ERR_OOM;
    if (s == FMM_OK &&
        (cudaMemcpy(sw->d_lv, lv.data(), sizeof(SweepLevel) * lv.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
         cudaMemcpy(sw->d_items, items.data(), sizeof(int4) * items.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
         cudaMemcpy(sw->d_errs, errs.data(), sizeof(int *) * errs.size(), cudaMemcpyHostToDevice) != cudaSuccess))
        s = FMM_ERR_CUDA;
    // as many pairs as can be resident (one CTA per SM), at most one per tile pair of the queue
    const int npad = 16 * sw->nch;
    sw->smem = tc_pair_smem_bytes(npad);
    SweepKernel k = pick_sweep_kernel(sw->nch);
    if (s == FMM_OK && cudaFuncSetAttribute((const void *)k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)sw->smem) != cudaSuccess)
        s = FMM_ERR_CUDA;
    if (s == FMM_OK) {
        int dev = 0, sms = 0, clusters = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(sms > 0 ? sms : 2));
        cfg.blockDim = dim3(TC_THREADS);
        cfg.dynamicSmemBytes = sw->smem;
        if (cudaOccupancyMaxActiveClusters(&clusters, (const void *)k, &cfg) != cudaSuccess || clusters < 1)
            clusters = sms / 2;
        cudaGetLastError();
        sw->pairs = clusters < m_items ? clusters : m_items;
        if (sw->pairs < 1) sw->pairs = 1;
    }
    if (s != FMM_OK) {
        sweep_destroy(sw);
        return s;
    }
    sweep_enable(sw, true);
    *out = sw;
    return FMM_OK;
}

fmm_status sweep_launch(Sweep *sw, cudaStream_t st, uint64_t wait_ns, bool stall, int max_pairs)
{
    if (!sw) return FMM_OK;
    FMM_CUDA_TRY(cudaMemsetAsync(sw->d_q, 0, sizeof(int) * (2 + 3 * (size_t)sw->n_lv), st));
    SweepKernel k = pick_sweep_kernel(sw->nch);
    const int pairs = max_pairs > 0 && max_pairs < sw->pairs ? max_pairs : sw->pairs;
    k<<<2u * (unsigned)pairs, TC_THREADS, sw->smem, st>>>(sw->d_lv, sw->d_items, sw->n_items, sw->stages, sw->d_q,
                                                              wait_ns, stall ? sw->stall_item : -1);
    FMM_CUDA_TRY(cudaGetLastError());
    const int n = (int)sw->plans.size();
    k_sweep_status<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(sw->d_q, sw->d_errs, n);
    FMM_CUDA_TRY(cudaGetLastError());
    return FMM_OK;
}

// Brick of the level-l tiles: bx x by x bz target cells of one parity class (the MMA's 128 rows), each
// dividing the class side 2^(l-1), an even number of tiles per class (CTA pairs); the level's plane maps
// are encoded for it.  Which targets share a tile changes, no target's arithmetic does.
fmm_status tc_set_brick(Plan &P, int l, int bx, int by, int bz)
{
    TcState *S = (TcState *)P.tc;
    if (!S) return FMM_ERR_UNSUPPORTED;
    if (l < 2 || l > P.d) return FMM_ERR_INVALID_ARG;
    const int np = 1 << (l - 1);
    if (bx < 1 || by < 1 || bz < 1 || bx * by * bz != TC_ROWS || np % bx || np % by || np % bz ||
        ((np / bx) * (np / by) * (np / bz)) % 2)
        return FMM_ERR_INVALID_ARG;
    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
    if (!enc) return FMM_ERR_INTERNAL;
    TcMaps m = S->maps[l];
    TRY_TC(encode_level(enc, S, l, np, P.ws, bx, by, bz, &m));
    S->maps[l] = m;
    S->bx[l] = bx;
    S->by[l] = by;
    S->bz[l] = bz;
    return FMM_OK;
}

void tc_get_brick(const Plan &P, int l, int *bx, int *by, int *bz)
{
    const TcState *S = (const TcState *)P.tc;
    *bx = S && l >= 1 && l <= P.d ? S->bx[l] : 0;
    *by = S && l >= 1 && l <= P.d ? S->by[l] : 0;
    *bz = S && l >= 1 && l <= P.d ? S->bz[l] : 0;
}

// The split operator tables depend only on p, ws and the split (the M2L and L2L operators are
// built for unit cells), so plans that agree on those can read one copy: dst drops its own and reads
// src's, which must outlive it.  A plan with another table is left alone.
fmm_status tc_share_operators(Plan &dst, const Plan &src)
{
    TcState *D = (TcState *)dst.tc;
    const TcState *S = (const TcState *)src.tc;
    if (!D || !S || D == S || D->ops == S->ops) return FMM_OK;
    if (dst.p != src.p || dst.ws != src.ws || D->f16 != S->f16 || D->pa != S->pa || D->pb != S->pb ||
        D->parts != S->parts || D->npad != S->npad || D->kp != S->kp || D->noff != S->noff || D->sw != S->sw ||
        D->ops_part_elems != S->ops_part_elems)
        return FMM_OK;
    FMM_CUDA_TRY(cudaDeviceSynchronize());  // nothing of dst's may still read its own table
    if (!D->ops_borrowed) cudaFree(D->ops);
    D->ops = S->ops;
    D->ops_borrowed = true;
    for (TcMaps &m : D->maps) {
        m.bS = S->maps[0].bS;
        m.bP = S->maps[0].bP;
        m.bC = S->maps[0].bC;
    }
    memcpy((void *)D->mapB2, (const void *)S->mapB2, sizeof(D->mapB2));
    return FMM_OK;
}

void tc_free(Plan &P)
{
    TcState *S = (TcState *)P.tc;
    if (!S) return;
    for (int l = 0; l < 9; ++l) cudaFree(S->planes[l]);
    if (!S->ops_borrowed) cudaFree(S->ops);
    cudaFree(S->Lpart);
    cudaFree(S->s32);
    cudaFree(S->s32inv);
    cudaFree(S->s64);
    cudaFree(S->amax);
    cudaFree(S->planesL);
    delete S;
    P.tc = nullptr;
}

}  // namespace fmm
