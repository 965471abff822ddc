// fmm_tc.cuh -- the tensor-core (tcgen05) product kernels of the M2L and fused L2L, shared by the mixed path
// (fmm_m2l_tc.cu: 16-bit operand splits) and the FP64 path (fmm_m2l_res.cu: exact residue products), with the
// host helpers that lay out their launches and tensor maps.
//
// Roles (6 warps): warp 0 issues TMA loads into a 2..6-stage ring, warp 1
// issues tcgen05.mma (both run with all lanes, one elected lane issues), warps
// 2..5 drain TMEM (warp w reads TMEM lanes 32 (w mod 4) .. +31, one target row
// per thread) and write the FP32 level array.
//
// The tensor pipe bounds the large launches: active in 91 % of a CTA's cycles
// (level 5 of 100,000 charges, p = 12; 75 % with the last wave).  It was the
// issuer's instruction stream: halving the copied bytes or the MMAs per stage
// moved the level-6 launch (N = 1M, p = 12) by 1-6 %, taking a quarter of the
// ring away by 2 %, while its per-stage code took ~900 cycles against 350-700
// of MMA time.  Issued from a single-lane branch every TMA / MMA operand is
// moved to uniform registers first; run by the whole warp, with the chunk
// structure fixed at compile time (NCH) and the grading unpacked once per tile,
// the launch went 3.69 -> 2.69 ms (N = 1M, p = 12), 24.9 -> 16.1 ms (N = 10M,
// p = 10) and 2.00 -> 1.51 ms (N = 100k, ws = 2, p = 8).  Every mbarrier wait is bounded (globaltimer); on a timeout the
// kernel records FMM_ERR_TIMEOUT, waits (bounded) for its copies and MMAs in
// flight, frees TMEM and returns.
#pragma once
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "fmm_internal.cuh"

namespace fmm {

namespace {

constexpr int TC_THREADS = 192;
constexpr int TC_MAX_STAGES = 6;
constexpr int TC_ROWS = 128;          // MMA M
// Operand rows in shared memory are SW = 64 (bf16 splits) or 128 (fp16 split)
// bytes wide, swizzled with the matching pattern: one copy box carries SW / 2
// K elements of 128 (A) or npad (B) rows.
constexpr int kchunk_of(int sw) { return sw / 2; }
constexpr uint32_t TMEM_COLS = 512;   // two accumulators of up to 256 columns
constexpr int TC_PMAX = 15;           // N = (p+1)^2 rounded to 16 must not exceed 256
constexpr uint64_t WAIT_LIMIT_NS = 2000000000ull;  // 2 s: the teardown's own limit (and the default budget)
constexpr int GAIN_T_EXP = 14;        // gT = 2^14 (fp16 split)
constexpr int GAIN_M_EXP = 14;        // gM = 2^(14 - E)
constexpr size_t TC_SMEM_BUDGET = 224 * 1024;

// Tensor maps of one launch.  Operand rows are stored chunk by chunk, [term][chunk][cell or operator row][KCH],
// so that a row of a copy box and the rows of neighbouring cells are contiguous; of A (halo'd planes), B
// (operators) and L (parent-level local expansions, natural order):
//   S  one box of one term and chunk (term and chunk folded into the slowest cell coordinate);
//   P  both terms of a chunk in one copy;  C  term 0 of two consecutive chunks in one copy (fp16 split).
struct TcMaps {
    CUtensorMap aS, aP, aC, bS, bP, bC, lS, lP;
};

struct TcArgs {
    int np, bx, by, bz, rows, tiles_x, tiles_y, tiles_per_class;
    int nc, npad, stages;
    int nslots;             // operator slots of the B tables
    int groups, per_group;  // the offsets split over `groups` CTAs per tile (small levels)
    int n_off;              // offsets: 189 or 875 (+1 with the fused L2L)
    int ws, n_il, noff;     // well-separatedness, interaction-list length, M2L operator slots
    const int *il;          // the interaction list of each class, [8][n_il] packed offsets (il_pack)
    uint32_t idesc;
    uint32_t gchunks;       // fp16x2 M2L offsets: products per K chunk, 2 bits per chunk (0 = all 3), FMM_OPT_M2L_GRADE
    uint32_t gsteps;        // in a 3-product chunk, the first K16 step from which x1 y0 is dropped, 3 bits per chunk
                            // (0: none)
    int acc_group;          // offsets summed in one TMEM accumulator before it is drained (>= 1)
    uint64_t wait_ns;       // budget of every pipeline wait (FMM_OPT_WAIT_BUDGET_NS); the teardown keeps its own
    int inject_stall;       // test hook (single-CTA kernel): the MMA issuer first waits on a barrier nothing arrives on
    float *L;               // output level array (L of the level)
    float *Lpart;           // [groups][level cells][nc] partial sums when groups > 1
    const float *post;      // fp16 split: s(j) per output coefficient, else null
    const unsigned *amax;   // fp16 split: largest |M^ s| of the A planes (gM follows from it)
    const unsigned *amaxL;  // fused L2L: largest |L^ / s| of the parent planes (gL), else null
    // residue products (FP64 path): modulus mod0 + m of `mods` in block order, planes and results by m
    int mod0;
    const int *mods;
    int16_t *resid;         // [groups][moduli of the launch][level cells][nc]
    int nmods;
    unsigned *amax_out;     // fp16 split, one offset group: fold max_i |out_i sx(i)| of the written rows in here
    const float *sx;        // with amax_out: 1 / s(i)
    int *err;
};

// 2^e as a float for |e| <= 126, built from its bits
__host__ __device__ inline float pow2f(int e)
{
    e = e < -126 ? -126 : (e > 126 ? 126 : e);
    union {
        uint32_t u;
        float f;
    } v;
    v.u = (uint32_t)(e + 127) << 23;
    return v.f;
}

// binary exponent E of a positive float given by its bits (value in [2^E, 2^(E+1)))
__device__ inline int exp_of_bits(unsigned bits) { return (int)((bits >> 23) & 0xFFu) - 127; }

// gM = 2^(GAIN_M_EXP - E), 1 when the level has no moments; kept within 2^+-100
__device__ inline int gain_m_exp(unsigned bits)
{
    if (bits == 0u) return 0;
    const int e = GAIN_M_EXP - exp_of_bits(bits);
    return e < -100 ? -100 : (e > 100 ? 100 : e);
}

// An offset of an interaction list: delta per axis in [-2 ws - c, 2 ws + 1 - c], the near (2 ws + 1)^3 block left
// out, in z, y, x order.  The producers read the list from a table: stepping through the cube and skipping what
// is not theirs took ~160 cycles a position, up to 17 us before and after the copies of a small launch (2,998
// charges at depth 3, p = 8: 682 -> 533 us a call; 100,000 at ws = 2: 2.9 -> 2.3 ms).
// A producer warp's walk through offsets o .. end of one class's list: 32 entries per load, one load ahead
struct IlWalk {
    const int *list;
    int o, end, lane, cur, next;
    __device__ __forceinline__ IlWalk(const int *l, int begin, int e, int ln) : list(l), o(begin), end(e), lane(ln)
    {
        cur = o + lane < end ? __ldg(list + o + lane) : 0;
        next = o + 32 + lane < end ? __ldg(list + o + 32 + lane) : 0;
    }
    // the offset of step k = 0, 1, .. (all lanes)
    __device__ __forceinline__ void get(int k, int &dx, int &dy, int &dz)
    {
        if (k > 0 && (k & 31) == 0) {
            cur = next;
            next = o + k + 32 + lane < end ? __ldg(list + o + k + 32 + lane) : 0;
        }
        const int e = __shfl_sync(0xffffffffu, cur, k & 31);
        il_unpack(e, dx, dy, dz);
    }
};

// Accumulation groups of one CTA's offsets: the M2L offsets, local indices 0 .. nm - 1, in runs
// of G that share one TMEM accumulator; the fused L2L offset (when present it is the CTA's last) alone,
// since its drain is scaled by gM / gL.
struct AccGroups {
    int nm, ng, G;
    __device__ AccGroups(int nloc, bool has_l2l, int g) : nm(nloc - (has_l2l ? 1 : 0)), ng(0), G(g < 1 ? 1 : g)
    {
        ng = (nm + G - 1) / G + (has_l2l ? 1 : 0);
    }
    __device__ int begin(int g) const { return g * G < nm ? g * G : nm; }
    __device__ int end(int g) const { return g * G < nm ? min((g + 1) * G, nm) : nm + 1; }
};

// ------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// 1 in one lane of a converged warp (the same lane every time a warp asks), 0 in the others
__device__ __forceinline__ uint32_t elect_one()
{
    uint32_t e;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(e));
    return e;
}

// a value that every lane of the warp holds alike, made visibly so (uniform registers)
__device__ __forceinline__ uint32_t warp_uniform(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// bounded wait on phase `parity`; false after limit_ns or when the CTA aborts
__device__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, uint64_t limit_ns = WAIT_LIMIT_NS)
{
    if (mbar_try(bar, parity)) return true;  // the usual case: no clock read
    uint64_t t0 = global_ns();
    for (uint32_t i = 0;; ++i) {
        if (mbar_try(bar, parity)) return true;
        if ((i & 63) == 63) {
            if (*abort_flag) return false;
            if (global_ns() - t0 > limit_ns) return false;
        }
    }
}

__device__ __forceinline__ bool mbar_try_cluster(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// The bounded wait of a whole converged warp: every lane gets the same answer (lanes that read the clock at
// different times must not leave a loop with warp-wide instructions in it one by one).  The clock is read out of
// line: the usual wait is one poll and one vote.
__device__ __forceinline__ bool mbar_poll_warp(uint32_t bar, uint32_t parity)
{
    return __all_sync(0xffffffffu, mbar_try(bar, parity)) != 0;
}

__device__ __noinline__ bool mbar_wait_warp_slow(uint32_t bar, uint32_t parity, volatile int *abort_flag,
                                                 uint64_t limit_ns)
{
    uint64_t t0 = global_ns();
    for (uint32_t i = 0;; ++i) {
        if (mbar_poll_warp(bar, parity)) return true;
        if ((i & 63) == 63 && __any_sync(0xffffffffu, *abort_flag != 0 || global_ns() - t0 > limit_ns)) return false;
    }
}

__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int *abort_flag,
                                               uint64_t limit_ns)
{
    return mbar_poll_warp(bar, parity) || mbar_wait_warp_slow(bar, parity, abort_flag, limit_ns);
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1, int c2,
                                            int c3)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1, int c2,
                                            int c3, int c4)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], "
        "[%7];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1, int c2)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::
            "r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}

// tcgen05 shared-memory matrix descriptor: K-major, SW-byte swizzle (layout
// code 4 for 64 bytes, 2 for 128 bytes), 8-row groups 8 SW bytes apart
// (stride byte offset), version field 1.  The high word is a constant; the low
// word holds the address in 16-byte units (14 bits: shared-memory addresses
// stay below 2^18) and the leading byte offset (unused for swizzled K-major),
// so an operand o bytes further on has the low word + o / 16.
template <int SW>
constexpr uint32_t sdesc_hi()
{
    return ((8u * SW) >> 4) | (1u << 14) | ((SW == 128 ? 2u : 4u) << 29);
}
__device__ __forceinline__ uint32_t sdesc_lo(uint32_t saddr) { return ((saddr >> 4) & 0x3FFFu) | (1u << 16); }

// D += A . B (acc = 0: D = A . B), both descriptors with the high word `hi`
template <bool PAIR>
__device__ __forceinline__ void mma_f16(uint32_t tmem_d, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc,
                                        uint32_t acc)
{
    if (PAIR)  // 2-SM: 128 rows of A and N / 2 rows of B per CTA, 128 lanes of D in each CTA's TMEM
        asm volatile(
            "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
            "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
            "setp.ne.b32 p, %5, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %4, p;\n\t}" ::"r"(tmem_d),
            "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(acc)
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
            "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
            "setp.ne.b32 p, %5, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}" ::"r"(tmem_d),
            "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(acc)
            : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
        "[%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Lr[i] += fac * accumulator column i of this warp's 32 TMEM lanes, i < 16 NCH; the loads go out in
// batches of 16-column pieces before one wait, as many as the registers left beside Lr allow
template <int NCH>
__device__ __forceinline__ void drain_accumulator(uint32_t taddr, float fac, float (&Lr)[NCH * 16])
{
    constexpr int DRAIN_BATCH = NCH * 16 + 64 <= 240 ? 4 : (NCH * 16 + 32 <= 240 ? 2 : 1);
#pragma unroll
    for (int c0 = 0; c0 < NCH; c0 += DRAIN_BATCH) {
        uint32_t r[DRAIN_BATCH][16];
#pragma unroll
        for (int c = 0; c < DRAIN_BATCH; ++c)
            if (c0 + c < NCH) tmem_ld16(taddr + (uint32_t)((c0 + c) * 16), r[c]);
        tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < DRAIN_BATCH; ++c)
            if (c0 + c < NCH)
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    Lr[(c0 + c) * 16 + j] = fmaf(__uint_as_float(r[c][j]), fac, Lr[(c0 + c) * 16 + j]);
    }
}

// The same for residue products: the accumulator columns are whole numbers of at most 2^24 and the sums are kept
// as 32-bit integers
template <int NCH>
__device__ __forceinline__ void drain_residues(uint32_t taddr, int (&acc)[NCH * 16])
{
    constexpr int DRAIN_BATCH = NCH * 16 + 64 <= 240 ? 4 : (NCH * 16 + 32 <= 240 ? 2 : 1);
#pragma unroll
    for (int c0 = 0; c0 < NCH; c0 += DRAIN_BATCH) {
        uint32_t r[DRAIN_BATCH][16];
#pragma unroll
        for (int c = 0; c < DRAIN_BATCH; ++c)
            if (c0 + c < NCH) tmem_ld16(taddr + (uint32_t)((c0 + c) * 16), r[c]);
        tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < DRAIN_BATCH; ++c)
            if (c0 + c < NCH)
#pragma unroll
                for (int j = 0; j < 16; ++j) acc[(c0 + c) * 16 + j] += __float2int_rn(__uint_as_float(r[c][j]));
    }
}

// a number congruent to v modulo p, |v| < 2^31, rp = 1 / p: the quotient has three FP32 roundings, so it is within
// p / 2 + 3 2^-24 |v| (up to p / 2 + 384)
__device__ __forceinline__ int mod_near(int v, int p, float rp) { return v - p * __float2int_rn((float)v * rp); }

// drains after which the 32-bit sums are taken modulo p: 96 x 2^24 and what mod_near leaves (moduli below 2^11) stay
// below 2^31; the sums that finish_residues stores fit 16 bits
constexpr int RES_DRAINS = 96;
static_assert((int64_t)RES_DRAINS * (1 << 24) + (1 << 10) + 384 < (int64_t)1 << 31, "sums between drains");
static_assert((1 << 10) + 384 < 1 << 15, "stored residues");

// One warp's 32 rows of residues (staged as 16-bit values, row stride srow) to out + idx(r) nc, as store_rows
template <int NCH>
__device__ __forceinline__ void store_rows16(const int16_t *stage, int srow, int r0, int rows, int64_t my_idx,
                                             int16_t *out, int nc, int lane)
{
#pragma unroll 1
    for (int r = 0; r < 32; r += 4) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t di = __shfl_sync(0xffffffffu, my_idx, r + u);
            if (r0 + r + u < rows) {
                int16_t *dst = out + di * nc;
                const int16_t *src = stage + (r0 + r + u) * srow;
#pragma unroll
                for (int c = 0; c < NCH * 16; c += 32)
                    if (c + lane < nc) dst[c + lane] = src[c + lane];
            }
        }
    }
}

// Rows r0 .. r0 + 31 (those below `rows`) of the staged output tile (row stride srow in shared memory) to
// out + idx(r) nc, idx(r) held by lane r - r0: one warp, coalesced stores, four rows in flight
template <int NCH>
__device__ __forceinline__ void store_rows(const float *stage, int srow, int r0, int rows, int64_t my_idx, float *out,
                                           int nc, int lane)
{
#pragma unroll 1
    for (int r = 0; r < 32; r += 4) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t di = __shfl_sync(0xffffffffu, my_idx, r + u);
            if (r0 + r + u < rows) {
                float *dst = out + di * nc;
                const float *src = stage + (r0 + r + u) * srow;
#pragma unroll
                for (int c = 0; c < NCH * 16; c += 32)
                    if (c + lane < nc) dst[c + lane] = src[c + lane];
            }
        }
    }
}

// The warp's rows r0 .. r0 + 31 (those below `rows`), lane r - r0 holding row r in x, to out + idx(r) nc,
// idx(r) held by lane r - r0, without shared memory: each 32 x 32 block of columns is transposed across
// the warp by a 5-step butterfly of shuffles (step m swaps the m-wide off-diagonal blocks between lanes
// l and l ^ m), after which lane l holds column 32 b + l of all 32 rows and every store is coalesced.
template <int NCH>
__device__ __forceinline__ void store_rows_shfl(float (&x)[NCH * 16], int64_t my_idx, int r0, int rows, float *out,
                                                int nc, int lane)
{
    constexpr int C = NCH * 16;
#pragma unroll
    for (int b = 0; b < (C + 31) / 32; ++b) {
        float v[32];
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = 32 * b + k < C ? x[32 * b + k] : 0.f;
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) {
            const bool up = (lane & m) != 0;
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                if (j & m) continue;
                const float recv = __shfl_xor_sync(0xffffffffu, up ? v[j] : v[j | m], m);
                if (up) v[j] = recv;
                else v[j | m] = recv;
            }
        }
        const int col = 32 * b + lane;
#pragma unroll
        for (int k = 0; k < 32; ++k) {
            const int64_t di = __shfl_sync(0xffffffffu, my_idx, k);
            if (r0 + k < rows && col < nc) out[di * nc + col] = v[k];
        }
    }
}

// ---- CTA pair (cluster of 2) helpers for the 2-SM MMA
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// shared::cluster address of the object at local shared address `a` in CTA `rank`
__device__ __forceinline__ uint32_t map_shared(uint32_t a, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// bounded wait with cluster-scope acquire (barriers that receive arrivals from the peer CTA)
__device__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int *abort_flag,
                                  uint64_t limit_ns = WAIT_LIMIT_NS)
{
    if (mbar_try_cluster(bar, parity)) return true;  // the usual case: no clock read
    uint64_t t0 = global_ns();
    for (uint32_t i = 0;; ++i) {
        if (mbar_try_cluster(bar, parity)) return true;
        if ((i & 63) == 63) {
            if (*abort_flag) return false;
            if (global_ns() - t0 > limit_ns) return false;
        }
    }
}

// arrive on an mbarrier of the peer CTA (shared::cluster address).  No cluster-scope release: what it orders
// are the epilogue's TMEM loads, which tcgen05.wait::ld has completed, and a release there is a memory barrier
// of ~2,400 cycles per drain while the copies stream in.
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_bar)
{
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}

// TMA loads into this CTA's shared memory whose completion is counted on the
// pair leader's mbarrier (`bar` a shared::cluster address)
__device__ __forceinline__ void tma_load_4d_pair(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1,
                                                 int c2, int c3)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
        "%4, %5}], [%6];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tma_load_5d_pair(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1,
                                                 int c2, int c3, int c4)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
        "%4, %5, %6}], [%7];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1,
                                                 int c2)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
        "%4}], [%5];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}

// arrive on the mbarrier at local offset `bar` in both CTAs of the pair once
// every MMA issued so far by this thread has completed
__device__ __forceinline__ void mma_commit_pair(uint32_t bar)
{
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
        "h"((uint16_t)3)
        : "memory");
}

// ------------------------------------------------------------------ the kernel
template <int PA, int PB>
struct Products;
template <>
struct Products<3, 3> {  // x_i y_j with i + j <= 2
    static constexpr int n = 6;
    __device__ static constexpr int a(int k) { return k == 0 ? 0 : k == 1 ? 0 : k == 2 ? 1 : k == 3 ? 0 : k == 4 ? 1 : 2; }
    __device__ static constexpr int b(int k) { return k == 0 ? 0 : k == 1 ? 1 : k == 2 ? 0 : k == 3 ? 2 : k == 4 ? 1 : 0; }
};
template <>
struct Products<2, 2> {  // i + j <= 1
    static constexpr int n = 3;
    __device__ static constexpr int a(int k) { return k == 2 ? 1 : 0; }
    __device__ static constexpr int b(int k) { return k == 1 ? 1 : 0; }
};
// moments in 2 terms, operator in 3: x0 y0, x0 y1, x1 y0, x0 y2.  The operator
// (the same table for every cell) keeps ~2^-24; the dropped products involve
// the moments' residual, whose error differs from cell to cell.
template <>
struct Products<2, 3> {
    static constexpr int n = 4;
    __device__ static constexpr int a(int k) { return k == 2 ? 1 : 0; }
    __device__ static constexpr int b(int k) { return k == 1 ? 1 : k == 3 ? 2 : 0; }
};

// What a pipeline stage holds, per K chunk of an offset: kind 1 one chunk with np products (of the third,
// x1 y0, the K16 steps below s2), kind 2 this chunk and the next with the product x0 y0 each, kind 0 nothing
// (the chunk went into the stage before).  Worked out once per tile; NCH fixes the number of chunks and of
// valid K16 steps, so the issuer's per-stage code is straight.
template <int KC>
struct ChunkPlan {
    int kind[KC], np[KC], s2[KC];
    __device__ __forceinline__ ChunkPlan(uint32_t gchunks, uint32_t gsteps, int nprod, int k16)
    {
        bool taken = false;
#pragma unroll
        for (int kc = 0; kc < KC; ++kc) {
            const int c = (int)((gchunks >> (2 * kc)) & 3u), st = (int)((gsteps >> (3 * kc)) & 7u);
            np[kc] = c == 0 ? nprod : c;
            s2[kc] = st == 0 ? k16 : st;
            const bool two = !taken && c == 1 && kc + 1 < KC && ((gchunks >> (2 * (kc + 1))) & 3u) == 1u;
            kind[kc] = taken ? 0 : two ? 2 : 1;
            taken = two;
        }
    }
};

// Bytes that the copies of one stage bring to this CTA (copy_bytes), and the copies: A from the box at (c1, c2, c3) of the planes (zspan slowest cells per chunk; the L
// planes when `l2l`), B rows n0 .. of operator slot `oslot`.  With at least 8 rows (`fused`) the two terms or
// the two chunks of an operand are one copy and lie rows * SW bytes apart: with four copies a stage the
// producer took ~550 cycles of its own code, as long as the MMAs of a stage at p <= 10.  Two copies a stage and
// the epilogue's scale factors in shared memory: level-d launch 16.1 -> 12.4 ms (N = 10M, p = 10), 2.69 -> 2.50 ms
// (N = 1M, p = 12), 1.51 -> 1.29 ms (N = 100k, ws = 2, p = 8), the upward pass 0.63 -> 0.56 ms at 1M.
template <int KC, int PA, int PB, int SW, bool PAIR>
__device__ __forceinline__ uint32_t copy_bytes(int kind, int np, uint32_t rows_bytes, uint32_t stageB)
{
    if (PA == 2 && PB == 2 && SW == 128) {
        if (kind == 2) return 2u * (rows_bytes + stageB);
        return (np == 3 ? 2u : 1u) * rows_bytes + (np >= 2 ? 2u : 1u) * stageB;
    }
    return (uint32_t)PA * rows_bytes + (uint32_t)PB * stageB;
}

template <int KC, int PA, int PB, int SW, bool PAIR>
__device__ __forceinline__ void issue_copies(const TcMaps &m, bool l2l, uint32_t full, uint32_t base, uint32_t sa,
                                             uint32_t stageA, uint32_t stageB, int kc, int kind, int np, bool fused,
                                             int c1, int c2, int c3, int zspan, int n0, int oslot, int nslots,
                                             int ta = 0, int tb = 0)
{
    const uint32_t bB = base + PA * stageA;
    auto a4 = [&](uint32_t dst, int term, int chunk) {
        const CUtensorMap *map = l2l ? &m.lS : &m.aS;
        if (PAIR) tma_load_4d_pair(dst, map, full, 0, c1, c2, ((ta + term) * KC + chunk) * zspan + c3);
        else tma_load_4d(dst, map, full, 0, c1, c2, ((ta + term) * KC + chunk) * zspan + c3);
    };
    auto b3 = [&](uint32_t dst, int term, int chunk) {
        if (PAIR) tma_load_3d_pair(dst, &m.bS, full, 0, n0, ((tb + term) * KC + chunk) * nslots + oslot);
        else tma_load_3d(dst, &m.bS, full, 0, n0, ((tb + term) * KC + chunk) * nslots + oslot);
    };
    if constexpr (PA == 2 && PB == 2 && SW == 128) {
        if (kind == 2) {
            if (!fused) {
                a4(base, 0, kc);
                a4(base + sa, 0, kc + 1);
            } else if (PAIR) tma_load_5d_pair(base, &m.aC, full, 0, c1, c2, c3, ta * KC + kc);
            else tma_load_5d(base, &m.aC, full, 0, c1, c2, c3, ta * KC + kc);
            if (PAIR) tma_load_4d_pair(bB, &m.bC, full, 0, n0, oslot, tb * KC + kc);
            else tma_load_4d(bB, &m.bC, full, 0, n0, oslot, tb * KC + kc);
            return;
        }
        if (np == 3 && fused) {
            const CUtensorMap *map = l2l ? &m.lP : &m.aP;
            if (PAIR) tma_load_5d_pair(base, map, full, 0, c1, c2, kc * zspan + c3, 0);
            else tma_load_5d(base, map, full, 0, c1, c2, kc * zspan + c3, 0);
        } else {
            a4(base, 0, kc);
            if (np == 3) a4(base + sa, 1, kc);
        }
        if (np == 1) b3(bB, 0, kc);
        else if (PAIR) tma_load_4d_pair(bB, &m.bP, full, 0, n0, kc * nslots + oslot, 0);
        else tma_load_4d(bB, &m.bP, full, 0, n0, kc * nslots + oslot, 0);
    } else {
#pragma unroll
        for (int i = 0; i < PA; ++i) a4(base + i * stageA, i, kc);
#pragma unroll
        for (int j = 0; j < PB; ++j) b3(bB + j * stageB, j, kc);
    }
}

// The MMAs of one stage (operand addresses are compile-time steps from the stage's descriptor words): nk valid
// K16 steps in the chunk, nk1 in the second one of a kind-2 stage; acc0 = 0 starts a new accumulator.  Products
// outer, K16 steps inner.
template <typename PR, int K16, int SW, bool PAIR>
__device__ __forceinline__ void issue_stage(uint32_t tmem_d, uint32_t a_lo, uint32_t b_lo, uint32_t sa, uint32_t sb,
                                            int nk, int nk1, int kind, int np, int s2, uint32_t idesc, uint32_t acc0)
{
    constexpr uint32_t hi = sdesc_hi<SW>();
    if (PR::n == 3 && kind == 2) {
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int k16 = 0; k16 < K16; ++k16) {
                if (k16 >= (t == 0 ? nk : nk1)) continue;
                mma_f16<PAIR>(tmem_d, a_lo + (uint32_t)t * sa + 2 * k16, b_lo + (uint32_t)t * sb + 2 * k16, hi, idesc,
                              (t == 0 && k16 == 0) ? acc0 : 1u);
            }
        return;
    }
#pragma unroll
    for (int pr = 0; pr < PR::n; ++pr) {
        if (PR::n == 3 && pr >= np) continue;
#pragma unroll
        for (int k16 = 0; k16 < K16; ++k16) {
            if (k16 >= nk || (PR::n == 3 && pr == 2 && k16 >= s2)) continue;
            mma_f16<PAIR>(tmem_d, a_lo + (uint32_t)PR::a(pr) * sa + 2 * k16, b_lo + (uint32_t)PR::b(pr) * sb + 2 * k16, hi,
                          idesc, (pr == 0 && k16 == 0) ? acc0 : 1u);
        }
    }
}

// Per output coefficient i: the factor that undoes the balancing and the gains, x^ = x~ post(i) / (gM gT), and
// s(i) or 1 / s(i) for the level maximum, in shared memory for the epilogue warps (threads t = 0 .. 127, their
// named barrier): read from global memory in the row loop, one dependent load after another, they took 31,000
// of the 381,000 cycles of a tile at p = 12.
__device__ __forceinline__ void load_scales(const TcArgs &a, float2 *sc, int n, int t)
{
    const float g = a.post ? pow2f(-gain_m_exp(__ldcg(a.amax)) - GAIN_T_EXP) : 1.f;
    asm volatile("bar.sync 1, 128;" ::: "memory");  // the tile before is done with them
    for (int i = t; i < n; i += 128)
        sc[i] = i < a.nc ? make_float2(a.post ? __ldg(a.post + i) * g : 1.f, a.amax_out ? __ldg(a.sx + i) : 0.f)
                         : make_float2(0.f, 0.f);
    asm volatile("bar.sync 1, 128;" ::: "memory");
}

// One row of results, scaled, to its place in the staging tile; returns its largest |value f.y|.  The factors of
// 16 columns are read before their values are stored (the compiler cannot move shared-memory reads over stores).
template <int NCH>
__device__ __forceinline__ float stage_row(const float (&Lr)[NCH * 16], const float2 *sc, float *dst, int nc)
{
    float mx = 0.f;
#pragma unroll
    for (int i0 = 0; i0 < NCH * 16; i0 += 16) {
        float2 f[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) f[i] = sc[i0 + i];
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (i0 < (NCH - 1) * 16 || i0 + i < nc) {
                const float v = Lr[i0 + i] * f[i].x;
                dst[i0 + i] = v;
                mx = fmaxf(mx, fabsf(v * f[i].y));
            }
    }
    return mx;
}

// The end of a residue tile: sums taken modulo p, staged as 16-bit rows in the idle ring, stored
template <int NCH>
__device__ __forceinline__ void finish_residues(int (&acc)[NCH * 16], const TcArgs &a, int mod, int grp, int p, float rp,
                                                int16_t *stage, int quad, int row, int64_t my_idx, int lane)
{
    const int srow = a.nc | 1;
    if (row < a.rows) {
#pragma unroll
        for (int i = 0; i < NCH * 16; ++i)
            if (i < (NCH - 1) * 16 || i < a.nc) stage[row * srow + i] = (int16_t)mod_near(acc[i], p, rp);
    }
    __syncwarp();
    const int64_t cells = 8 * (int64_t)a.np * a.np * a.np;
    store_rows16<NCH>(stage, srow, quad * 32, a.rows, my_idx,
                      a.resid + ((int64_t)grp * a.nmods + mod) * cells * a.nc, a.nc, lane);
}

// One CTA sums, for 128 target rows, the products of a list of offsets: the
// 189 (875) interaction-list offsets of parity class `cls`, A from the halo'd
// source planes of the level; with fused L2L (fp16 split) one more offset whose
// A is the parent level's local expansion at the targets' parents (natural-order
// planes) and whose B is the L2L operator of child octant `cls`; its accumulator
// is scaled by gM / gL.
// PA, PB: terms of the A and B operands; NCH: output coefficients / 16 (the
// accumulator width held in registers); SW: bytes per swizzled operand row.
template <int PA, int PB, int NCH, int SW, bool RES = false>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_m2l_tc(const __grid_constant__ TcMaps maps, TcArgs a)
{
    extern __shared__ uint8_t smem_dyn[];
    __shared__ __align__(8) uint64_t bar_full[TC_MAX_STAGES];
    __shared__ __align__(8) uint64_t bar_empty[TC_MAX_STAGES];
    __shared__ __align__(8) uint64_t bar_tfull[2];
    __shared__ __align__(8) uint64_t bar_tempty[2];
    __shared__ __align__(8) uint64_t bar_done;
    __shared__ __align__(8) uint64_t bar_never;  // test hook: initialised, never arrived on
    __shared__ uint32_t tmem_sh;
    __shared__ int abort_sh;
    __shared__ int produced_sh, consumed_sh;
    __shared__ float2 scale_sh[NCH * 16];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t smem0 = warp_uniform((smem_u32(smem_dyn) + 1023u) & ~1023u);
    constexpr int KCH = kchunk_of(SW);  // K elements per stage
    constexpr int K16 = SW / 32;        // MMAs (K = 16) per stage and product
    constexpr uint32_t stageA = TC_ROWS * SW;
    constexpr uint32_t stageB = NCH * 16u * SW;
    constexpr uint32_t stage_bytes = PA * stageA + PB * stageB;
    constexpr bool kGradable = PA == 2 && PB == 2;  // the degree grading applies to the 2 x 2-term products

    // M2L: the 8 parity classes of one brick run side by side, so CTAs resident
    // at the same time read overlapping shifted bricks, which stay in L2
    const int per_mod = 8 * a.tiles_per_class * a.groups;  // residues: the modulus outermost
    const int mod = RES ? (int)blockIdx.x / per_mod : 0;
    const int block = (int)blockIdx.x - mod * per_mod;
    const int grp = block % a.groups;
    const int cls = (block / a.groups) & 7;
    const int tile = (block / a.groups) >> 3;
    const int o_begin = grp * a.per_group;
    const int o_end = o_begin + a.per_group < a.n_off ? o_begin + a.per_group : a.n_off;
    const int nloc = o_end > o_begin ? o_end - o_begin : 0;
    const bool has_l2l = a.n_off > a.n_il && a.n_il >= o_begin && a.n_il < o_end;
    const AccGroups groups(nloc, has_l2l, a.acc_group);
    const int x0 = (tile % a.tiles_x) * a.bx;
    const int y0 = ((tile / a.tiles_x) % a.tiles_y) * a.by;
    const int z0 = (tile / (a.tiles_x * a.tiles_y)) * a.bz;
    const int cx = cls & 1, cy = (cls >> 1) & 1, cz = (cls >> 2) & 1;
    const int np2 = a.np + 2 * a.ws;
    // the second term (or chunk) of A lies right behind the tile's rows when it comes with the first in one copy
    const bool fused = kGradable && SW == 128 && a.rows >= 8;
    const uint32_t rows_bytes = (uint32_t)(a.rows * SW);
    const uint32_t sa = fused ? rows_bytes : stageA;

    if (threadIdx.x == 0) {
        for (int s = 0; s < a.stages; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&bar_tfull[b]), 1);
            mbar_init(smem_u32(&bar_tempty[b]), 4);  // one arrival per epilogue warp
        }
        mbar_init(smem_u32(&bar_done), 1);
        mbar_init(smem_u32(&bar_never), 1);
        abort_sh = 0;
        produced_sh = 0;
        consumed_sh = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_sh)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = warp_uniform(tmem_sh);
    volatile int *abort_flag = &abort_sh;

    // The producer and issuer warps run their loops with all lanes (waits and ring arithmetic are the same in
    // every lane) and one elected lane issues: operands of a TMA copy or an MMA then come from uniform
    // registers, where a single-lane branch has to move each of them there per instruction.
    const uint32_t el = elect_one();
    if (warp == 0) {
        {
            // ---------------- producer: TMA loads of the A brick and the B operator
            constexpr int KC = (NCH + K16 - 1) / K16;
            const ChunkPlan<KC> graded_plan(kGradable ? a.gchunks : 0u,
                                            kGradable ? a.gsteps : 0u, PB == 2 ? 3 : PA + PB, K16);
            const uint32_t full0 = smem_u32(&bar_full[0]), empty0 = smem_u32(&bar_empty[0]);
            int it = 0, s = 0;
            uint32_t phase = 1;
            bool ok = true;
            // all K chunks of one offset: A from the planes (or the L planes) at (c1, c2, c3), B at operator slot
            // `oslot`; a graded (M2L) offset copies only the terms its chunk's products read
            auto load_offset = [&](bool l2l, int c1, int c2, int c3, int zspan, int oslot, bool graded) {
#pragma unroll
                for (int kc = 0; kc < KC; ++kc) {
                    const int kind = graded ? graded_plan.kind[kc] : 1;
                    const int np = graded ? graded_plan.np[kc] : 3;
                    if (kind == 0 || !ok) continue;
                    if (it >= a.stages && !mbar_wait_warp(empty0 + 8u * (uint32_t)s, phase, abort_flag, a.wait_ns)) {
                        ok = false;
                        continue;
                    }
                    if (el) {
                        const uint32_t full = full0 + 8u * (uint32_t)s, base = smem0 + (uint32_t)s * stage_bytes;
                        mbar_expect_tx(full, copy_bytes<KC, PA, PB, SW, false>(kind, np, rows_bytes, stageB));
                        issue_copies<KC, PA, PB, SW, false>(maps, l2l, full, base, sa, stageA, stageB, kc, kind, np, fused,
                                                            c1, c2, c3, zspan, 0, oslot, a.nslots, mod, RES ? a.mod0 + mod : 0);
                    }
                    __syncwarp();
                    ++it;
                    if (++s == a.stages) {
                        s = 0;
                        phase ^= 1u;
                    }
                }
            };
            // the source brick sits at parent offset (c + delta) >> 1 in [-ws, ws], halo width ws
            const int w = a.ws, o_il = o_end < a.n_il ? o_end : a.n_il;
            IlWalk walk(a.il + cls * a.n_il, o_begin, o_il, lane);
            for (int k = 0; k < o_il - o_begin && ok; ++k) {
                int dx, dy, dz;
                walk.get(k, dx, dy, dz);
                const int sx = cx + dx, sy = cy + dy, sz = cz + dz;
                const int scls = (sx & 1) | ((sy & 1) << 1) | ((sz & 1) << 2);
                load_offset(false, x0 + (sx >> 1) + w, y0 + (sy >> 1) + w, scls * np2 + z0 + (sz >> 1) + w, 8 * np2,
                            off_slot(dx, dy, dz, w), true);
            }
            // fused L2L: the parents' local expansions (natural order, no halo)
            if (ok && a.n_off > a.n_il && a.n_il >= o_begin && a.n_il < o_end)
                load_offset(true, x0, y0, z0, a.np, a.noff + cls, false);
            if (el) {
                produced_sh = it;
                if (!ok) {
                    abort_sh = 1;
                    atomicOr(a.err, ERRF_TIMEOUT);
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        {
            // ---------------- MMA issuer: one fresh accumulator per group of offsets
            using PR = Products<PA, PB>;
            constexpr int KC = (NCH + K16 - 1) / K16;
            const ChunkPlan<KC> graded_plan(kGradable ? a.gchunks : 0u,
                                            kGradable ? a.gsteps : 0u, PR::n, K16);
            const uint32_t a_lo0 = sdesc_lo(smem0), b_lo0 = sdesc_lo(smem0 + PA * stageA);
            const uint32_t full0 = smem_u32(&bar_full[0]), empty0 = smem_u32(&bar_empty[0]);
            int it = 0, s = 0;
            uint32_t phase = 0;
            // the test hook makes this thread's first wait run out (its budget), as a lost copy would
            bool ok = !(a.inject_stall && !mbar_wait_warp(smem_u32(&bar_never), 0, abort_flag, a.wait_ns));
            for (int g = 0; g < groups.ng && ok; ++g) {
                const int acc = g & 1;
                const uint32_t use = (uint32_t)(g >> 1);
                if (g >= 2 && !mbar_wait_warp(smem_u32(&bar_tempty[acc]), (use - 1u) & 1u, abort_flag, a.wait_ns)) {
                    ok = false;
                    break;
                }
                fence_after();
                const uint32_t tmem_d = tmem + (uint32_t)(acc * 256);
                uint32_t acc0 = 0;  // the group's first MMA overwrites the accumulator
                for (int o = groups.begin(g); o < groups.end(g) && ok; ++o) {
                    const bool graded = o_begin + o < a.n_il;
#pragma unroll
                    for (int kc = 0; kc < KC; ++kc) {
                        const int kind = graded ? graded_plan.kind[kc] : 1;
                        if (kind == 0 || !ok) continue;
                        if (!mbar_wait_warp(full0 + 8u * (uint32_t)s, phase, abort_flag, a.wait_ns)) {
                            ok = false;
                            continue;
                        }
                        fence_after();
                        if (el) {
                            const uint32_t at = (uint32_t)s * (stage_bytes >> 4);
                            const int nk = NCH - K16 * kc < K16 ? NCH - K16 * kc : K16;
                            const int nk1 = NCH - K16 * (kc + 1) < K16 ? NCH - K16 * (kc + 1) : K16;
                            issue_stage<PR, K16, SW, false>(tmem_d, a_lo0 + at, b_lo0 + at, sa >> 4, stageB >> 4, nk, nk1,
                                                            kind, graded ? graded_plan.np[kc] : PR::n,
                                                            graded ? graded_plan.s2[kc] : K16, a.idesc, acc0);
                            mma_commit(empty0 + 8u * (uint32_t)s);
                        }
                        __syncwarp();
                        acc0 = 1;
                        ++it;
                        if (++s == a.stages) {
                            s = 0;
                            phase ^= 1u;
                        }
                    }
                }
                if (ok && el) mma_commit(smem_u32(&bar_tfull[acc]));
                __syncwarp();
            }
            if (el) {
                consumed_sh = it;
                if (!ok) {
                    abort_sh = 1;
                    atomicOr(a.err, ERRF_TIMEOUT);
                }
                mma_commit(smem_u32(&bar_done));  // arrives once every issued MMA has completed
            }
        }
        __syncwarp();
    } else {
        // ---------------- epilogue warps: drain each group's accumulator into FP32 registers
        const int quad = warp & 3;
        const int row = quad * 32 + lane;
        if constexpr (RES) {
            const int p = a.mods[a.mod0 + mod];
            const float rp = 1.f / (float)p;
            int acc[NCH * 16];
#pragma unroll
            for (int i = 0; i < NCH * 16; ++i) acc[i] = 0;
            bool ok = true;
            for (int g = 0; g < groups.ng; ++g) {
                const int b = g & 1;
                if (!mbar_wait_warp(smem_u32(&bar_tfull[b]), (uint32_t)(g >> 1) & 1u, abort_flag, a.wait_ns)) {
                    ok = false;
                    break;
                }
                fence_after();
                drain_residues<NCH>(tmem + (uint32_t)(b * 256) + ((uint32_t)(quad * 32) << 16), acc);
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bar_tempty[b]));
                if ((g + 1) % RES_DRAINS == 0)
#pragma unroll
                    for (int i = 0; i < NCH * 16; ++i) acc[i] = mod_near(acc[i], p, rp);
            }
            if (!ok) {
                abort_sh = 1;
                if (lane == 0) atomicOr(a.err, ERRF_TIMEOUT);
            } else {
                const int64_t np = a.np;
                const int tx = row % a.bx, ty = (row / a.bx) % a.by, tz = row / (a.bx * a.by);
                finish_residues<NCH>(acc, a, mod, grp, p, rp,
                                     reinterpret_cast<int16_t *>(smem_dyn + (smem0 - smem_u32(smem_dyn))), quad, row,
                                     (int64_t)cls * np * np * np + (x0 + tx) + np * ((y0 + ty) + np * (int64_t)(z0 + tz)),
                                     lane);
            }
        } else {
        load_scales(a, scale_sh, NCH * 16, quad * 32 + lane);
        // fused L2L offset: its A planes carry the gain gL instead of gM
        const float l2l_fac =
            a.amaxL ? pow2f(gain_m_exp(*a.amax) - gain_m_exp(*a.amaxL)) : 1.f;
        float Lr[NCH * 16];
#pragma unroll
        for (int i = 0; i < NCH * 16; ++i) Lr[i] = 0.f;
        bool ok = true;
        for (int g = 0; g < groups.ng; ++g) {
            const int acc = g & 1;
            const uint32_t use = (uint32_t)(g >> 1);
            if (!mbar_wait_warp(smem_u32(&bar_tfull[acc]), use & 1u, abort_flag, a.wait_ns)) {
                ok = false;
                break;
            }
            fence_after();
            const float fac = (has_l2l && g == groups.ng - 1) ? l2l_fac : 1.f;
            drain_accumulator<NCH>(tmem + (uint32_t)(acc * 256) + ((uint32_t)(quad * 32) << 16), fac, Lr);
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bar_tempty[acc]));
        }
        float mx = 0.f;  // largest |out_i sx(i)| of this thread's row (a.amax_out)
        if (!ok) {
            abort_sh = 1;
            if (lane == 0) atomicOr(a.err, ERRF_TIMEOUT);
        } else {
            // every MMA has completed, so the stage ring is idle: the rows go through shared memory (stride
            // srow, odd) and leave in coalesced stores, a warp per 32 rows
            float *stage = reinterpret_cast<float *>(smem_dyn + (smem0 - smem_u32(smem_dyn)));
            const int srow = a.nc | 1;
            if (row < a.rows) {
                mx = stage_row<NCH>(Lr, scale_sh, stage + row * srow, a.nc);
            }
            const int64_t np = a.np;
            const int64_t level_cells = 8 * np * np * np;
            float *out = a.groups == 1 ? a.L : a.Lpart + (int64_t)grp * level_cells * a.nc;
            const int tx = row % a.bx, ty = (row / a.bx) % a.by, tz = row / (a.bx * a.by);
            const int64_t my_idx =
                (int64_t)cls * np * np * np + (x0 + tx) + np * ((y0 + ty) + np * (int64_t)(z0 + tz));
            __syncwarp();
            store_rows<NCH>(stage, srow, quad * 32, a.rows, my_idx, out, a.nc, lane);
        }
        if (a.amax_out) {  // the whole warp is here
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            if (lane == 0 && mx > 0.f) atomicMax(a.amax_out, __float_as_uint(mx));
        }
        }
    }

    // ---------------- teardown: wait (bounded) for MMAs and copies in flight, free TMEM
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile int no_abort = 0;
        if (!mbar_wait(smem_u32(&bar_done), 0, &no_abort)) atomicOr(a.err, ERRF_TIMEOUT);
        if (abort_sh)
            for (int it = consumed_sh; it < produced_sh; ++it)
                mbar_wait(smem_u32(&bar_full[it % a.stages]), (uint32_t)(it / a.stages) & 1u, &no_abort);
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
}

// Pair variant for the fp16 split (128-byte rows): a cluster of two
// CTAs computes 256 target rows, tiles 2t and 2t + 1 of one class, with 2-SM
// MMAs (M = 256).  Each CTA copies its own 128-row A brick and half of every
// operator tile (N/2 rows); the MMAs, issued by the even CTA, read both CTAs'
// shared memory and leave each CTA's 128 rows in its own TMEM, so each SM
// streams half of the operator bytes of the single-CTA kernel.
//   full[s]   even CTA only: its expect-tx covers both CTAs' copies, which all
//             complete on it
//   empty[s]  both CTAs: the even CTA's MMA commit, multicast to the pair
//   tfull[b]  both CTAs: multicast commit; tempty[b] on the even CTA counts
//             the 4 local and 4 remote epilogue warps
//   done      both CTAs: multicast commit after the last MMA
// Barriers are initialised and TMEM is allocated (collectively) only after a
// cluster barrier, and both CTAs pass a cluster barrier before the collective
// TMEM release, so neither touches the other after it has exited.
struct PairBars {
    uint64_t full[TC_MAX_STAGES];
    uint64_t empty[TC_MAX_STAGES];
    uint64_t tfull[2];
    uint64_t tempty[2];
    uint64_t done;
    float2 scale[256];  // the epilogue's per-coefficient factors (load_scales)
};

// Pipeline positions of one role thread, carried from tile to tile when a pair runs several tiles (the
// persistent sweep): stages issued, ring stage and pass, accumulator groups used.
struct PairPipe {
    int it = 0, s = 0;
    uint32_t round = 0, g = 0;
};

__device__ __forceinline__ void pair_bars_init(PairBars &b, int stages)
{
    for (int s = 0; s < stages; ++s) {
        mbar_init(smem_u32(&b.full[s]), 1);
        mbar_init(smem_u32(&b.empty[s]), 1);
    }
    for (int i = 0; i < 2; ++i) {
        mbar_init(smem_u32(&b.tfull[i]), 1);
        mbar_init(smem_u32(&b.tempty[i]), 8);  // 4 epilogue warps in each CTA
    }
    mbar_init(smem_u32(&b.done), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// The roles of both CTAs for pair `pair` of the launch arguments `a` (tiles 2t and 2t + 1 of one class,
// one offset group).  The ring and accumulator phases continue from `pp`; the caller commits `done` after
// its last tile.  A wait that runs out sets *abort_flag and records FMM_ERR_TIMEOUT.  `staged`: the caller
// issues no copies until every thread is done with this tile, so the epilogue may stage the output rows
// in the ring (`stage`, generic address of its start); otherwise each thread writes its row directly.
template <int NCH, bool RES = false>
__device__ __forceinline__ void pair_tile(const TcMaps &maps, const TcArgs &a, int pair, uint32_t rank, uint32_t smem0, float *stage,
                                          bool staged, PairBars &bars, uint32_t tmem, volatile int *abort_flag,
                                          PairPipe &pp, uint32_t el)
{
    constexpr int PA = 2, PB = 2, SW = 128;
    constexpr int K16 = SW / 32, KC = (NCH + K16 - 1) / K16;
    using PR = Products<PA, PB>;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool leader = rank == 0;
    constexpr uint32_t halfN = NCH * 8u;  // rows of B per CTA
    constexpr uint32_t stageA = TC_ROWS * SW;
    constexpr uint32_t stageB = halfN * SW;
    constexpr uint32_t stage_bytes = PA * stageA + PB * stageB;

    const int per_mod = 4 * a.tiles_per_class * a.groups;  // residues: the modulus outermost
    const int mod = RES ? pair / per_mod : 0;
    pair -= mod * per_mod;
    const int grp = pair % a.groups;
    const int cls = (pair / a.groups) & 7;
    const int tile = 2 * ((pair / a.groups) >> 3) + (int)rank;
    const int o_begin = grp * a.per_group;
    const int o_end = o_begin + a.per_group < a.n_off ? o_begin + a.per_group : a.n_off;
    const int nloc = o_end > o_begin ? o_end - o_begin : 0;
    const bool has_l2l = a.n_off > a.n_il && a.n_il >= o_begin && a.n_il < o_end;
    const AccGroups groups(nloc, has_l2l, a.acc_group);
    const int x0 = (tile % a.tiles_x) * a.bx;
    const int y0 = ((tile / a.tiles_x) % a.tiles_y) * a.by;
    const int z0 = (tile / (a.tiles_x * a.tiles_y)) * a.bz;
    const int cx = cls & 1, cy = (cls >> 1) & 1, cz = (cls >> 2) & 1;
    const int np2 = a.np + 2 * a.ws;

    // as in k_m2l_tc, the producer and issuer warps run with all lanes and the elected lane `el` issues
    if (warp == 0) {
        {
            // ---------------- producer (both CTAs): own A brick, own half of B, completing on the leader's barrier
            const ChunkPlan<KC> graded_plan(a.gchunks, a.gsteps, PR::n, K16);
            const uint32_t full_local0 = smem_u32(&bars.full[0]), empty0 = smem_u32(&bars.empty[0]);
            const uint32_t full_lead0 = warp_uniform(map_shared(full_local0, 0));
            int it = pp.it, s = pp.s;
            uint32_t phase = (pp.round & 1u) ^ 1u;
            bool ok = true;
            auto load_offset = [&](bool l2l, int c1, int c2, int c3, int zspan, int oslot, bool graded) {
#pragma unroll
                for (int kc = 0; kc < KC; ++kc) {
                    const int kind = graded ? graded_plan.kind[kc] : 1;
                    const int np = graded ? graded_plan.np[kc] : 3;
                    if (kind == 0 || !ok) continue;
                    if (it >= a.stages && !mbar_wait_warp(empty0 + 8u * (uint32_t)s, phase, abort_flag, a.wait_ns)) {
                        ok = false;
                        continue;
                    }
                    if (el) {
                        const uint32_t base = smem0 + (uint32_t)s * stage_bytes;
                        // the leader's barrier counts both CTAs' copies (the same boxes in each)
                        if (leader)
                            mbar_expect_tx(full_local0 + 8u * (uint32_t)s,
                                           2u * copy_bytes<KC, PA, PB, SW, true>(kind, np, stageA, stageB));
                        issue_copies<KC, PA, PB, SW, true>(maps, l2l, full_lead0 + 8u * (uint32_t)s, base, stageA, stageA,
                                                           stageB, kc, kind, np, true, c1, c2, c3, zspan,
                                                           (int)(rank * halfN), oslot, a.nslots, mod, RES ? a.mod0 + mod : 0);
                    }
                    __syncwarp();
                    if (it < a.stages) ++it;
                    if (++s == a.stages) {
                        s = 0;
                        phase ^= 1u;
                    }
                }
            };
            const int w = a.ws, o_il = o_end < a.n_il ? o_end : a.n_il;
            IlWalk walk(a.il + cls * a.n_il, o_begin, o_il, lane);
            for (int k = 0; k < o_il - o_begin && ok; ++k) {
                int dx, dy, dz;
                walk.get(k, dx, dy, dz);
                const int sx = cx + dx, sy = cy + dy, sz = cz + dz;
                const int scls = (sx & 1) | ((sy & 1) << 1) | ((sz & 1) << 2);
                load_offset(false, x0 + (sx >> 1) + w, y0 + (sy >> 1) + w, scls * np2 + z0 + (sz >> 1) + w, 8 * np2,
                            off_slot(dx, dy, dz, w), true);
            }
            if (ok && a.n_off > a.n_il && a.n_il >= o_begin && a.n_il < o_end)
                load_offset(true, x0, y0, z0, a.np, a.noff + cls, false);
            pp.it = it;
            pp.s = s;
            pp.round = phase ^ 1u;
            if (!ok && el) {
                *abort_flag = 1;
                atomicOr(a.err, ERRF_TIMEOUT);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (leader) {
            // ---------------- MMA issuer (even CTA): 256-row MMAs over both CTAs' operands
            const ChunkPlan<KC> graded_plan(a.gchunks, a.gsteps, PR::n, K16);
            const uint32_t a_lo0 = sdesc_lo(smem0), b_lo0 = sdesc_lo(smem0 + PA * stageA);
            const uint32_t full0 = smem_u32(&bars.full[0]), empty0 = smem_u32(&bars.empty[0]);
            int s = pp.s;
            uint32_t phase = pp.round & 1u;
            bool ok = true;
            for (int g = 0; g < groups.ng && ok; ++g) {
                const uint32_t gg = pp.g + (uint32_t)g;
                const int acc = (int)(gg & 1u);
                const uint32_t use = gg >> 1;
                if (gg >= 2 && !mbar_wait_warp(smem_u32(&bars.tempty[acc]), (use - 1u) & 1u, abort_flag, a.wait_ns)) {
                    ok = false;
                    break;
                }
                fence_after();
                const uint32_t tmem_d = tmem + (uint32_t)(acc * 256);
                uint32_t acc0 = 0;  // the group's first MMA overwrites the accumulator
                for (int o = groups.begin(g); o < groups.end(g) && ok; ++o) {
                    const bool graded = o_begin + o < a.n_il;
#pragma unroll
                    for (int kc = 0; kc < KC; ++kc) {
                        const int kind = graded ? graded_plan.kind[kc] : 1;
                        if (kind == 0 || !ok) continue;
                        if (!mbar_wait_warp(full0 + 8u * (uint32_t)s, phase, abort_flag, a.wait_ns)) {
                            ok = false;
                            continue;
                        }
                        fence_after();
                        if (el) {
                            const uint32_t at = (uint32_t)s * (stage_bytes >> 4);
                            const int nk = NCH - K16 * kc < K16 ? NCH - K16 * kc : K16;
                            const int nk1 = NCH - K16 * (kc + 1) < K16 ? NCH - K16 * (kc + 1) : K16;
                            issue_stage<PR, K16, SW, true>(tmem_d, a_lo0 + at, b_lo0 + at, stageA >> 4, stageB >> 4, nk, nk1,
                                                           kind, graded ? graded_plan.np[kc] : PR::n,
                                                           graded ? graded_plan.s2[kc] : K16, a.idesc, acc0);
                            mma_commit_pair(empty0 + 8u * (uint32_t)s);
                        }
                        __syncwarp();
                        acc0 = 1;
                        if (++s == a.stages) {
                            s = 0;
                            phase ^= 1u;
                        }
                    }
                }
                if (ok && el) mma_commit_pair(smem_u32(&bars.tfull[acc]));
                __syncwarp();
            }
            pp.s = s;
            pp.round = phase;
            pp.g += (uint32_t)groups.ng;
            if (!ok && el) {
                *abort_flag = 1;
                atomicOr(a.err, ERRF_TIMEOUT);
            }
        }
        __syncwarp();
    } else {
        // ---------------- epilogue warps (both CTAs): drain this CTA's 128 rows
        const int quad = warp & 3;
        const int row = quad * 32 + lane;
        if constexpr (RES) {
            const int p = a.mods[a.mod0 + mod];
            const float rp = 1.f / (float)p;
            int acc[NCH * 16];
#pragma unroll
            for (int i = 0; i < NCH * 16; ++i) acc[i] = 0;
            bool ok = true;
            for (int g = 0; g < groups.ng; ++g) {
                const uint32_t gg = pp.g + (uint32_t)g;
                const int b = (int)(gg & 1u);
                if (!mbar_wait_warp(smem_u32(&bars.tfull[b]), (gg >> 1) & 1u, abort_flag, a.wait_ns)) {
                    ok = false;
                    break;
                }
                fence_after();
                drain_residues<NCH>(tmem + (uint32_t)(b * 256) + ((uint32_t)(quad * 32) << 16), acc);
                fence_before();
                __syncwarp();
                if (lane == 0) {
                    const uint32_t te = smem_u32(&bars.tempty[b]);
                    if (leader) mbar_arrive(te);
                    else mbar_arrive_remote(map_shared(te, 0));
                }
                if ((g + 1) % RES_DRAINS == 0)
#pragma unroll
                    for (int i = 0; i < NCH * 16; ++i) acc[i] = mod_near(acc[i], p, rp);
            }
            pp.g += (uint32_t)groups.ng;
            if (!ok) {
                *abort_flag = 1;
                if (lane == 0) atomicOr(a.err, ERRF_TIMEOUT);
            } else {
                const int64_t np = a.np;
                const int tx = row % a.bx, ty = (row / a.bx) % a.by, tz = row / (a.bx * a.by);
                finish_residues<NCH>(acc, a, mod, grp, p, rp, reinterpret_cast<int16_t *>(stage), quad, row,
                                     (int64_t)cls * np * np * np + (x0 + tx) + np * ((y0 + ty) + np * (int64_t)(z0 + tz)),
                                     lane);
            }
        } else {
        load_scales(a, bars.scale, NCH * 16, row);
        const float l2l_fac = a.amaxL ? pow2f(gain_m_exp(__ldcg(a.amax)) - gain_m_exp(__ldcg(a.amaxL))) : 1.f;
        float Lr[NCH * 16];
#pragma unroll
        for (int i = 0; i < NCH * 16; ++i) Lr[i] = 0.f;
        bool ok = true;
        for (int g = 0; g < groups.ng; ++g) {
            const uint32_t gg = pp.g + (uint32_t)g;
            const int acc = (int)(gg & 1u);
            const uint32_t use = gg >> 1;
            if (!mbar_wait_warp(smem_u32(&bars.tfull[acc]), use & 1u, abort_flag, a.wait_ns)) {
                ok = false;
                break;
            }
            fence_after();
            const float fac = (has_l2l && g == groups.ng - 1) ? l2l_fac : 1.f;
            drain_accumulator<NCH>(tmem + (uint32_t)(acc * 256) + ((uint32_t)(quad * 32) << 16), fac, Lr);
            fence_before();
            __syncwarp();
            if (lane == 0) {
                const uint32_t te = smem_u32(&bars.tempty[acc]);
                if (leader) mbar_arrive(te);
                else mbar_arrive_remote(map_shared(te, 0));
            }
        }
        pp.g += (uint32_t)groups.ng;
        float mx = 0.f;  // largest |out_i sx(i)| of this thread's row (a.amax_out)
        if (!ok) {
            *abort_flag = 1;
            if (lane == 0) atomicOr(a.err, ERRF_TIMEOUT);
        } else if (!staged) {
            // the ring may already hold the next tile's copies: the rows are transposed across each warp in
            // registers for coalesced stores
#pragma unroll
            for (int i = 0; i < NCH * 16; ++i) {
                const float2 f = bars.scale[i];  // zeros beyond nc
                Lr[i] = (i < (NCH - 1) * 16 || i < a.nc) ? Lr[i] * f.x : 0.f;
                mx = fmaxf(mx, fabsf(Lr[i] * f.y));
            }
            const int64_t np = a.np;
            float *out = a.groups == 1 ? a.L : a.Lpart + (int64_t)grp * 8 * np * np * np * a.nc;
            const int tx = row % a.bx, ty = (row / a.bx) % a.by, tz = row / (a.bx * a.by);
            const int64_t my_idx = (int64_t)cls * np * np * np + (x0 + tx) + np * ((y0 + ty) + np * (int64_t)(z0 + tz));
            store_rows_shfl<NCH>(Lr, my_idx, quad * 32, a.rows, out, a.nc, lane);
        } else {
            // every MMA of the tile has completed and no copy is pending, so the stage ring is idle: the rows
            // go through shared memory (stride srow, odd) and leave in coalesced stores, a warp per 32 rows
            const int srow = a.nc | 1;
            mx = stage_row<NCH>(Lr, bars.scale, stage + row * srow, a.nc);
            const int64_t np = a.np;
            float *out = a.groups == 1 ? a.L : a.Lpart + (int64_t)grp * 8 * np * np * np * a.nc;
            const int tx = row % a.bx, ty = (row / a.bx) % a.by, tz = row / (a.bx * a.by);
            const int64_t my_idx = (int64_t)cls * np * np * np + (x0 + tx) + np * ((y0 + ty) + np * (int64_t)(z0 + tz));
            __syncwarp();
            store_rows<NCH>(stage, srow, quad * 32, a.rows, my_idx, out, a.nc, lane);
        }
        if (a.amax_out) {  // the whole warp is here
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            if (lane == 0 && mx > 0.f) atomicMax(a.amax_out, __float_as_uint(mx));
        }
        }
    }
}

template <int NCH, bool RES = false>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TC_THREADS, 1)
    k_m2l_tc_pair(const __grid_constant__ TcMaps maps, TcArgs a)
{
    extern __shared__ uint8_t smem_dyn[];
    __shared__ __align__(8) PairBars bars;
    __shared__ uint32_t tmem_sh;
    __shared__ int abort_sh;

    const int warp = threadIdx.x >> 5;
    const uint32_t rank = warp_uniform(cluster_rank());
    const uint32_t smem0 = warp_uniform((smem_u32(smem_dyn) + 1023u) & ~1023u);
    if (threadIdx.x == 0) {
        pair_bars_init(bars, a.stages);
        abort_sh = 0;
    }
    cluster_sync_all();  // the pair's barriers are initialised and both CTAs are running
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
    PairPipe pp;
    float *stage = reinterpret_cast<float *>(smem_dyn + (smem0 - smem_u32(smem_dyn)));
    pair_tile<NCH, RES>(maps, a, (int)(blockIdx.x >> 1), rank, smem0, stage, true, bars,
                   tmem, &abort_sh, pp, el);
    if (warp == 1 && el && rank == 0)
        mma_commit_pair(smem_u32(&bars.done));  // arrives in both CTAs once every MMA has completed

    // ---------------- teardown: every MMA done (bounded wait), pair barrier, collective TMEM release
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile int no_abort = 0;
        if (!mbar_wait_cluster(smem_u32(&bars.done), 0, &no_abort)) atomicOr(a.err, ERRF_TIMEOUT);
    }
    fence_before();
    __syncthreads();
    cluster_sync_all();
    fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    cluster_sync_all();
}

// ------------------------------------------------------------------ operand layout
// element of coefficient k of cell (or operator row) `cell` of `ncell` in one term of an operand array, chunks
// of kch coefficients outermost
__device__ __forceinline__ int64_t chunk_at(int64_t cell, int64_t ncell, int k, int kch)
{
    return ((int64_t)(k / kch) * ncell + cell) * kch + k % kch;
}

// ------------------------------------------------------------------ host helpers
PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    return fn;
}

int tile_dim(int np, int cap) { return np < cap ? np : cap; }

// Whether a plan's levels may run on CTA pairs.  When a wait runs out, the pair kernel does not wait for its partner's
// copies in flight, as the single-CTA kernel does for its own; with the default budget every copy has had two seconds
// to land by then, a shorter one keeps to single CTAs.
bool pairs_allowed(const Plan &P) { return P.tc_pair && P.wait_ns >= WAIT_LIMIT_NS; }

// stage ring of the split (pa, pb): as many stages as the shared-memory budget allows, 2..6
int tc_stages(int pa, int pb, int npad, int sw)
{
    const size_t stage = (size_t)pa * TC_ROWS * sw + (size_t)pb * npad * sw;
    size_t n = (TC_SMEM_BUDGET - 1024) / stage;
    if (n > (size_t)TC_MAX_STAGES) n = TC_MAX_STAGES;
    return n < 2 ? 2 : (int)n;
}

size_t tc_smem_bytes(int pa, int pb, int npad, int sw)
{
    // at least 120 KB so that a second CTA (and its 512 TMEM columns) never shares the SM
    size_t need = (size_t)tc_stages(pa, pb, npad, sw) * (pa * TC_ROWS * sw + pb * npad * sw) + 1024;
    return need < 120 * 1024 ? 120 * 1024 : need;
}

typedef void (*TcKernel)(TcMaps, TcArgs);  // single CTAs and CTA pairs alike

// CTA-pair kernel (fp16, 128-byte rows): stage = 2 A terms of 128 rows + 2 B terms of npad / 2 rows
int tc_pair_stages(int npad)
{
    const size_t stage = (size_t)2 * TC_ROWS * 128 + (size_t)2 * (npad / 2) * 128;
    size_t n = (TC_SMEM_BUDGET - 1024) / stage;
    if (n > (size_t)TC_MAX_STAGES) n = TC_MAX_STAGES;
    return n < 2 ? 2 : (int)n;
}

size_t tc_pair_smem_bytes(int npad)
{
    size_t need = (size_t)tc_pair_stages(npad) * ((size_t)2 * TC_ROWS * 128 + (size_t)2 * (npad / 2) * 128) + 1024;
    return need < 120 * 1024 ? 120 * 1024 : need;
}

// Offsets split over `groups` CTAs per tile, per_group offsets each.  With one CTA per SM a launch of
// tiles x g CTAs takes ceil(tiles g / sms) waves of ceil(n_off / g) offsets plus a fixed cost per CTA
// (pipeline fill and the exposed epilogue: about SPLIT_FIXED offsets' worth); g is the smallest that
// minimises that product.
constexpr int SPLIT_FIXED = 10;

void split_offsets(int n_off, int tiles, int max_groups, int sms, int &groups, int &per_group)
{
    long long best = -1;
    int g_best = 1;
    for (int g = 1; g <= max_groups && g <= n_off; ++g) {
        const int per = (n_off + g - 1) / g;
        const int used = (n_off + per - 1) / per;  // groups that actually hold offsets
        if (used != g) continue;
        const long long waves = ((long long)tiles * g + sms - 1) / sms;
        const long long cost = waves * (per + SPLIT_FIXED);
        if (best < 0 || cost < best) {
            best = cost;
            g_best = g;
        }
    }
    per_group = (n_off + g_best - 1) / g_best;
    groups = (n_off + per_group - 1) / per_group;
}

CUtensorMapSwizzle swizzle_of(int sw) { return sw == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B; }

// One map over `base`: rank-n extents, strides (bytes) of all but the innermost, box
fmm_status encode_map(PFN_cuTensorMapEncodeTiled_v12000 enc, CUtensorMap *map, CUtensorMapDataType dt, void *base,
                      int rank, const cuuint64_t *dims, const cuuint64_t *strides, const cuuint32_t *box, int sw)
{
    const cuuint32_t es[5] = {1, 1, 1, 1, 1};
    return enc(map, dt, (cuuint32_t)rank, base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(sw),
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
               ? FMM_OK
               : FMM_ERR_INTERNAL;
}

// The S, P and C maps (TcMaps) of a cell array [terms][kc chunks][d3][d2][d1][KCH], boxes b1 x b2 x b3 cells
fmm_status encode_planes(PFN_cuTensorMapEncodeTiled_v12000 enc, CUtensorMap *mS, CUtensorMap *mP, CUtensorMap *mC,
                         CUtensorMapDataType dt, void *base, int kc, int terms, int64_t d1, int64_t d2, int64_t d3,
                         int b1, int b2, int b3, int sw)
{
    const cuuint64_t row = (cuuint64_t)sw, k = (cuuint64_t)kchunk_of(sw), chunk = row * d1 * d2 * d3;
    const cuuint32_t box[5] = {(cuuint32_t)k, (cuuint32_t)b1, (cuuint32_t)b2, (cuuint32_t)b3, 2};
    const cuuint64_t dS[4] = {k, (cuuint64_t)d1, (cuuint64_t)d2, (cuuint64_t)(d3 * kc * terms)};
    const cuuint64_t dP[5] = {k, (cuuint64_t)d1, (cuuint64_t)d2, (cuuint64_t)(d3 * kc), (cuuint64_t)terms};
    const cuuint64_t dC[5] = {k, (cuuint64_t)d1, (cuuint64_t)d2, (cuuint64_t)d3, (cuuint64_t)(kc * terms)};
    const cuuint64_t sP[4] = {row, row * d1, row * d1 * d2, chunk * kc}, sC[4] = {row, row * d1, row * d1 * d2, chunk};
    fmm_status st = encode_map(enc, mS, dt, base, 4, dS, sP, box, sw);
    if (st == FMM_OK && mP) st = encode_map(enc, mP, dt, base, 5, dP, sP, box, sw);
    if (st == FMM_OK && mC) st = encode_map(enc, mC, dt, base, 5, dC, sC, box, sw);
    return st;
}

// The same of the operator tables [terms][kc chunks][slots][npad][KCH], boxes of n rows of one slot
fmm_status encode_operators(PFN_cuTensorMapEncodeTiled_v12000 enc, CUtensorMap *mS, CUtensorMap *mP, CUtensorMap *mC,
                            CUtensorMapDataType dt, void *base, int kc, int terms, int npad, int slots, int n, int sw)
{
    const cuuint64_t row = (cuuint64_t)sw, k = (cuuint64_t)kchunk_of(sw), slot = row * npad, chunk = slot * slots;
    const cuuint32_t box[4] = {(cuuint32_t)k, (cuuint32_t)n, 1, 2};
    const cuuint64_t dS[3] = {k, (cuuint64_t)npad, (cuuint64_t)slots * kc * terms};
    const cuuint64_t dP[4] = {k, (cuuint64_t)npad, (cuuint64_t)slots * kc, (cuuint64_t)terms};
    const cuuint64_t dC[4] = {k, (cuuint64_t)npad, (cuuint64_t)slots, (cuuint64_t)(kc * terms)};
    const cuuint64_t sP[3] = {row, slot, chunk * kc}, sC[3] = {row, slot, chunk};
    fmm_status st = encode_map(enc, mS, dt, base, 3, dS, sP, box, sw);
    if (st == FMM_OK && mP) st = encode_map(enc, mP, dt, base, 4, dP, sP, box, sw);
    if (st == FMM_OK && mC) st = encode_map(enc, mC, dt, base, 4, dC, sC, box, sw);
    return st;
}

}  // namespace

}  // namespace fmm
