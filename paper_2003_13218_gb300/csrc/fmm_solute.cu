// fmm_solute.cu -- the solute-only far-field pass of the reduced scheme for the
// solute-solvent energy (Eq. FMMcalc): Phi_u^FF at every charge, from the
// solute charges alone.
//
// With a handful of solute charges only the leaves holding them and their
// ancestors carry solute moments.  The pass therefore
//  * builds the list of active cells per level (at most NU_MAX per level) and
//    their solute moments, each straight from the charges (Eq. P2M about that
//    cell's centre, which is what M2M would carry up, up to rounding);
//  * on the coarse levels 1..ld, ld = min(3, depth), computes the local
//    expansion of every cell in the pass's own arrays: level 1 by the top
//    operator, then per level the M2L terms of the active cells (one block per
//    active cell and offset, every periodic image counted) summed per target
//    with the L2L of its parent, giving the full local expansion at level ld;
//  * on the finer levels evaluates M2L only onto the targets whose interaction
//    list contains an active source (at most n_il(ws) per source);
//  * evaluates Phi_u at every charge as the level-ld expansion plus the sparse
//    contributions found at its finer ancestors.  A local expansion is a
//    polynomial of degree p, so evaluating it at a charge directly equals
//    shifting it to the leaf with L2L first (Appendix B) up to rounding.
// The work of all levels that does not depend on another level shares one
// launch (grids of blocks that take work items in turn, since the host does not
// know the number of active cells): the pass is a chain of small kernels, and
// as ~60 of them, level by level, it took 0.57 ms of a call on 100,000 charges.
// None of it needs more than the sort, so it starts beside the upward pass.  At
// depth 3 and less, where the dense pass used to run, it saves a second far-field
// pass.  Calls with E_uv: 100,000 charges from host arrays 1.87 -> 1.18 ms, 16
// coupling windows 6.96 -> 5.48 ms, 2,998 charges in FP64 1.36 -> 1.02 ms.
// When more than NU_MAX charges are solute the caller runs the dense pass instead.
#include <math.h>

#include <new>
#include <type_traits>

#include "fmm_internal.cuh"

namespace fmm {

namespace {

constexpr int NU_MAX = 64;      // solute charges handled by the sparse pass
constexpr int LD_MAX = 3;       // levels 1..min(3, depth) treated densely
constexpr int ACT_OFFS = 3;     // interaction-list offsets per block of the solvent field (n_il is a multiple of it
                                // or the last block takes fewer)
constexpr int ITEM_BLOCKS = 912;  // 6 x 152 SMs: blocks of the launches that loop over work items
// targets per fine level: at most NU_MAX * n_il(ws) (mt below)
__host__ __device__ inline int max_tgt(int ws) { return NU_MAX * n_il(ws); }
__host__ __device__ inline int act_groups(int ws) { return (n_il(ws) + ACT_OFFS - 1) / ACT_OFFS; }

struct SoluteScratch {
    int *list = nullptr;     // [NU_MAX] sorted slots of solute charges as found; the count is P.d_err[1]
    int *slots = nullptr;    // [NU_MAX] the same in slot order
    int *cells = nullptr;    // [9][NU_MAX] active cell (linear index) per level
    int *ncells = nullptr;   // [9] active cells, [16 + l] targets of fine level l
    void *MU = nullptr;      // [9][NU_MAX][nc] solute moments of the active cells
    int *map = nullptr;      // per fine level [8^l]: 1 + index of a target cell in tlist, 0: no target
    size_t map_bytes = 0;
    int *tlist = nullptr;    // [9][mt] targets per fine level, in no particular order
    void *contrib = nullptr; // [9][mt][nc] M2L sums at those targets; rows of levels 0..ld: M2L terms of the dense levels
    int *h_count = nullptr;  // pinned
    cudaStream_t side = nullptr;       // high-priority stream of the pass (overlaps the full pass)
    cudaEvent_t ev_count = nullptr;    // count copied to h_count
    cudaEvent_t ev_sort = nullptr;     // sort done (fork)
    cudaEvent_t ev_up = nullptr;       // full upward pass done
    cudaEvent_t ev_ready = nullptr;    // expansions ready (Phi_u on the near stream waits)
    cudaEvent_t ev_done = nullptr;     // everything on the side stream done (join)
    bool forked = false, act_done = false;
    double *Lt = nullptr;    // [9][NU_MAX][nc] the solvent's M2L sums at the active cells (FP64)
    void *Lu = nullptr;      // solute-only local expansions of every cell of levels 1..ld (class layout), T
    double *part = nullptr;  // [level][NU_MAX][act_groups][nc] partial sums of Lt
};

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

__device__ inline void cell_xyz(int64_t lin, int n, int &x, int &y, int &z)
{
    x = (int)(lin % n);
    y = (int)((lin / n) % n);
    z = (int)(lin / ((int64_t)n * n));
}

// One block of 64 threads: the solute slots in order, then per level the active cells -- the leaves of the solute
// charges and their ancestors, each list sorted by linear index and without repeats.  Every thread ranks its own
// key among the at most 64 (a serial sort by one thread took 7 us with one charge and far more with 64).
__global__ void __launch_bounds__(NU_MAX) k_sol_cells(int d, const int *__restrict__ count, const int *__restrict__ list,
                                                      const int *__restrict__ sleaf, int *__restrict__ slots,
                                                      int *__restrict__ cells, int *__restrict__ ncells)
{
    __shared__ int key[NU_MAX], first[NU_MAX];
    const int i = threadIdx.x;
    int n = *count;
    if (n > NU_MAX) n = 0;  // the dense pass runs instead: no active cells
    key[i] = i < n ? list[i] : 0;
    __syncthreads();
    int x = 0, y = 0, z = 0;
    if (i < n) {
        int r = 0;
        for (int j = 0; j < n; ++j) r += key[j] < key[i];
        slots[r] = key[i];
        cell_xyz(sleaf[key[i]], 1 << d, x, y, z);
    }
    for (int l = d; l >= 1; --l) {
        const int nl = 1 << l;
        __syncthreads();
        const int k = x + nl * (y + nl * z);
        key[i] = k;
        __syncthreads();
        int f = i < n;
        for (int j = 0; j < i && f; ++j) f = key[j] != k;
        first[i] = f;
        const int cnt = __syncthreads_count(f);
        if (f) {
            int r = 0;
            for (int j = 0; j < n; ++j) r += first[j] && key[j] < k;
            cells[l * NU_MAX + r] = k;
        }
        if (i == 0) {
            ncells[l] = cnt;
            ncells[16 + l] = 0;
        }
        x >>= 1;
        y >>= 1;
        z >>= 1;
    }
}

// reciprocals of the harmonics' recurrences, once per block: -1/(2m) and 1/((n+m)(n-m))
template <typename T>
__device__ __forceinline__ void recurrence_tables(int p, T *s_half, T *s_inv)
{
    for (int e = threadIdx.x; e < (p + 1) * (p + 1); e += blockDim.x) {
        const int n = e / (p + 1), mm = e % (p + 1);
        s_inv[e] = n > mm ? T(1) / T((n + mm) * (n - mm)) : T(0);
        if (e <= p) s_half[e] = e > 0 ? T(-0.5) / T(e) : T(0);
    }
}

// Solute moments of active cell blockIdx.x of level blockIdx.y + 1 about the cell's centre; thread m = column m
template <typename T>
__global__ void k_sol_p2m(int p, int d, T h, const int *__restrict__ count, const int *__restrict__ slots,
                          const int *__restrict__ sleaf, const int *__restrict__ cells, const int *__restrict__ ncells,
                          const Particle<T> *__restrict__ sp, T *__restrict__ MU)
{
    __shared__ T s_half[P_MAX + 1], s_inv[(P_MAX + 1) * (P_MAX + 1)];
    const int i = blockIdx.x, l = blockIdx.y + 1;
    if (i >= ncells[l]) return;
    recurrence_tables<T>(p, s_half, s_inv);
    __syncthreads();
    const int m = threadIdx.x;
    if (m > p) return;
    const int nc = ncoef(p), nu = *count, sh = d - l;
    int cx, cy, cz;
    cell_xyz(cells[l * NU_MAX + i], 1 << l, cx, cy, cz);
    const T inv_h = T(1) / (h * T(1 << sh));
    T accr[P_MAX + 1], acci[P_MAX + 1];
    for (int n = 0; n <= p; ++n) accr[n] = acci[n] = 0;
    for (int u = 0; u < nu; ++u) {
        const int s = slots[u];
        int x, y, z;
        cell_xyz(sleaf[s], 1 << d, x, y, z);
        if ((x >> sh) != cx || (y >> sh) != cy || (z >> sh) != cz) continue;
        const Particle<T> pt = sp[s];
        // the leaf's centre relative to the cell's, in leaf units
        const T ox = T((x - (cx << sh)) + 0.5) - T(0.5) * T(1 << sh), oy = T((y - (cy << sh)) + 0.5) - T(0.5) * T(1 << sh),
                oz = T((z - (cz << sh)) + 0.5) - T(0.5) * T(1 << sh);
        const T vx = -(pt.x + ox * h) * inv_h, vy = -(pt.y + oy * h) * inv_h, vz = -(pt.z + oz * h) * inv_h;
        const T r2 = vx * vx + vy * vy + vz * vz;
        T dre = pt.q, dim = 0;
        for (int k = 1; k <= m; ++k) {
            const T nre = s_half[k] * (vx * dre - vy * dim), nim = s_half[k] * (vx * dim + vy * dre);
            dre = nre;
            dim = nim;
        }
        T p2re = 0, p2im = 0, p1re = dre, p1im = dim;
        accr[m] += dre;
        acci[m] += dim;
        for (int n = m + 1; n <= p; ++n) {
            const T a = T(2 * n - 1) * vz, inv = s_inv[n * (p + 1) + m];
            const T cr = (a * p1re - r2 * p2re) * inv, ci = (a * p1im - r2 * p2im) * inv;
            accr[n] += cr;
            acci[n] += ci;
            p2re = p1re;
            p2im = p1im;
            p1re = cr;
            p1im = ci;
        }
    }
    T *out = MU + ((size_t)l * NU_MAX + i) * nc;
    for (int n = m; n <= p; ++n) {
        out[cre(n, m)] = accr[n];
        if (m > 0) out[cim(n, m)] = acci[n];
    }
}

// interaction-list test: is s = t + delta in IL(t)?  (per axis delta in
// [-2 ws - c, 2 ws + 1 - c] for target parity c, and not all |delta| <= ws)
__device__ inline bool in_il(int dx, int dy, int dz, int tx, int ty, int tz, int ws)
{
    if (dx >= -ws && dx <= ws && dy >= -ws && dy <= ws && dz >= -ws && dz <= ws) return false;
    int cx = tx & 1, cy = ty & 1, cz = tz & 1;
    return dx >= -2 * ws - cx && dx <= 2 * ws + 1 - cx && dy >= -2 * ws - cy && dy <= 2 * ws + 1 - cy &&
           dz >= -2 * ws - cz && dz <= 2 * ws + 1 - cz;
}

__device__ inline int wrap_delta(int d, int n)  // representative of d mod n in [-n/2, n/2)
{
    d %= n;
    if (d < -n / 2) d += n;
    if (d >= n / 2) d -= n;
    return d;
}

// offset of level l >= 1 in the dense arrays of levels 1..ld (8^1 + ... + 8^(l-1) cells before it)
__host__ __device__ inline int64_t dense_off(int l, int nc) { return ((((int64_t)1 << (3 * l)) - 1) / 7 - 1) * nc; }

// offset of fine level l in the target map (levels l0 + 1 .. l - 1 before it)
__host__ __device__ inline int64_t map_off(int l, int l0)
{
    return ((((int64_t)1 << (3 * l)) - 1) / 7) - ((((int64_t)1 << (3 * (l0 + 1))) - 1) / 7);
}

// sum_k a[k stride] b[k], k < n, in 4 partial sums with 8 loads in flight (a column of an operator against a row of
// coefficients: the loads' latency is what these small kernels wait for)
template <typename T>
__device__ __forceinline__ T dot8(const T *__restrict__ a, size_t stride, const T *b, int n)
{
    T s0 = 0, s1 = 0, s2 = 0, s3 = 0;
    int k = 0;
    for (; k + 8 <= n; k += 8) {
        T v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = a[(size_t)(k + u) * stride];
        s0 += v[0] * b[k];
        s1 += v[1] * b[k + 1];
        s2 += v[2] * b[k + 2];
        s3 += v[3] * b[k + 3];
        s0 += v[4] * b[k + 4];
        s1 += v[5] * b[k + 5];
        s2 += v[6] * b[k + 6];
        s3 += v[7] * b[k + 7];
    }
    for (; k < n; ++k) s0 += a[(size_t)k * stride] * b[k];
    return (s0 + s1) + (s2 + s3);
}

// M2L terms of the dense levels 2..ld, one work item per (level, active source a, offset d of the window
// [-2ws-1, 2ws+1]^3): part[l - 2][a][d] = T(d) . MU_a (Eq. Lcoeffdef) when the source lies in the interaction
// list of the target t = s_a - d (wrapped).  At coarse levels several offsets reach the same target (its
// periodic images): each has its own term.
template <typename T>
__global__ void k_sol_dense_m2l(int p, int ld, int ws, const int *__restrict__ cells, const int *__restrict__ ncells,
                                const T *__restrict__ Top, const T *__restrict__ MU, T *__restrict__ part)
{
    const int nc = ncoef(p), h = 2 * ws + 1, side = 2 * h + 1, W = side * side * side;
    int total = 0;
    for (int l = 2; l <= ld; ++l) total += ncells[l] * W;
    for (int it = blockIdx.x; it < total; it += gridDim.x) {
        int l = 2, r = it;
        while (r >= ncells[l] * W) r -= ncells[l++] * W;
        const int a = r / W, b = r - a * W, n = 1 << l;
        const int dx = b % side - h, dy = (b / side) % side - h, dz = b / (side * side) - h;
        int sx, sy, sz;
        cell_xyz(cells[l * NU_MAX + a], n, sx, sy, sz);
        const int tx = (sx - dx + 4 * n) & (n - 1), ty = (sy - dy + 4 * n) & (n - 1), tz = (sz - dz + 4 * n) & (n - 1);
        if (!in_il(dx, dy, dz, tx, ty, tz, ws)) continue;
        const T *Tp = Top + (size_t)off_slot(dx, dy, dz, ws) * nc * nc;
        const T *Ms = MU + ((size_t)l * NU_MAX + a) * nc;
        T *out = part + (((size_t)(l - 2) * NU_MAX + a) * W + b) * nc;
        for (int j = threadIdx.x; j < nc; j += blockDim.x) {
            out[j] = dot8<T>(Tp + j, nc, Ms, nc);
        }
    }
}

// dense level 2 <= l <= ld of the solute-only pass, every target cell (one block each, thread j =
// coefficient j): the L2L of the parent's expansion (the octant's operator, transposed [nc][8 nc]) plus the M2L
// terms of k_sol_dense_m2l whose target this is, summed in the window's offset order (the sums do not depend on
// the schedule)
template <typename T>
__global__ void k_sol_dense(int p, int l, int ws, const int *__restrict__ cells, const int *__restrict__ ncells,
                            const T *__restrict__ part, const T *__restrict__ l2lT, const T *__restrict__ Lpar,
                            T *__restrict__ Lout)
{
    constexpr int W_MAX = (4 * WS_MAX + 3) * (4 * WS_MAX + 3) * (4 * WS_MAX + 3);
    __shared__ int hit[W_MAX];  // part rows of this target, in offset order
    __shared__ int nhit;
    __shared__ T sL[NC_MAX];
    const int nc = ncoef(p), n = 1 << l, h = 2 * ws + 1, side = 2 * h + 1, W = side * side * side;
    int tx, ty, tz;
    cell_xyz(blockIdx.x, n, tx, ty, tz);
    const int na = ncells[l];
    const int *act = cells + l * NU_MAX;
    const int oct = (tx & 1) | ((ty & 1) << 1) | ((tz & 1) << 2);
    const T *Lp = Lpar + cell_index(l - 1, tx >> 1, ty >> 1, tz >> 1) * nc;
    for (int j = threadIdx.x; j < nc; j += blockDim.x) sL[j] = Lp[j];
    if (threadIdx.x < 32) {  // the first warp collects the hits in order
        int cnt = 0;
        for (int b0 = 0; b0 < W; b0 += 32) {
            const int b = b0 + threadIdx.x;
            const int dx = b % side - h, dy = (b / side) % side - h, dz = b / (side * side) - h;
            int a = -1;
            if (b < W && in_il(dx, dy, dz, tx, ty, tz, ws)) {
                const int key = ((tx + dx + 4 * n) & (n - 1)) + n * (((ty + dy + 4 * n) & (n - 1)) +
                                                                     n * ((tz + dz + 4 * n) & (n - 1)));
                int lo = 0, hi = na;  // active cells are sorted and unique
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (act[mid] < key) lo = mid + 1;
                    else hi = mid;
                }
                if (lo < na && act[lo] == key) a = lo;
            }
            const unsigned m = __ballot_sync(0xffffffffu, a >= 0);
            if (a >= 0) hit[cnt + __popc(m & ((1u << threadIdx.x) - 1u))] = a * W + b;
            cnt += __popc(m);
        }
        if (threadIdx.x == 0) nhit = cnt;
    }
    __syncthreads();
    const T *pl = part + (size_t)(l - 2) * NU_MAX * W * nc;
    for (int j = threadIdx.x; j < nc; j += blockDim.x) {
        T acc = dot8<T>(l2lT + oct * nc + j, 8 * nc, sL, nc);
        const int nh = nhit;
        T a0 = 0, a1 = 0;
        int b = 0;
#pragma unroll 4
        for (; b + 1 < nh; b += 2) {
            a0 += pl[(size_t)hit[b] * nc + j];
            a1 += pl[(size_t)hit[b + 1] * nc + j];
        }
        if (b < nh) a0 += pl[(size_t)hit[b] * nc + j];
        acc += a0 + a1;
        Lout[cell_index(l, tx, ty, tz) * nc + j] = acc;
    }
}

// the targets of active source blockIdx.x at fine level ld + 1 + blockIdx.y (threads over the candidate offsets):
// the first source to reach a cell gives it a place in the level's target list
__global__ void k_sol_mark(int ld, int ws, int mt, const int *__restrict__ cells, int *__restrict__ ncells,
                           int *__restrict__ map, int *__restrict__ tlist)
{
    const int i = blockIdx.x, l = ld + 1 + blockIdx.y;
    if (i >= ncells[l]) return;
    const int side = off_side(ws), h = 2 * ws + 1;
    const int n = 1 << l;
    int *mp = map + map_off(l, ld);
    int sx, sy, sz;
    cell_xyz(cells[l * NU_MAX + i], n, sx, sy, sz);
    for (int o = threadIdx.x; o < side * side * side; o += blockDim.x) {
        const int dx = o % side - h, dy = (o / side) % side - h, dz = o / (side * side) - h;
        const int tx = (sx - dx + 2 * n) & (n - 1), ty = (sy - dy + 2 * n) & (n - 1), tz = (sz - dz + 2 * n) & (n - 1);
        if (!in_il(dx, dy, dz, tx, ty, tz, ws)) continue;
        const int t = tx + n * (ty + n * tz);
        if (atomicCAS(mp + t, 0, -1) != 0) continue;
        const int k = atomicAdd(ncells + 16 + l, 1);  // below mt: n_il targets per source
        tlist[(size_t)l * mt + k] = t;
        mp[t] = k + 1;
    }
}

// contribution of every active source to the targets of the fine levels (Eq. Lcoeffdef), one target per work item,
// the sources in the order of their list
template <typename T>
__global__ void k_sol_m2l(int p, int d, int ld, int ws, const int *__restrict__ cells, const int *__restrict__ ncells,
                          const int *__restrict__ tlist, const T *__restrict__ Top, const T *__restrict__ MU,
                          T *__restrict__ contrib)
{
    const int nc = ncoef(p), mt = max_tgt(ws);
    int total = 0;
    for (int l = ld + 1; l <= d; ++l) total += ncells[16 + l];
    for (int it = blockIdx.x; it < total; it += gridDim.x) {
        int l = ld + 1, b = it;
        while (b >= ncells[16 + l]) b -= ncells[16 + l++];
        const int n = 1 << l;
        int tx, ty, tz;
        cell_xyz(tlist[(size_t)l * mt + b], n, tx, ty, tz);
        for (int j = threadIdx.x; j < nc; j += blockDim.x) {
            T acc = 0;
            for (int s = 0; s < ncells[l]; ++s) {
                int sx, sy, sz;
                cell_xyz(cells[l * NU_MAX + s], n, sx, sy, sz);
                const int dx = wrap_delta(sx - tx, n), dy = wrap_delta(sy - ty, n), dz = wrap_delta(sz - tz, n);
                if (!in_il(dx, dy, dz, tx, ty, tz, ws)) continue;
                const T *Tp = Top + (size_t)off_slot(dx, dy, dz, ws) * nc * nc + j;
                const T *Ms = MU + ((size_t)l * NU_MAX + s) * nc;
                acc += dot8<T>(Tp, nc, Ms, nc);
            }
            contrib[((size_t)l * mt + b) * nc + j] = acc;
        }
    }
}

// ---- full-field potential at the solute charges (the A of Eq. FMMcalc): M2L over the interaction list of
// each active cell from the full pass's moments in FP64 (CUDA cores, no operand splitting; level 1 and above by
// the FP64 top operator), on the solvent moments M - M_u, and each level's sum evaluated at the charge itself.
// The few solute charges cannot average out the split-operand rounding of the tensor-core M2L, so A is taken
// from here.

// part[l][i][g] = the M2L terms of ACT_OFFS offsets of active cell i at level l >= 2, one work item each.  Bound by
// the FP64 pipe (2 operations per SM and clock): the moments are converted once per block, not per thread.
template <typename T>
__global__ void k_act_m2l(int p, int d, int ws, const int *__restrict__ il, const int *__restrict__ cells,
                          const int *__restrict__ ncells, const double *__restrict__ Top, const T *const *__restrict__ Mlev,
                          const T *__restrict__ MU, double *__restrict__ part)
{
    __shared__ double sM[NC_MAX];
    const int nc = ncoef(p), nil = n_il(ws), ng = act_groups(ws);
    int total = 0;
    for (int l = 2; l <= d; ++l) total += ncells[l] * ng;
    for (int it = blockIdx.x; it < total; it += gridDim.x) {
        int l = 2, r = it;
        while (r >= ncells[l] * ng) r -= ncells[l++] * ng;
        const int i = r / ng, g = r - i * ng, n = 1 << l;
        const T *M = Mlev[l];
        int tx, ty, tz;
        cell_xyz(cells[l * NU_MAX + i], n, tx, ty, tz);
        const int cls = (tx & 1) | ((ty & 1) << 1) | ((tz & 1) << 2);
        double acc[(NC_MAX + 191) / 192] = {};  // coefficients threadIdx.x, + blockDim.x, ...
        for (int o = g * ACT_OFFS; o < nil && o < (g + 1) * ACT_OFFS; ++o) {
            int dx, dy, dz;
            il_unpack(il[cls * nil + o], dx, dy, dz);
            const int sx = (tx + dx + 4 * n) & (n - 1), sy = (ty + dy + 4 * n) & (n - 1), sz = (tz + dz + 4 * n) & (n - 1);
            const T *Ms = M + cell_index(l, sx, sy, sz) * nc;
            const T *Mu = nullptr;  // the solute part of this source, if it is an active cell
            const int slin = sx + n * (sy + n * sz);
            for (int k = 0; k < ncells[l]; ++k)
                if (cells[l * NU_MAX + k] == slin) Mu = MU + ((size_t)l * NU_MAX + k) * nc;
            __syncthreads();
            for (int k = threadIdx.x; k < nc; k += blockDim.x) sM[k] = Mu ? (double)Ms[k] - (double)Mu[k] : (double)Ms[k];
            __syncthreads();
            const double *Tp = Top + (size_t)off_slot(dx, dy, dz, ws) * nc * nc;
#pragma unroll
            for (int q = 0; q < (NC_MAX + 191) / 192; ++q) {
                const int j = threadIdx.x + q * blockDim.x;
                if (j >= nc) break;
                acc[q] += dot8<double>(Tp + j, nc, sM, nc);
            }
        }
        double *out = part + ((size_t)((l - 2) * NU_MAX + i) * ng + g) * nc;
#pragma unroll
        for (int q = 0; q < (NC_MAX + 191) / 192; ++q) {
            const int j = threadIdx.x + q * blockDim.x;
            if (j < nc) out[j] = acc[q];
        }
    }
}

// Lt[l][i] = sum of the groups' terms, level 2 + blockIdx.z: one warp per (active cell, coefficient j), lanes take
// every 32nd group, then a fixed shuffle tree (deterministic)
__global__ void k_act_sum(int p, int ng, const int *__restrict__ ncells, const double *__restrict__ part,
                          double *__restrict__ Lt)
{
    const int nc = ncoef(p), l = 2 + blockIdx.z;
    const int j = blockIdx.y * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (j >= nc) return;
    for (int i = blockIdx.x; i < ncells[l]; i += gridDim.x) {
        double s = 0;
        for (int o = lane; o < ng; o += 32) s += part[((size_t)((l - 2) * NU_MAX + i) * ng + o) * nc + j];
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (lane == 0) Lt[((size_t)l * NU_MAX + i) * nc + j] = s;
    }
}

// at solute charge blockIdx.x: phi_ff = (solvent field: every level's Lt at the charge) + phi_u (solute field of
// the solute-only pass), so that A - B = sum_u q Phi_v holds term by term.  Warp w takes levels w + 1, w + 9, ...,
// lane m the column m of the harmonics (one thread doing all of it, a division per term, took 66 us); the levels
// are added in order.
template <typename T>
__global__ void __launch_bounds__(256) k_act_l2p(int p, int d, double h, const int *__restrict__ count,
                                                 const int *__restrict__ slots, const int *__restrict__ cells,
                                                 const int *__restrict__ ncells, const int *__restrict__ sleaf,
                                                 const Particle<T> *__restrict__ sp, const double *__restrict__ Lt,
                                                 const T *__restrict__ phi_u, T *__restrict__ phi)
{
    __shared__ double s_half[P_MAX + 1], s_inv[(P_MAX + 1) * (P_MAX + 1)], s_lev[9];
    const int n = *count;
    if (n > NU_MAX || (int)blockIdx.x >= n) return;
    recurrence_tables<double>(p, s_half, s_inv);
    __syncthreads();
    const int s = slots[blockIdx.x], nc = ncoef(p);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int x, y, z;
    cell_xyz(sleaf[s], 1 << d, x, y, z);
    const Particle<T> pt = sp[s];
    for (int l = w + 1; l <= d; l += 8) {
        const int sh = d - l, nl = 1 << l;
        const int ax = x >> sh, ay = y >> sh, az = z >> sh, key = ax + nl * (ay + nl * az);
        int i = 0;
        while (i < ncells[l] - 1 && cells[l * NU_MAX + i] != key) ++i;
        const double inv = 1.0 / (h * (double)(1 << sh));
        const double vx = ((double)pt.x + ((x - (ax << sh)) + 0.5 - 0.5 * (1 << sh)) * h) * inv,
                     vy = ((double)pt.y + ((y - (ay << sh)) + 0.5 - 0.5 * (1 << sh)) * h) * inv,
                     vz = ((double)pt.z + ((z - (az << sh)) + 0.5 - 0.5 * (1 << sh)) * h) * inv;
        const double r2 = vx * vx + vy * vy + vz * vz;
        const double *Lc = Lt + ((size_t)l * NU_MAX + i) * nc;
        double pot = 0;
        if (lane <= p) {
            const int m = lane;
            double dre = 1, dim = 0;
            for (int k = 1; k <= m; ++k) {
                const double nre = s_half[k] * (vx * dre - vy * dim), nim = s_half[k] * (vx * dim + vy * dre);
                dre = nre;
                dim = nim;
            }
            double p2re = 0, p2im = 0, rre = dre, rim = dim;
            for (int k = m; k <= p; ++k) {
                if (k > m) {
                    const double a = (2 * k - 1) * vz, iv = s_inv[k * (p + 1) + m];
                    const double cr = (a * rre - r2 * p2re) * iv, ci = (a * rim - r2 * p2im) * iv;
                    p2re = rre;
                    p2im = rim;
                    rre = cr;
                    rim = ci;
                }
                const Cx<double> L = coef(Lc, k, m);
                pot += L.re * rre - L.im * rim;
            }
            if (m > 0) pot *= 2.0;
        }
        for (int o = 16; o > 0; o >>= 1) pot += __shfl_xor_sync(0xffffffffu, pot, o);
        if (lane == 0) s_lev[l] = pot * inv;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0;
        for (int l = 1; l <= d; ++l) v += s_lev[l];
        phi[s] = (T)(v + (double)phi_u[s]);
    }
}

// Phi at (v) from the real-layout local coefficients Lc (scaled), v in cell units;
// s_half[m] = -1/(2m) and s_inv[n (p+1) + m] = 1/((n+m)(n-m))
template <typename T>
__device__ T l2p_value(int p, const T *__restrict__ Lc, T vx, T vy, T vz, const T *s_half, const T *s_inv)
{
    T r2 = vx * vx + vy * vy + vz * vz;
    T pot = 0, dre = 1, dim = 0;
    for (int m = 0; m <= p; ++m) {
        if (m > 0) {
            T sc = s_half[m];
            T nre = sc * (vx * dre - vy * dim), nim = sc * (vx * dim + vy * dre);
            dre = nre;
            dim = nim;
        }
        T w = m == 0 ? T(1) : T(2);
        T p2re = 0, p2im = 0, rre = dre, rim = dim;
        for (int n = m; n <= p; ++n) {
            if (n > m) {
                T a = T(2 * n - 1) * vz, inv = s_inv[n * (p + 1) + m];
                T cr = (a * rre - r2 * p2re) * inv, ci = (a * rim - r2 * p2im) * inv;
                p2re = rre;
                p2im = rim;
                rre = cr;
                rim = ci;
            }
            Cx<T> L = coef(Lc, n, m);
            pot += w * (L.re * rre - L.im * rim);
        }
    }
    return pot;
}

// Phi_u at every charge: level-ld expansion plus the sparse finer-level sums
template <typename T>
__global__ void k_sol_eval(int p, int d, int ld, int mt, int64_t N, T h_leaf, const int *__restrict__ sleaf,
                           const Particle<T> *__restrict__ sp, const T *__restrict__ Lld, const int *__restrict__ map,
                           const T *__restrict__ contrib, T *__restrict__ phi)
{
    __shared__ T s_half[P_MAX + 1];
    __shared__ T s_inv[(P_MAX + 1) * (P_MAX + 1)];
    recurrence_tables<T>(p, s_half, s_inv);
    __syncthreads();
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= N) return;
    int nc = ncoef(p);
    int nside = 1 << d;
    int leaf = sleaf[s];
    int x, y, z;
    cell_xyz(leaf, nside, x, y, z);
    Particle<T> pt = sp[s];
    T total = 0;
    for (int l = ld; l <= d; ++l) {
        int sh = d - l;
        int ax = x >> sh, ay = y >> sh, az = z >> sh;
        const T *Lc;
        if (l == ld) Lc = Lld + cell_index(l, ax, ay, az) * nc;
        else {
            const int k = map[map_off(l, ld) + ax + (1 << l) * (ay + ((int64_t)az << l))];
            if (k <= 0) continue;
            Lc = contrib + ((size_t)l * mt + k - 1) * nc;
        }
        // centre of the leaf relative to the centre of its level-l ancestor, in leaf units
        T ox = T((x - (ax << sh)) + 0.5) - T(0.5) * T(1 << sh);
        T oy = T((y - (ay << sh)) + 0.5) - T(0.5) * T(1 << sh);
        T oz = T((z - (az << sh)) + 0.5) - T(0.5) * T(1 << sh);
        T inv = T(1) / (h_leaf * T(1 << sh));
        T vx = (pt.x + ox * h_leaf) * inv, vy = (pt.y + oy * h_leaf) * inv, vz = (pt.z + oz * h_leaf) * inv;
        total += l2p_value<T>(p, Lc, vx, vy, vz, s_half, s_inv) * inv;
    }
    phi[s] = total;
}

// the solute-only expansions, on stream `st` (needs the sort only); the device count decides how many cells are
// active (none when the sparse pass does not apply)
template <typename T>
fmm_status solute_expand_t(Plan &P, SoluteScratch &S, cudaStream_t st)
{
    const int p = P.p, d = P.d, nc = P.nc, ld = d < LD_MAX ? d : LD_MAX, mt = max_tgt(P.ws);
    const bool f64 = std::is_same<T, double>::value;
    const T h = (T)(P.box / (1 << d));
    const T *Top = f64 ? (const T *)P.tab.Top64 : (const T *)P.tab.Top32;
    const T *l2lT = (f64 ? (const T *)P.tab.l2l64 : (const T *)P.tab.l2l32) + (size_t)8 * nc * nc;
    const int *count = P.d_err + 1;
    T *MU = (T *)S.MU, *Lu = (T *)S.Lu, *part = (T *)S.contrib;
    const int nth = ((nc + 31) / 32) * 32;
    k_sol_cells<<<1, NU_MAX, 0, st>>>(d, count, S.list, P.sleaf, S.slots, S.cells, S.ncells);
    FMM_LAUNCH_CHECK(P);
    k_sol_p2m<T><<<dim3(NU_MAX, d), 32, 0, st>>>(p, d, h, count, S.slots, P.sleaf, S.cells, S.ncells,
                                                 (const Particle<T> *)P.sorted, MU);
    FMM_LAUNCH_CHECK(P);
    fmm_status s = launch_top_solute(P, st, MU + (size_t)NU_MAX * nc, S.cells + NU_MAX, S.ncells + 1, Lu + dense_off(1, nc));
    if (s != FMM_OK) return s;
    k_sol_dense_m2l<T><<<ITEM_BLOCKS, nth, 0, st>>>(p, ld, P.ws, S.cells, S.ncells, Top, MU, part);
    FMM_LAUNCH_CHECK(P);
    for (int l = 2; l <= ld; ++l) {
        k_sol_dense<T><<<1u << (3 * l), nth, 0, st>>>(p, l, P.ws, S.cells, S.ncells, part, l2lT, Lu + dense_off(l - 1, nc),
                                                      Lu + dense_off(l, nc));
        FMM_LAUNCH_CHECK(P);
    }
    if (d > ld) {
        FMM_CUDA_TRY(cudaMemsetAsync(S.map, 0, S.map_bytes, st));
        k_sol_mark<<<dim3(NU_MAX, d - ld), 256, 0, st>>>(ld, P.ws, mt, S.cells, S.ncells, S.map, S.tlist);
        FMM_LAUNCH_CHECK(P);
        k_sol_m2l<T><<<ITEM_BLOCKS, nth, 0, st>>>(p, d, ld, P.ws, S.cells, S.ncells, S.tlist, Top, MU, (T *)S.contrib);
        FMM_LAUNCH_CHECK(P);
    }
    return FMM_OK;
}

// the solvent's FP64 field at the active cells, on stream `st` (needs the full pass's moments of all levels)
template <typename T>
fmm_status solute_act_t(Plan &P, SoluteScratch &S, cudaStream_t st)
{
    const int p = P.p, d = P.d, nc = P.nc, ng = act_groups(P.ws);
    const T *MU = (const T *)S.MU;
    const int nth = nc < 192 ? ((nc + 31) / 32) * 32 : 192;
    k_act_m2l<T><<<ITEM_BLOCKS, nth, 0, st>>>(p, d, P.ws, P.tab.il, S.cells, S.ncells, P.tab.Top64,
                                              (const T *const *)P.d_M, MU, S.part);
    FMM_LAUNCH_CHECK(P);
    fmm_status s = launch_top_active(P, st, MU + (size_t)NU_MAX * nc, S.cells + NU_MAX, S.ncells + 1,
                                     S.Lt + (size_t)NU_MAX * nc);
    if (s != FMM_OK) return s;
    k_act_sum<<<dim3(8, (nc + 7) / 8, d - 1), 256, 0, st>>>(p, ng, S.ncells, S.part, S.Lt);
    FMM_LAUNCH_CHECK(P);
    return FMM_OK;
}

// Phi_u at every charge: the level-ld expansion plus the sparse finer-level sums
template <typename T>
fmm_status solute_eval_t(Plan &P, SoluteScratch &S, cudaStream_t st)
{
    const double h = P.box / (1 << P.d);
    const int ld = P.d < LD_MAX ? P.d : LD_MAX;
    k_sol_eval<T><<<blocks_for(P.N, 128), 128, 0, st>>>(P.p, P.d, ld, max_tgt(P.ws), P.N, (T)h, P.sleaf,
                                                        (const Particle<T> *)P.sorted,
                                                        (const T *)S.Lu + dense_off(ld, P.nc), S.map,
                                                        (const T *)S.contrib, (T *)P.phi_u);
    FMM_LAUNCH_CHECK(P);
    return FMM_OK;
}

// full-field potential at the solute charges (solvent field + solute field) into phi_ff, after the full
// pass's L2P has written phi_ff
template <typename T>
fmm_status solute_act_l2p_t(Plan &P, SoluteScratch &S)
{
    const double h = P.box / (1 << P.d);
    k_act_l2p<T><<<NU_MAX, 256, 0, P.stream>>>(P.p, P.d, h, P.d_err + 1, S.slots, S.cells, S.ncells, P.sleaf,
                                               (const Particle<T> *)P.sorted, S.Lt, (const T *)P.phi_u, (T *)P.phi_ff);
    FMM_LAUNCH_CHECK(P);
    return FMM_OK;
}

// the sparse pass applies to this call as far as the host knows
bool solute_may_run(const Plan &P) { return P.known_count < 0 || (P.known_count > 0 && P.known_count <= NU_MAX); }

}  // namespace

fmm_status solute_prepare(Plan &P)
{
    solute_free(P);
    SoluteScratch *S = new (std::nothrow) SoluteScratch();
    if (!S) return FMM_ERR_OOM;
    P.sol = S;
    const int ld = P.d < LD_MAX ? P.d : LD_MAX;
    FMM_CUDA_TRY(cudaMalloc(&S->list, sizeof(int) * NU_MAX));
    FMM_CUDA_TRY(cudaMalloc(&S->slots, sizeof(int) * NU_MAX));
    FMM_CUDA_TRY(cudaMalloc(&S->cells, sizeof(int) * 9 * NU_MAX));
    FMM_CUDA_TRY(cudaMalloc(&S->ncells, sizeof(int) * 32));
    FMM_CUDA_TRY(cudaMalloc(&S->MU, sizeof(double) * 9 * NU_MAX * P.nc));
    S->map_bytes = sizeof(int) * (size_t)(P.d > ld ? map_off(P.d + 1, ld) : 0);
    FMM_CUDA_TRY(cudaMalloc(&S->map, S->map_bytes + 16));
    FMM_CUDA_TRY(cudaMalloc(&S->tlist, sizeof(int) * 9 * max_tgt(P.ws)));
    FMM_CUDA_TRY(cudaMalloc(&S->contrib, sizeof(double) * (size_t)(P.d + 1) * max_tgt(P.ws) * P.nc));
    FMM_CUDA_TRY(cudaMallocHost((void **)&S->h_count, sizeof(int)));
    int lo = 0, hi = 0;
    FMM_CUDA_TRY(cudaDeviceGetStreamPriorityRange(&lo, &hi));
    FMM_CUDA_TRY(cudaStreamCreateWithPriority(&S->side, cudaStreamNonBlocking, hi));
    for (cudaEvent_t *e : {&S->ev_count, &S->ev_sort, &S->ev_up, &S->ev_ready, &S->ev_done})
        FMM_CUDA_TRY(cudaEventCreateWithFlags(e, cudaEventDisableTiming));
    FMM_CUDA_TRY(cudaMalloc(&S->Lt, sizeof(double) * 9 * NU_MAX * P.nc));
    FMM_CUDA_TRY(cudaMalloc(&S->Lu, sizeof(double) * dense_off(ld + 1, P.nc)));
    FMM_CUDA_TRY(cudaMalloc(&S->part, sizeof(double) * (size_t)(P.d - 1) * NU_MAX * act_groups(P.ws) * P.nc));
    return FMM_OK;
}

void solute_free(Plan &P)
{
    SoluteScratch *S = (SoluteScratch *)P.sol;
    if (!S) return;
    cudaFree(S->list);
    cudaFree(S->slots);
    cudaFree(S->cells);
    cudaFree(S->ncells);
    cudaFree(S->MU);
    cudaFree(S->map);
    cudaFree(S->tlist);
    cudaFree(S->contrib);
    cudaFree(S->Lt);
    cudaFree(S->Lu);
    cudaFree(S->part);
    if (S->h_count) cudaFreeHost(S->h_count);
    if (S->side) {
        cudaStreamSynchronize(S->side);
        cudaStreamDestroy(S->side);
    }
    for (cudaEvent_t e : {S->ev_count, S->ev_sort, S->ev_up, S->ev_ready, S->ev_done})
        if (e) cudaEventDestroy(e);
    delete S;
    P.sol = nullptr;
}

int solute_count_host(const Plan &P)
{
    const SoluteScratch *S = (const SoluteScratch *)P.sol;
    return S ? *S->h_count : -1;
}

int *solute_list(Plan &P, int *cap)
{
    SoluteScratch *S = (SoluteScratch *)P.sol;
    *cap = NU_MAX;
    return S ? S->list : nullptr;
}

fmm_status solute_count(Plan &P)
{
    SoluteScratch *S = (SoluteScratch *)P.sol;
    if (!S) return FMM_ERR_INTERNAL;
    S->forked = S->act_done = false;  // a new call (a failed one may have left them set)
    FMM_CUDA_TRY(cudaEventRecord(S->ev_sort, P.stream));
    FMM_CUDA_TRY(cudaMemcpyAsync(S->h_count, P.d_err + 1, sizeof(int), cudaMemcpyDeviceToHost, P.stream));
    FMM_CUDA_TRY(cudaEventRecord(S->ev_count, P.stream));
    return FMM_OK;
}

fmm_status solute_fork(Plan &P)
{
    SoluteScratch *S = (SoluteScratch *)P.sol;
    if (!S || !P.overlap || !solute_may_run(P)) return FMM_OK;
    FMM_CUDA_TRY(cudaStreamWaitEvent(S->side, S->ev_sort, 0));
    S->forked = true;
    fmm_status s = P.precision == FMM_PREC_FP64 ? solute_expand_t<double>(P, *S, S->side)
                                                : solute_expand_t<float>(P, *S, S->side);
    if (s != FMM_OK) return s;
    // Phi_u at every charge (a full-size launch) on the near stream, where it fills idle SMs instead of taking
    // them from the far field
    cudaStream_t st = S->side;
    if (P.near_forked) {
        FMM_CUDA_TRY(cudaEventRecord(S->ev_ready, S->side));
        FMM_CUDA_TRY(cudaStreamWaitEvent(P.near, S->ev_ready, 0));
        st = P.near;
    }
    return P.precision == FMM_PREC_FP64 ? solute_eval_t<double>(P, *S, st) : solute_eval_t<float>(P, *S, st);
}

fmm_status solute_active(Plan &P)
{
    SoluteScratch *S = (SoluteScratch *)P.sol;
    if (!S || !S->forked) return FMM_OK;
    FMM_CUDA_TRY(cudaEventRecord(S->ev_up, P.stream));
    FMM_CUDA_TRY(cudaStreamWaitEvent(S->side, S->ev_up, 0));
    fmm_status s = P.precision == FMM_PREC_FP64 ? solute_act_t<double>(P, *S, S->side)
                                                : solute_act_t<float>(P, *S, S->side);
    if (s != FMM_OK) return s;
    S->act_done = true;
    return FMM_OK;
}

fmm_status solute_join(Plan &P)
{
    SoluteScratch *S = (SoluteScratch *)P.sol;
    if (!S || !S->forked) return FMM_OK;
    S->forked = false;
    FMM_CUDA_TRY(cudaEventRecord(S->ev_done, S->side));
    FMM_CUDA_TRY(cudaStreamWaitEvent(P.stream, S->ev_done, 0));
    return FMM_OK;
}

// Phi_u into P.phi_u by the sparse pass; *done = false asks for the dense pass
fmm_status launch_solute_pass(Plan &P, bool *done)
{
    *done = false;
    SoluteScratch *S = (SoluteScratch *)P.sol;
    if (!S) return FMM_ERR_INTERNAL;
    const bool expanded = S->forked && S->act_done;
    fmm_status s = solute_join(P);
    if (s != FMM_OK) return s;
    // the count was copied right after the sort, or the caller knows it
    if (P.known_count < 0) FMM_CUDA_TRY(cudaEventSynchronize(S->ev_count));
    S->act_done = false;
    const int n = P.known_count >= 0 ? P.known_count : *S->h_count;
    if (n > NU_MAX) return FMM_OK;  // the dense pass overwrites the (empty) result
    if (n == 0) {
        size_t bytes = (P.precision == FMM_PREC_FP64 ? sizeof(double) : sizeof(float)) * P.N;
        FMM_CUDA_TRY(cudaMemsetAsync(P.phi_u, 0, bytes, P.stream));
        *done = true;
        return FMM_OK;
    }
    const bool f64 = P.precision == FMM_PREC_FP64;
    if (!expanded) {  // in order on the plan's stream
        s = f64 ? solute_expand_t<double>(P, *S, P.stream) : solute_expand_t<float>(P, *S, P.stream);
        if (s == FMM_OK) s = f64 ? solute_act_t<double>(P, *S, P.stream) : solute_act_t<float>(P, *S, P.stream);
        if (s == FMM_OK) s = f64 ? solute_eval_t<double>(P, *S, P.stream) : solute_eval_t<float>(P, *S, P.stream);
    }
    if (s == FMM_OK) s = f64 ? solute_act_l2p_t<double>(P, *S) : solute_act_l2p_t<float>(P, *S);
    if (s == FMM_OK) *done = true;
    return s;
}

}  // namespace fmm
