// fmm_p2p.cu -- near field (Eq. EqNF): direct Coulomb sums over the
// (2 ws + 1)^3 leaves around each charge's leaf (27 for ws = 1, 125 for ws = 2),
// periodic, j != i.
//
// Coordinates are relative to each leaf's centre, so the separation of a
// charge in leaf c from one in neighbour leaf c + delta is
// loc_i - loc_j - delta h: the periodic image shift is implicit and the FP32
// path keeps full precision in boxes of any size.
#include <math.h>

#include "fmm_internal.cuh"

namespace fmm {

namespace {

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

template <typename T>
__device__ inline T inv_sqrt(T x);
template <>
__device__ inline float inv_sqrt<float>(float x) { return rsqrtf(x); }
template <>
__device__ inline double inv_sqrt<double>(double x) { return rsqrt(x); }  // within 1 ulp; 1.0 / sqrt(x) is twice the instructions

// One source of the near field: adds q_j / r and q_j r / r^3 for r = (ox, oy, oz) - x_j.  A source at r = 0
// (the target itself: the same stored coordinates) adds nothing; the near field never holds a charge's own
// periodic image (2^depth > 2 ws + 1).
template <typename T>
__device__ __forceinline__ void p2p_pair(const Particle<T> &pj, T ox, T oy, T oz, T &acc, T &ex, T &ey, T &ez)
{
    const T rx = ox - pj.x, ry = oy - pj.y, rz = oz - pj.z;
    const T r2 = rx * rx + ry * ry + rz * rz;
    const T ir = r2 > T(0) ? inv_sqrt<T>(r2) : T(0);
    const T qir = pj.q * ir;
    acc += qir;
    const T qir3 = qir * ir * ir;
    ex += qir3 * rx;
    ey += qir3 * ry;
    ez += qir3 * rz;
}

// The near field with the neighbour particles staged in shared memory: phi_i = sum q_j / r_ij and
// e_i = sum q_j r_ij / r_ij^3 per sorted charge i.  A block takes a row segment of BX consecutive leaves
// along x at (y, z) -- their charges are contiguous in the sorted order -- and copies the particles of the
// (2 ws + 1)^2 rows around it, each BX + 2 ws leaves long (x wrapped periodically, a leaf may appear twice
// when BX + 2 ws exceeds the side), into shared memory with 16-byte cp.async copies.  Then each thread
// takes one target charge of the segment and sums over its (2 ws + 1)^3 neighbour leaves in a fixed
// order; a block whose rows hold more than `cap` particles reads them from global memory with the same
// arithmetic in the same order, so the staged and unstaged blocks give identical results.
//   shared memory: pre[R W + 1] (staged start of leaf f = r W + i, row r = (dz + ws)(2 ws + 1) + dy + ws,
//   i = x - x0 + ws), gst[R W] (the leaf's first sorted index), then the staged records.
constexpr int P2P_THREADS = 128;

__device__ __forceinline__ void cp_async16(void *smem_dst, const void *gsrc)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem_dst)),
                 "l"(gsrc)
                 : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <typename T>
__device__ __forceinline__ void stage_copy(Particle<T> *dst, const Particle<T> *src)
{
    if (sizeof(Particle<T>) == 16) {
        cp_async16(dst, src);
    } else {
        cp_async16(dst, src);
        cp_async16(reinterpret_cast<char *>(dst) + 16, reinterpret_cast<const char *>(src) + 16);
    }
}

// The FP64 target loop.  GB300's FP64 pipe takes 16 cycles per warp instruction however many lanes are active, so the
// loops run over whole rows of neighbours (the 2 WS + 1 leaves of a row are contiguous; which leaf, hence which shift, a
// source is in follows from integer compares): the lanes of a warp differ by 14 sources in 9 where leaf by leaf they
// wait for the fullest leaf, 6 in 3.  In small systems `split` neighbouring lanes share a target and take its rows in
// turn.  100,000 charges at depth 5: 1,240 us leaf by leaf with 1 / sqrt, 631 us here; 2,998 at depth 3 278 and 88 us.
template <int WS, bool STAGED>
__device__ __forceinline__ void p2p_rows(int W, int it, int lane_of, int split, double h, const Particle<double> &pi,
                                         const int *pre, const int *gst, const Particle<double> *stg,
                                         const Particle<double> *__restrict__ sp, double (&out)[4])
{
    constexpr int SIDE = 2 * WS + 1;
    double ox[SIDE];
#pragma unroll
    for (int t = 0; t < SIDE; ++t) ox[t] = pi.x - (double)(t - WS) * h;
#pragma unroll
    for (int k = 0; k < 4; ++k) out[k] = 0.0;
    for (int r = lane_of; r < SIDE * SIDE; r += split) {
        const double oy = pi.y - (double)(r % SIDE - WS) * h, oz = pi.z - (double)(r / SIDE - WS) * h;
        const int f = r * W + it - WS;
        int b[SIDE], off[SIDE];  // each leaf's first staged index and its distance from the sorted one
#pragma unroll
        for (int t = 0; t < SIDE; ++t) {
            b[t] = pre[f + t];
            off[t] = STAGED ? 0 : gst[f + t] - b[t];
        }
        const int je = pre[f + SIDE];
        double acc = 0.0, ex = 0.0, ey = 0.0, ez = 0.0;
        for (int j = b[0]; j < je; ++j) {
            double x = ox[0];
            int o = off[0];
#pragma unroll
            for (int t = 1; t < SIDE; ++t) {
                x = j >= b[t] ? ox[t] : x;
                o = j >= b[t] ? off[t] : o;
            }
            p2p_pair<double>(STAGED ? stg[j] : sp[j + o], x, oy, oz, acc, ex, ey, ez);
        }
        out[0] += acc;
        out[1] += ex;
        out[2] += ey;
        out[3] += ez;
    }
    for (int o = 1; o < split; o <<= 1)  // the whole warp is here
#pragma unroll
        for (int k = 0; k < 4; ++k) out[k] += __shfl_xor_sync(0xffffffffu, out[k], o);
}

template <typename T>
__global__ void __launch_bounds__(P2P_THREADS) k_p2p_tile(int d, int ws, int bx, int cap, int split, T h,
                                                          const int *__restrict__ start,
                                                          const Particle<T> *__restrict__ sp, T *__restrict__ phi,
                                                          T *__restrict__ field)
{
    extern __shared__ __align__(16) unsigned char p2p_smem[];
    const int n = 1 << d, mask = n - 1;
    const int side = 2 * ws + 1, R = side * side, W = bx + 2 * ws, F = R * W;
    const int tiles_x = n / bx;
    const int x0 = (blockIdx.x % tiles_x) * bx;
    const int y = (blockIdx.x / tiles_x) & mask, z = blockIdx.x / (tiles_x * n);
    int *pre = reinterpret_cast<int *>(p2p_smem);
    int *gst = pre + F + 1;
    Particle<T> *stg = reinterpret_cast<Particle<T> *>(p2p_smem + ((sizeof(int) * (2 * F + 1) + 15) / 16) * 16);
    __shared__ int warp_tot[P2P_THREADS / 32];

    auto gleaf = [&](int f) {  // global leaf of staged leaf f
        const int r = f / W, i = f - r * W;
        const int dy = r % side - ws, dz = r / side - ws;
        return ((x0 - ws + i) & mask) + n * (((y + dy) & mask) + n * ((z + dz) & mask));
    };
    // 1. per-leaf counts -> exclusive prefix pre[] (each thread a run of consecutive entries, then a scan of
    //    the run totals across the block)
    const int per = (F + P2P_THREADS - 1) / P2P_THREADS;
    const int f0 = threadIdx.x * per;
    int run = 0;
    for (int f = f0; f < f0 + per && f < F; ++f) {
        const int g = gleaf(f);
        const int b = start[g];
        const int c = start[g + 1] - b;
        gst[f] = b;
        pre[f + 1] = c;
        run += c;
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int incl = run;
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) warp_tot[w] = incl;
    if (threadIdx.x == 0) pre[0] = 0;
    __syncthreads();
    int base = incl - run;
    for (int k = 0; k < w; ++k) base += warp_tot[k];
    for (int f = f0; f < f0 + per && f < F; ++f) {
        const int c = pre[f + 1];
        base += c;
        pre[f + 1] = base;
    }
    __syncthreads();
    const int total = pre[F];
    const bool staged = total <= cap;
    // 2. stage the rows: thread per staged leaf, its records by independent 16-byte copies
    if (staged) {
        for (int f = threadIdx.x; f < F; f += P2P_THREADS) {
            const int b = pre[f], n = pre[f + 1] - b;
            const Particle<T> *src = sp + gst[f];
            for (int k = 0; k < n; ++k) stage_copy<T>(stg + b + k, src + k);
        }
        cp_async_wait_all();
    }
    __syncthreads();
    // 3. targets: the leaves x0 .. x0 + bx - 1 of the centre row
    const int rc = ws * side + ws;
    const int tb = pre[rc * W + ws], te = pre[rc * W + ws + bx];
    if constexpr (sizeof(T) == 8) {
        for (int u0 = 0; u0 < (te - tb) * split; u0 += P2P_THREADS) {
            const int u = u0 + (int)threadIdx.x;
            const bool on = u < (te - tb) * split;
            const int st = on ? tb + u / split : te - 1;  // spare lanes redo the last target and store nothing
            int lo = rc * W + ws, hi = rc * W + ws + bx;
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (pre[mid] <= st) lo = mid;
                else hi = mid;
            }
            const int it = lo - rc * W, s = gst[lo] + (st - pre[lo]);
            // a warp with no target of its own: nothing to do (the shuffles stay within a warp)
            if (__ballot_sync(0xffffffffu, on) == 0) continue;
            const Particle<T> pi = staged ? stg[st] : sp[s];
            T v[4];
            if (ws == 1) {
                if (staged) p2p_rows<1, true>(W, it, u % split, split, h, pi, pre, gst, stg, sp, v);
                else p2p_rows<1, false>(W, it, u % split, split, h, pi, pre, gst, stg, sp, v);
            } else {
                if (staged) p2p_rows<2, true>(W, it, u % split, split, h, pi, pre, gst, stg, sp, v);
                else p2p_rows<2, false>(W, it, u % split, split, h, pi, pre, gst, stg, sp, v);
            }
            if (on && u % split == 0) {
                phi[s] = v[0];
                if (field) {
                    field[3 * s] = v[1];
                    field[3 * s + 1] = v[2];
                    field[3 * s + 2] = v[3];
                }
            }
        }
    } else {
        for (int st = tb + (int)threadIdx.x; st < te; st += P2P_THREADS) {
            int lo = rc * W + ws, hi = rc * W + ws + bx;  // the target's staged leaf
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (pre[mid] <= st) lo = mid;
                else hi = mid;
            }
            const int it = lo - rc * W;  // index of the target leaf within its row
            const int s = gst[lo] + (st - pre[lo]);  // sorted index of the target
            const Particle<T> pi = staged ? stg[st] : sp[s];
            // four independent partial sums (sources j, j + 1, j + 2, j + 3 of each leaf), so that the loads and
            // the dependent additions of consecutive pairs overlap; added in a fixed order at the end
            T a[4] = {0, 0, 0, 0}, fx[4] = {0, 0, 0, 0}, fy[4] = {0, 0, 0, 0}, fz[4] = {0, 0, 0, 0};
            for (int dz = -ws; dz <= ws; ++dz)
                for (int dy = -ws; dy <= ws; ++dy)
                    for (int dx = -ws; dx <= ws; ++dx) {
                        const int f = ((dz + ws) * side + dy + ws) * W + it + dx;
                        const T ox = pi.x - T(dx) * h, oy = pi.y - T(dy) * h, oz = pi.z - T(dz) * h;
                        int jb, je;
                        const Particle<T> *src;
                        if (staged) {
                            jb = pre[f];
                            je = pre[f + 1];
                            src = stg;
                        } else {  // the leaf's records in the sorted array
                            jb = gst[f];
                            je = jb + (pre[f + 1] - pre[f]);
                            src = sp;
                        }
                        int j = jb;
                        for (; j + 4 <= je; j += 4) {
                            Particle<T> q4[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u) q4[u] = src[j + u];
#pragma unroll
                            for (int u = 0; u < 4; ++u) p2p_pair<T>(q4[u], ox, oy, oz, a[u], fx[u], fy[u], fz[u]);
                        }
                        if (j < je) {
                            p2p_pair<T>(src[j], ox, oy, oz, a[0], fx[0], fy[0], fz[0]);
                            if (j + 1 < je) {
                                p2p_pair<T>(src[j + 1], ox, oy, oz, a[1], fx[1], fy[1], fz[1]);
                                if (j + 2 < je) p2p_pair<T>(src[j + 2], ox, oy, oz, a[2], fx[2], fy[2], fz[2]);
                            }
                        }
                    }
            phi[s] = (a[0] + a[1]) + (a[2] + a[3]);
            if (field) {
                field[3 * s] = (fx[0] + fx[1]) + (fx[2] + fx[3]);
                field[3 * s + 1] = (fy[0] + fy[1]) + (fy[2] + fy[3]);
                field[3 * s + 2] = (fz[0] + fz[1]) + (fz[2] + fz[3]);
            }
        }
    }
}

// near-field solute-solvent pair sum of every solute slot: out_i = q_i sum_{j in NF(i), j solvent} q_j / r_ij (the
// slots of the solvent are not read).  The sum runs over the neighbour leaves and their charges in order, in T: the
// solute-solvent energy is a small difference of it and the far field, so another order would show.
// A block looks at 128 slots.  Where only a few are solute, it takes them one at a time, all threads computing the
// terms and one adding them up from shared memory: as one thread's whole work a lone ion's ~1,000 sources took
// 31-127 us, each term a chain of loads.  Where many are, each of their threads sums its own.
// SC: also the soft-core form of these pairs, r -> reff = (alpha lambda A^c + r^c)^(1/c) (the paper's soft-core
// form, which it notes applies to the electrostatic NF term), in FP64 from the stored coordinates:
// sc[s] = q_i sum_j q_j / reff and sc[N + s] = -(alpha A^c / c) q_i sum_j q_j / (reff (alpha lambda A^c + r^c)).
// alpha_Ac = alpha A^c; lambda is read from device memory.
constexpr int UV_THREADS = 128;
constexpr int UV_FEW = 6;       // solute slots of a block up to which it works on one at a time
constexpr int UV_CHUNK = 1024;  // terms staged at once

struct UvSoft {
    int c;
    double b0, ic;  // alpha lambda A^c and 1/c
};

template <typename T>
__device__ __forceinline__ void uv_soft_term(const Particle<T> &pi, const Particle<T> &pj, int dx, int dy, int dz, T h,
                                             const UvSoft &f, double &e, double &de)
{
    const double ux = (double)pi.x - (double)dx * (double)h - (double)pj.x,
                 uy = (double)pi.y - (double)dy * (double)h - (double)pj.y,
                 uz = (double)pi.z - (double)dz * (double)h - (double)pj.z;
    const double base = f.b0 + pow(sqrt(ux * ux + uy * uy + uz * uz), (double)f.c);
    const double reff = pow(base, f.ic);
    e += (double)pj.q / reff;
    de += (double)pj.q / (reff * base);
}

template <typename T>
__device__ __forceinline__ T uv_term(const Particle<T> &pj, T ox, T oy, T oz)
{
    const T rx = ox - pj.x, ry = oy - pj.y, rz = oz - pj.z;
    return pj.q * inv_sqrt<T>(rx * rx + ry * ry + rz * rz);
}

__device__ __forceinline__ double uv_block_sum(double v, double *part, int lane, int w)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) part[w] = v;
    __syncthreads();
    double a = part[0];
    for (int k = 1; k < UV_THREADS / 32; ++k) a += part[k];
    __syncthreads();
    return a;
}

template <typename T, bool SC>
__global__ void __launch_bounds__(UV_THREADS) k_p2p_uv(int64_t N, int d, int ws, T h, const int *__restrict__ start,
                                                       const int *__restrict__ sleaf, const Particle<T> *__restrict__ sp,
                                                       const uint8_t *__restrict__ sol, T *__restrict__ out, int c,
                                                       double alpha_Ac, const double *__restrict__ lambda,
                                                       double *__restrict__ sc)
{
    constexpr int NL_MAX = (2 * WS_MAX + 1) * (2 * WS_MAX + 1) * (2 * WS_MAX + 1);
    __shared__ unsigned found[UV_THREADS / 32];
    __shared__ int first[NL_MAX], pre[NL_MAX + 1];  // a neighbour leaf's first charge; charges of the leaves before it
    __shared__ T term[UV_CHUNK];
    __shared__ double part[UV_THREADS / 32];
    const int64_t s0 = blockIdx.x * (int64_t)UV_THREADS;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const bool mine = s0 + threadIdx.x < N && sol[s0 + threadIdx.x];
    const unsigned m = __ballot_sync(0xffffffffu, mine);
    if (lane == 0) found[w] = m;
    const int nsol = __syncthreads_count(mine);
    if (nsol == 0) return;
    const int side = 2 * ws + 1, nl = side * side * side, nside = 1 << d;
    UvSoft f{};
    if (SC) f = {c, alpha_Ac * *lambda, 1.0 / (double)c};
    auto neighbour = [&](int leaf, int l, int &dx, int &dy, int &dz) {  // l-th neighbour leaf, x fastest
        dx = l % side - ws;
        dy = (l / side) % side - ws;
        dz = l / (side * side) - ws;
        const int x = leaf & (nside - 1), y = (leaf >> d) & (nside - 1), z = leaf >> (2 * d);
        return ((x + dx) & (nside - 1)) + nside * (((y + dy) & (nside - 1)) + nside * ((z + dz) & (nside - 1)));
    };
    if (nsol > UV_FEW) {
        if (!mine) return;
        const int64_t s = s0 + threadIdx.x;
        const int leaf = sleaf[s];
        const Particle<T> pi = sp[s];
        T acc = 0;
        double e = 0.0, de = 0.0;
        for (int l = 0; l < nl; ++l) {
            int dx, dy, dz;
            const int lc = neighbour(leaf, l, dx, dy, dz);
            const T ox = pi.x - T(dx) * h, oy = pi.y - T(dy) * h, oz = pi.z - T(dz) * h;
            for (int j = start[lc]; j < start[lc + 1]; ++j) {
                if (sol[j]) continue;
                const Particle<T> pj = sp[j];
                acc += uv_term<T>(pj, ox, oy, oz);
                if (SC) uv_soft_term<T>(pi, pj, dx, dy, dz, h, f, e, de);
            }
        }
        out[s] = pi.q * acc;
        if (SC) {
            sc[s] = (double)pi.q * e;
            sc[N + s] = -(alpha_Ac * f.ic) * (double)pi.q * de;
        }
        return;
    }
    for (int v = 0; v < UV_THREADS / 32; ++v)
        for (unsigned fm = found[v]; fm; fm &= fm - 1) {
            const int64_t s = s0 + 32 * v + __ffs(fm) - 1;
            const int leaf = sleaf[s];
            const Particle<T> pi = sp[s];
            for (int l = threadIdx.x; l < nl; l += UV_THREADS) {
                int dx, dy, dz;
                const int lc = neighbour(leaf, l, dx, dy, dz);
                first[l] = start[lc];
                pre[l + 1] = start[lc + 1] - start[lc];
            }
            if (threadIdx.x == 0) pre[0] = 0;
            __syncthreads();
            if (w == 0) {  // counts -> exclusive prefix
                int base = 0;
                for (int l0 = 0; l0 < nl; l0 += 32) {
                    const int l = l0 + lane;
                    int x = l < nl ? pre[l + 1] : 0;
                    for (int o = 1; o < 32; o <<= 1) {
                        const int y = __shfl_up_sync(0xffffffffu, x, o);
                        if (lane >= o) x += y;
                    }
                    if (l < nl) pre[l + 1] = base + x;
                    base += __shfl_sync(0xffffffffu, x, 31);
                }
            }
            __syncthreads();
            const int total = pre[nl];
            T acc = 0;
            double e = 0.0, de = 0.0;
            for (int t0 = 0; t0 < total; t0 += UV_CHUNK) {
                const int n = total - t0 < UV_CHUNK ? total - t0 : UV_CHUNK;
                for (int t = threadIdx.x; t < n; t += UV_THREADS) {
                    int lo = 0, hi = nl;  // the leaf of term t0 + t
                    while (hi - lo > 1) {
                        const int mid = (lo + hi) >> 1;
                        if (pre[mid] <= t0 + t) lo = mid;
                        else hi = mid;
                    }
                    int dx, dy, dz;
                    neighbour(leaf, lo, dx, dy, dz);
                    const int j = first[lo] + t0 + t - pre[lo];
                    const Particle<T> pj = sp[j];
                    const T g = uv_term<T>(pj, pi.x - T(dx) * h, pi.y - T(dy) * h, pi.z - T(dz) * h);
                    const bool solvent = !sol[j];
                    term[t] = solvent ? g : T(0);
                    if (SC && solvent) uv_soft_term<T>(pi, pj, dx, dy, dz, h, f, e, de);
                }
                __syncthreads();
                if (threadIdx.x == 0) {
                    int t = 0;
                    for (; t + 8 <= n; t += 8) {
                        T g[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) g[u] = term[t + u];
#pragma unroll
                        for (int u = 0; u < 8; ++u) acc += g[u];
                    }
                    for (; t < n; ++t) acc += term[t];
                }
                __syncthreads();
            }
            if (SC) {
                e = uv_block_sum(e, part, lane, w);
                de = uv_block_sum(de, part, lane, w);
            }
            if (threadIdx.x == 0) {
                out[s] = pi.q * acc;
                if (SC) {
                    sc[s] = (double)pi.q * e;
                    sc[N + s] = -(alpha_Ac * f.ic) * (double)pi.q * de;
                }
            }
        }
}

}  // namespace

namespace {

// staged-tile launch: rows of BX leaves, BX a power of two up to min(32, side) chosen so that a row holds
// about 128 target charges at the mean leaf occupancy (dense leaves: short rows, more blocks); the staging
// capacity is 1.25 times the expected particle count of a tile's rows plus 256 (a tile beyond it reads global memory;
// twice the count plus 512 left room for one block less per SM: 10M charges 23.1 -> 22.2 ms, 100k at ws = 2 1.62 ->
// 1.53 ms), within 96 KB of shared memory.  Boxes filled to half or an eighth of their volume, the near field alone: 447 ->
// 424 and 1,320 -> 1,007 us (1M, d = 6), 428 -> 358 us (100k, ws = 2, half); but 172 -> 238 us (61k, d = 4, half) and 61
// -> 76 us (100k, d = 5, half), where it runs beside a longer far field.  The FP32 path keeps one thread per target for
// the same reason
template <typename T>
fmm_status launch_p2p_tile(Plan &P, T h, T *phi, T *field)
{
    static bool attr = false;
    const size_t smem_max = 96 * 1024;
    if (!attr) {
        FMM_CUDA_TRY(cudaFuncSetAttribute(k_p2p_tile<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max));
        attr = true;
    }
    const int n = 1 << P.d;
    const double occ = (double)P.N / (double)P.nleaf;
    // FP64: lanes per target until every SM has 8 warps, and tiles for two blocks per SM
    int split = 1;
    if (sizeof(T) == 8)
        while (split < 8 && P.N * split < 152 * 8 * 32) split *= 2;
    int bx = 1;
    while (bx < 32 && bx < n && (double)(2 * bx) * occ * split <= 128.0) bx *= 2;
    if (sizeof(T) == 8)
        while (bx > 1 && (int64_t)n * n * (n / bx) < 304) bx /= 2;
    const int side = 2 * P.ws + 1, F = side * side * (bx + 2 * P.ws);
    const size_t head = ((sizeof(int) * (2 * F + 1) + 15) / 16) * 16;
    const double expect = (double)P.N / (double)P.nleaf * F;
    size_t cap = (size_t)(1.25 * expect) + 256;
    const size_t cap_max = (smem_max - head) / sizeof(Particle<T>);
    if (cap > cap_max) cap = cap_max;
    const unsigned blocks = (unsigned)((int64_t)n * n * (n / bx));
    k_p2p_tile<T><<<blocks, P2P_THREADS, head + cap * sizeof(Particle<T>), P.stream>>>(
        P.d, P.ws, bx, (int)cap, split, h, P.cell_start, (const Particle<T> *)P.sorted, phi, field);
    return FMM_OK;
}

}  // namespace

fmm_status launch_p2p(Plan &P, bool forces)
{
    int nside = 1 << P.d;
    double h = P.box / nside;
    fmm_status st;
    if (P.precision == FMM_PREC_FP64)
        st = launch_p2p_tile<double>(P, h, (double *)P.phi_nf, forces ? (double *)P.f_nf : nullptr);
    else
        st = launch_p2p_tile<float>(P, (float)h, (float *)P.phi_nf, forces ? (float *)P.f_nf : nullptr);
    if (st != FMM_OK) return st;
    FMM_LAUNCH_CHECK(P);
    return FMM_OK;
}

template <typename T>
static void run_p2p_uv(Plan &P, T h)
{
    const unsigned blocks = blocks_for(P.N, UV_THREADS);
    const Particle<T> *sp = (const Particle<T> *)P.sorted;
    T *out = (T *)P.phi_nf + P.N;
    if (P.sc_c > 0)
        k_p2p_uv<T, true><<<blocks, UV_THREADS, 0, P.stream>>>(P.N, P.d, P.ws, h, P.cell_start, P.sleaf, sp, P.sorted_sol,
                                                               out, P.sc_c, P.sc_alpha * pow(P.sc_A, (double)P.sc_c),
                                                               P.sc_lambda, P.sc_out);
    else
        k_p2p_uv<T, false><<<blocks, UV_THREADS, 0, P.stream>>>(P.N, P.d, P.ws, h, P.cell_start, P.sleaf, sp,
                                                                P.sorted_sol, out, 0, 0.0, nullptr, nullptr);
}

fmm_status launch_p2p_uv(Plan &P)
{
    const double h = P.box / (1 << P.d);
    if (P.precision == FMM_PREC_FP64) run_p2p_uv<double>(P, h);
    else run_p2p_uv<float>(P, (float)h);
    FMM_LAUNCH_CHECK(P);
    return FMM_OK;
}

}  // namespace fmm
