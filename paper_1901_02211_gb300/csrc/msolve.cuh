// Multi-shift CG for (D_W^dag D_W + q_i) x_i = b, all shifts in one Krylov
// space (Sec. 2.1, Eqs. 6-8; Frommer et al. 1995, Jegerlehner hep-lat/9612014),
// for a batch of B right-hand sides, accumulating y = sum_i c_i x_i (Eq. 4) on
// the support the trace needs.
//
// One iteration is three launches, with no host synchronisation:
//   A   t = D_W p, per-block partials |t|^2, |p|^2; the last block to finish
//       an RHS tile sums the tile's partials and runs the first scalar step of
//       its columns: alpha = <r,r> / (|t|^2 + s0 |p|^2), zeta_{k+1} and
//       alpha_i of every shift
//   B   r -= alpha (D_W^dag t + s0 p) [x_lo += alpha p], partials |r|^2; the
//       last block of a tile runs the second scalar step: beta, beta_i,
//       convergence |zeta_i| ||r|| <= tol ||b||, residual-replacement request
//   YP  on the support: r into the history; on the lattice: p = r + beta p
//       [x += alpha p for the true residual]
// The "last block" is found with one atomic counter per RHS tile (the CUDA
// threadfence-reduction pattern): no block ever waits for another.
// Base vectors (p, t, r) live on the whole lattice in the iteration precision T.
// Shifted directions p_i are pointwise in x (the matrix never touches them):
// p_i = zeta_i r + beta_i p_i and y += c_i alpha_i p_i make y a sum of the
// residuals r_k with weights that only the scalars decide.  So an iteration
// keeps r where y is read later (the 9-site star around every site of the
// right-hand side's colour class; the full lattice for smpq_apply_dov) and the
// scalars of its shifts, and y is formed once, at the end of the solve
// ("the residual history" below).
// FP32 path: x_hi (FP64) += x_lo at every residual replacement, where the FP64
// residual b - (A + s0) x_hi replaces r (reliable updates, Sleijpen & van der
// Vorst 1996); scalars, reductions and y stay FP64 throughout.
//
// Reductions are deterministic: per-block partial sums in a fixed tree/sequence,
// then a fixed-order sum over the blocks of a tile in the tile's last block.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <initializer_list>

#include "bfp.cuh"
#include "half.cuh"
#include "smpq_internal.cuh"
#include "stage.cuh"
#include "wilson.cuh"

namespace {

// Each block of a lattice kernel handles TPB consecutive tiles of one RHS
// tile, and blocks are numbered site-major inside an RHS tile, so the blocks
// resident at any moment cover a narrow band of the lattice for few RHS tiles:
// the +-t neighbours (V/n_t sites away) are still in L2 when they are read.
// (The D_W kernels take the count as an argument, chosen by the autotuner.)
constexpr int TPB = 4;

// minimum resident blocks per SM requested from the register allocator for
// the FP32 lattice kernels (240-thread blocks: 2 -> <= 136 registers, 3 -> <= 91)
#ifndef SMPQ_FP32_MIN_BLOCKS
#define SMPQ_FP32_MIN_BLOCKS 3
#endif
template <typename T> struct MinBlocks { static constexpr int value = SMPQ_FP32_MIN_BLOCKS; };
template <> struct MinBlocks<double> { static constexpr int value = 1; };
#ifndef SMPQ_DF64_MIN_BLOCKS
#define SMPQ_DF64_MIN_BLOCKS 2
#endif
template <> struct MinBlocks<df64> { static constexpr int value = SMPQ_DF64_MIN_BLOCKS; };

// link copy matching the iteration precision
template <typename T> struct Links;
template <> struct Links<double> { static const void *get(const smpq_ctx *c) { return c->Ubf.p; } }; // (block fixed point)
template <> struct Links<float> { static const void *get(const smpq_ctx *c) { return c->U32.p; } };
template <> struct Links<df64> { static const void *get(const smpq_ctx *c) { return c->Udf.p; } };


// ------------------------------------------------------------------ block reduction per column
template <int BC, int THREADS = TileMap<BC>::THREADS>
__device__ __forceinline__ double block_sum(double v, double *sm) {
    double s = 0;
    if constexpr (32 % BC == 0) {
#pragma unroll
        for (int o = 16; o >= BC; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        if (lane < BC) sm[warp * BC + lane] = v;
        __syncthreads();
        if (threadIdx.x < BC)
            for (int w = 0; w < THREADS / 32; ++w) s += sm[w * BC + threadIdx.x];
        __syncthreads();
    } else {
        sm[threadIdx.x] = v;
        __syncthreads();
        if (threadIdx.x < BC)
            for (int k = threadIdx.x; k < THREADS; k += BC) s += sm[k];
        __syncthreads();
    }
    return s;
}

constexpr int NFLAGS = 5; // the flags the host reads after each check interval
struct Scal {
    double *rr, *bb, *alpha, *beta, *alpha_prev, *beta_prev, *rr_ref; // [B]
    int *act_rhs, *upd_rhs, *iters;                                  // [B]
    double *zeta, *zeta_prev;                                        // [n][B]
    int *act, *upd;                                                  // [n][B]
    // per iteration of the history (row slot[j] of column j): zeta_{k+1} and the
    // zeta_k before it of every shift, [rows][n][B] (hz 0 in an iteration that
    // left the shift's direction alone), alpha and beta of the column, [rows][B].
    // The shift's own alpha_i = alpha zeta_{k+1} / zeta_k and beta_i = beta
    // (zeta_{k+1} / zeta_k)^2 are formed from them at the end (their divisions
    // were half of the scalar steps' FP64 work, which every launch waits for).
    double *hz, *ho, *hal, *hbe;
    int *slot;    // [B] history row of the column's current iteration
    int slot_inc; // 1; 0 without a history (every row is row 0)
    int *flags; // [0] active rhs count, [1] residual replacement requested, [2] breakdown,
                // [3] active rhs still above the precision-switch residual,
                // [4] a staging wait of the FP32 D_W ran out (stage.cuh)
    double *hist; // Lanczos: [2][hist_len] alpha_k, beta_k of rhs 0 (nullable)
    int hist_len;
    int *iter_counter; // [1] global iteration count (for the history index)
};

// source value of component c of rhs j at site s
struct Source {
    const int *colour;     // [V] (class-based sources)
    const int *src_class;  // [B] colour class carrying rhs j (-1: zero source)
    const int *src_comp;   // [B] spin*3 + colour index of rhs j
    const double2 *b64;    // tiled FP64 explicit source (nullable)
};

template <int BC>
__device__ __forceinline__ double2 source_at(const Source &src, int V, int s, int c, int j, size_t tiled_idx) {
    if (src.b64) return src.b64[tiled_idx];
    int cl = src.src_class[j];
    return make_double2((cl >= 0 && src.colour[s] == cl && c == src.src_comp[j]) ? 1.0 : 0.0, 0.0);
}

// ------------------------------------------------------------------ the lattices of a launch
// The RHS tiles of a launch (blockIdx.y) belong to one lattice, or to several
// of different sizes (the uneven batch of smpq_compute_qx_batch): lattice l
// owns the tiles from chunk0_l on, and its part of every field buffer starts
// at element f0_l.  The iteration kernels take this table; M = false is the
// one-lattice form (entry 0, known at compile time).
constexpr int MAX_LAT = 4;
struct Lat {
    Geom g;
    const void *U;  // links in the launch's precision
    long long f0;   // first element (complex value) of the lattice's fields
    long long p0;   // first partial-sum row of the lattice in this launch
    int chunk0;     // first RHS tile
    int G;          // blocks per tile in this launch (launch YP: lattice blocks)
    double s0;      // base (smallest) shift of the lattice's rational
    int n_sup, Gs;  // launch YP: support entries per rhs, support blocks per tile
    int B;          // right-hand sides of the lattice
    const int *supsite;
    long long sup0; // first element of the lattice's support fields (y; ps shift by shift)
};
struct Lats {
    int n;
    Lat l[MAX_LAT];
};
template <bool M> __device__ __forceinline__ int lat_index(const Lats &L) {
    if constexpr (!M) return 0;
    int l = 0;
    while (l + 1 < L.n && (int)blockIdx.y >= L.l[l + 1].chunk0) ++l;
    return l;
}

// ------------------------------------------------------------------ scalar steps
// Run by one block of NT threads for the BC columns of an RHS tile (from the
// solve's column j0): thread t < BC has column t's sum and does the column's
// own scalars, then NT / BC threads share its shifts (one thread per column took 14
// of them in a row, divisions and dependent loads: 5 us at the end of every
// D_W launch).
// First step: alpha and the shift recurrences zeta_{k+1}, alpha_i (tt = |D_W
// p|^2, pp = |p|^2, so <p, A p> = tt + s0 pp).
template <int BC, int NT>
__device__ void s1_tile(int j0, double tt, double pp, const Scal &sc, const ShiftParams &sp, int B, double *sm) {
    __shared__ int mode[BC]; // 0 idle, 1 active
    const int t = threadIdx.x;
    if (t < BC) {
        const int j = j0 + t;
        if (j == 0) {
            sc.flags[0] = 0;
            sc.flags[3] = 0;
            if (sc.hist) {
                int it = sc.iter_counter[0];
                if (it < sc.hist_len) sc.hist[it] = 0; // filled below when rhs 0 is active
            }
        }
        int m = sc.act_rhs[j] != 0;
        double a = 0;
        if (m) {
            const double pAp = tt + sp.s0 * pp;
            if (!(pAp > 0) || !isfinite(pAp)) {
                atomicOr(&sc.flags[2], 1);
                sc.act_rhs[j] = 0;
                m = 0;
            } else {
                a = sc.rr[j] / pAp;
                if (sc.hist && j == 0) {
                    int it = sc.iter_counter[0];
                    if (it < sc.hist_len) sc.hist[it] = a;
                }
            }
        }
        sc.alpha[j] = a;
        sc.upd_rhs[j] = m;
        mode[t] = m;
        sm[t] = a;
    }
    __syncthreads();
    constexpr int K = NT / BC;
    const int q = t % BC, j = j0 + q;
    if (t < K * BC) {
        const size_t row = (size_t)sc.slot[j] * sp.n * B + j;
        const bool on = mode[q];
        const double a = sm[q], ap = sc.alpha_prev[j], bp = sc.beta_prev[j];
        for (int i = t / BC; i < sp.n; i += K) {
            const int ix = i * B + j;
            const size_t hx = row + (size_t)i * B;
            if (!on || !sc.act[ix]) { sc.upd[ix] = 0; continue; }
            double z = sc.zeta[ix], zp = sc.zeta_prev[ix];
            double den = a * bp * (zp - z) + zp * ap * (1.0 + sp.sig[i] * a);
            double zn = z * zp * ap / den;
            sc.hz[hx] = zn;
            sc.ho[hx] = z;
            sc.upd[ix] = 1;
        }
    }
}

// Second step (rrn = |r_{k+1}|^2): beta, beta_i, the convergence of every
// shift, the residual-replacement request and the count of columns still above
// the precision-switch residual.
template <int BC, int NT>
__device__ void s2_tile(int j0, double rrn, const Scal &sc, const ShiftParams &sp, int B, double tol2, double delta2,
                        double theta2, double *sm) {
    __shared__ int any[BC]; // some shift is active
    const int t = threadIdx.x;
    if (t < BC) {
        const int j = j0 + t;
        if (j == 0) {
            if (sc.hist) {
                int it = sc.iter_counter[0];
                if (it < sc.hist_len) sc.hist[sc.hist_len + it] = sc.upd_rhs[0] ? rrn / sc.rr[0] : 0.0;
            }
            sc.iter_counter[0] += 1;
        }
        any[t] = 0;
        sm[t] = rrn;
        sm[BC + t] = sc.upd_rhs[j] ? rrn / sc.rr[j] : 0.0;
    }
    __syncthreads();
    constexpr int K = NT / BC;
    if (t < K * BC) {
        const int q = t % BC, j = j0 + q;
        const size_t row = (size_t)sc.slot[j] * sp.n * B + j;
        const bool on = sc.upd_rhs[j];
        const double r2 = sm[q], bb = sc.bb[j];
        for (int i = t / BC; i < sp.n; i += K) {
            const int ix = i * B + j;
            const size_t hx = row + (size_t)i * B;
            if (!on || !sc.upd[ix]) {
                if (on && sc.act[ix]) any[q] = 1;
                sc.hz[hx] = 0;
                continue;
            }
            const double z = sc.ho[hx], zn = sc.hz[hx];
            sc.zeta_prev[ix] = z;
            sc.zeta[ix] = zn;
            int a = zn * zn * r2 > tol2 * bb;
            sc.act[ix] = a;
            if (a) any[q] = 1;
        }
    }
    __syncthreads();
    if (t < BC) {
        const int j = j0 + t;
        const size_t h = (size_t)sc.slot[j] * B + j;
        sc.hal[h] = sc.alpha[j];
        sc.hbe[h] = sm[BC + t];
        sc.slot[j] += sc.slot_inc;
        if (!sc.upd_rhs[j]) return;
        const double bb = sc.bb[j];
        sc.beta[j] = sm[BC + t];
        sc.alpha_prev[j] = sc.alpha[j];
        sc.beta_prev[j] = sm[BC + t];
        sc.rr[j] = rrn;
        sc.iters[j] += 1;
        sc.act_rhs[j] = any[t];
        if (any[t]) atomicAdd(&sc.flags[0], 1);
        if (delta2 > 0 && rrn < delta2 * sc.rr_ref[j]) atomicOr(&sc.flags[1], 1);
        if (any[t] && rrn > theta2 * bb) atomicAdd(&sc.flags[3], 1); // still above the precision switch
    }
}

// What the lattice kernels A and B need for the scalar step of an RHS tile.
// count == nullptr: no scalar step (the autotuner's timing launches).
struct Fuse {
    int *count; // [tiles] blocks of the tile that have stored their partials; back to 0 after each launch
    int *gcount; // [tiles][ngroups] the same for groups of 64 blocks
    int ngroups;
    Scal sc;
    const ShiftParams *sp; // [lattices] each lattice's shifts (device memory)
    int B;                 // right-hand sides of the solve (stride of the shift-major scalars)
    double tol2, delta2, theta2; // (second step only)
};

// Called by every thread of a block after its partial sums are stored: true
// in every thread of the block that arrives last among the G blocks of RHS
// tile blockIdx.y.  The threads that stored partials (wrote) fence them before
// the arrival count, so the last block sees every partial of its tile; the
// other threads' stores need no fence (the next launch sees them).
__device__ __forceinline__ bool last_block_of_tile(int *count, int G, bool wrote) {
    __shared__ int last;
    if (wrote) __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const int ticket = atomicAdd(&count[blockIdx.y], 1);
        last = ticket == G - 1;
        if (last) count[blockIdx.y] = 0; // every block of the tile has arrived: reset for the next launch
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// Sum over the G blocks of an RHS tile (partial rows prow...) of each column, in
// a fixed order (NT / BC lanes per column, then the lanes in order); every
// thread of the block calls it, threads < BC receive their column's total.
// (rows: every step-th)
template <int BC, int NT> __device__ double tile_sum(const double *part, size_t prow, int G, double *sm, int step = 1) {
    constexpr int K = NT / BC;
    const int t = threadIdx.x, jj = t % BC, k = t / BC;
    double v = 0;
    if (k < K)
        for (int b = k; b < G; b += K) v += __ldcg(part + (prow + (size_t)b * step) * BC + jj);
    if (k < K) sm[t] = v;
    __syncthreads();
    double tot = 0;
    if constexpr (BC == 1) { // K = NT values: a tree (a chain of FP64 additions costs 70 cycles each)
        for (int w = NT / 2; w > 0; w >>= 1) {
            if (t < w) sm[t] += sm[t + w];
            __syncthreads();
        }
        tot = sm[0];
    } else if (t < BC) {
        for (int q = 0; q < K; ++q) tot += sm[q * BC + t];
    }
    __syncthreads();
    return tot;
}

// A tile with many blocks sums its rows in two levels (GROUPS): the last block of
// each 64 sums their rows into the first of them, the last of those sums the
// groups.  In one level one SM adds G x BC numbers at 2 FP64 additions a clock:
// for 16^3x32 (G = 6554, 48 columns) 80 us at the end of every launch.  The
// float-float iterations keep one level, and with it the order of their sums: the
// mixed solve's q(x) follows every rounding of alpha there by 1e-9 of its norm.
constexpr int GROUP = 64;
// true in every thread of the block that arrives last of all; nv sums v[q]
template <int BC, int NT, int NV>
__device__ __forceinline__ bool last_in_groups(const Fuse &f, double *const *v, size_t prow, int G, double *sm) {
    const int grp = blockIdx.x / GROUP, first = grp * GROUP, n = min(GROUP, G - first);
    __shared__ int last;
    if (threadIdx.x < BC) __threadfence();
    __syncthreads();
    int *gc = f.gcount + (size_t)blockIdx.y * f.ngroups + grp;
    if (threadIdx.x == 0) {
        last = atomicAdd(gc, 1) == n - 1;
        if (last) *gc = 0;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        const double s = tile_sum<BC, NT>(v[q], prow + first, n, sm);
        if (threadIdx.x < BC) v[q][(prow + first) * BC + threadIdx.x] = s;
    }
    return last_block_of_tile(f.count, (G + GROUP - 1) / GROUP, threadIdx.x < BC);
}

// end of lattice kernel A: the tile's last block runs the first scalar step
// (lattice l, its tile's partial rows from prow)
template <int BC, int NT, bool GROUPS = false>
__device__ __forceinline__ void fuse_step1(const Fuse &f, int l, double *part_t, double *part_p, size_t prow, int G,
                                           double *sm) {
    if (!f.count) return;
    int step = 1;
    if (GROUPS && G > 4 * GROUP) {
        double *const v[2] = {part_t, part_p};
        if (!last_in_groups<BC, NT, 2>(f, v, prow, G, sm)) return;
        step = GROUP;
        G = (G + GROUP - 1) / GROUP;
    } else if (!last_block_of_tile(f.count, G, threadIdx.x < BC)) return;
    const double tt = tile_sum<BC, NT>(part_t, prow, G, sm, step);
    const double pp = tile_sum<BC, NT>(part_p, prow, G, sm, step);
    s1_tile<BC, NT>(blockIdx.y * BC, tt, pp, f.sc, f.sp[l], f.B, sm);
}
// end of lattice kernel B: the tile's last block runs the second scalar step
template <int BC, int NT, bool GROUPS = false>
__device__ __forceinline__ void fuse_step2(const Fuse &f, int l, double *part_r, size_t prow, int G, double *sm) {
    if (!f.count) return;
    int step = 1;
    if (GROUPS && G > 4 * GROUP) {
        double *const v[1] = {part_r};
        if (!last_in_groups<BC, NT, 1>(f, v, prow, G, sm)) return;
        step = GROUP;
        G = (G + GROUP - 1) / GROUP;
    } else if (!last_block_of_tile(f.count, G, threadIdx.x < BC)) return;
    const double rr = tile_sum<BC, NT>(part_r, prow, G, sm, step);
    s2_tile<BC, NT>(blockIdx.y * BC, rr, f.sc, f.sp[l], f.B, f.tol2, f.delta2, f.theta2, sm);
}

// ------------------------------------------------------------------ lattice kernels
template <typename T, int BC>
__global__ void __launch_bounds__(TileMap<BC>::THREADS)
    k_init(Geom g, Source src, typename cplx_t<T>::type *r, typename cplx_t<T>::type *p,
           typename cplx_t<T>::type *xlo, df64c *xhi, double *part, int G) {
    typedef typename cplx_t<T>::type C;
    __shared__ double sm[TileMap<BC>::THREADS];
    const int jj = threadIdx.x % BC, chunk = blockIdx.y, j = chunk * BC + jj;
    const size_t base = (size_t)chunk * 12 * g.V * BC + jj;
    const int ntiles = (g.V + TileMap<BC>::SPB - 1) / TileMap<BC>::SPB;
    double acc = 0;
    for (int tile = blockIdx.x * TPB, tend = min(ntiles, tile + TPB); tile < tend; ++tile) {
        int s = tile * TileMap<BC>::SPB + threadIdx.x / BC;
        if (s >= g.V) continue;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            size_t o = base + ((size_t)s * 12 + c) * BC;
            double2 b = source_at<BC>(src, g.V, s, c, j, o);
            C v = mkc<C>(b.x, b.y);
            r[o] = v;
            p[o] = v;
            if (xlo) xlo[o] = mkc<C>(0, 0);
            if (xhi) xhi[o] = df64c{df64(0.f), df64(0.f)};
            acc += b.x * b.x + b.y * b.y;
        }
    }
    double s = block_sum<BC>(acc, sm);
    if (threadIdx.x < BC) part[((size_t)chunk * G + blockIdx.x) * BC + threadIdx.x] = s;
}

// per-column sums over a block of the NR-column kernels (sites x columns in
// shared memory, then a fixed-order sum down each column); threads < BC return
// the total of column threadIdx.x
template <int BC, int NR>
__device__ __forceinline__ double block_sum_cols(const double v[NR], double *sm) {
    constexpr int TPS = TileMap<BC, NR>::TPS, SPB = TileMap<BC, NR>::SPB;
    const int row = threadIdx.x / TPS, col0 = (threadIdx.x % TPS) * NR;
#pragma unroll
    for (int r = 0; r < NR; ++r) sm[row * BC + col0 + r] = v[r];
    __syncthreads();
    double s = 0;
    if (threadIdx.x < BC)
        for (int k = 0; k < SPB; ++k) s += sm[k * BC + threadIdx.x];
    __syncthreads();
    return s;
}

template <int BC, int NR>
__device__ __forceinline__ double block_total(const double v[NR], double *sm) {
    if constexpr (NR == 1) return block_sum<BC>(v[0], sm);
    else return block_sum_cols<BC, NR>(v, sm);
}

template <int BC, int NR> struct SmemCols {
    static constexpr int N = TileMap<BC, NR>::THREADS > TileMap<BC, NR>::SPB * BC ? TileMap<BC, NR>::THREADS
                                                                                   : TileMap<BC, NR>::SPB * BC;
};

// t = D_W p ; partials |t|^2 -> part_t, |p|^2 -> part_p (NR columns per thread)
template <typename T, int BC, int NR, bool M>
__global__ void __launch_bounds__(TileMap<BC, NR>::THREADS, MinBlocks<T>::value)
    k_apply_a(Lats L, const typename cplx_t<T>::type *__restrict__ p, typename cplx_t<T>::type *__restrict__ t,
              double kd, double *part_t, double *part_p, int tpb, Fuse f) {
    typedef typename cplx_t<T>::type C;
    typedef TileMap<BC, NR> TM;
    const T kappa = (T)kd;
    __shared__ double sm[SmemCols<BC, NR>::N];
    const int l = lat_index<M>(L);
    const Lat &la = L.l[l];
    if ((int)blockIdx.x >= la.G) return; // beyond this lattice's blocks (uneven batch)
    const Geom &g = la.g;
    const C *__restrict__ U = (const C *)la.U;
    const int G = la.G, cl = blockIdx.y - la.chunk0;
    const size_t prow = la.p0 + (size_t)cl * G;
    const int jj = (threadIdx.x % TM::TPS) * NR;
    const size_t base = la.f0 + (size_t)cl * 12 * g.V * BC + jj;
    const int ntiles = (g.V + TM::SPB - 1) / TM::SPB;
    double at[NR], ap[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) at[r] = ap[r] = 0;
    for (int tile = blockIdx.x * tpb, tend = min(ntiles, tile + tpb); tile < tend; ++tile) {
        int s = tile * TM::SPB + threadIdx.x / TM::TPS;
        if (s >= g.V) continue;
        C acc[12][NR];
        wilson_hop_auto<T, false, BC, NR>(g, U, p + base, s, acc);
        T st[NR], sp[NR]; // per-site sums in the iteration precision, one FP64 add per site
#pragma unroll
        for (int r = 0; r < NR; ++r) st[r] = sp[r] = 0;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            size_t o = base + ((size_t)s * 12 + c) * BC;
            C v[NR];
            Cols<C, NR>::load(p + o, v);
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                sp[r] += v[r].x * v[r].x + v[r].y * v[r].y;
                v[r].x -= kappa * acc[c][r].x;
                v[r].y -= kappa * acc[c][r].y;
                st[r] += v[r].x * v[r].x + v[r].y * v[r].y;
            }
            Cols<C, NR>::store(t + o, v);
        }
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            at[r] += (double)st[r];
            ap[r] += (double)sp[r];
        }
    }
    double s1 = block_total<BC, NR>(at, sm);
    double s2 = block_total<BC, NR>(ap, sm);
    if (threadIdx.x < BC) {
        part_t[(prow + blockIdx.x) * BC + threadIdx.x] = s1;
        part_p[(prow + blockIdx.x) * BC + threadIdx.x] = s2;
    }
    fuse_step1<BC, TM::THREADS, !std::is_same<T, df64>::value>(f, l, part_t, part_p, prow, G, sm);
}

// r -= alpha (D_W^dag t + s0 p); partial |r|^2 (NR columns per thread)
template <typename T, int BC, int NR, bool M>
__global__ void __launch_bounds__(TileMap<BC, NR>::THREADS, MinBlocks<T>::value)
    k_apply_b(Lats L, const typename cplx_t<T>::type *__restrict__ t, const typename cplx_t<T>::type *__restrict__ p,
              typename cplx_t<T>::type *__restrict__ r, const double *__restrict__ alpha, double kd, double *part_r,
              int tpb, Fuse f) {
    typedef typename cplx_t<T>::type C;
    typedef TileMap<BC, NR> TM;
    const T kappa = (T)kd;
    __shared__ double sm[SmemCols<BC, NR>::N];
    const int l = lat_index<M>(L);
    const Lat &la = L.l[l];
    if ((int)blockIdx.x >= la.G) return;
    const Geom &g = la.g;
    const C *__restrict__ U = (const C *)la.U;
    const int G = la.G, cl = blockIdx.y - la.chunk0;
    const size_t prow = la.p0 + (size_t)cl * G;
    const double s0 = la.s0;
    const int jj = (threadIdx.x % TM::TPS) * NR, j = blockIdx.y * BC + jj;
    const size_t base = la.f0 + (size_t)cl * 12 * g.V * BC + jj;
    const int ntiles = (g.V + TM::SPB - 1) / TM::SPB;
    T a[NR];
#pragma unroll
    for (int q = 0; q < NR; ++q) a[q] = (T)alpha[j + q];
    const T sh = (T)s0;
    double ar[NR];
#pragma unroll
    for (int q = 0; q < NR; ++q) ar[q] = 0;
    for (int tile = blockIdx.x * tpb, tend = min(ntiles, tile + tpb); tile < tend; ++tile) {
        int s = tile * TM::SPB + threadIdx.x / TM::TPS;
        if (s >= g.V) continue;
        C acc[12][NR];
        wilson_hop_auto<T, true, BC, NR>(g, U, t + base, s, acc);
        T sr[NR];
#pragma unroll
        for (int q = 0; q < NR; ++q) sr[q] = 0;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            size_t o = base + ((size_t)s * 12 + c) * BC;
            C tv[NR], pv[NR], rv[NR];
            Cols<C, NR>::load(t + o, tv);
            Cols<C, NR>::load(p + o, pv);
            Cols<C, NR>::load(r + o, rv);
#pragma unroll
            for (int q = 0; q < NR; ++q) {
                C ap;
                ap.x = tv[q].x - kappa * acc[c][q].x + sh * pv[q].x;
                ap.y = tv[q].y - kappa * acc[c][q].y + sh * pv[q].y;
                rv[q].x -= a[q] * ap.x;
                rv[q].y -= a[q] * ap.y;
                sr[q] += rv[q].x * rv[q].x + rv[q].y * rv[q].y;
            }
            Cols<C, NR>::store(r + o, rv);
        }
#pragma unroll
        for (int q = 0; q < NR; ++q) ar[q] += (double)sr[q];
    }
    double s1 = block_total<BC, NR>(ar, sm);
    if (threadIdx.x < BC) part_r[(prow + blockIdx.x) * BC + threadIdx.x] = s1;
    fuse_step2<BC, TM::THREADS, !std::is_same<T, df64>::value>(f, l, part_r, prow, G, sm);
}

// ------------------------------------------------------------------ FP32 D_W pair, neighbours staged
// k_apply_a / k_apply_b for FP32 iterations (one column per thread) with the
// neighbour sites brought into shared memory by bulk asynchronous copies
// (stage.cuh): the same arithmetic in the same order, NS stages of SPB sites
// in dynamic shared memory, *err set if a copy wait runs out.
// three 240-thread blocks per SM (<= 91 registers a thread; 3 x 71 KB of shared memory)
template <int BC, bool M>
__global__ void __launch_bounds__(TileMap<BC>::THREADS, 3)
    k_apply_a_st(Lats L, const float2 *__restrict__ p, float2 *__restrict__ t, double kd, double *part_t,
                 double *part_p, int tpb, Fuse f, int *err) {
    typedef TileMap<BC> TM;
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ double sm[SmemCols<BC, 1>::N];
    const int l = lat_index<M>(L);
    const Lat &la = L.l[l];
    if ((int)blockIdx.x >= la.G) return;
    const Geom &g = la.g;
    const int G = la.G, cl = blockIdx.y - la.chunk0;
    const size_t prow = la.p0 + (size_t)cl * G;
    const int jj = threadIdx.x % BC;
    const size_t tb = la.f0 + (size_t)cl * 12 * g.V * BC; // this RHS tile of the fields
    const int ntiles = (g.V + TM::SPB - 1) / TM::SPB;
    const int tile0 = blockIdx.x * tpb, ntb = min(ntiles, tile0 + tpb) - tile0;
    const float kappa = (float)kd;
    stage::Runner<false, BC, stage::NSTAGE> run(dsm, g, (const float2 *)la.U, p + tb, tile0, ntb, err);
    double at = 0, ap = 0;
    for (int tl = 0; tl < ntb; ++tl) {
        const int s = (tile0 + tl) * TM::SPB + threadIdx.x / BC;
        const bool valid = s < g.V;
        float2 acc[12][1];
        run.hops(tl, s, valid, acc);
        if (!valid) continue;
        float st = 0, sp = 0;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const size_t o = tb + ((size_t)s * 12 + c) * BC + jj;
            float2 v = p[o];
            sp += v.x * v.x + v.y * v.y;
            v.x -= kappa * acc[c][0].x;
            v.y -= kappa * acc[c][0].y;
            st += v.x * v.x + v.y * v.y;
            t[o] = v;
        }
        at += (double)st;
        ap += (double)sp;
    }
    const double s1 = block_sum<BC>(at, sm);
    const double s2 = block_sum<BC>(ap, sm);
    if (threadIdx.x < BC) {
        part_t[(prow + blockIdx.x) * BC + threadIdx.x] = s1;
        part_p[(prow + blockIdx.x) * BC + threadIdx.x] = s2;
    }
    fuse_step1<BC, TM::THREADS, true>(f, l, part_t, part_p, prow, G, sm);
}

template <int BC, bool M>
__global__ void __launch_bounds__(TileMap<BC>::THREADS, 3)
    k_apply_b_st(Lats L, const float2 *__restrict__ t, const float2 *__restrict__ p, float2 *__restrict__ r,
                 const double *__restrict__ alpha, double kd, double *part_r, int tpb, Fuse f, int *err) {
    typedef TileMap<BC> TM;
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ double sm[SmemCols<BC, 1>::N];
    const int l = lat_index<M>(L);
    const Lat &la = L.l[l];
    if ((int)blockIdx.x >= la.G) return;
    const Geom &g = la.g;
    const int G = la.G, cl = blockIdx.y - la.chunk0;
    const size_t prow = la.p0 + (size_t)cl * G;
    const int jj = threadIdx.x % BC, j = blockIdx.y * BC + jj;
    const size_t tb = la.f0 + (size_t)cl * 12 * g.V * BC;
    const int ntiles = (g.V + TM::SPB - 1) / TM::SPB;
    const int tile0 = blockIdx.x * tpb, ntb = min(ntiles, tile0 + tpb) - tile0;
    const float a = (float)alpha[j], sh = (float)la.s0, kappa = (float)kd;
    stage::Runner<true, BC, stage::NSTAGE> run(dsm, g, (const float2 *)la.U, t + tb, tile0, ntb, err);
    double ar = 0;
    for (int tl = 0; tl < ntb; ++tl) {
        const int s = (tile0 + tl) * TM::SPB + threadIdx.x / BC;
        const bool valid = s < g.V;
        float2 acc[12][1];
        run.hops(tl, s, valid, acc);
        if (!valid) continue;
        float sr = 0;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const size_t o = tb + ((size_t)s * 12 + c) * BC + jj;
            const float2 tv = t[o], pv = p[o];
            float2 rv = r[o];
            const float apx = tv.x - kappa * acc[c][0].x + sh * pv.x;
            const float apy = tv.y - kappa * acc[c][0].y + sh * pv.y;
            rv.x -= a * apx;
            rv.y -= a * apy;
            sr += rv.x * rv.x + rv.y * rv.y;
            r[o] = rv;
        }
        ar += (double)sr;
    }
    const double s1 = block_sum<BC>(ar, sm);
    if (threadIdx.x < BC) part_r[(prow + blockIdx.x) * BC + threadIdx.x] = s1;
    fuse_step2<BC, TM::THREADS, true>(f, l, part_r, prow, G, sm);
}

// The float-float pair (the first phase of SMPQ_MIXED) with staged neighbours
// and links (stage.cuh, two stages): the epilogues of k_apply_a / k_apply_b.
template <int BC, bool M>
__global__ void __launch_bounds__(TileMap<BC>::THREADS, MinBlocks<df64>::value)
    k_apply_a_dfst(Lats L, const df64c *__restrict__ p, df64c *__restrict__ t, df64 kappa, double *part_t,
                   double *part_p, int tpb, Fuse f, int *err) {
    typedef TileMap<BC> TM;
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ double sm[SmemCols<BC, 1>::N];
    const int l = lat_index<M>(L);
    const Lat &la = L.l[l];
    if ((int)blockIdx.x >= la.G) return;
    const Geom &g = la.g;
    const int G = la.G, cl = blockIdx.y - la.chunk0;
    const size_t prow = la.p0 + (size_t)cl * G;
    const int jj = threadIdx.x % BC;
    const size_t tb = la.f0 + (size_t)cl * 12 * g.V * BC;
    const int ntiles = (g.V + TM::SPB - 1) / TM::SPB;
    const int tile0 = blockIdx.x * tpb, ntb = min(ntiles, tile0 + tpb) - tile0;
    stage::RunnerDF<false, BC, stage::NSTAGE_DF> run(dsm, g, (const df64c *)la.U, p + tb, tile0, ntb, err);
    double at = 0, ap = 0;
    for (int tl = 0; tl < ntb; ++tl) {
        const int s = (tile0 + tl) * TM::SPB + threadIdx.x / BC;
        const bool valid = s < g.V;
        df64c acc[12][1];
        run.hops(tl, s, valid, acc);
        if (!valid) continue;
        df64 st = 0, sp = 0;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const size_t o = tb + ((size_t)s * 12 + c) * BC + jj;
            df64c v = p[o];
            sp += v.x * v.x + v.y * v.y;
            v.x -= kappa * acc[c][0].x;
            v.y -= kappa * acc[c][0].y;
            st += v.x * v.x + v.y * v.y;
            t[o] = v;
        }
        at += (double)st;
        ap += (double)sp;
    }
    const double s1 = block_sum<BC>(at, sm);
    const double s2 = block_sum<BC>(ap, sm);
    if (threadIdx.x < BC) {
        part_t[(prow + blockIdx.x) * BC + threadIdx.x] = s1;
        part_p[(prow + blockIdx.x) * BC + threadIdx.x] = s2;
    }
    fuse_step1<BC, TM::THREADS, false>(f, l, part_t, part_p, prow, G, sm);
}

template <int BC, bool M>
__global__ void __launch_bounds__(TileMap<BC>::THREADS, MinBlocks<df64>::value)
    k_apply_b_dfst(Lats L, const df64c *__restrict__ t, const df64c *__restrict__ p, df64c *__restrict__ r,
                   const double *__restrict__ alpha, df64 kappa, double *part_r, int tpb, Fuse f, int *err) {
    typedef TileMap<BC> TM;
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ double sm[SmemCols<BC, 1>::N];
    const int l = lat_index<M>(L);
    const Lat &la = L.l[l];
    if ((int)blockIdx.x >= la.G) return;
    const Geom &g = la.g;
    const int G = la.G, cl = blockIdx.y - la.chunk0;
    const size_t prow = la.p0 + (size_t)cl * G;
    const int jj = threadIdx.x % BC, j = blockIdx.y * BC + jj;
    const size_t tb = la.f0 + (size_t)cl * 12 * g.V * BC;
    const int ntiles = (g.V + TM::SPB - 1) / TM::SPB;
    const int tile0 = blockIdx.x * tpb, ntb = min(ntiles, tile0 + tpb) - tile0;
    const df64 a(alpha[j]), sh(la.s0);
    stage::RunnerDF<true, BC, stage::NSTAGE_DF> run(dsm, g, (const df64c *)la.U, t + tb, tile0, ntb, err);
    double ar = 0;
    for (int tl = 0; tl < ntb; ++tl) {
        const int s = (tile0 + tl) * TM::SPB + threadIdx.x / BC;
        const bool valid = s < g.V;
        df64c acc[12][1];
        run.hops(tl, s, valid, acc);
        if (!valid) continue;
        df64 sr = 0;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const size_t o = tb + ((size_t)s * 12 + c) * BC + jj;
            const df64c tv = t[o], pv = p[o];
            df64c rv = r[o];
            df64c apv;
            apv.x = tv.x - kappa * acc[c][0].x + sh * pv.x;
            apv.y = tv.y - kappa * acc[c][0].y + sh * pv.y;
            rv.x -= a * apv.x;
            rv.y -= a * apv.y;
            sr += rv.x * rv.x + rv.y * rv.y;
            r[o] = rv;
        }
        ar += (double)sr;
    }
    const double s1 = block_sum<BC>(ar, sm);
    if (threadIdx.x < BC) part_r[(prow + blockIdx.x) * BC + threadIdx.x] = s1;
    fuse_step2<BC, TM::THREADS, false>(f, l, part_r, prow, G, sm);
}

template <int BC, bool M> cudaError_t staged_df_attrs() {
    static bool done = false;
    if (done) return cudaSuccess;
    const int bytes = (int)stage::DimsDF<BC, stage::NSTAGE_DF>::SMEM;
    cudaError_t e = cudaFuncSetAttribute(k_apply_a_dfst<BC, M>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_apply_b_dfst<BC, M>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    done = e == cudaSuccess;
    return e;
}

// the dynamic shared memory of the staged pair (above the 48 KB default)
template <int BC, bool M> cudaError_t staged_attrs() {
    static bool done = false;
    if (done) return cudaSuccess;
    const int bytes = (int)stage::Dims<BC, stage::NSTAGE>::SMEM;
    cudaError_t e = cudaFuncSetAttribute(k_apply_a_st<BC, M>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_apply_b_st<BC, M>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    done = e == cudaSuccess;
    return e;
}

// The base system's solution x accumulated by the p update: FP64 for the FP64
// iterations (the true-residual check), float-float for the FP64-accurate
// first phase of the mixed solve (the x_hi its FP32 phase's reliable updates
// continue from).
template <typename T> struct XAcc { typedef double2 type; };
template <> struct XAcc<df64> { typedef df64c type; };

// p = r + beta p on the lattice tiles of tile group bx; with x64, first
// x64 += alpha p, with xlo, first xlo += alpha p in T (the part of the base
// solution that the next residual replacement folds into x_hi)
// (tile0: first element of the block's RHS tile in the fields; the tile is
// blockIdx.y of the solve, so rhs j = blockIdx.y * BC + column)
template <typename T, int BC>
__device__ __forceinline__ void update_p_tiles(int bx, int tpb, int V, size_t tile0,
                                               const typename cplx_t<T>::type *__restrict__ r,
                                               typename cplx_t<T>::type *__restrict__ p, const Scal &sc,
                                               typename XAcc<T>::type *__restrict__ x64,
                                               typename cplx_t<T>::type *__restrict__ xlo) {
    typedef typename cplx_t<T>::type C;
    const int jj = threadIdx.x % BC, j = blockIdx.y * BC + jj;
    if (!sc.upd_rhs[j]) return;
    const size_t base = tile0 + jj;
    const int ntiles = (V + TileMap<BC>::SPB - 1) / TileMap<BC>::SPB;
    const T b = (T)sc.beta[j];
    const double a = sc.alpha[j];
    for (int tile = bx * tpb, tend = min(ntiles, tile + tpb); tile < tend; ++tile) {
        int s = tile * TileMap<BC>::SPB + threadIdx.x / BC;
        if (s >= V) continue;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            size_t o = base + ((size_t)s * 12 + c) * BC;
            C rv = r[o], pv = p[o];
            if (xlo) {
                C xv = xlo[o];
                xv.x += (T)a * pv.x;
                xv.y += (T)a * pv.y;
                xlo[o] = xv;
            }
            if (x64) {
                if constexpr (std::is_same<T, df64>::value) {
                    df64c xv = x64[o];
                    const df64 ad(a);
                    xv.x = fma_df(ad, pv.x, xv.x);
                    xv.y = fma_df(ad, pv.y, xv.y);
                    x64[o] = xv;
                } else {
                    double2 xv = x64[o];
                    xv.x += a * to_d(pv.x);
                    xv.y += a * to_d(pv.y);
                    x64[o] = xv;
                }
            }
            pv.x = rv.x + b * pv.x;
            pv.y = rv.y + b * pv.y;
            p[o] = pv;
        }
    }
}

// ------------------------------------------------------------------ FP64 iterations
// SMPQ_FP64: p, t and r in block fixed point (bfp.cuh), one thread per site and
// column.  Bound by the integer pipe: 300 us a launch for 72 columns of 8^3x16
// (1340 us in FP64 arithmetic); 24 576 sites and columns take 30 us (325 us in
// blocks of 256 threads, 4 tiles each: 24 blocks on 152 SMs).
template <int BC>
__global__ void __launch_bounds__(BfMap<BC>::THREADS)
    k_init_bf(Geom g, Source src, BFF r, BFF p, double *part, int G) {
    typedef BfMap<BC> TM;
    __shared__ double sm[2 * TM::THREADS];
    const int jj = threadIdx.x % BC, chunk = blockIdx.y, j = chunk * BC + jj;
    const size_t base = (size_t)chunk * 12 * g.V * BC + jj, ebase = (size_t)chunk * g.V * BC + jj;
    const BfOff<BC> off{g.V};
    const int s = blockIdx.x * TM::SPB + threadIdx.x / BC;
    double acc = 0;
    if (s < g.V) {
        double2 b[12];
        bfc v[12];
        int e;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            b[c] = source_at<BC>(src, g.V, s, c, j, base + ((size_t)s * 12 + c) * BC);
            acc += b[c].x * b[c].x + b[c].y * b[c].y;
        }
        bf_from_double(b, v, e);
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            r.v[base + off(s, c)] = v[c];
            p.v[base + off(s, c)] = v[c];
        }
        r.e[ebase + off.exp(s)] = e;
        p.e[ebase + off.exp(s)] = e;
    }
    const double sum = block_sum<BC, TM::THREADS>(acc, sm);
    if (threadIdx.x < BC) part[((size_t)chunk * G + blockIdx.x) * BC + threadIdx.x] = sum;
}

// t = D_W p; partials |t|^2, |p|^2
template <int BC, bool M>
__global__ void __launch_bounds__(BfMap<BC>::THREADS, BfMap<BC>::BLOCKS)
    k_apply_a_bf(Lats L, BFF p, BFF t, BfScal kappa, double *part_t, double *part_p, int tpb, Fuse f) {
    typedef BfMap<BC> TM;
    __shared__ double sm[2 * TM::THREADS];
    const int l = lat_index<M>(L);
    const Lat &la = L.l[l];
    if ((int)blockIdx.x >= la.G) return;
    const Geom &g = la.g;
    const int G = la.G, cl = blockIdx.y - la.chunk0;
    const size_t prow = la.p0 + (size_t)cl * G;
    const int jj = threadIdx.x % BC;
    const size_t base = la.f0 + (size_t)cl * 12 * g.V * BC + jj, ebase = la.f0 / 12 + (size_t)cl * g.V * BC + jj;
    const BfOff<BC> off{g.V};
    const int ntiles = (g.V + TM::SPB - 1) / TM::SPB;
    const int one = opaque_one();
    double at = 0, ap = 0;
    for (int tile = blockIdx.x * tpb, tend = min(ntiles, tile + tpb); tile < tend; ++tile) {
        const int s = tile * TM::SPB + threadIdx.x / BC;
        if (s >= g.V) continue;
        bfc acc[12], own[12];
        int eown, eref, e;
        bf_wilson<false>(g, (const int4 *)la.U, p.v + base, p.e + ebase, off, s, one, acc, eown, eref);
#pragma unroll
        for (int c = 0; c < 12; ++c) own[c] = p.v[base + off(s, c)];
        ap += bf_norm2(own, eown, one);
        bf_dw<12>(own, eown, acc, eref, kappa, eown + 2, one, acc, e);
        bf_normalise(acc, e);
        at += bf_norm2(acc, e, one);
#pragma unroll
        for (int c = 0; c < 12; ++c) t.v[base + off(s, c)] = acc[c];
        t.e[ebase + off.exp(s)] = e;
    }
    const double s1 = block_sum<BC, TM::THREADS>(at, sm);
    const double s2 = block_sum<BC, TM::THREADS>(ap, sm);
    if (threadIdx.x < BC) {
        part_t[(prow + blockIdx.x) * BC + threadIdx.x] = s1;
        part_p[(prow + blockIdx.x) * BC + threadIdx.x] = s2;
    }
    fuse_step1<BC, TM::THREADS, true>(f, l, part_t, part_p, prow, G, sm);
}

// r -= alpha (D_W^dag t + s0 p); partial |r|^2
template <int BC, bool M>
__global__ void __launch_bounds__(BfMap<BC>::THREADS, BfMap<BC>::BLOCKS)
    k_apply_b_bf(Lats L, BFF t, BFF p, BFF r, const double *__restrict__ alpha, BfScal kappa, double *part_r, int tpb,
                 Fuse f) {
    typedef BfMap<BC> TM;
    __shared__ double sm[2 * TM::THREADS];
    const int l = lat_index<M>(L);
    const Lat &la = L.l[l];
    if ((int)blockIdx.x >= la.G) return;
    const Geom &g = la.g;
    const int G = la.G, cl = blockIdx.y - la.chunk0;
    const size_t prow = la.p0 + (size_t)cl * G;
    const int jj = threadIdx.x % BC, j = blockIdx.y * BC + jj;
    const size_t base = la.f0 + (size_t)cl * 12 * g.V * BC + jj, ebase = la.f0 / 12 + (size_t)cl * g.V * BC + jj;
    const BfOff<BC> off{g.V};
    const int ntiles = (g.V + TM::SPB - 1) / TM::SPB;
    const int one = opaque_one();
    const BfScal s0 = bf_scal(la.s0), a = bf_scal(alpha[j]);
    double ar = 0;
    for (int tile = blockIdx.x * tpb, tend = min(ntiles, tile + tpb); tile < tend; ++tile) {
        const int s = tile * TM::SPB + threadIdx.x / BC;
        if (s >= g.V) continue;
        bfc acc[12], own[12];
        int eown, eref, eu;
        bf_wilson<true>(g, (const int4 *)la.U, t.v + base, t.e + ebase, off, s, one, acc, eown, eref);
#pragma unroll
        for (int c = 0; c < 12; ++c) own[c] = t.v[base + off(s, c)];
        // the unit of A p = D_W^dag t + s0 p: its last term takes part in the choice
        const int ep = p.e[ebase + off.exp(s)], ew = ep + s0.e + 64;
        bf_dw<12>(own, eown, acc, eref, kappa, max(eown + 3, ew + 1), one, acc, eu);
        const int nw = eu - ew;
        // r - alpha A p
        int er = r.e[ebase + off.exp(s)];
        const int ez = eu + a.e + 64, em = max(ez, er + 2), nz = em - ez, nr = em - er;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const size_t o = base + off(s, c);
            const bfc pv = p.v[o], rv = r.v[o];
            const long long x = acc[c].x + bf_shr(bf_mul(pv.x, s0, one), nw),
                            y = acc[c].y + bf_shr(bf_mul(pv.y, s0, one), nw);
            acc[c] = {bf_shr(rv.x, nr) - bf_shr(bf_mul(x, a, one), nz),
                      bf_shr(rv.y, nr) - bf_shr(bf_mul(y, a, one), nz)};
        }
        er = max(eu, max(er, ep)) >= BF_BAD / 2 || a.e >= BF_BAD / 2 ? BF_BAD : em;
        bf_normalise(acc, er);
        ar += bf_norm2(acc, er, one);
#pragma unroll
        for (int c = 0; c < 12; ++c) r.v[base + off(s, c)] = acc[c];
        r.e[ebase + off.exp(s)] = er;
    }
    const double s1 = block_sum<BC, TM::THREADS>(ar, sm);
    if (threadIdx.x < BC) part_r[(prow + blockIdx.x) * BC + threadIdx.x] = s1;
    fuse_step2<BC, TM::THREADS, true>(f, l, part_r, prow, G, sm);
}

// Launch YP of an FP64 iteration: r on the support into the history (as
// doubles), p = r + beta p and, with x64, first x64 += alpha p on the lattice
// (x64 in the tile layout).  tpb tiles of BfMap per block.
template <int BC, bool M>
__global__ void __launch_bounds__(BfMap<BC>::THREADS, 640 / BfMap<BC>::THREADS)
    k_yp_bf(Lats L, int tpb, const int *__restrict__ rhs_class, BFF r, double2 *__restrict__ h, size_t stride, Scal sc,
            BFF p, double2 *__restrict__ x64) {
    typedef BfMap<BC> TM;
    const int l = lat_index<M>(L);
    const Lat &la = L.l[l];
    const int cl = blockIdx.y - la.chunk0, V = la.g.V;
    const int jj = threadIdx.x % BC, j = blockIdx.y * BC + jj;
    if (!sc.upd_rhs[j]) return;
    const size_t base = la.f0 + (size_t)cl * 12 * V * BC + jj, ebase = la.f0 / 12 + (size_t)cl * V * BC + jj;
    const BfOff<BC> off{V};
    if ((int)blockIdx.x < la.Gs) {
        const int cls = rhs_class[j];
        if (cls < 0) return;
        double2 *o = h + la.sup0 + (size_t)(sc.slot[j] - 1) * stride + (size_t)cl * 12 * la.n_sup * BC + jj;
        const int nt = (la.n_sup + TM::SPB - 1) / TM::SPB;
        for (int tile = blockIdx.x * tpb, tend = min(nt, tile + tpb); tile < tend; ++tile) {
            const int k = tile * TM::SPB + threadIdx.x / BC;
            if (k >= la.n_sup) continue;
            const int site = la.supsite ? la.supsite[(size_t)cls * la.n_sup + k] : k;
            const int e = r.e[ebase + off.exp(site)];
            bfc v[12];
#pragma unroll
            for (int c = 0; c < 12; ++c) v[c] = r.v[base + off(site, c)];
#pragma unroll
            for (int c = 0; c < 12; ++c)
                o[((size_t)k * 12 + c) * BC] = make_double2(bf_double(v[c].x, e), bf_double(v[c].y, e));
        }
        return;
    }
    const int bx = blockIdx.x - la.Gs;
    if (bx >= la.G) return;
    const int nt = (V + TM::SPB - 1) / TM::SPB;
    const int one = opaque_one();
    const BfScal b = bf_scal(sc.beta[j]);
    const double al = sc.alpha[j];
    for (int tile = bx * tpb, tend = min(nt, tile + tpb); tile < tend; ++tile) {
        const int s = tile * TM::SPB + threadIdx.x / BC;
        if (s >= V) continue;
        const int er = r.e[ebase + off.exp(s)];
        int ep = p.e[ebase + off.exp(s)];
        const int ez = ep + b.e + 64, em = max(ez, er + 2), nz = em - ez, nr = em - er;
        bfc v[12], rv[12];
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            rv[c] = r.v[base + off(s, c)];
            v[c] = p.v[base + off(s, c)];
        }
        if (x64)
#pragma unroll
            for (int c = 0; c < 12; ++c) {
                double2 &x = x64[base + ((size_t)s * 12 + c) * BC];
                x = make_double2(fma(al, bf_double(v[c].x, ep), x.x), fma(al, bf_double(v[c].y, ep), x.y));
            }
#pragma unroll
        for (int c = 0; c < 12; ++c)
            v[c] = {bf_shr(rv[c].x, nr) + bf_shr(bf_mul(v[c].x, b, one), nz),
                    bf_shr(rv[c].y, nr) + bf_shr(bf_mul(v[c].y, b, one), nz)};
        ep = max(er, ep) >= BF_BAD / 2 || b.e >= BF_BAD / 2 ? BF_BAD : em;
        bf_normalise(v, ep);
#pragma unroll
        for (int c = 0; c < 12; ++c) p.v[base + off(s, c)] = v[c];
        p.e[ebase + off.exp(s)] = ep;
    }
}

// ------------------------------------------------------------------ half-storage iterations
// SMPQ_FP16N / SMPQ_BF16N: the FP32 path (FP64 reliable updates, FP32 r, x_lo
// and shifted directions) with p and t -- the input and output of D_W --
// stored in the half format of half.cuh and the links in reconstruct-12 form.
// One thread per site and column (TileMap<BC>), FP32 arithmetic.
template <typename HT> struct HF {
    typename HT::h2 *v; // components, tiled like the FP32 fields
    float *n;           // norms [j / BC][V][BC]
};
template <typename HT> struct HLinks;
template <> struct HLinks<H16> { static const void *get(const smpq_ctx *c) { return c->Uh16.p; } };
template <> struct HLinks<B16> { static const void *get(const smpq_ctx *c) { return c->Ub16.p; } };

// r = p = b (p in the half format), x_lo = x_hi = 0; partial |b|^2
template <typename HT, int BC>
__global__ void __launch_bounds__(TileMap<BC>::THREADS)
    k_init_h(Geom g, Source src, float2 *r, HF<HT> p, float2 *xlo, df64c *xhi, double *part, int G) {
    __shared__ double sm[TileMap<BC>::THREADS];
    const int jj = threadIdx.x % BC, chunk = blockIdx.y, j = chunk * BC + jj;
    const size_t base = (size_t)chunk * 12 * g.V * BC + jj, nbase = (size_t)chunk * g.V * BC + jj;
    const int ntiles = (g.V + TileMap<BC>::SPB - 1) / TileMap<BC>::SPB;
    double acc = 0;
    for (int tile = blockIdx.x * TPB, tend = min(ntiles, tile + TPB); tile < tend; ++tile) {
        const int s = tile * TileMap<BC>::SPB + threadIdx.x / BC;
        if (s >= g.V) continue;
        float2 v[12];
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const size_t o = base + ((size_t)s * 12 + c) * BC;
            const double2 b = source_at<BC>(src, g.V, s, c, j, o);
            v[c] = make_float2((float)b.x, (float)b.y);
            r[o] = v[c];
            xlo[o] = make_float2(0.f, 0.f);
            xhi[o] = df64c{df64(0.f), df64(0.f)};
            acc += b.x * b.x + b.y * b.y;
        }
        st_site_half<HT, BC>(p.v + base + (size_t)s * 12 * BC, p.n + nbase + (size_t)s * BC, v);
    }
    const double t = block_sum<BC>(acc, sm);
    if (threadIdx.x < BC) part[((size_t)chunk * G + blockIdx.x) * BC + threadIdx.x] = t;
}

// t = D_W p in the half format; partials |t|^2 (before rounding) and |p|^2
template <typename HT, int BC, bool M>
__global__ void __launch_bounds__(TileMap<BC>::THREADS, 3)
    k_apply_a_h(Lats L, HF<HT> p, HF<HT> t, float kappa, double *part_t, double *part_p, int tpb, Fuse f) {
    __shared__ double sm[TileMap<BC>::THREADS];
    const int l = lat_index<M>(L);
    const Lat &la = L.l[l];
    if ((int)blockIdx.x >= la.G) return;
    const Geom &g = la.g;
    const typename HT::h2 *__restrict__ U = (const typename HT::h2 *)la.U;
    const int G = la.G, cl = blockIdx.y - la.chunk0;
    const size_t prow = la.p0 + (size_t)cl * G;
    const int jj = threadIdx.x % BC;
    const size_t base = la.f0 + (size_t)cl * 12 * g.V * BC + jj, nbase = la.f0 / 12 + (size_t)cl * g.V * BC + jj;
    const int ntiles = (g.V + TileMap<BC>::SPB - 1) / TileMap<BC>::SPB;
    double at = 0, ap = 0;
    for (int tile = blockIdx.x * tpb, tend = min(ntiles, tile + tpb); tile < tend; ++tile) {
        const int s = tile * TileMap<BC>::SPB + threadIdx.x / BC;
        if (s >= g.V) continue;
        float2 acc[12][1];
        wilson_hop_half<HT, false, BC>(g, U, p.v + base, p.n + nbase, s, acc);
        const typename HT::h2 *ps = p.v + base + (size_t)s * 12 * BC;
        const float n = p.n[nbase + (size_t)s * BC];
        float sp = 0.f, st = 0.f;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const float2 f = HT::f2(ps[c * BC]);
            const float2 v = make_float2(n * f.x, n * f.y);
            sp += v.x * v.x + v.y * v.y;
            acc[c][0] = make_float2(fmaf(-kappa, acc[c][0].x, v.x), fmaf(-kappa, acc[c][0].y, v.y));
            st += acc[c][0].x * acc[c][0].x + acc[c][0].y * acc[c][0].y;
        }
        float2 w[12];
#pragma unroll
        for (int c = 0; c < 12; ++c) w[c] = acc[c][0];
        st_site_half<HT, BC>(t.v + base + (size_t)s * 12 * BC, t.n + nbase + (size_t)s * BC, w);
        at += (double)st;
        ap += (double)sp;
    }
    const double s1 = block_sum<BC>(at, sm);
    const double s2 = block_sum<BC>(ap, sm);
    if (threadIdx.x < BC) {
        part_t[(prow + blockIdx.x) * BC + threadIdx.x] = s1;
        part_p[(prow + blockIdx.x) * BC + threadIdx.x] = s2;
    }
    fuse_step1<BC, TileMap<BC>::THREADS, true>(f, l, part_t, part_p, prow, G, sm);
}

// r -= alpha (D_W^dag t + s0 p); partial |r|^2
template <typename HT, int BC, bool M>
__global__ void __launch_bounds__(TileMap<BC>::THREADS, 3)
    k_apply_b_h(Lats L, HF<HT> t, HF<HT> p, float2 *__restrict__ r, const double *__restrict__ alpha, float kappa,
                double *part_r, int tpb, Fuse f) {
    __shared__ double sm[TileMap<BC>::THREADS];
    const int l = lat_index<M>(L);
    const Lat &la = L.l[l];
    if ((int)blockIdx.x >= la.G) return;
    const Geom &g = la.g;
    const typename HT::h2 *__restrict__ U = (const typename HT::h2 *)la.U;
    const int G = la.G, cl = blockIdx.y - la.chunk0;
    const size_t prow = la.p0 + (size_t)cl * G;
    const double s0 = la.s0;
    const int jj = threadIdx.x % BC, j = blockIdx.y * BC + jj;
    const size_t base = la.f0 + (size_t)cl * 12 * g.V * BC + jj, nbase = la.f0 / 12 + (size_t)cl * g.V * BC + jj;
    const int ntiles = (g.V + TileMap<BC>::SPB - 1) / TileMap<BC>::SPB;
    const float a = (float)alpha[j], sh = (float)s0;
    double ar = 0;
    for (int tile = blockIdx.x * tpb, tend = min(ntiles, tile + tpb); tile < tend; ++tile) {
        const int s = tile * TileMap<BC>::SPB + threadIdx.x / BC;
        if (s >= g.V) continue;
        float2 acc[12][1];
        wilson_hop_half<HT, true, BC>(g, U, t.v + base, t.n + nbase, s, acc);
        const typename HT::h2 *ts = t.v + base + (size_t)s * 12 * BC, *pq = p.v + base + (size_t)s * 12 * BC;
        const float nt = t.n[nbase + (size_t)s * BC], np = p.n[nbase + (size_t)s * BC];
        float sr = 0.f;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const size_t o = base + ((size_t)s * 12 + c) * BC;
            const float2 tf = HT::f2(ts[c * BC]), pf = HT::f2(pq[c * BC]);
            const float2 pv = make_float2(np * pf.x, np * pf.y);
            float2 apv;
            apv.x = fmaf(sh, pv.x, fmaf(-kappa, acc[c][0].x, nt * tf.x));
            apv.y = fmaf(sh, pv.y, fmaf(-kappa, acc[c][0].y, nt * tf.y));
            float2 rv = r[o];
            rv.x = fmaf(-a, apv.x, rv.x);
            rv.y = fmaf(-a, apv.y, rv.y);
            r[o] = rv;
            sr += rv.x * rv.x + rv.y * rv.y;
        }
        ar += (double)sr;
    }
    const double s1 = block_sum<BC>(ar, sm);
    if (threadIdx.x < BC) part_r[(prow + blockIdx.x) * BC + threadIdx.x] = s1;
    fuse_step2<BC, TileMap<BC>::THREADS, true>(f, l, part_r, prow, G, sm);
}

// p = r + beta p on the lattice tiles of tile group bx, p in the half format
template <typename HT, int BC>
__device__ __forceinline__ void update_p_h_tiles(int bx, int tpb, int V, size_t tile0, const float2 *__restrict__ r,
                                                 HF<HT> p, const Scal &sc, float2 *__restrict__ xlo) {
    const int jj = threadIdx.x % BC, j = blockIdx.y * BC + jj;
    if (!sc.upd_rhs[j]) return;
    const size_t base = tile0 + jj, nbase = tile0 / 12 + jj;
    const int ntiles = (V + TileMap<BC>::SPB - 1) / TileMap<BC>::SPB;
    const float b = (float)sc.beta[j], a = (float)sc.alpha[j];
    for (int tile = bx * tpb, tend = min(ntiles, tile + tpb); tile < tend; ++tile) {
        const int s = tile * TileMap<BC>::SPB + threadIdx.x / BC;
        if (s >= V) continue;
        typename HT::h2 *ps = p.v + base + (size_t)s * 12 * BC;
        float *pn = p.n + nbase + (size_t)s * BC;
        const float n = *pn;
        float2 v[12];
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const size_t o = base + ((size_t)s * 12 + c) * BC;
            const float2 f = HT::f2(ps[c * BC]), rv = r[o];
            if (xlo) { // x_lo += alpha p (p as stored: n times the half value)
                float2 xv = xlo[o];
                xv.x = fmaf(a * n, f.x, xv.x);
                xv.y = fmaf(a * n, f.y, xv.y);
                xlo[o] = xv;
            }
            v[c] = make_float2(fmaf(b * n, f.x, rv.x), fmaf(b * n, f.y, rv.y));
        }
        st_site_half<HT, BC>(ps, pn, v);
    }
}

// Two columns per thread (the packed lanes of half.cuh) forms of k_apply_a_h
// and k_apply_b_h, used for even tile widths: half the FP32 instructions and
// one link reconstruction per two columns; r and x_lo move as 16-byte pairs.
template <int BC> __device__ __forceinline__ void ld_rx2(const float2 *p, float2 &re, float2 &im) {
    const float4 q = *reinterpret_cast<const float4 *>(p);
    re = make_float2(q.x, q.z);
    im = make_float2(q.y, q.w);
}
template <int BC> __device__ __forceinline__ void st_rx2(float2 *p, float2 re, float2 im) {
    *reinterpret_cast<float4 *>(p) = make_float4(re.x, im.x, re.y, im.y);
}

template <typename HT, int BC, bool M>
__global__ void __launch_bounds__(TileMap<BC, 2>::THREADS, 2)
    k_apply_a_h2(Lats L, HF<HT> p, HF<HT> t, float kappa, double *part_t, double *part_p, int tpb, Fuse f) {
    typedef TileMap<BC, 2> TM;
    __shared__ double sm[SmemCols<BC, 2>::N];
    const int l = lat_index<M>(L);
    const Lat &la = L.l[l];
    if ((int)blockIdx.x >= la.G) return;
    const Geom &g = la.g;
    const typename HT::h2 *__restrict__ U = (const typename HT::h2 *)la.U;
    const int G = la.G, cl = blockIdx.y - la.chunk0;
    const size_t prow = la.p0 + (size_t)cl * G;
    const int jj = (threadIdx.x % TM::TPS) * 2;
    const size_t base = la.f0 + (size_t)cl * 12 * g.V * BC + jj, nbase = la.f0 / 12 + (size_t)cl * g.V * BC + jj;
    const int ntiles = (g.V + TM::SPB - 1) / TM::SPB;
    double at[2] = {0, 0}, ap[2] = {0, 0};
    const float2 nk = bc2(-kappa);
    for (int tile = blockIdx.x * tpb, tend = min(ntiles, tile + tpb); tile < tend; ++tile) {
        const int s = tile * TM::SPB + threadIdx.x / TM::TPS;
        if (s >= g.V) continue;
        c2 acc[12];
        wilson_hop_half_c2<HT, false, BC>(g, U, p.v + base, p.n + nbase, s, acc);
        const typename HT::h2 *ps = p.v + base + (size_t)s * 12 * BC;
        const float2 np = *reinterpret_cast<const float2 *>(p.n + nbase + (size_t)s * BC);
        float2 sp = bc2(0.f), st = bc2(0.f);
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const c2 f = ld_c2<HT>(ps + c * BC);
            const float2 vr = __fmul2_rn(np, f.r), vi = __fmul2_rn(np, f.i);
            sp = __ffma2_rn(vr, vr, __ffma2_rn(vi, vi, sp));
            acc[c].r = __ffma2_rn(nk, acc[c].r, vr);
            acc[c].i = __ffma2_rn(nk, acc[c].i, vi);
            st = __ffma2_rn(acc[c].r, acc[c].r, __ffma2_rn(acc[c].i, acc[c].i, st));
        }
        st_site_half_c2<HT, BC>(t.v + base + (size_t)s * 12 * BC, t.n + nbase + (size_t)s * BC, acc);
        at[0] += (double)st.x;
        at[1] += (double)st.y;
        ap[0] += (double)sp.x;
        ap[1] += (double)sp.y;
    }
    const double s1 = block_total<BC, 2>(at, sm);
    const double s2 = block_total<BC, 2>(ap, sm);
    if (threadIdx.x < BC) {
        part_t[(prow + blockIdx.x) * BC + threadIdx.x] = s1;
        part_p[(prow + blockIdx.x) * BC + threadIdx.x] = s2;
    }
    fuse_step1<BC, TM::THREADS, true>(f, l, part_t, part_p, prow, G, sm);
}

template <typename HT, int BC, bool M>
__global__ void __launch_bounds__(TileMap<BC, 2>::THREADS, 2)
    k_apply_b_h2(Lats L, HF<HT> t, HF<HT> p, float2 *__restrict__ r, const double *__restrict__ alpha, float kappa,
                 double *part_r, int tpb, Fuse f) {
    typedef TileMap<BC, 2> TM;
    __shared__ double sm[SmemCols<BC, 2>::N];
    const int l = lat_index<M>(L);
    const Lat &la = L.l[l];
    if ((int)blockIdx.x >= la.G) return;
    const Geom &g = la.g;
    const typename HT::h2 *__restrict__ U = (const typename HT::h2 *)la.U;
    const int G = la.G, cl = blockIdx.y - la.chunk0;
    const size_t prow = la.p0 + (size_t)cl * G;
    const double s0 = la.s0;
    const int jj = (threadIdx.x % TM::TPS) * 2, j = blockIdx.y * BC + jj;
    const size_t base = la.f0 + (size_t)cl * 12 * g.V * BC + jj, nbase = la.f0 / 12 + (size_t)cl * g.V * BC + jj;
    const int ntiles = (g.V + TM::SPB - 1) / TM::SPB;
    const float2 a = make_float2((float)alpha[j], (float)alpha[j + 1]), na = make_float2(-a.x, -a.y);
    const float2 sh = bc2((float)s0), nk = bc2(-kappa);
    double ar[2] = {0, 0};
    for (int tile = blockIdx.x * tpb, tend = min(ntiles, tile + tpb); tile < tend; ++tile) {
        const int s = tile * TM::SPB + threadIdx.x / TM::TPS;
        if (s >= g.V) continue;
        c2 acc[12];
        wilson_hop_half_c2<HT, true, BC>(g, U, t.v + base, t.n + nbase, s, acc);
        const typename HT::h2 *ts = t.v + base + (size_t)s * 12 * BC, *pq = p.v + base + (size_t)s * 12 * BC;
        const float2 nt = *reinterpret_cast<const float2 *>(t.n + nbase + (size_t)s * BC);
        const float2 np = *reinterpret_cast<const float2 *>(p.n + nbase + (size_t)s * BC);
        float2 sr = bc2(0.f);
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const size_t o = base + ((size_t)s * 12 + c) * BC;
            const c2 tf = ld_c2<HT>(ts + c * BC), pf = ld_c2<HT>(pq + c * BC);
            const float2 pr = __fmul2_rn(np, pf.r), pi = __fmul2_rn(np, pf.i);
            // A p = D_W^dag t + s0 p
            const float2 apr = __ffma2_rn(sh, pr, __ffma2_rn(nk, acc[c].r, __fmul2_rn(nt, tf.r)));
            const float2 api = __ffma2_rn(sh, pi, __ffma2_rn(nk, acc[c].i, __fmul2_rn(nt, tf.i)));
            float2 rr, ri;
            ld_rx2<BC>(r + o, rr, ri);
            rr = __ffma2_rn(na, apr, rr);
            ri = __ffma2_rn(na, api, ri);
            st_rx2<BC>(r + o, rr, ri);
            sr = __ffma2_rn(rr, rr, __ffma2_rn(ri, ri, sr));
        }
        ar[0] += (double)sr.x;
        ar[1] += (double)sr.y;
    }
    const double s1 = block_total<BC, 2>(ar, sm);
    if (threadIdx.x < BC) part_r[(prow + blockIdx.x) * BC + threadIdx.x] = s1;
    fuse_step2<BC, TM::THREADS, true>(f, l, part_r, prow, G, sm);
}

// ------------------------------------------------------------------ the residual history
// Shift i of a column starts from p_i = b and repeats
//     x_i += alpha_i p_i,   p_i = zeta_i r + beta_i p_i
// with the r of each iteration, at every site alike.  An iteration therefore
// only writes r on the support into the next slot of the history (16 bytes a
// value in the FP64-accurate iterations, 8 in the others); p_i and y = sum_i
// c_i x_i are formed when the solve, its FP64-accurate phase or the slots end.
// Before, launch YP read and wrote n shifted directions and y (32 n + 32 bytes
// a value) with 6 n FP64 operations on them: with 14 shifts on 9/16 of the
// lattice (r = 2) two thirds of a mixed solve (2.1 / 0.52 ms per FP64-accurate
// / FP32 iteration of three lattices; the copy and p take 0.15 / 0.06 ms).
//
// FP64-accurate iterations (k_hist_w, k_hist_y, k_hist_p): over n iterations k
// (r_k the residual after iteration k), with the scalars run backwards from
// S_n = 0, P_n = 1 as S_k = alpha_k + beta_k S_{k+1}, P_k = beta_k P_{k+1},
//     x_i += S_0 p_i + sum_k zeta_k S_{k+1} r_k,
//     p_i  = P_0 p_i + sum_k zeta_k P_{k+1} r_k,
// so y needs one weight per iteration, w_k = sum_i c_i zeta_k S_{k+1}, whatever
// the number of shifts: one FP64 operation a real value and iteration.  All
// terms have the sign of r_k's coefficient in x_i (every factor is positive).
// FP32 iterations (k_hist_run): the directions are FP32 there, and so is their
// rounding, which weights would not reproduce: the recurrences run as written,
// with the directions in registers and each r_k read once.
//
// slot q of a lattice: H[q * stride + element], elements [tile][n_sup][12][BC]

__device__ __forceinline__ double2 hist_value(double2 v) { return v; }
__device__ __forceinline__ double2 hist_value(float2 v) { return make_double2(exact_d(v.x), exact_d(v.y)); }
__device__ __forceinline__ double2 hist_value(df64c v) {
    return make_double2(exact_d(v.x.hi) + exact_d(v.x.lo), exact_d(v.y.hi) + exact_d(v.y.lo));
}

// r of one iteration into the history, for the support tiles of block group bx
// (one lattice: rtile0 is the first element of the RHS tile in r, cl the tile
// within the lattice, h the lattice's part of slot 0)
template <typename T, int BC>
__device__ __forceinline__ void hist_tiles(int bx, int tpb, int cl, int j0, size_t rtile0, int n_sup,
                                           const int *__restrict__ supsite, const int *__restrict__ rhs_class,
                                           const typename cplx_t<T>::type *__restrict__ r,
                                           typename cplx_t<T>::type *__restrict__ h, size_t stride, const Scal &sc) {
    typedef typename cplx_t<T>::type C;
    const int jj = threadIdx.x % BC, j = j0 + jj;
    const int cls = rhs_class[j];
    if (cls < 0 || !sc.upd_rhs[j]) return; // (an idle column's weights are zero: its slot is not read)
    C *o = h + (size_t)(sc.slot[j] - 1) * stride + (size_t)cl * 12 * n_sup * BC + jj;
    const C *q = r + rtile0 + jj;
    const int ntiles = (n_sup + TileMap<BC>::SPB - 1) / TileMap<BC>::SPB;
    for (int tile = bx * tpb, tend = min(ntiles, tile + tpb); tile < tend; ++tile) {
        const int k = tile * TileMap<BC>::SPB + threadIdx.x / BC;
        if (k >= n_sup) continue;
        const int site = supsite ? supsite[(size_t)cls * n_sup + k] : k;
        C v[12];
#pragma unroll
        for (int c = 0; c < 12; ++c) v[c] = q[((size_t)site * 12 + c) * BC];
#pragma unroll
        for (int c = 0; c < 12; ++c) o[((size_t)k * 12 + c) * BC] = v[c];
    }
}

// Two FP32 values whose sum is v to about 2^-49, in place of it
__device__ __forceinline__ double hi_lo(double v) {
    const float h = (float)v;
    return __hiloint2double(__float_as_int((float)(v - (double)h)), __float_as_int(h));
}
// alpha_i and beta_i of shift i in row k (0 and 1 where its direction was left alone)
__device__ __forceinline__ void shift_scalars(const Scal &sc, int k, int i, int j, int nshift, int B, double &a,
                                              double &b, double &z) {
    const size_t o = ((size_t)k * nshift + i) * B + j;
    z = sc.hz[o];
    a = 0;
    b = 1;
    if (z != 0) {
        const double zo = sc.ho[o], w = z / zo;
        a = sc.hal[(size_t)k * B + j] * z / zo;
        b = sc.hbe[(size_t)k * B + j] * w * w;
    }
}
// The weights of a chunk of n iterations, one thread per shift and column of a
// lattice (columns j0 <= j < j0 + Bl): hz <- c_i zeta_k S_{k+1}, ho <- zeta_k
// P_{k+1} (packed: as two FP32 values, for k_hist_p<.., true>); v0 <- c_i S_0,
// d0 <- P_0.
__global__ void k_hist_w(int n, int nshift, int B, int j0, int Bl, const ShiftParams *__restrict__ sp, Scal sc,
                         double *__restrict__ v0, double *__restrict__ d0, bool packed) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nshift * Bl) return;
    const int i = t / Bl, j = j0 + t % Bl;
    const size_t step = (size_t)nshift * B;
    const double c = sp->c[i];
    double S = 0, P = 1;
    size_t o = (size_t)n * step + (size_t)i * B + j;
    for (int k = n - 1; k >= 0; --k) {
        o -= step;
        double a, b, z;
        shift_scalars(sc, k, i, j, nshift, B, a, b, z);
        sc.hz[o] = c * (z * S);
        sc.ho[o] = packed ? hi_lo(z * P) : z * P;
        S = fma(b, S, a);
        P *= b;
    }
    v0[(size_t)i * B + j] = c * S;
    d0[(size_t)i * B + j] = P;
}
// hw[k][j] = sum over the shifts of a row's weights, rows 0..n-1 (hz) and row n (v0)
__global__ void k_hist_sum(int n, int nshift, int B, const double *__restrict__ hz, const double *__restrict__ v0,
                           double *__restrict__ hw) {
    const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (t >= (size_t)(n + 1) * B) return;
    const int k = (int)(t / B), j = (int)(t % B);
    const double *q = (k < n ? hz + (size_t)k * nshift * B : v0) + j;
    double w = 0;
    for (int i = 0; i < nshift; ++i) w += q[(size_t)i * B];
    hw[t] = w;
}

// what the history kernels know of a lattice's support and of the chunk
struct HistLat {
    size_t ne; // elements of the lattice: 12 n_sup columns
    int n_sup, V, j0, nshift, B;
    const int *supsite, *rhs_class;
    Source src;
    const void *h; // slot 0
    size_t stride; // elements of one slot, and of one shift's directions
    int n;         // iterations in the chunk
    bool first;    // it starts from p_i = b, y = 0 (else from the directions and y kept)
};
template <int BC> __device__ __forceinline__ int hist_col(const HistLat &L, size_t e) {
    return L.j0 + (int)(e / ((size_t)12 * L.n_sup * BC)) * BC + (int)(e % BC);
}
// b at element e of a lattice's support
template <int BC> __device__ __forceinline__ double2 hist_b(const HistLat &L, size_t e, int j, int cls) {
    const size_t q = e / BC;
    const int c = (int)(q % 12), k = (int)(q / 12 % L.n_sup);
    const size_t tile = q / 12 / L.n_sup;
    const int site = L.supsite ? L.supsite[(size_t)cls * L.n_sup + k] : k;
    return source_at<BC>(L.src, L.V, site, c, j - L.j0, ((tile * L.V + site) * 12 + c) * BC + e % BC);
}

// y += the share of a chunk of FP64-accurate iterations, one thread per
// element: every slot read once, consecutive threads on consecutive values
// (bound by HBM: 16 bytes and two FP64 operations a value and slot)
template <typename C, int BC>
__global__ void __launch_bounds__(256) k_hist_y(HistLat L, const double *__restrict__ hw,
                                                const double *__restrict__ v0, const double2 *__restrict__ ps,
                                                double2 *__restrict__ y) {
    const size_t e = blockIdx.x * (size_t)256 + threadIdx.x;
    if (e >= L.ne) return;
    const int j = hist_col<BC>(L, e), cls = L.rhs_class[j];
    if (cls < 0) return;
    double2 acc;
    if (L.first) {
        const double2 b = hist_b<BC>(L, e, j, cls);
        const double w = hw[(size_t)L.n * L.B + j];
        acc = make_double2(w * b.x, w * b.y);
    } else {
        acc = y[e];
        for (int i = 0; i < L.nshift; ++i) {
            const double w = v0[(size_t)i * L.B + j];
            const double2 q = ps[i * L.stride + e];
            acc.x = fma(w, q.x, acc.x);
            acc.y = fma(w, q.y, acc.y);
        }
    }
    const C *h = (const C *)L.h + e;
#pragma unroll 4
    for (int k = 0; k < L.n; ++k) {
        const double w = hw[(size_t)k * L.B + j];
        if (w != 0) { // (weight 0: the column was idle, its slot is unset)
            const double2 v = hist_value(h[k * L.stride]);
            acc.x = fma(w, v.x, acc.x);
            acc.y = fma(w, v.y, acc.y);
        }
    }
    y[e] = acc;
}

// The kernels below go over the support rows (component, support entry) of one
// RHS tile (blockIdx.y) with a thread for each column and HROWS rows of it: the
// scalars of NG shifts and HK iterations wait in shared memory, loaded by the
// block at once, and serve the HROWS values of a thread from there (read from
// global memory shift by shift they were the latency of the whole kernel: 100
// ms of a 266 ms solve of three r = 2 lattices).
//   NG is 14, or 1 for solves of one shift (the trace: with 14 it took 140 ms for 192
// mixed sources of 8^3x16, 124 with 1).
constexpr int HROWS = 2;
template <int BC, typename V, int NG> struct HistTile {
    typedef TileMap<BC> TM;
    int jj, j, cls;      // column within the tile and the solve, its class
    size_t e[HROWS];     // elements, valid where ok
    bool ok[HROWS];
    __device__ __forceinline__ explicit HistTile(const HistLat &L) {
        jj = threadIdx.x % BC;
        j = L.j0 + blockIdx.y * BC + jj;
        cls = L.rhs_class[j];
#pragma unroll
        for (int q = 0; q < HROWS; ++q) {
            const int row = (blockIdx.x * HROWS + q) * TM::SPB + threadIdx.x / BC;
            ok[q] = row < 12 * L.n_sup && cls >= 0;
            e[q] = ((size_t)blockIdx.y * 12 * L.n_sup + row) * BC + jj;
        }
    }
    // the scalars of iterations k0.. and shifts i0.. of the tile's columns (zeros beyond the last)
    template <int HK>
    __device__ __forceinline__ static void load(const HistLat &L, const V *__restrict__ c, int k0, int i0,
                                                V (*sm)[NG][BC], V zero) {
        for (int t = threadIdx.x; t < HK * NG * BC; t += TM::THREADS) {
            const int q = t % BC, g = t / BC % NG, k = t / BC / NG;
            const bool in = k0 + k < L.n && i0 + g < L.nshift;
            sm[k][g][q] = in ? c[((size_t)(k0 + k) * L.nshift + i0 + g) * L.B + L.j0 + blockIdx.y * BC + q] : zero;
        }
    }
};
template <int BC> static dim3 hist_grid(const HistLat &L) {
    const int per = HROWS * TileMap<BC>::SPB;
    return dim3((unsigned)((12 * (size_t)L.n_sup + per - 1) / per), (unsigned)(L.ne / ((size_t)12 * L.n_sup * BC)));
}

// p_i = P_0 p_i + sum_k zeta_k P_{k+1} r_k for every shift after a chunk of
// FP64-accurate iterations.  Into ps (FP64; more such iterations follow): FP64
// weights and sums.  Into ps32 (the mixed solve's switch to FP32): float-float
// ones (48 bits, re and im packed: 12 FP32 instructions of 2 cycles for the two
// FP64 ones of 66), rounded to FP32 at the end.  The weights then fall like
// (|r_n| / |r_k|)^2: one below the FP32 range belongs to a term that far below
// the last ones.
template <typename C, int BC, bool F32, int NG>
__global__ void __launch_bounds__(TileMap<BC>::THREADS) k_hist_p(HistLat L, const double *__restrict__ hp,
                                                                 const double *__restrict__ d0,
                                                                 double2 *__restrict__ ps,
                                                                 float2 *__restrict__ ps32) {
    constexpr int HK = 8;
    __shared__ double sm[HK][NG][BC];
    const HistTile<BC, double, NG> T(L);
    for (int i0 = 0; i0 < L.nshift; i0 += NG) {
        for (int q = 0; q < HROWS; ++q) {
            double2 acc[F32 ? 1 : NG];
            float2 sh[F32 ? NG : 1], sl[F32 ? NG : 1];
            double2 b = make_double2(0, 0);
            if (T.ok[q] && L.first) b = hist_b<BC>(L, T.e[q], T.j, T.cls);
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                double2 v = make_double2(0, 0);
                if (T.ok[q] && i0 + g < L.nshift) {
                    const double2 w = L.first ? b : ps[(i0 + g) * L.stride + T.e[q]];
                    const double d = d0[(size_t)(i0 + g) * L.B + T.j];
                    v = make_double2(d * w.x, d * w.y);
                }
                if constexpr (F32) {
                    sh[g] = make_float2((float)v.x, (float)v.y);
                    sl[g] = make_float2((float)(v.x - (double)sh[g].x), (float)(v.y - (double)sh[g].y));
                } else {
                    acc[g] = v;
                }
            }
            for (int k0 = 0; k0 < L.n; k0 += HK) {
                __syncthreads();
                HistTile<BC, double, NG>::template load<HK>(L, hp, k0, i0, sm, 0.0);
                __syncthreads();
                if (!T.ok[q]) continue;
#pragma unroll
                for (int k = 0; k < HK; ++k) {
                    // every shift's zeta is 0 where the column was idle, and only there is the slot unset
                    const double w0 = sm[k][0][T.jj];
                    if (F32 ? __double2loint(w0) == 0 : w0 == 0) continue;
                    const C v = ((const C *)L.h)[(k0 + k) * L.stride + T.e[q]];
#pragma unroll
                    for (int g = 0; g < NG; ++g) {
                        const double w = sm[k][g][T.jj];
                        if constexpr (F32 && std::is_same<C, df64c>::value) {
                            const float wh = __int_as_float(__double2loint(w)), wl = __int_as_float(__double2hiint(w));
                            ff_acc2(sh[g], sl[g], f2b(wh), f2b(wl), make_float2(v.x.hi, v.y.hi),
                                    make_float2(v.x.lo, v.y.lo));
                        } else if constexpr (!F32) {
                            const double2 d = hist_value(v);
                            acc[g].x = fma(w, d.x, acc[g].x);
                            acc[g].y = fma(w, d.y, acc[g].y);
                        }
                    }
                }
            }
            if (!T.ok[q]) continue;
#pragma unroll
            for (int g = 0; g < NG; ++g)
                if (i0 + g < L.nshift) {
                    const size_t o = (i0 + g) * L.stride + T.e[q];
                    if constexpr (F32) ps32[o] = make_float2(sh[g].x + sl[g].x, sh[g].y + sl[g].y);
                    else ps[o] = acc[g];
                }
        }
    }
}

// what a chunk of FP32 iterations needs of its scalars, for every (row, shift,
// column) of a lattice: {c_i alpha_i as two FP32 values, zeta, beta}
__global__ void k_hist_coef(int n, int nshift, int B, int j0, int Bl, const ShiftParams *__restrict__ sp, Scal sc,
                            float4 *__restrict__ ct) {
    const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (t >= (size_t)n * nshift * Bl) return;
    const size_t ki = t / Bl; // row * nshift + shift
    const int i = (int)(ki % nshift), j = j0 + (int)(t % Bl);
    double a, b, z;
    shift_scalars(sc, (int)(ki / nshift), i, j, nshift, B, a, b, z);
    const size_t o = ki * B + j;
    const double ca = sp->c[i] * a, w = hi_lo(ca);
    sc.ho[o] = ca;
    // a converged shift's row (alpha 0) leaves y and its direction alone
    ct[o] = make_float4(__int_as_float(__double2loint(w)), __int_as_float(__double2hiint(w)), (float)z, (float)b);
}

// A chunk of FP32 iterations: y += c_i alpha_i p_i, p_i = zeta r + beta p_i for
// every shift, in the order of the iterations, the directions in registers.
// EXACT: y in FP64 all through (hist_exact).  Else the chunk's share is summed in
// float-float and added to y in FP64: 10 packed FP32 instructions a value instead
// of FP64 ones of 66 cycles.  Bound by those.
//   Float-float coefficients and sums round at about 2^-48 of the share, FP64 ones at
// 2^-53 of y in every addition.  In the mixed solve the share is what is left of y
// below the switch residual theta (times a factor of order 1): for theta up to 2^-8
// (the default is 1e-3) its rounding is no larger than FP64's.  Above that, and where
// y starts here (SMPQ_FP32 and the half storage), the sums are FP64.
constexpr double HIST_FF_THETA = 1.0 / 256;
inline bool hist_exact(int prec, double theta) { return prec != SMPQ_MIXED || theta > HIST_FF_THETA; }
template <int BC, bool EXACT, int NG>
__global__ void __launch_bounds__(TileMap<BC>::THREADS) k_hist_run(HistLat L, const double *__restrict__ ca,
                                                                   const float4 *__restrict__ ct,
                                                                   float2 *__restrict__ ps32,
                                                                   double2 *__restrict__ y, bool last) {
    constexpr int HK = NG == 1 ? 8 : EXACT ? 2 : 4;
    __shared__ float4 sm[HK][NG][BC];
    __shared__ double sa[EXACT ? HK : 1][NG][BC];
    const HistTile<BC, float4, NG> T(L);
    for (int i0 = 0; i0 < L.nshift; i0 += NG) {
        float2 p[HROWS][NG], s[HROWS], d[HROWS];
        double2 yv[HROWS];
#pragma unroll
        for (int q = 0; q < HROWS; ++q) {
            s[q] = d[q] = make_float2(0.f, 0.f);
            yv[q] = make_double2(0, 0);
            float2 b = make_float2(0.f, 0.f);
            if (T.ok[q] && L.first) {
                const double2 v = hist_b<BC>(L, T.e[q], T.j, T.cls);
                b = make_float2((float)v.x, (float)v.y);
            }
            if (T.ok[q] && !(L.first && i0 == 0)) yv[q] = y[T.e[q]];
#pragma unroll
            for (int g = 0; g < NG; ++g)
                p[q][g] = T.ok[q] && !L.first && i0 + g < L.nshift ? ps32[(i0 + g) * L.stride + T.e[q]] : b;
        }
        for (int k0 = 0; k0 < L.n; k0 += HK) {
            __syncthreads();
            HistTile<BC, float4, NG>::template load<HK>(L, ct, k0, i0, sm, make_float4(0.f, 0.f, 0.f, 0.f));
            if constexpr (EXACT) HistTile<BC, double, NG>::template load<HK>(L, ca, k0, i0, sa, 0.0);
            __syncthreads();
            float2 rv[HK][HROWS];
#pragma unroll
            for (int k = 0; k < HK; ++k)
#pragma unroll
                for (int q = 0; q < HROWS; ++q)
                    rv[k][q] = T.ok[q] && k0 + k < L.n ? ((const float2 *)L.h)[(k0 + k) * L.stride + T.e[q]]
                                                       : make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < HK; ++k)
#pragma unroll
                for (int g = 0; g < NG; ++g) {
                    const float4 c = sm[k][g][T.jj];
                    if (c.x == 0.f) continue; // converged: y and the direction stay
                    const float2 ah = f2b(c.x), al = f2b(c.y);
#pragma unroll
                    for (int q = 0; q < HROWS; ++q) {
                        float2 &pv = p[q][g];
                        if constexpr (EXACT) {
                            const double a = sa[k][g][T.jj];
                            yv[q].x += a * exact_d(pv.x);
                            yv[q].y += a * exact_d(pv.y);
                        } else {
                            const float2 t = __fmul2_rn(ah, pv);
                            const float2 u = __ffma2_rn(al, pv, __ffma2_rn(ah, pv, f2neg(t)));
                            float2 w, x;
                            two_sum2(s[q], t, w, x);
                            s[q] = w;
                            d[q] = __fadd2_rn(d[q], __fadd2_rn(u, x));
                        }
                        pv = __ffma2_rn(f2b(c.w), pv, __fmul2_rn(f2b(c.z), rv[k][q]));
                    }
                }
        }
#pragma unroll
        for (int q = 0; q < HROWS; ++q) {
            if (!T.ok[q]) continue;
            if constexpr (!EXACT) {
                yv[q].x += (double)s[q].x + (double)d[q].x;
                yv[q].y += (double)s[q].y + (double)d[q].y;
            }
            y[T.e[q]] = yv[q];
            if (!last)
#pragma unroll
                for (int g = 0; g < NG; ++g)
                    if (i0 + g < L.nshift) ps32[(i0 + g) * L.stride + T.e[q]] = p[q][g];
        }
    }
}

// Launch YP of an iteration: blocks x < Gs keep r on the support in the
// history, the others update p (and x64, xlo) on the lattice.  Bound by HBM:
// 36 e bytes a site and column for p, 24 e on the support.  tpb tiles per
// block: 4, fewer where that would leave SMs without a block.
template <typename T, int BC, bool M>
__global__ void __launch_bounds__(TileMap<BC>::THREADS)
    k_yp(Lats L, int tpb, const int *__restrict__ rhs_class, const typename cplx_t<T>::type *__restrict__ r,
         typename cplx_t<T>::type *__restrict__ h, size_t stride, Scal sc,
         typename cplx_t<T>::type *__restrict__ p, typename XAcc<T>::type *__restrict__ x64,
         typename cplx_t<T>::type *__restrict__ xlo) {
    const int l = lat_index<M>(L);
    const Lat &la = L.l[l];
    const int cl = blockIdx.y - la.chunk0, bx = blockIdx.x;
    const size_t tile0 = la.f0 + (size_t)cl * 12 * la.g.V * BC;
    if (bx < la.Gs)
        hist_tiles<T, BC>(bx, tpb, cl, blockIdx.y * BC, tile0, la.n_sup, la.supsite, rhs_class, r, h + la.sup0, stride,
                          sc);
    else if (bx < la.Gs + la.G)
        update_p_tiles<T, BC>(bx - la.Gs, tpb, la.g.V, tile0, r, p, sc, x64, xlo);
}

// Launch YP of a half-storage iteration (p in the half format)
template <typename HT, int BC, bool M>
__global__ void __launch_bounds__(TileMap<BC>::THREADS)
    k_yp_h(Lats L, int tpb, const int *__restrict__ rhs_class, const float2 *__restrict__ r, float2 *__restrict__ h,
           size_t stride, Scal sc, HF<HT> p, float2 *__restrict__ xlo) {
    const int l = lat_index<M>(L);
    const Lat &la = L.l[l];
    const int cl = blockIdx.y - la.chunk0, bx = blockIdx.x;
    const size_t tile0 = la.f0 + (size_t)cl * 12 * la.g.V * BC;
    if (bx < la.Gs)
        hist_tiles<float, BC>(bx, tpb, cl, blockIdx.y * BC, tile0, la.n_sup, la.supsite, rhs_class, r, h + la.sup0,
                              stride, sc);
    else if (bx < la.Gs + la.G)
        update_p_h_tiles<HT, BC>(bx - la.Gs, tpb, la.g.V, tile0, r, p, sc, xlo);
}

// x_hi += x_lo ; x_lo = 0 (x_hi in float-float: FP64 accuracy on the FP32 pipes)
template <typename T, int BC>
__global__ void __launch_bounds__(TileMap<BC>::THREADS)
    k_rel_accum(int V, df64c *__restrict__ xhi, typename cplx_t<T>::type *__restrict__ xlo, int G) {
    typedef typename cplx_t<T>::type C;
    const int jj = threadIdx.x % BC, chunk = blockIdx.y;
    const size_t base = (size_t)chunk * 12 * V * BC + jj;
    const int ntiles = (V + TileMap<BC>::SPB - 1) / TileMap<BC>::SPB;
    for (int tile = blockIdx.x * TPB, tend = min(ntiles, tile + TPB); tile < tend; ++tile) {
        int s = tile * TileMap<BC>::SPB + threadIdx.x / BC;
        if (s >= V) continue;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            size_t o = base + ((size_t)s * 12 + c) * BC;
            C xl = xlo[o];
            df64c xh = xhi[o];
            xh.x = xh.x + df64(xl.x);
            xh.y = xh.y + df64(xl.y);
            xhi[o] = xh;
            xlo[o] = mkc<C>(0, 0);
        }
    }
}

// r_hi = b - (D_W^dag t64 + s0 x_hi) in FP64 (t64 = D_W x_hi); r = T(r_hi); partial |r_hi|^2
template <typename T, int BC>
__global__ void __launch_bounds__(TileMap<BC>::THREADS)
    k_rel_resid(Geom g, const double2 *__restrict__ U64, const double2 *__restrict__ t64,
                const double2 *__restrict__ xhi, Source src, typename cplx_t<T>::type *__restrict__ r, double s0,
                double kappa, double *part_r, int G) {
    typedef typename cplx_t<T>::type C;
    __shared__ double sm[TileMap<BC>::THREADS];
    const int jj = threadIdx.x % BC, chunk = blockIdx.y, j = chunk * BC + jj;
    const size_t base = (size_t)chunk * 12 * g.V * BC + jj;
    const int ntiles = (g.V + TileMap<BC>::SPB - 1) / TileMap<BC>::SPB;
    double ar = 0;
    for (int tile = blockIdx.x * TPB, tend = min(ntiles, tile + TPB); tile < tend; ++tile) {
        int s = tile * TileMap<BC>::SPB + threadIdx.x / BC;
        if (s >= g.V) continue;
        double2 acc[12][1];
        wilson_hop<double, true, BC>(g, U64, t64 + base, s, acc);
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            size_t o = base + ((size_t)s * 12 + c) * BC;
            double2 tv = t64[o], xv = xhi[o];
            double2 b = source_at<BC>(src, g.V, s, c, j, o);
            double2 rv;
            rv.x = b.x - (tv.x - kappa * acc[c][0].x + s0 * xv.x);
            rv.y = b.y - (tv.y - kappa * acc[c][0].y + s0 * xv.y);
            r[o] = mkc<C>(rv.x, rv.y);
            ar += rv.x * rv.x + rv.y * rv.y;
        }
    }
    double s1 = block_sum<BC>(ar, sm);
    if (threadIdx.x < BC) part_r[((size_t)chunk * G + blockIdx.x) * BC + threadIdx.x] = s1;
}

// Residual replacement in float-float (FP64-accurate, on the FP32 pipes):
// r_hi = b - (D_W^dag t + s0 x_hi) with t = D_W x_hi (both float-float fields);
// r = T(r_hi); partial |r_hi|^2 (per-site sums of the high parts in FP32: the
// norm only steers the recurrences and the convergence test).
template <typename T, int BC>
__global__ void __launch_bounds__(TileMap<BC>::THREADS, MinBlocks<df64>::value)
    k_rel_resid_df(Geom g, const df64c *__restrict__ U, const df64c *__restrict__ t, const df64c *__restrict__ xhi,
                   Source src, typename cplx_t<T>::type *__restrict__ r, double s0, df64 kappa, double *part_r,
                   int G) {
    typedef typename cplx_t<T>::type C;
    __shared__ double sm[TileMap<BC>::THREADS];
    const int jj = threadIdx.x % BC, chunk = blockIdx.y, j = chunk * BC + jj;
    const size_t base = (size_t)chunk * 12 * g.V * BC + jj;
    const int ntiles = (g.V + TileMap<BC>::SPB - 1) / TileMap<BC>::SPB;
    const df64 sh(s0);
    const int cls = src.b64 ? -1 : src.src_class[j], comp = src.b64 ? -1 : src.src_comp[j];
    double ar = 0;
    for (int tile = blockIdx.x * TPB, tend = min(ntiles, tile + TPB); tile < tend; ++tile) {
        int s = tile * TileMap<BC>::SPB + threadIdx.x / BC;
        if (s >= g.V) continue;
        df64c acc[12][1];
        wilson_hop_auto<df64, true, BC>(g, U, t + base, s, acc);
        const bool in_class = cls >= 0 && src.colour[s] == cls;
        float sr = 0.f;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            size_t o = base + ((size_t)s * 12 + c) * BC;
            const df64c tv = t[o], xv = xhi[o];
            df64c bv;
            if (src.b64) bv = df64c{df64(src.b64[o].x), df64(src.b64[o].y)}; // explicit source (rare)
            else bv = df64c{df64((in_class && c == comp) ? 1.f : 0.f), df64(0.f)};
            df64c rv;
            rv.x = bv.x - (tv.x - kappa * acc[c][0].x + sh * xv.x);
            rv.y = bv.y - (tv.y - kappa * acc[c][0].y + sh * xv.y);
            if constexpr (std::is_same<T, float>::value) r[o] = make_float2(rv.x.hi + rv.x.lo, rv.y.hi + rv.y.lo);
            else if constexpr (std::is_same<T, df64>::value) r[o] = rv;
            else r[o] = mkc<C>(to_d(rv.x), to_d(rv.y));
            sr += rv.x.hi * rv.x.hi + rv.y.hi * rv.y.hi;
        }
        ar += (double)sr;
    }
    double s1 = block_sum<BC>(ar, sm);
    if (threadIdx.x < BC) part_r[((size_t)chunk * G + blockIdx.x) * BC + threadIdx.x] = s1;
}

// ------------------------------------------------------------------ scalar kernels (one block per rhs)
constexpr int SCAL_THREADS = 128;

// sum over blocks of the partials of rhs j: strided per-thread sums, then a
// fixed tree (deterministic)
__device__ __forceinline__ double part_sum(const double *part, int j, int BC, int G, double *sm) {
    const int chunk = j / BC, jj = j % BC;
    double s = 0;
    for (int b = threadIdx.x; b < G; b += SCAL_THREADS) s += part[((size_t)chunk * G + b) * BC + jj];
    sm[threadIdx.x] = s;
    __syncthreads();
    for (int st = SCAL_THREADS / 2; st > 0; st >>= 1) {
        if (threadIdx.x < st) sm[threadIdx.x] += sm[threadIdx.x + st];
        __syncthreads();
    }
    double r = sm[0];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(SCAL_THREADS)
    s_init(int B, int BC, int G, const double *part_b, Scal sc, ShiftParams sp, double tol) {
    __shared__ double sm[SCAL_THREADS];
    const int j = blockIdx.x;
    double bb = part_sum(part_b, j, BC, G, sm);
    if (threadIdx.x) return;
    sc.bb[j] = bb;
    sc.rr[j] = bb;
    sc.rr_ref[j] = bb;
    sc.alpha[j] = 0;
    sc.beta[j] = 0;
    sc.alpha_prev[j] = 1;
    sc.beta_prev[j] = 0;
    sc.iters[j] = 0;
    sc.slot[j] = 0;
    int any = 0;
    for (int i = 0; i < sp.n; ++i) {
        sc.zeta[i * B + j] = 1;
        sc.zeta_prev[i * B + j] = 1;
        sc.upd[i * B + j] = 0;
        int a = bb > 0;
        sc.act[i * B + j] = a;
        any |= a;
    }
    sc.act_rhs[j] = any;
    sc.upd_rhs[j] = 0;
    if (any) atomicAdd(&sc.flags[0], 1);
}

// out[j] = sum over the blocks of the partials of rhs j (one block per rhs)
__global__ void __launch_bounds__(SCAL_THREADS) s_sum_rhs(int BC, int G, const double *part, double *out) {
    __shared__ double sm[SCAL_THREADS];
    const double v = part_sum(part, blockIdx.x, BC, G, sm);
    if (threadIdx.x == 0) out[blockIdx.x] = v;
}

// after a residual replacement: rr = |r_hi|^2, the base shift re-activates if
// its true residual is above tolerance (flags[0] and flags[1] are cleared by
// the host before the launch)
__global__ void __launch_bounds__(SCAL_THREADS)
    s_rel(int B, int BC, int G, const double *part_r, Scal sc, ShiftParams sp, double tol2, int base) {
    __shared__ double sm[SCAL_THREADS];
    const int j = blockIdx.x;
    double rr = part_sum(part_r, j, BC, G, sm);
    if (threadIdx.x || !(sc.bb[j] > 0)) return;
    sc.rr[j] = rr;
    sc.rr_ref[j] = rr;
    int any = 0;
    for (int i = 0; i < sp.n; ++i) {
        int ix = i * B + j;
        if (i == base) sc.act[ix] = sc.zeta[ix] * sc.zeta[ix] * rr > tol2 * sc.bb[j];
        any |= sc.act[ix];
    }
    sc.act_rhs[j] = any;
    if (any) atomicAdd(&sc.flags[0], 1);
}

// ------------------------------------------------------------------ driver

// p = r for every right-hand side whose base shift a residual replacement has
// re-activated (a restart of its CG from the true residual)
template <typename C>
__global__ void k_restart_p(const C *__restrict__ r, C *__restrict__ p, size_t n, int BC, int V,
                            const int *__restrict__ act_rhs) {
    size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int j = (int)(i / ((size_t)12 * V * BC)) * BC + (int)(i % BC); // tile layout [j/BC][V][12][BC]
    if (act_rhs[j]) p[i] = r[i];
}

// elementwise float-float -> FP32 copy of a field (same tiled layout)
__global__ void k_to_fp32(const df64c *__restrict__ in, float2 *__restrict__ out, size_t n) {
    size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i < n) out[i] = make_float2((float)in[i].x, (float)in[i].y);
}

// One multi-shift solve of B right-hand sides in tiles of BC columns, over
// one lattice or several of different sizes in the same launches.  The
// solve runs in one or two phases:
//   SMPQ_FP64  : FP64 iterations (vectors, D_W, residual history);
//   SMPQ_FP32  : FP32 iterations with FP64 reliable updates of the base system;
//   SMPQ_FP16N / SMPQ_BF16N : the same with p and t stored in FP16 / BF16 with
//                per-site norms and reconstruct-12 links;
//   SMPQ_MIXED : FP64-accurate iterations until every right-hand side has
//                ||r|| <= theta ||b||, then FP32 iterations; the residual
//                history is kept in the precision of r.
// Scalars, reductions and y are FP64 in every mode.  The fields of all
// lattices share one buffer per vector: lattice l's part starts at element
// f0[l] (its tiles first come at tile ch0[l] of the solve).
template <int BC> struct Solve {
    smpq_ctx *ctx; // the first lattice's context: stream, workspace, options
    std::vector<LatIn> in;
    int nl;
    // per lattice: sites, right-hand sides, tiles, first tile, first rhs, blocks
    // per tile of the one-column lattice kernels (TPB tiles each), of the
    // support kernels, one-column tiles; field, support-field and partial-row offsets
    std::vector<int> V, Bl, nch, ch0, j0, G1, Gs1, nt1;
    std::vector<size_t> f0, s0, p0;
    std::vector<Source> srcl;
    std::vector<ShiftParams> sph; // host copies behind spd
    int B = 0, nchunk = 0, nshift = 0;
    size_t nfield = 0, nsupf = 0, npart = 0;
    cudaStream_t st;
    Scal sc;
    const ShiftParams *spd = nullptr; // [nl] device copies
    double *part0, *part1, *part2;
    double2 *y = nullptr;
    // the residual history: bytes per support element in W_HIST, rows of scalars,
    // iterations in the chunk
    size_t hcap = 0;
    int hrows = 1, hn = 0;
    bool hfirst = true;
    double *hw = nullptr, *hv0 = nullptr, *hd0 = nullptr;
    float4 *hct = nullptr;
    double tol2;
    int *hflags = nullptr;
    int *count = nullptr;       // [nchunk] arrival counters of the fused scalar steps, [nchunk][ngroups] of groups
    int ngroups = 1;
    std::vector<int> rows1;     // per lattice: the most partial rows a launch has per tile
    double2 *x64 = nullptr;     // base-system solution in FP64 (true residual), nullable
    double *true_rr = nullptr;  // [B] |b - (A + s0) x64|^2
    int iters = 0, nrel = 0;
    bool prof;
    int chk;
    bool shifts;
    int tpb_hi = TPB, tpb_lo = TPB, nr = 1;
    bool stg = false;    // FP32 iterations: the D_W pair with staged neighbours (stage.cuh)
    bool stg_df = false; // float-float iterations: likewise

    explicit Solve(const std::vector<LatIn> &lats) : ctx(lats[0].ctx), in(lats), nl((int)lats.size()) {}

    // the per-rhs scalars of lattice l (the shift-major ones keep the solve's stride B)
    Scal scal_of(int l) const {
        Scal s = sc;
        const int o = j0[l];
        s.rr += o; s.bb += o; s.alpha += o; s.beta += o; s.alpha_prev += o; s.beta_prev += o; s.rr_ref += o;
        s.act_rhs += o; s.upd_rhs += o; s.iters += o;
        s.zeta += o; s.zeta_prev += o; s.act += o; s.upd += o; s.slot += o;
        return s;
    }

    int setup(double tol, double *hist, int hist_len) {
        st = ctx->stream;
        shifts = in[0].spec->n_sup > 0;
        nshift = in[0].sp.n;
        V.resize(nl); Bl.resize(nl); nch.resize(nl); ch0.resize(nl); j0.resize(nl); G1.resize(nl); Gs1.resize(nl);
        nt1.resize(nl); f0.resize(nl); s0.resize(nl); p0.resize(nl); srcl.resize(nl); sph.resize(nl);
        for (int l = 0; l < nl; ++l) {
            const SolveSpec &sp = *in[l].spec;
            if (sp.B % BC || in[l].sp.n != nshift || (sp.n_sup > 0) != shifts || in[l].ctx->device != ctx->device)
                return set_err(ctx, SMPQ_EINVAL, "lattices of one solve need the same tile width, poles, support "
                                                 "kind and device");
            V[l] = in[l].ctx->V;
            Bl[l] = sp.B;
            nch[l] = sp.B / BC;
            ch0[l] = nchunk;
            j0[l] = B;
            nt1[l] = (V[l] + TileMap<BC>::SPB - 1) / TileMap<BC>::SPB;
            G1[l] = (nt1[l] + TPB - 1) / TPB;
            const int nsup_tiles = (sp.n_sup + TileMap<BC>::SPB - 1) / TileMap<BC>::SPB;
            Gs1[l] = std::max(1, (nsup_tiles + TPB - 1) / TPB);
            f0[l] = nfield;
            s0[l] = nsupf;
            p0[l] = npart / BC;
            nchunk += nch[l];
            B += sp.B;
            nfield += (size_t)sp.B * 12 * V[l];
            nsupf += (size_t)sp.B * 12 * sp.n_sup;
            // partial rows per tile: the most blocks any launch has per tile (the
            // D_W launches at one tile per block have nt1; the support kernels Gs1)
            const int ntb = (V[l] + BfMap<BC>::SPB - 1) / BfMap<BC>::SPB;
            rows1.push_back(std::max(std::max(nt1[l], ntb), Gs1[l]));
            npart += (size_t)nch[l] * rows1[l] * BC;
            sph[l] = in[l].sp;
        }
        tpb_hi = std::max(1, in[0].spec->tpb_hi > 0 ? in[0].spec->tpb_hi : TPB);
        tpb_lo = std::max(1, in[0].spec->tpb_lo > 0 ? in[0].spec->tpb_lo : TPB);
        nr = in[0].spec->nr == 2 ? 2 : 1;
        stg = (in[0].spec->staged & 1) && BC >= 12; // (one-column tiles: plain loads)
        stg_df = (in[0].spec->staged & 2) && BC >= 12;
        if (stg && nr == 2) return set_err(ctx, SMPQ_EINVAL, "internal: the staged D_W has one column per thread");
        std::vector<Buf> &ws = ctx->ws;
        if (ws.size() < W_COUNT) ws.resize(W_COUNT);
        int rc;
        if ((rc = ensure(ctx, ws[W_PART], 3 * npart * sizeof(double)))) return rc;
        const size_t nscal = (size_t)B * 8 + (size_t)nshift * B * 2;
        ngroups = 1;
        for (int l = 0; l < nl; ++l) ngroups = std::max(ngroups, (rows1[l] + GROUP - 1) / GROUP);
        const size_t nint = (size_t)B * 4 + (size_t)nshift * B * 2 + 12 + (size_t)nchunk * (1 + ngroups);
        if (shifts && (rc = plan_history())) return rc;
        const size_t rowlen = (size_t)nshift * B;
        if ((rc = ensure(ctx, ws[W_HCOEF], (size_t)hrows * rowlen * (2 * sizeof(double) + sizeof(float4)) +
                                                ((3 * (size_t)hrows + 1) * B + 2 * rowlen) * sizeof(double))))
            return rc;
        hct = (float4 *)ws[W_HCOEF].p;
        sc.hz = (double *)(hct + hrows * rowlen);
        sc.ho = sc.hz + hrows * rowlen;
        sc.hal = sc.ho + hrows * rowlen;
        sc.hbe = sc.hal + (size_t)hrows * B;
        hw = sc.hbe + (size_t)hrows * B;
        hv0 = hw + ((size_t)hrows + 1) * B;
        hd0 = hv0 + rowlen;
        sc.slot_inc = shifts ? 1 : 0;
        const size_t spbytes = ((size_t)nl * sizeof(ShiftParams) + 255) / 256 * 256;
        if ((rc = ensure(ctx, ws[W_SCAL], spbytes + nscal * sizeof(double) + nint * sizeof(int)))) return rc;
        part0 = (double *)ws[W_PART].p;
        part1 = part0 + npart;
        part2 = part1 + npart;
        spd = (const ShiftParams *)ws[W_SCAL].p;
        cudaMemcpyAsync((void *)spd, sph.data(), nl * sizeof(ShiftParams), cudaMemcpyHostToDevice, st);
        double *d = (double *)((char *)ws[W_SCAL].p + spbytes);
        sc.rr = d; d += B; sc.bb = d; d += B; sc.alpha = d; d += B; sc.beta = d; d += B;
        sc.alpha_prev = d; d += B; sc.beta_prev = d; d += B; sc.rr_ref = d; d += B;
        sc.zeta = d; d += nshift * B; sc.zeta_prev = d; d += nshift * B;
        true_rr = d; d += B;
        int *ip = (int *)d;
        sc.act_rhs = ip; ip += B; sc.upd_rhs = ip; ip += B; sc.iters = ip; ip += B; sc.slot = ip; ip += B;
        sc.act = ip; ip += nshift * B; sc.upd = ip; ip += nshift * B;
        sc.flags = ip; ip += 8; sc.iter_counter = ip; ip += 4;
        count = ip;
        sc.hist = hist;
        sc.hist_len = hist_len;
        for (int l = 0; l < nl; ++l) { // the lattice's sources, its per-rhs tables at its first rhs
            const SolveSpec &sp = *in[l].spec;
            srcl[l].colour = sp.d_colour;
            srcl[l].src_class = sp.d_src_class ? sp.d_src_class + j0[l] : nullptr;
            srcl[l].src_comp = sp.d_src_comp ? sp.d_src_comp + j0[l] : nullptr;
            srcl[l].b64 = sp.d_src_field ? (const double2 *)sp.d_src_field + f0[l] : nullptr;
        }
        tol2 = tol * tol;
        prof = ctx->opt.profile != 0;
        chk = std::max(1, ctx->opt.iters_per_check);
        if (prof) {
            while ((int)ctx->prof_ev.size() < 4 * chk) {
                cudaEvent_t ev;
                if (cudaEventCreate(&ev) != cudaSuccess) return cuda_check(ctx, cudaGetLastError(), "event");
                ctx->prof_ev.push_back(ev);
            }
        }
        if (cudaMallocHost(&hflags, NFLAGS * sizeof(int)) != cudaSuccess) {
            cudaGetLastError();
            return set_err(ctx, SMPQ_ENOMEM, "pinned host flags");
        }
        cudaMemsetAsync(sc.flags, 0, (12 + (size_t)nchunk * (1 + ngroups)) * sizeof(int), st); // flags, counter, arrivals
        return SMPQ_OK;
    }

    ~Solve() {
        if (hflags) cudaFreeHost(hflags);
    }

    // The lattice table of a D_W launch: blocks per tile for spb sites per tile
    // and tpb tiles per block; partial rows lattice after lattice.  *gx: the
    // grid's x extent (the largest lattice's blocks).
    template <typename T, typename HT = void> Lats lats_dw(int spb, int tpb, int *gx) const {
        Lats L{};
        L.n = nl;
        size_t prow = 0;
        *gx = 1;
        for (int l = 0; l < nl; ++l) {
            Lat &a = L.l[l];
            a.g = in[l].ctx->geom;
            if constexpr (std::is_void<HT>::value) a.U = Links<T>::get(in[l].ctx);
            else a.U = HLinks<HT>::get(in[l].ctx);
            a.f0 = (long long)f0[l];
            a.chunk0 = ch0[l];
            a.G = ((V[l] + spb - 1) / spb + tpb - 1) / tpb;
            a.p0 = (long long)prow;
            a.s0 = sph[l].s0;
            a.B = Bl[l];
            prow += (size_t)nch[l] * a.G;
            *gx = std::max(*gx, a.G);
        }
        return L;
    }
    // the lattice table of launch YP: support blocks, then lattice blocks (one
    // column per thread, *tpb tiles per block: as many as leave each SM several blocks)
    Lats lats_yp(int spb, int *gx, int *tpb) const {
        size_t tiles = 0;
        for (int l = 0; l < nl; ++l) tiles += (size_t)nch[l] * ((V[l] + spb - 1) / spb);
        *tpb = TPB;
        while (*tpb > 1 && tiles / *tpb < 2048) *tpb /= 2;
        Lats L{};
        L.n = nl;
        *gx = 1;
        for (int l = 0; l < nl; ++l) {
            Lat &a = L.l[l];
            a.g = in[l].ctx->geom;
            a.f0 = (long long)f0[l];
            a.chunk0 = ch0[l];
            const int nst = (in[l].spec->n_sup + spb - 1) / spb;
            a.G = ((V[l] + spb - 1) / spb + *tpb - 1) / *tpb;
            a.Gs = shifts ? (nst + *tpb - 1) / *tpb : 0;
            a.n_sup = in[l].spec->n_sup;
            a.supsite = in[l].spec->d_supsite;
            a.sup0 = (long long)s0[l];
            a.B = Bl[l];
            a.s0 = sph[l].s0;
            *gx = std::max(*gx, a.Gs + a.G);
        }
        return L;
    }
    // one lattice alone (its part of every buffer), for the per-lattice launches
    template <typename T> Lats lats_one(int l) const {
        Lats L{};
        L.n = 1;
        Lat &a = L.l[0];
        a.g = in[l].ctx->geom;
        a.U = Links<T>::get(in[l].ctx);
        a.f0 = (long long)f0[l];
        a.chunk0 = 0;
        a.G = G1[l];
        a.p0 = (long long)p0[l];
        a.s0 = sph[l].s0;
        a.B = Bl[l];
        return L;
    }

    void collect(int n, bool hi) {
        if (!prof) return;
        for (int k = 0; k < n; ++k) {
            float a = 0, b = 0;
            if (cudaEventElapsedTime(&a, ctx->prof_ev[4 * k], ctx->prof_ev[4 * k + 1]) != cudaSuccess ||
                cudaEventElapsedTime(&b, ctx->prof_ev[4 * k + 2], ctx->prof_ev[4 * k + 3]) != cudaSuccess) {
                cudaGetLastError();
                a = b = 0;
            }
            (hi ? ctx->prof_a_hi_ms : ctx->prof_a_ms) += a;
            (hi ? ctx->prof_b_hi_ms : ctx->prof_b_ms) += b;
        }
        (hi ? ctx->prof_a_hi_n : ctx->prof_a_n) += n;
        (hi ? ctx->prof_b_hi_n : ctx->prof_b_n) += n;
    }

    // a block-fixed-point field of this solve passed through a double2 pointer, from element o on
    BFF bfield(void *f, size_t o = 0) const {
        bfc *v = (bfc *)f;
        return BFF{v + o, (int *)(v + nfield) + o / 12};
    }

    // a half-format field of this solve passed through a float2 pointer
    template <typename HT> HF<HT> hfield(void *f) const {
        typename HT::h2 *v = (typename HT::h2 *)f;
        return HF<HT>{v, (float *)(v + nfield)};
    }

    // Capacity of the history for this solve: hist_bytes_wanted per support element,
    // at most a twelfth of the GPU's memory or what the directions p_i take (a
    // chunk's end needs them, so that the solve can go on with less).  The solve's
    // fields and the directions come first: where the rest of the free memory does not
    // hold the history as well, the directions are set aside at once and it takes
    // three quarters of what is left then.
    int plan_history() {
        std::vector<Buf> &ws = ctx->ws;
        Buf &hist = ws[W_HIST];
        const int prec = in[0].spec->prec;
        const bool fp64 = prec == SMPQ_FP64, both = prec == SMPQ_MIXED;
        const size_t eb = fp64 || both ? sizeof(double2) : sizeof(float2);
        const size_t dirs = (size_t)nshift * ((fp64 || both ? sizeof(double2) : 0) + (fp64 ? 0 : sizeof(float2)));
        const size_t most = std::max(dirs, ctx->mem_total / 12 / nsupf / eb * eb);
        size_t want = std::min(hist_bytes_wanted(prec, ctx->opt.max_iter), most);
        const size_t fields = missing_fields();
        if (hist.bytes < want * nsupf || fields > 0) {
            auto room = [&]() { // free for the history, less a little for buffers of a few bytes a source
                size_t freeb = 0, totb = 0;
                cudaMemGetInfo(&freeb, &totb);
                const size_t rows = want / (fp64 ? sizeof(double2) : sizeof(float2));
                const size_t need = missing_fields() + missing_dirs() + rows * nshift * B * 32;
                const size_t have = (freeb + hist.bytes) / 64 * 63;
                return have > need ? have - need : 0;
            };
            int rc;
            const size_t r = room();
            if (hist.bytes > r) release(hist);
            if (want * nsupf > r) {
                if ((eb == sizeof(double2) && (rc = hist_dirs(W_PS, sizeof(double2)))) ||
                    (!fp64 && (rc = hist_dirs(W_PS32, sizeof(float2)))))
                    return rc;
                // (a history kept from the same call before stays as it is: the same chunks)
                const size_t give = std::max(room() / 4 * 3, hist.bytes);
                want = std::min(want, std::max(eb, give / nsupf / eb * eb));
            }
            if (hist.bytes < want * nsupf && (rc = ensure(ctx, hist, want * nsupf))) return rc;
        }
        hcap = want;
        hrows = (int)(hcap / (fp64 ? sizeof(double2) : sizeof(float2)));
        return SMPQ_OK;
    }
    size_t missing(int w, size_t bytes) const {
        const size_t held = ctx->ws[w].bytes;
        return bytes > held ? bytes - held : 0;
    }
    // bytes of the solve's whole-lattice fields and y that are not allocated yet (run())
    size_t missing_fields() const {
        const size_t nf = nfield, d = nf * sizeof(double2), f = nf * sizeof(float2), hf = nf * 4 + nf / 12 * 4 + 256;
        size_t m = missing(W_Y, nsupf * sizeof(double2));
        if (in[0].spec->full_support) m += missing(W_OUT, d);
        auto add = [&](size_t b, std::initializer_list<int> l) {
            for (int w : l) m += missing(w, b);
        };
        switch (in[0].spec->prec) {
        case SMPQ_FP64:
            add(d + nf / 12 * sizeof(int), {W_P, W_T, W_R});
            if (ctx->opt.true_residual) add(d, {W_XHI, W_T64});
            break;
        case SMPQ_MIXED:
            add(d, {W_P, W_T, W_R});
            if (ctx->opt.true_residual) add(d, {W_XHI});
            add(4 * f, {W_XLO});
            break;
        case SMPQ_FP32:
            add(f, {W_P, W_T, W_R, W_XLO});
            add(d, {W_XHI, W_T64});
            break;
        default:
            add(hf, {W_P, W_T});
            add(f, {W_R, W_XLO});
            add(d, {W_XHI, W_T64});
        }
        return m;
    }
    // bytes of the directions that are not allocated yet
    size_t missing_dirs() const {
        const int prec = in[0].spec->prec;
        const size_t n = (size_t)nshift * nsupf;
        return (prec == SMPQ_FP64 || prec == SMPQ_MIXED ? missing(W_PS, n * sizeof(double2)) : 0) +
               (prec == SMPQ_FP64 ? 0 : missing(W_PS32, n * sizeof(float2)));
    }

    // the slots left in the chunk for iterations of an eb-byte residual
    int hist_left(size_t eb) const { return std::min(hrows, (int)(hcap / eb)) - hn; }

    // the directions that outlive a chunk: ps (FP64) and ps32 in one buffer each
    int hist_dirs(int w, size_t eb) { return ensure(ctx, ctx->ws[w], (size_t)nshift * nsupf * eb); }
    HistLat hist_lat(int l) const {
        HistLat L{};
        L.ne = (size_t)Bl[l] * 12 * in[l].spec->n_sup;
        L.n_sup = in[l].spec->n_sup;
        L.V = V[l];
        L.j0 = j0[l];
        L.nshift = nshift;
        L.B = B;
        L.supsite = in[l].spec->d_supsite;
        L.rhs_class = in[l].spec->d_rhs_class;
        L.src = srcl[l];
        L.stride = nsupf;
        L.n = hn;
        L.first = hfirst;
        return L;
    }
    template <typename F> void shift_groups(F launch) const {
        if (nshift == 1) launch(std::integral_constant<int, 1>());
        else launch(std::integral_constant<int, 14>());
    }
    int hist_next(bool last, int launched) {
        ctx->launches += launched;
        if (!last) cudaMemsetAsync(sc.slot, 0, (size_t)B * sizeof(int), st);
        hn = 0;
        hfirst = false;
        return cuda_check(ctx, cudaGetLastError(), "residual history");
    }
    // The end of a chunk of FP64-accurate iterations with slots of type C: its
    // share of y, and the directions if the solve goes on (next: 0 it ends, 1
    // more such iterations, 2 FP32 ones).  Then the slots are free again.
    template <typename C> int hist_flush(int next) {
        std::vector<Buf> &ws = ctx->ws;
        const int n = hn;
        int rc;
        if (next == 1 && (rc = hist_dirs(W_PS, sizeof(double2)))) return rc;
        if (next == 2 && (rc = hist_dirs(W_PS32, sizeof(float2)))) return rc;
        for (int l = 0; l < nl; ++l)
            k_hist_w<<<(nshift * Bl[l] + 127) / 128, 128, 0, st>>>(n, nshift, B, j0[l], Bl[l], spd + l, sc, hv0, hd0, next == 2);
        k_hist_sum<<<(unsigned)(((size_t)(n + 1) * B + 255) / 256), 256, 0, st>>>(n, nshift, B, sc.hz, hv0, hw);
        for (int l = 0; l < nl; ++l) {
            HistLat L = hist_lat(l);
            L.h = (const C *)ws[W_HIST].p + s0[l];
            double2 *ps = (double2 *)ws[W_PS].p + s0[l];
            float2 *ps32 = (float2 *)ws[W_PS32].p + s0[l];
            const unsigned nb = (unsigned)((L.ne + 255) / 256);
            k_hist_y<C, BC><<<nb, 256, 0, st>>>(L, hw, hv0, ps, y + s0[l]);
            const dim3 grid = hist_grid<BC>(L);
            const int TH = TileMap<BC>::THREADS;
            shift_groups([&](auto ng) {
                constexpr int NG = decltype(ng)::value;
                if (next == 1) k_hist_p<C, BC, false, NG><<<grid, TH, 0, st>>>(L, sc.ho, hd0, ps, ps32);
                if constexpr (std::is_same<C, df64c>::value)
                    if (next == 2) k_hist_p<C, BC, true, NG><<<grid, TH, 0, st>>>(L, sc.ho, hd0, ps, ps32);
            });
        }
        return hist_next(next == 0, 1 + (next ? 3 : 2) * nl);
    }
    // the end of a chunk of FP32 iterations
    int hist_flush32(bool last) {
        std::vector<Buf> &ws = ctx->ws;
        const bool exact = hist_exact(in[0].spec->prec, ctx->opt.switch_residual);
        int rc;
        if (!last && (rc = hist_dirs(W_PS32, sizeof(float2)))) return rc;
        for (int l = 0; l < nl; ++l) {
            const size_t nc = (size_t)hn * nshift * Bl[l];
            if (nc) k_hist_coef<<<(unsigned)((nc + 255) / 256), 256, 0, st>>>(hn, nshift, B, j0[l], Bl[l], spd + l, sc, hct);
            HistLat L = hist_lat(l);
            L.h = (const float2 *)ws[W_HIST].p + s0[l];
            float2 *ps32 = (float2 *)ws[W_PS32].p + s0[l];
            const dim3 nb = hist_grid<BC>(L);
            const int TH = TileMap<BC>::THREADS;
            shift_groups([&](auto ng) {
                constexpr int NG = decltype(ng)::value;
                if (exact) k_hist_run<BC, true, NG><<<nb, TH, 0, st>>>(L, sc.ho, hct, ps32, y + s0[l], last);
                else k_hist_run<BC, false, NG><<<nb, TH, 0, st>>>(L, sc.ho, hct, ps32, y + s0[l], last);
            });
        }
        return hist_next(last, 2 * nl);
    }

    // Iterate with vectors of precision T (residual history likewise).
    // init: start from x = 0 (sources); otherwise continue from the current state.
    // rel: FP64 reliable updates (needs xlo, xhi, t64).  theta2 > 0: return once
    // every active right-hand side has ||r||^2 <= theta2 ||b||^2.
    // fixed > 0: exactly `fixed` iterations, no checks (Lanczos).
    // HT (H16 or B16, T = float): p and t are half-format fields (components,
    // then norms) passed through the float2 pointers.
    // xacc (nullable): the base solution accumulated by the p updates (FP64 for
    // FP64 iterations, float-float for the mixed solve's first phase).
    template <typename T, typename HT = void>
    int phase(typename cplx_t<T>::type *p, typename cplx_t<T>::type *t, typename cplx_t<T>::type *r,
              typename cplx_t<T>::type *xlo, df64c *xhi, df64c *t64, bool init, bool rel, double theta2, int fixed, int max_iter, typename XAcc<T>::type *xacc = nullptr,
              bool replace_mid = true) {
        typedef typename cplx_t<T>::type C;
        constexpr bool half = !std::is_void<HT>::value;
        constexpr bool fixed_point = std::is_same<T, double>::value; // p, t, r through double2 pointers
        const int TH = TileMap<BC>::THREADS;
        const bool hi = sizeof(T) != sizeof(float); // FP64 or float-float iterations
        const bool multi = nl > 1;
        // kernel shape of the D_W launches (the autotuner's choice): tiles per
        // block, per phase, and for the FP32 kernels one or two columns per thread
        int tpb = hi ? tpb_hi : tpb_lo;
        if (fixed_point && in[0].spec->tpb_hi == 0) { // no tuned shape: several blocks for each SM
            size_t tiles = 0;
            for (int l = 0; l < nl; ++l) tiles += (size_t)nch[l] * ((V[l] + BfMap<BC>::SPB - 1) / BfMap<BC>::SPB);
            while (tpb > 1 && tiles / tpb < 2048) tpb /= 2;
        }
        const bool two_cols = std::is_same<T, float>::value && !half && nr == 2 && BC % 2 == 0 && !multi;
        constexpr bool can_stage = std::is_same<T, float>::value && !half && BC >= 12;
        constexpr bool can_stage_df = std::is_same<T, df64>::value && BC >= 12;
        const bool staged = can_stage && stg;
        const bool staged_df = can_stage_df && stg_df;
        if constexpr (can_stage) {
            if (staged) { // before any capture: the kernels' shared-memory limit
                const cudaError_t e = multi ? staged_attrs<BC, true>() : staged_attrs<BC, false>();
                if (e != cudaSuccess) return cuda_check(ctx, e, "staged D_W attributes");
            }
        }
        if constexpr (can_stage_df) {
            if (staged_df) {
                const cudaError_t e = multi ? staged_df_attrs<BC, true>() : staged_df_attrs<BC, false>();
                if (e != cudaSuccess) return cuda_check(ctx, e, "staged D_W attributes");
            }
        }
        // Half-storage iterations replace the residual at least every 10x drop:
        // their iterated residual drifts from the true one by about the format's
        // rounding times the condition number per iteration, so a 1000x drop
        // (the FP32 default) would outlast its meaning.
        const double delta = half ? std::max(ctx->opt.reliable_delta, 0.1) : ctx->opt.reliable_delta;
        // replace_mid = false: one replacement when every shift has converged
        // (then only the base shift can re-activate, so the replacement never
        // enters the shifted systems; the mixed solve's FP32 phase)
        const double delta2 = rel && replace_mid ? delta * delta : 0.0;
        const T kappa = (T)ctx->opt.kappa;
        const double kd = ctx->opt.kappa;
        const int per_iter = 3;
        if constexpr (half) {
            if (!rel || !xlo || !xhi || !t64)
                return set_err(ctx, SMPQ_EINVAL, "internal: half-storage iterations need FP64 reliable updates");
        }
        // every launch's partial rows must fit the partial buffers (npart per
        // buffer): the D_W launches at this tpb (one column: the most blocks)
        // and the one-column lattice kernels
        {
            size_t rows = 0;
            const int spb = fixed_point ? BfMap<BC>::SPB : TileMap<BC>::SPB;
            for (int l = 0; l < nl; ++l)
                rows += (size_t)nch[l] * std::max(((V[l] + spb - 1) / spb + tpb - 1) / tpb, G1[l]);
            if (rows * BC > npart)
                return set_err(ctx, SMPQ_EINVAL, "internal: launch shape exceeds the partial-sum buffers");
        }
        if (init) {
            for (int l = 0; l < nl; ++l) {
                const dim3 grid(G1[l], nch[l]);
                const Geom &g = in[l].ctx->geom;
                const size_t o = f0[l];
                double *pl = part0 + p0[l] * BC;
                int G = G1[l];
                if constexpr (fixed_point) {
                    G = (V[l] + BfMap<BC>::SPB - 1) / BfMap<BC>::SPB;
                    k_init_bf<BC><<<dim3(G, nch[l]), BfMap<BC>::THREADS, 0, st>>>(g, srcl[l], bfield(r, o), bfield(p, o),
                                                                                 pl, G);
                } else if constexpr (half)
                    k_init_h<HT, BC><<<grid, TH, 0, st>>>(g, srcl[l], (float2 *)r + o, hfield_at<HT>(p, o),
                                                          (float2 *)xlo + o, xhi + o, pl, G1[l]);
                else
                    k_init<T, BC><<<grid, TH, 0, st>>>(g, srcl[l], r + o, p + o, xlo ? xlo + o : nullptr,
                                                       xhi ? xhi + o : nullptr, pl, G1[l]);
                s_init<<<Bl[l], SCAL_THREADS, 0, st>>>(B, BC, G, pl, scal_of(l), sph[l], sqrt(tol2));
                ctx->launches += 2;
            }
        }
        // the scalar steps ride on the last block of each RHS tile of launches A and B
        const Fuse f1{count, count + nchunk, ngroups, sc, spd, B, 0.0, 0.0, 0.0};
        const Fuse f2{count, count + nchunk, ngroups, sc, spd, B, tol2, delta2, theta2};
        int gyp, tyy;
        const Lats Lyp = lats_yp(fixed_point ? BfMap<BC>::SPB : TileMap<BC>::SPB, &gyp, &tyy);
        C *hbase = shifts ? (C *)ctx->ws[W_HIST].p : nullptr;
        const dim3 gridyp(gyp, nchunk);
        const int *rhs_class = in[0].spec->d_rhs_class;
        // two columns per thread for even tiles (SMPQ_HALF_SOLVE_NR=1: one)
#ifndef SMPQ_HALF_SOLVE_NR
#define SMPQ_HALF_SOLVE_NR 2
#endif
        constexpr bool h2cols = SMPQ_HALF_SOLVE_NR == 2 && BC % 2 == 0;
        typedef TileMap<BC, h2cols ? 2 : 1> TMH;
        auto iteration_half = [&](int k) {
            if constexpr (half) {
                const HF<HT> hp = hfield<HT>(p), ht = hfield<HT>(t);
                constexpr int THH = TMH::THREADS;
                int gx;
                const Lats Ld = lats_dw<T, HT>(TMH::SPB, tpb, &gx);
                const dim3 gridh(gx, nchunk);
                auto launch = [&](auto m) {
                    constexpr bool M = decltype(m)::value;
                    if (prof) cudaEventRecord(ctx->prof_ev[4 * k], st);
                    if constexpr (h2cols)
                        k_apply_a_h2<HT, BC, M><<<gridh, THH, 0, st>>>(Ld, hp, ht, (float)kappa, part0, part1, tpb, f1);
                    else
                        k_apply_a_h<HT, BC, M><<<gridh, THH, 0, st>>>(Ld, hp, ht, (float)kappa, part0, part1, tpb, f1);
                    if (prof) cudaEventRecord(ctx->prof_ev[4 * k + 1], st);
                    if (prof) cudaEventRecord(ctx->prof_ev[4 * k + 2], st);
                    if constexpr (h2cols)
                        k_apply_b_h2<HT, BC, M><<<gridh, THH, 0, st>>>(Ld, ht, hp, (float2 *)r, sc.alpha, (float)kappa,
                                                                       part2, tpb, f2);
                    else
                        k_apply_b_h<HT, BC, M><<<gridh, THH, 0, st>>>(Ld, ht, hp, (float2 *)r, sc.alpha, (float)kappa,
                                                                      part2, tpb, f2);
                    if (prof) cudaEventRecord(ctx->prof_ev[4 * k + 3], st);
                    k_yp_h<HT, BC, M><<<gridyp, TH, 0, st>>>(Lyp, tyy, rhs_class, (const float2 *)r, (float2 *)hbase,
                                                             nsupf, sc, hp, (float2 *)xlo);
                };
                if (multi) launch(std::true_type());
                else launch(std::false_type());
            }
        };
        auto iteration = [&](int k) {
            if constexpr (half) {
                iteration_half(k);
                return;
            }
            // the D_W pair with NR columns per thread, then launch YP
            auto launch = [&](auto nr_c, auto m) {
                constexpr int NR = decltype(nr_c)::value;
                constexpr bool M = decltype(m)::value;
                if constexpr (fixed_point) {
                    if constexpr (NR == 1) {
                        int gx;
                        const Lats Ld = lats_dw<T>(BfMap<BC>::SPB, tpb, &gx);
                        const BFF bp = bfield(p), bt = bfield(t), br = bfield(r);
                        const BfScal ks = bf_scal(kd);
                        constexpr int THB = BfMap<BC>::THREADS;
                        if (prof) cudaEventRecord(ctx->prof_ev[4 * k], st);
                        k_apply_a_bf<BC, M><<<dim3(gx, nchunk), THB, 0, st>>>(Ld, bp, bt, ks, part0, part1, tpb, f1);
                        if (prof) cudaEventRecord(ctx->prof_ev[4 * k + 1], st);
                        if (prof) cudaEventRecord(ctx->prof_ev[4 * k + 2], st);
                        k_apply_b_bf<BC, M><<<dim3(gx, nchunk), THB, 0, st>>>(Ld, bt, bp, br, sc.alpha, ks, part2, tpb,
                                                                              f2);
                        if (prof) cudaEventRecord(ctx->prof_ev[4 * k + 3], st);
                        k_yp_bf<BC, M><<<gridyp, THB, 0, st>>>(Lyp, tyy, rhs_class, br, (double2 *)hbase, nsupf, sc, bp,
                                                               (double2 *)xacc);
                    }
                    return;
                }
                if constexpr (can_stage && NR == 1) {
                    if (staged) {
                        int gx;
                        const Lats Ld = lats_dw<T>(TileMap<BC>::SPB, tpb, &gx);
                        const dim3 gridn(gx, nchunk);
                        const size_t smem = stage::Dims<BC, stage::NSTAGE>::SMEM;
                        if (prof) cudaEventRecord(ctx->prof_ev[4 * k], st);
                        k_apply_a_st<BC, M><<<gridn, TH, smem, st>>>(Ld, p, t, kd, part0, part1, tpb, f1,
                                                                      sc.flags + 4);
                        if (prof) cudaEventRecord(ctx->prof_ev[4 * k + 1], st);
                        if (prof) cudaEventRecord(ctx->prof_ev[4 * k + 2], st);
                        k_apply_b_st<BC, M><<<gridn, TH, smem, st>>>(Ld, t, p, r, sc.alpha, kd, part2, tpb, f2,
                                                                      sc.flags + 4);
                        if (prof) cudaEventRecord(ctx->prof_ev[4 * k + 3], st);
                        k_yp<T, BC, M><<<gridyp, TH, 0, st>>>(Lyp, tyy, rhs_class, r, hbase, nsupf, sc, p, xacc, xlo);
                        return;
                    }
                }
                if constexpr (can_stage_df && NR == 1) {
                    if (staged_df) {
                        int gx;
                        const Lats Ld = lats_dw<T>(TileMap<BC>::SPB, tpb, &gx);
                        const dim3 gridn(gx, nchunk);
                        const size_t smem = stage::DimsDF<BC, stage::NSTAGE_DF>::SMEM;
                        if (prof) cudaEventRecord(ctx->prof_ev[4 * k], st);
                        k_apply_a_dfst<BC, M><<<gridn, TH, smem, st>>>(Ld, p, t, kappa, part0, part1, tpb, f1,
                                                                        sc.flags + 4);
                        if (prof) cudaEventRecord(ctx->prof_ev[4 * k + 1], st);
                        if (prof) cudaEventRecord(ctx->prof_ev[4 * k + 2], st);
                        k_apply_b_dfst<BC, M><<<gridn, TH, smem, st>>>(Ld, t, p, r, sc.alpha, kappa, part2, tpb, f2,
                                                                        sc.flags + 4);
                        if (prof) cudaEventRecord(ctx->prof_ev[4 * k + 3], st);
                        k_yp<T, BC, M><<<gridyp, TH, 0, st>>>(Lyp, tyy, rhs_class, r, hbase, nsupf, sc, p, xacc, xlo);
                        return;
                    }
                }
                if constexpr (!fixed_point && (NR == 1 || (std::is_same<T, float>::value && BC % 2 == 0 && !M))) {
                    typedef TileMap<BC, NR> TMN;
                    int gx;
                    const Lats Ld = lats_dw<T>(TMN::SPB, tpb, &gx);
                    const dim3 gridn(gx, nchunk);
                    if (prof) cudaEventRecord(ctx->prof_ev[4 * k], st);
                    k_apply_a<T, BC, NR, M><<<gridn, TMN::THREADS, 0, st>>>(Ld, p, t, kd, part0, part1, tpb, f1);
                    if (prof) cudaEventRecord(ctx->prof_ev[4 * k + 1], st);
                    if (prof) cudaEventRecord(ctx->prof_ev[4 * k + 2], st);
                    k_apply_b<T, BC, NR, M><<<gridn, TMN::THREADS, 0, st>>>(Ld, t, p, r, sc.alpha, kd, part2, tpb,
                                                                            f2);
                    if (prof) cudaEventRecord(ctx->prof_ev[4 * k + 3], st);
                    k_yp<T, BC, M><<<gridyp, TH, 0, st>>>(Lyp, tyy, rhs_class, r, hbase, nsupf, sc, p, xacc, xlo);
                }
            };
            if (multi) launch(std::integral_constant<int, 1>(), std::true_type());
            else if (two_cols) launch(std::integral_constant<int, 2>(), std::false_type());
            else launch(std::integral_constant<int, 1>(), std::false_type());
        };
        // residual replacement, lattice by lattice: x_hi += x_lo, r = b - (A + s0) x_hi in float-float
        auto reliable = [&]() {
            if constexpr (fixed_point) return; // (no residual replacement in FP64)
            else {
            const df64 kdf(ctx->opt.kappa);
            Fuse none{};
            for (int l = 0; l < nl; ++l) {
                const dim3 grid(G1[l], nch[l]);
                const size_t o = f0[l];
                const Geom &g = in[l].ctx->geom;
                const df64c *Udf = (const df64c *)in[l].ctx->Udf.p;
                k_rel_accum<T, BC><<<grid, TH, 0, st>>>(V[l], xhi + o, xlo + o, G1[l]);
                k_apply_a<df64, BC, 1, false><<<grid, TH, 0, st>>>(lats_one<df64>(l), xhi, t64, ctx->opt.kappa, part0,
                                                                   part1, TPB, none);
                k_rel_resid_df<T, BC><<<grid, TH, 0, st>>>(g, Udf, t64 + o, xhi + o, srcl[l], r + o, sph[l].s0, kdf,
                                                           part2 + p0[l] * BC, G1[l]);
                ctx->launches += 3;
            }
            cudaMemsetAsync(sc.flags, 0, 2 * sizeof(int), st);
            for (int l = 0; l < nl; ++l) {
                int base = 0;
                for (int i = 1; i < nshift; ++i)
                    if (sph[l].sig[i] < sph[l].sig[base]) base = i;
                s_rel<<<Bl[l], SCAL_THREADS, 0, st>>>(B, BC, G1[l], part2 + p0[l] * BC, scal_of(l), sph[l], tol2, base);
                ctx->launches += 1;
            }
            // A replacement once every shift has converged (replace_mid = false)
            // re-activates at most the base shift, whose true residual can then be
            // many times the iterated one: its CG restarts from p = r (the old
            // direction belongs to the drifted residual history).
            if (!replace_mid && !half) {
                for (int l = 0; l < nl; ++l) {
                    const size_t nfl = (size_t)12 * V[l] * Bl[l];
                    k_restart_p<C><<<(unsigned)((nfl + 255) / 256), 256, 0, st>>>(r + f0[l], p + f0[l], nfl, BC, V[l],
                                                                                   sc.act_rhs + j0[l]);
                    ctx->launches += 1;
                }
            }
            }
        };
        if (fixed > 0) {
            for (int k = 0; k < fixed; ++k) {
                iteration(prof ? k % chk : 0);
                if (prof && k % chk == chk - 1) {
                    cudaStreamSynchronize(st);
                    collect(chk, hi);
                }
            }
            ctx->launches += (long long)fixed * per_iter;
            iters += fixed;
            return SMPQ_OK;
        }
        // (profiling records CUDA events between launches, so it runs without a graph)
        cudaGraphExec_t gexec = nullptr;
        bool graph_ok = false;
        // the phase that ends at the switch residual checks every 2 iterations:
        // its iterations are the expensive ones, and overshoot would waste them
        // (no longer than the history can take between two checks)
        const size_t he = hi ? sizeof(double2) : sizeof(float2);
        int ck = theta2 > 0 ? std::min(chk, 2) : chk;
        if (shifts) ck = std::max(1, std::min(ck, std::min(hrows, (int)(hcap / he))));
        if (ctx->opt.use_graphs && !prof) {
            cudaGraph_t graph;
            if (cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
                for (int k = 0; k < ck; ++k) iteration(k);
                if (cudaStreamEndCapture(st, &graph) == cudaSuccess) {
                    if (cudaGraphInstantiate(&gexec, graph, 0) == cudaSuccess) graph_ok = true;
                    cudaGraphDestroy(graph);
                }
            }
            cudaGetLastError();
        }
        int status = SMPQ_OK;
        for (;;) {
            if (shifts && hist_left(he) < ck) {
                if constexpr (std::is_same<T, float>::value) status = hist_flush32(false);
                else status = hist_flush<C>(1);
                if (status) break;
            }
            if (graph_ok) cudaGraphLaunch(gexec, st);
            else
                for (int k = 0; k < ck; ++k) iteration(k);
            ctx->launches += (long long)ck * per_iter;
            iters += ck;
            if (shifts) hn += ck;
            cudaMemcpyAsync(hflags, sc.flags, NFLAGS * sizeof(int), cudaMemcpyDeviceToHost, st);
            cudaError_t e = cudaStreamSynchronize(st);
            if (e != cudaSuccess) { status = cuda_check(ctx, e, "multishift iteration"); break; }
            collect(ck, hi);
            if (hflags[4]) {
                status = set_err(ctx, SMPQ_ECUDA, "a shared-memory staging wait of the D_W timed out");
                break;
            }
            if (hflags[2]) { status = set_err(ctx, SMPQ_EBREAKDOWN, "CG breakdown: <p,Ap> <= 0 or not finite"); break; }
            bool done = hflags[0] == 0;
            if (rel && (hflags[1] || done)) {
                reliable();
                ++nrel;
                cudaMemcpyAsync(hflags, sc.flags, NFLAGS * sizeof(int), cudaMemcpyDeviceToHost, st);
                e = cudaStreamSynchronize(st);
                if (e != cudaSuccess) { status = cuda_check(ctx, e, "residual replacement"); break; }
                done = hflags[0] == 0;
            }
            if (done) break;
            if (theta2 > 0 && hflags[3] == 0) break; // every rhs below the switch residual
            if (iters >= max_iter) {
                // the largest relative residual reached, for the message
                std::vector<double> hrr(B), hbb(B);
                cudaMemcpy(hrr.data(), sc.rr, B * sizeof(double), cudaMemcpyDeviceToHost);
                cudaMemcpy(hbb.data(), sc.bb, B * sizeof(double), cudaMemcpyDeviceToHost);
                double worst = 0;
                for (int j = 0; j < B; ++j)
                    if (hbb[j] > 0) worst = std::max(worst, std::sqrt(hrr[j] / hbb[j]));
                char msg[160];
                std::snprintf(msg, sizeof msg, "multishift CG reached max_iter (%d iterations, base residual %.3e)",
                              iters, worst);
                status = set_err(ctx, SMPQ_ENOCONV, msg);
                break;
            }
        }
        if (gexec) cudaGraphExecDestroy(gexec);
        return status;
    }

    // a half field's view at element offset o (components o..., norms o / 12...)
    template <typename HT> HF<HT> hfield_at(void *f, size_t o) const {
        HF<HT> h = hfield<HT>(f);
        return HF<HT>{h.v + o, h.n + o / 12};
    }

    bool relpath = false; // FP32 / half / mixed: the last reliable update left |b - (A + s0) x_hi|^2 in sc.rr

    // True residual of the base system from the FP64 solution x64 (FP64 path):
    // t64 = D_W x64, |b - (D_W^dag t64 + s0 x64)|^2 per rhs into rr_out (the
    // residual itself goes to the scratch field rs).
    int true_residual(double2 *t64, double2 *rs, double *rr_out) {
        const int TH = TileMap<BC>::THREADS;
        for (int l = 0; l < nl; ++l) {
            const dim3 grid(G1[l], nch[l]);
            const size_t o = f0[l];
            smpq_ctx *c = in[l].ctx;
            launch_dslash<double>(c->geom, c->U64.p, x64 + o, t64 + o, Bl[l], BC, 0, ctx->opt.kappa, st);
            k_rel_resid<double, BC><<<grid, TH, 0, st>>>(c->geom, (const double2 *)c->U64.p, t64 + o, x64 + o,
                                                         srcl[l], rs + o, sph[l].s0, ctx->opt.kappa,
                                                         part2 + p0[l] * BC, G1[l]);
            s_sum_rhs<<<Bl[l], SCAL_THREADS, 0, st>>>(BC, G1[l], part2 + p0[l] * BC, rr_out + j0[l]);
            ctx->launches += 3;
        }
        return cuda_check(ctx, cudaGetLastError(), "true residual");
    }

    // The base system's true residual in float-float without replacing r:
    // x_hi += x_lo, t = D_W x_hi, |b - (A + s0) x_hi|^2 per rhs into true_rr
    // (rs: scratch for the residual itself).
    int measure_residual_df(df64c *xhi, float2 *xlo, df64c *t64, float2 *rs) {
        const int TH = TileMap<BC>::THREADS;
        const df64 kdf(ctx->opt.kappa);
        Fuse none{};
        for (int l = 0; l < nl; ++l) {
            const dim3 grid(G1[l], nch[l]);
            const size_t o = f0[l];
            const df64c *Udf = (const df64c *)in[l].ctx->Udf.p;
            k_rel_accum<float, BC><<<grid, TH, 0, st>>>(V[l], xhi + o, xlo + o, G1[l]);
            k_apply_a<df64, BC, 1, false><<<grid, TH, 0, st>>>(lats_one<df64>(l), xhi, t64, ctx->opt.kappa, part0, part1, TPB,
                                                               none);
            k_rel_resid_df<float, BC><<<grid, TH, 0, st>>>(in[l].ctx->geom, Udf, t64 + o, xhi + o, srcl[l], rs + o,
                                                           sph[l].s0, kdf, part2 + p0[l] * BC, G1[l]);
            s_sum_rhs<<<Bl[l], SCAL_THREADS, 0, st>>>(BC, G1[l], part2 + p0[l] * BC, true_rr + j0[l]);
            ctx->launches += 4;
        }
        return cuda_check(ctx, cudaGetLastError(), "true residual");
    }

    int finish(int fixed, const double *d_true_rr = nullptr) {
        cudaEventRecord(ctx->ev2, st);
        std::vector<double> hz((size_t)nshift * B), hrr(B), hbb(B);
        std::vector<int> hit(B);
        std::vector<double> htr(d_true_rr ? B : 0);
        if (d_true_rr) cudaMemcpyAsync(htr.data(), d_true_rr, B * sizeof(double), cudaMemcpyDeviceToHost, st);
        cudaMemcpyAsync(hz.data(), sc.zeta, hz.size() * sizeof(double), cudaMemcpyDeviceToHost, st);
        cudaMemcpyAsync(hrr.data(), sc.rr, B * sizeof(double), cudaMemcpyDeviceToHost, st);
        cudaMemcpyAsync(hbb.data(), sc.bb, B * sizeof(double), cudaMemcpyDeviceToHost, st);
        cudaMemcpyAsync(hit.data(), sc.iters, B * sizeof(int), cudaMemcpyDeviceToHost, st);
        cudaError_t e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return cuda_check(ctx, e, "multishift statistics");
        float ms = 0;
        cudaEventElapsedTime(&ms, ctx->ev1, ctx->ev2);
        for (int l = 0; l < nl; ++l) {
            double worst = 0, tr = 0;
            int maxit = 0;
            for (int j = j0[l]; j < j0[l] + Bl[l]; ++j) {
                if (!(hbb[j] > 0)) continue;
                for (int i = 0; i < nshift; ++i)
                    worst = std::max(worst, std::fabs(hz[(size_t)i * B + j]) * std::sqrt(hrr[j] / hbb[j]));
                maxit = std::max(maxit, hit[j]);
                tr = std::max(tr, std::sqrt((d_true_rr ? htr[j] : hrr[j]) / hbb[j]));
            }
            SolveOut *out = in[l].out;
            out->y = y + s0[l];
            out->iterations = fixed > 0 ? fixed : maxit;
            out->reliable_updates = nrel;
            out->max_resid = worst;
            out->true_resid = (relpath || d_true_rr) ? tr : -1;
            out->solve_ms = ms;
        }
        return cuda_check(ctx, cudaGetLastError(), "multishift launch");
    }

    // FP64 path with the true_residual option: x64 (and t64 for the final
    // check) on the whole lattice, x64 starting at 0
    int alloc_x64() {
        if (!ctx->opt.true_residual || !shifts) return SMPQ_OK;
        std::vector<Buf> &ws = ctx->ws;
        int rc;
        if ((rc = ensure(ctx, ws[W_XHI], nfield * sizeof(double2)))) return rc;
        if ((rc = ensure(ctx, ws[W_T64], nfield * sizeof(double2)))) return rc;
        x64 = (double2 *)ws[W_XHI].p;
        cudaMemsetAsync(x64, 0, nfield * sizeof(double2), st);
        return SMPQ_OK;
    }

    static int run(const std::vector<LatIn> &lats, double tol, int max_iter, double *hist, int hist_len, int fixed) {
        Solve S(lats);
        smpq_ctx *ctx = S.ctx;
        int rc = S.setup(tol, hist, hist_len);
        if (rc) return rc;
        std::vector<Buf> &ws = ctx->ws;
        const size_t nf = S.nfield;
        const bool shifts = S.shifts;
        const int prec = lats[0].spec->prec;
        cudaEventRecord(ctx->ev1, S.st);
        if (prec == SMPQ_FP64) {
            const size_t fb = nf * sizeof(bfc) + nf / 12 * sizeof(int);
            if ((rc = ensure(ctx, ws[W_P], fb))) return rc;
            if ((rc = ensure(ctx, ws[W_T], fb))) return rc;
            if ((rc = ensure(ctx, ws[W_R], fb))) return rc;
            if (shifts && (rc = ensure(ctx, ws[W_Y], S.nsupf * sizeof(double2)))) return rc;
            S.y = shifts ? (double2 *)ws[W_Y].p : nullptr;
            if ((rc = S.alloc_x64())) return rc;
            rc = S.template phase<double>((double2 *)ws[W_P].p, (double2 *)ws[W_T].p, (double2 *)ws[W_R].p, nullptr,
                                          nullptr, nullptr, true, false, 0.0, fixed, max_iter, S.x64);
            if (rc) return rc;
            if (shifts && (rc = S.template hist_flush<double2>(0))) return rc;
            if (S.x64 && (rc = S.true_residual((double2 *)ws[W_T64].p, (double2 *)ws[W_R].p, S.true_rr))) return rc;
        } else if (prec == SMPQ_MIXED) {
            // true_residual 0: no base solution is kept (the fastest form);
            // 1: x_hi (float-float, phase 1) and x_lo (FP32, phase 2) accumulate
            // the base solution and its true residual is measured at the end;
            // 2: as 1, and the base system is driven to a true residual below
            // tol (see phase 2)
            const int tres = ctx->opt.true_residual;
            // phase 1: float-float (FP64-accurate) vectors and D_W down to the switch residual
            if ((rc = ensure(ctx, ws[W_P], nf * sizeof(df64c)))) return rc;
            if ((rc = ensure(ctx, ws[W_T], nf * sizeof(df64c)))) return rc;
            if ((rc = ensure(ctx, ws[W_R], nf * sizeof(df64c)))) return rc;
            if (tres && (rc = ensure(ctx, ws[W_XHI], nf * sizeof(df64c)))) return rc;
            if (shifts && (rc = ensure(ctx, ws[W_Y], S.nsupf * sizeof(double2)))) return rc;
            S.y = shifts ? (double2 *)ws[W_Y].p : nullptr;
            df64c *p = (df64c *)ws[W_P].p, *t = (df64c *)ws[W_T].p, *r = (df64c *)ws[W_R].p;
            df64c *xh = tres ? (df64c *)ws[W_XHI].p : nullptr;
            const double theta = ctx->opt.switch_residual;
            rc = S.template phase<df64>(p, t, r, nullptr, xh, nullptr, true, false, theta * theta, 0, max_iter, xh);
            if (rc) return rc;
            // phase 2: FP32 vectors and D_W from the phase-1 state, without
            // residual replacement: the FP32 rounding of these iterations makes
            // the base residual drift from the true one by about u_32 theta
            // times a growth factor (measured about 64 u_32 theta: 2.7e-8 at
            // theta = 7e-3), and the shifted systems drift alike.  The drift
            // is smooth over the lattice, so its share of Q = sum_x q(x) does
            // not average out: at theta >= 2e-3 |dQ| over 8^3 x 16 reached
            // 0.5-1.4e-9 for some switch points, at 1e-3 it stays below 3e-11.  With true_residual 2 the base system alone is
            // corrected once every shift has converged (one replacement, then
            // its CG restarts from the true residual): its residual meets tol,
            // but the correction no longer cancels against the other shifts'
            // drift.
            if ((rc = ensure(ctx, ws[W_XLO], 4 * nf * sizeof(float2)))) return rc;
            float2 *p32 = (float2 *)ws[W_XLO].p, *t32 = p32 + nf, *r32 = t32 + nf, *xl32 = tres ? r32 + nf : nullptr;
            const unsigned nb = (unsigned)((nf + 255) / 256);
            k_to_fp32<<<nb, 256, 0, S.st>>>(p, p32, nf);
            k_to_fp32<<<nb, 256, 0, S.st>>>(r, r32, nf);
            if (xl32) cudaMemsetAsync(xl32, 0, nf * sizeof(float2), S.st);
            ctx->launches += 2;
            cudaMemcpyAsync(S.hflags, S.sc.flags, sizeof(int), cudaMemcpyDeviceToHost, S.st);
            cudaStreamSynchronize(S.st);
            const bool enforce = tres == 2;
            if (S.hflags[0] > 0 && enforce) S.relpath = true;
            const bool more = S.hflags[0] > 0;
            if (shifts && (rc = S.template hist_flush<df64c>(more ? 2 : 0))) return rc;
            if (more) {
                rc = S.template phase<float>(p32, t32, r32, xl32, xh, t, false, enforce, 0.0, 0, max_iter, nullptr,
                                             false);
                if (rc) return rc;
                if (shifts && (rc = S.hist_flush32(true))) return rc;
            }
            if (tres == 1) { // measure the base system's true residual (x_hi += x_lo, b - (A + s0) x_hi)
                if ((rc = S.measure_residual_df(xh, xl32, t, r32))) return rc;
                return S.finish(0, S.true_rr);
            }
        } else if (prec == SMPQ_FP16N || prec == SMPQ_BF16N) {
            // p and t in the half format, the rest as in the FP32 path
            const size_t hb = (nf * 4 + nf / 12 * 4 + 255) / 256 * 256;
            if ((rc = ensure(ctx, ws[W_P], hb))) return rc;
            if ((rc = ensure(ctx, ws[W_T], hb))) return rc;
            if ((rc = ensure(ctx, ws[W_R], nf * sizeof(float2)))) return rc;
            if ((rc = ensure(ctx, ws[W_XLO], nf * sizeof(float2)))) return rc;
            if ((rc = ensure(ctx, ws[W_XHI], nf * sizeof(df64c)))) return rc;
            if ((rc = ensure(ctx, ws[W_T64], nf * sizeof(df64c)))) return rc;
            if (shifts && (rc = ensure(ctx, ws[W_Y], S.nsupf * sizeof(double2)))) return rc;
            S.y = shifts ? (double2 *)ws[W_Y].p : nullptr;
            float2 *pp = (float2 *)ws[W_P].p, *tt = (float2 *)ws[W_T].p, *rr = (float2 *)ws[W_R].p;
            float2 *xl = (float2 *)ws[W_XLO].p;
            df64c *xh = (df64c *)ws[W_XHI].p, *t64 = (df64c *)ws[W_T64].p;
            S.relpath = true;
            if (prec == SMPQ_BF16N)
                rc = S.template phase<float, B16>(pp, tt, rr, xl, xh, t64, true, true, 0.0, fixed, max_iter);
            else
                rc = S.template phase<float, H16>(pp, tt, rr, xl, xh, t64, true, true, 0.0, fixed, max_iter);
            if (rc) return rc;
            if (shifts && (rc = S.hist_flush32(true))) return rc;
        } else {
            if ((rc = ensure(ctx, ws[W_P], nf * sizeof(float2)))) return rc;
            if ((rc = ensure(ctx, ws[W_T], nf * sizeof(float2)))) return rc;
            if ((rc = ensure(ctx, ws[W_R], nf * sizeof(float2)))) return rc;
            if ((rc = ensure(ctx, ws[W_XLO], nf * sizeof(float2)))) return rc;
            if ((rc = ensure(ctx, ws[W_XHI], nf * sizeof(df64c)))) return rc;
            if ((rc = ensure(ctx, ws[W_T64], nf * sizeof(df64c)))) return rc;
            if (shifts && (rc = ensure(ctx, ws[W_Y], S.nsupf * sizeof(double2)))) return rc;
            S.y = shifts ? (double2 *)ws[W_Y].p : nullptr;
            S.relpath = true;
            rc = S.template phase<float>((float2 *)ws[W_P].p, (float2 *)ws[W_T].p, (float2 *)ws[W_R].p,
                                         (float2 *)ws[W_XLO].p, (df64c *)ws[W_XHI].p, (df64c *)ws[W_T64].p, true,
                                         true, 0.0, fixed, max_iter);
            if (rc) return rc;
            if (shifts && (rc = S.hist_flush32(true))) return rc;
        }
        return S.finish(fixed, S.x64 ? S.true_rr : nullptr);
    }
};

} // namespace

// ------------------------------------------------------------------ autotuner support
// Average time (ms) of one t = D_W p plus one r -= alpha (D_W^dag t + s0 p)
// launch (the two D_W launches of an iteration, without their scalar steps)
// for B right-hand sides in tiles of BC, tpb tiles per block and NR columns
// per thread, on scratch fields (their values do not change the work).
// reps launches each, after one untimed pair.
namespace {
template <typename F> float time_launches(smpq_ctx *ctx, int reps, F once) {
    cudaStream_t st = ctx->stream;
    once(); // warm-up
    cudaEventRecord(ctx->ev1, st);
    for (int k = 0; k < reps; ++k) once();
    cudaEventRecord(ctx->ev2, st);
    if (cudaEventSynchronize(ctx->ev2) != cudaSuccess) {
        cudaGetLastError();
        return -1.f;
    }
    float ms = 0;
    cudaEventElapsedTime(&ms, ctx->ev1, ctx->ev2);
    return ms / reps;
}

// the table of a single-lattice launch over the context's lattice
Lats lats_single(smpq_ctx *ctx, const void *U, int G) {
    Lats L{};
    L.n = 1;
    L.l[0].g = ctx->geom;
    L.l[0].U = U;
    L.l[0].G = G;
    return L;
}

template <typename T, int BC, int NR>
float time_pair(smpq_ctx *ctx, int B, int tpb, int reps, void *buf, double *part, double *alpha) {
    typedef typename cplx_t<T>::type C;
    typedef TileMap<BC, NR> TM;
    const int V = ctx->V, nchunk = B / BC;
    const int GN = ((V + TM::SPB - 1) / TM::SPB + tpb - 1) / tpb;
    const size_t nf = (size_t)B * 12 * V;
    C *p = (C *)buf, *t = p + nf, *r = t + nf;
    const Lats L = lats_single(ctx, Links<T>::get(ctx), GN);
    cudaStream_t st = ctx->stream;
    const dim3 gridn(GN, nchunk);
    Fuse none{}; // timing only: no scalar step
    return time_launches(ctx, reps, [&]() {
        k_apply_a<T, BC, NR, false><<<gridn, TM::THREADS, 0, st>>>(L, p, t, ctx->opt.kappa, part,
                                                                    part + (size_t)nchunk * GN * BC, tpb, none);
        k_apply_b<T, BC, NR, false><<<gridn, TM::THREADS, 0, st>>>(L, t, p, r, alpha, ctx->opt.kappa, part, tpb, none);
    });
}

// the FP64 pair (block fixed point)
template <int BC> float time_pair_bf(smpq_ctx *ctx, int B, int tpb, int reps, void *buf, double *part, double *alpha) {
    typedef BfMap<BC> TM;
    const int V = ctx->V, nchunk = B / BC;
    const int GN = ((V + TM::SPB - 1) / TM::SPB + tpb - 1) / tpb;
    const size_t nf = (size_t)B * 12 * V;
    bfc *v = (bfc *)buf;
    int *e = (int *)(v + 3 * nf);
    const BFF p{v, e}, t{v + nf, e + nf / 12}, r{v + 2 * nf, e + 2 * (nf / 12)};
    const Lats L = lats_single(ctx, ctx->Ubf.p, GN);
    const BfScal ks = bf_scal(ctx->opt.kappa);
    cudaStream_t st = ctx->stream;
    const dim3 gridn(GN, nchunk);
    Fuse none{};
    return time_launches(ctx, reps, [&]() {
        k_apply_a_bf<BC, false><<<gridn, TM::THREADS, 0, st>>>(L, p, t, ks, part, part + (size_t)nchunk * GN * BC, tpb,
                                                               none);
        k_apply_b_bf<BC, false><<<gridn, TM::THREADS, 0, st>>>(L, t, p, r, alpha, ks, part, tpb, none);
    });
}

// the FP32 pair with staged neighbours (one column per thread); -1 if a
// staging wait ran out (*err, zero on entry)
template <int BC>
float time_pair_staged(smpq_ctx *ctx, int B, int tpb, int reps, void *buf, double *part, double *alpha, int *err) {
    typedef TileMap<BC> TM;
    const int V = ctx->V, nchunk = B / BC;
    const int GN = ((V + TM::SPB - 1) / TM::SPB + tpb - 1) / tpb;
    const size_t nf = (size_t)B * 12 * V;
    float2 *p = (float2 *)buf, *t = p + nf, *r = t + nf;
    const Lats L = lats_single(ctx, Links<float>::get(ctx), GN);
    const double kappa = ctx->opt.kappa;
    cudaStream_t st = ctx->stream;
    const dim3 gridn(GN, nchunk);
    const size_t smem = stage::Dims<BC, stage::NSTAGE>::SMEM;
    if (staged_attrs<BC, false>() != cudaSuccess) {
        cudaGetLastError();
        return -1.f;
    }
    Fuse none{};
    const float ms = time_launches(ctx, reps, [&]() {
        k_apply_a_st<BC, false><<<gridn, TM::THREADS, smem, st>>>(L, p, t, kappa, part,
                                                                   part + (size_t)nchunk * GN * BC, tpb, none, err);
        k_apply_b_st<BC, false><<<gridn, TM::THREADS, smem, st>>>(L, t, p, r, alpha, kappa, part, tpb, none, err);
    });
    int h = 0;
    if (ms < 0 || cudaMemcpy(&h, err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess || h) {
        cudaGetLastError();
        return -1.f;
    }
    return ms;
}

// the float-float pair with staged neighbours; -1 if a staging wait ran out
template <int BC>
float time_pair_dfstaged(smpq_ctx *ctx, int B, int tpb, int reps, void *buf, double *part, double *alpha, int *err) {
    typedef TileMap<BC> TM;
    const int V = ctx->V, nchunk = B / BC;
    const int GN = ((V + TM::SPB - 1) / TM::SPB + tpb - 1) / tpb;
    const size_t nf = (size_t)B * 12 * V;
    df64c *p = (df64c *)buf, *t = p + nf, *r = t + nf;
    const Lats L = lats_single(ctx, Links<df64>::get(ctx), GN);
    const df64 kappa(ctx->opt.kappa);
    cudaStream_t st = ctx->stream;
    const dim3 gridn(GN, nchunk);
    const size_t smem = stage::DimsDF<BC, stage::NSTAGE_DF>::SMEM;
    if (staged_df_attrs<BC, false>() != cudaSuccess) {
        cudaGetLastError();
        return -1.f;
    }
    Fuse none{};
    const float ms = time_launches(ctx, reps, [&]() {
        k_apply_a_dfst<BC, false><<<gridn, TM::THREADS, smem, st>>>(L, p, t, kappa, part,
                                                                     part + (size_t)nchunk * GN * BC, tpb, none, err);
        k_apply_b_dfst<BC, false><<<gridn, TM::THREADS, smem, st>>>(L, t, p, r, alpha, kappa, part, tpb, none, err);
    });
    int h = 0;
    if (ms < 0 || cudaMemcpy(&h, err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess || h) {
        cudaGetLastError();
        return -1.f;
    }
    return ms;
}

// the half-storage pair (two columns per thread, r and x_lo in FP32)
template <typename HT, int BC>
float time_pair_half(smpq_ctx *ctx, int B, int tpb, int reps, void *buf, double *part, double *alpha) {
    typedef TileMap<BC, 2> TM;
    const int V = ctx->V, nchunk = B / BC;
    const int GN = ((V + TM::SPB - 1) / TM::SPB + tpb - 1) / tpb;
    const size_t nf = (size_t)B * 12 * V;
    const size_t hb = (half_field_bytes(V, B) + 255) / 256 * 256;
    typename HT::h2 *pv = (typename HT::h2 *)buf, *tv = (typename HT::h2 *)((char *)buf + hb);
    const HF<HT> hp{pv, (float *)(pv + nf)}, ht{tv, (float *)(tv + nf)};
    float2 *r = (float2 *)((char *)buf + 2 * hb);
    const Lats L = lats_single(ctx, HLinks<HT>::get(ctx), GN);
    const float kappa = (float)ctx->opt.kappa;
    cudaStream_t st = ctx->stream;
    const dim3 gridn(GN, nchunk);
    Fuse none{};
    return time_launches(ctx, reps, [&]() {
        k_apply_a_h2<HT, BC, false><<<gridn, TM::THREADS, 0, st>>>(L, hp, ht, kappa, part,
                                                                    part + (size_t)nchunk * GN * BC, tpb, none);
        k_apply_b_h2<HT, BC, false><<<gridn, TM::THREADS, 0, st>>>(L, ht, hp, r, alpha, kappa, part, tpb, none);
    });
}

template <int BC> float time_kind(smpq_ctx *ctx, int kind, int B, int tpb, int nr, int reps, void *buf, double *part,
                                  double *alpha, int *err) {
    switch (kind) {
    case 0: return time_pair_bf<BC>(ctx, B, tpb, reps, buf, part, alpha);
    case 1:
        return nr == 2 ? time_pair<float, BC, 2>(ctx, B, tpb, reps, buf, part, alpha)
                       : time_pair<float, BC, 1>(ctx, B, tpb, reps, buf, part, alpha);
    case 2: return time_pair<df64, BC, 1>(ctx, B, tpb, reps, buf, part, alpha);
    case 3: return time_pair_half<H16, BC>(ctx, B, tpb, reps, buf, part, alpha);
    case 4: return time_pair_half<B16, BC>(ctx, B, tpb, reps, buf, part, alpha);
    case 5: return time_pair_staged<BC>(ctx, B, tpb, reps, buf, part, alpha, err);
    case 6: return time_pair_dfstaged<BC>(ctx, B, tpb, reps, buf, part, alpha, err);
    default: return -1.f;
    }
}
} // namespace

// each RHS tile width is a translation unit of its own (msolve_bc*.cu)
template <int BC>
int solve_bc(const std::vector<LatIn> &lats, double tol, int max_iter, double *hist, int hist_len, int fixed) {
    return Solve<BC>::run(lats, tol, max_iter, hist, hist_len, fixed);
}
template <int BC> float time_kind_bc(smpq_ctx *ctx, int kind, int B, int tpb, int nr, int reps, void *buf, double *part,
                                     double *alpha, int *err) {
    if constexpr (BC == 1) return -1.f;
    else return time_kind<BC>(ctx, kind, B, tpb, nr, reps, buf, part, alpha, err);
}
