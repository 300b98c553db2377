// Link packing, SU(3) check, layout conversion and the stand-alone Wilson
// dslash D_W / D_W^dag (Sec. 2.1, around Eq. 3) used by smpq_dslash.
#include <string>

#include "bfp.cuh"
#include "smpq_internal.cuh"
#include "stage.cuh"
#include "wilson.cuh"

// ------------------------------------------------------------------ links
// U_aos: double[V][4][3][3][2] -> U64/U32: [(mu * V + s) * 9 + e] complex
__global__ void pack_links_kernel(const double2 *__restrict__ Uaos, double2 *__restrict__ U64,
                                  float2 *__restrict__ U32, df64c *__restrict__ Udf, int4 *__restrict__ Ubf, int V) {
    long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= (long)V * 36) return;
    int s = (int)(i / 36), k = (int)(i % 36); // k = mu*9 + e
    double2 u = Uaos[i];
    size_t o = ((size_t)(k / 9) * V + s) * 9 + (k % 9);
    U64[o] = u;
    U32[o] = make_float2((float)u.x, (float)u.y);
    Udf[o] = df64c{df64(u.x), df64(u.y)};
    // units of 2^-60 as two signed words; the low one can be negated
    const double q[2] = {u.x, u.y};
    int w[4];
    for (int k = 0; k < 2; ++k) {
        const double c = fmin(fmax(q[k], -2.0), 2.0); // (a link that is not SU(3) is refused afterwards)
        bf_split(__double2ll_rn(c * 1152921504606846976.0), w[2 * k], w[2 * k + 1]);
        if (w[2 * k + 1] == (int)0x80000000) w[2 * k + 1] += 1;
    }
    Ubf[o] = make_int4(w[0], w[1], w[2], w[3]);
}

void launch_pack_links(const double *U_aos, double *U64, float *U32, void *Udf, void *Ubf, int V, cudaStream_t st) {
    long n = (long)V * 36;
    pack_links_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>((const double2 *)U_aos, (double2 *)U64,
                                                                     (float2 *)U32, (df64c *)Udf, (int4 *)Ubf, V);
}

// max over links of max(|U U^dag - 1|, |det U - 1|), as the bit pattern of a
// non-negative double (ordered like unsigned integers) for atomicMax.
__global__ void su3_check_kernel(const double2 *__restrict__ U, int V, unsigned long long *out) {
    long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    double err = 0;
    if (i < (long)V * 4) {
        int s = (int)(i / 4), mu = (int)(i % 4);
        double2 u[9];
        for (int e = 0; e < 9; ++e) u[e] = U[((size_t)mu * V + s) * 9 + e];
        for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b) {
                double2 t = make_double2(0, 0);
                for (int k = 0; k < 3; ++k) t = cfmac(u[b * 3 + k], u[a * 3 + k], t); // (U U^dag)_ab
                double d = sqrt((t.x - (a == b)) * (t.x - (a == b)) + t.y * t.y);
                err = fmax(err, d);
            }
        // det by cofactor expansion along row 0
        double2 m0 = csub(cmul(u[4], u[8]), cmul(u[5], u[7]));
        double2 m1 = csub(cmul(u[3], u[8]), cmul(u[5], u[6]));
        double2 m2 = csub(cmul(u[3], u[7]), cmul(u[4], u[6]));
        double2 det = cadd(csub(cmul(u[0], m0), cmul(u[1], m1)), cmul(u[2], m2));
        err = fmax(err, sqrt((det.x - 1) * (det.x - 1) + det.y * det.y));
        if (!(err == err)) err = 1e300; // NaN
    }
    // block max then one atomic
    __shared__ double sm[256];
    sm[threadIdx.x] = err;
    __syncthreads();
    for (int st = blockDim.x / 2; st > 0; st >>= 1) {
        if (threadIdx.x < st) sm[threadIdx.x] = fmax(sm[threadIdx.x], sm[threadIdx.x + st]);
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicMax(out, (unsigned long long)__double_as_longlong(sm[0]));
}

void launch_su3_check(const double *U64, int V, double *dev_maxerr, cudaStream_t st) {
    cudaMemsetAsync(dev_maxerr, 0, sizeof(double), st);
    long n = (long)V * 4;
    su3_check_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>((const double2 *)U64, V,
                                                                   (unsigned long long *)dev_maxerr);
}

// ------------------------------------------------------------------ layout conversion
// ABI [V][12][B] double2  <->  tiled [j/BC][V][12][BC] of complex T
template <typename T>
__global__ void to_tiled_kernel(const double2 *__restrict__ in, typename cplx_t<T>::type *__restrict__ out, int V,
                                int B, int BC) {
    long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= (long)V * 12 * B) return;
    int j = (int)(i % B);
    long r = i / B;
    int c = (int)(r % 12);
    int s = (int)(r / 12);
    double2 v = in[i];
    size_t o = (((size_t)(j / BC) * V + s) * 12 + c) * BC + (j % BC);
    out[o] = mkc<typename cplx_t<T>::type>(v.x, v.y);
}

template <typename T>
__global__ void from_tiled_kernel(const typename cplx_t<T>::type *__restrict__ in, double2 *__restrict__ out, int V,
                                  int B, int BC) {
    long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= (long)V * 12 * B) return;
    int j = (int)(i % B);
    long r = i / B;
    int c = (int)(r % 12);
    int s = (int)(r / 12);
    size_t o = (((size_t)(j / BC) * V + s) * 12 + c) * BC + (j % BC);
    typename cplx_t<T>::type v = in[o];
    out[i] = make_double2((double)v.x, (double)v.y);
}

template <typename T> void launch_to_tiled(const double *in, void *out, int V, int B, int BC, cudaStream_t st) {
    long n = (long)V * 12 * B;
    to_tiled_kernel<T><<<(unsigned)((n + 255) / 256), 256, 0, st>>>((const double2 *)in,
                                                                     (typename cplx_t<T>::type *)out, V, B, BC);
}
template <typename T> void launch_from_tiled(const void *in, double *out, int V, int B, int BC, cudaStream_t st) {
    long n = (long)V * 12 * B;
    from_tiled_kernel<T><<<(unsigned)((n + 255) / 256), 256, 0, st>>>((const typename cplx_t<T>::type *)in,
                                                                       (double2 *)out, V, B, BC);
}
template void launch_to_tiled<double>(const double *, void *, int, int, int, cudaStream_t);
template void launch_from_tiled<double>(const void *, double *, int, int, int, cudaStream_t);

// ------------------------------------------------------------------ stand-alone dslash
template <typename T, bool DAG, int BC>
__global__ void __launch_bounds__(TileMap<BC>::THREADS)
    dslash_kernel(Geom g, const typename cplx_t<T>::type *__restrict__ U, const typename cplx_t<T>::type *__restrict__ in,
                  typename cplx_t<T>::type *__restrict__ out, T kappa) {
    typedef typename cplx_t<T>::type C;
    int s = blockIdx.x * TileMap<BC>::SPB + threadIdx.x / BC;
    int jj = threadIdx.x % BC;
    if (s >= g.V) return;
    size_t base = (size_t)blockIdx.y * 12 * g.V * BC + jj;
    const C *pin = in + base;
    C acc[12][1];
    wilson_hop<T, DAG, BC>(g, U, pin, s, acc);
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        size_t o = ((size_t)s * 12 + c) * BC;
        C v = pin[o];
        v.x -= kappa * acc[c][0].x;
        v.y -= kappa * acc[c][0].y;
        out[base + o] = v;
    }
}

template <typename T, int BC>
static void dslash_bc(const Geom &g, const void *U, const void *in, void *out, int B, int dagger, double kappa,
                      cudaStream_t st) {
    typedef typename cplx_t<T>::type C;
    dim3 grid((g.V + TileMap<BC>::SPB - 1) / TileMap<BC>::SPB, B / BC);
    if (dagger)
        dslash_kernel<T, true, BC><<<grid, TileMap<BC>::THREADS, 0, st>>>(g, (const C *)U, (const C *)in, (C *)out,
                                                                           (T)kappa);
    else
        dslash_kernel<T, false, BC><<<grid, TileMap<BC>::THREADS, 0, st>>>(g, (const C *)U, (const C *)in, (C *)out,
                                                                            (T)kappa);
}

// The FP32 D_W with the neighbour sites staged in shared memory (stage.cuh):
// out = in - kappa hop(in), tpb lattice tiles per block.
template <bool DAG, int BC>
__global__ void __launch_bounds__(TileMap<BC>::THREADS, 3)
    dslash_staged_kernel(Geom g, const float2 *__restrict__ U, const float2 *__restrict__ in, float2 *__restrict__ out,
                         double kd, int tpb, int *err) {
    typedef TileMap<BC> TM;
    extern __shared__ __align__(128) unsigned char dsm[];
    const int jj = threadIdx.x % BC;
    const size_t tb = (size_t)blockIdx.y * 12 * g.V * BC;
    const int ntiles = (g.V + TM::SPB - 1) / TM::SPB;
    const int tile0 = blockIdx.x * tpb, ntb = min(ntiles, tile0 + tpb) - tile0;
    const float kappa = (float)kd;
    stage::Runner<DAG, BC, stage::NSTAGE> run(dsm, g, U, in + tb, tile0, ntb, err);
    for (int tl = 0; tl < ntb; ++tl) {
        const int s = (tile0 + tl) * TM::SPB + threadIdx.x / BC;
        const bool valid = s < g.V;
        float2 acc[12][1];
        run.hops(tl, s, valid, acc);
        if (!valid) continue;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const size_t o = tb + ((size_t)s * 12 + c) * BC + jj;
            float2 v = in[o];
            v.x -= kappa * acc[c][0].x;
            v.y -= kappa * acc[c][0].y;
            out[o] = v;
        }
    }
}

template <int BC>
static cudaError_t dslash_staged_bc(const Geom &g, const void *U, const void *in, void *out, int B, int dagger,
                                    double kappa, int *err, cudaStream_t st) {
    constexpr int TPB_ST = 4; // lattice tiles per block
    const int bytes = (int)stage::Dims<BC, stage::NSTAGE>::SMEM;
    static bool attrs = false;
    if (!attrs) {
        cudaError_t e = cudaFuncSetAttribute(dslash_staged_kernel<false, BC>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(dslash_staged_kernel<true, BC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     bytes);
        if (e != cudaSuccess) return e;
        attrs = true;
    }
    const int ntiles = (g.V + TileMap<BC>::SPB - 1) / TileMap<BC>::SPB;
    const dim3 grid((ntiles + TPB_ST - 1) / TPB_ST, B / BC);
    if (dagger)
        dslash_staged_kernel<true, BC><<<grid, TileMap<BC>::THREADS, bytes, st>>>(
            g, (const float2 *)U, (const float2 *)in, (float2 *)out, kappa, TPB_ST, err);
    else
        dslash_staged_kernel<false, BC><<<grid, TileMap<BC>::THREADS, bytes, st>>>(
            g, (const float2 *)U, (const float2 *)in, (float2 *)out, kappa, TPB_ST, err);
    return cudaSuccess;
}

cudaError_t launch_dslash_staged(const Geom &g, const void *U, const void *in, void *out, int B, int BC, int dagger,
                                 double kappa, int *err, cudaStream_t st) {
    switch (BC) {
    case 12: return dslash_staged_bc<12>(g, U, in, out, B, dagger, kappa, err, st);
    case 24: return dslash_staged_bc<24>(g, U, in, out, B, dagger, kappa, err, st);
    case 48: return dslash_staged_bc<48>(g, U, in, out, B, dagger, kappa, err, st);
    default: return cudaErrorInvalidValue;
    }
}

template <typename T>
void launch_dslash(const Geom &g, const void *U, const void *in, void *out, int B, int BC, int dagger, double kappa,
                   cudaStream_t st) {
    switch (BC) {
    case 1: dslash_bc<T, 1>(g, U, in, out, B, dagger, kappa, st); break;
    case 4: dslash_bc<T, 4>(g, U, in, out, B, dagger, kappa, st); break;
    case 12: dslash_bc<T, 12>(g, U, in, out, B, dagger, kappa, st); break;
    case 24: dslash_bc<T, 24>(g, U, in, out, B, dagger, kappa, st); break;
    case 48: dslash_bc<T, 48>(g, U, in, out, B, dagger, kappa, st); break;
    default: break;
    }
}
template void launch_dslash<double>(const Geom &, const void *, const void *, void *, int, int, int, double,
                                    cudaStream_t);
template void launch_dslash<float>(const Geom &, const void *, const void *, void *, int, int, int, double,
                                   cudaStream_t);

// ------------------------------------------------------------------ D_W on the caller's fields
// The ABI layout [V][12][B] is one RHS tile of B columns, so the stencil reads it
// as it is: the input is converted once (to block fixed point, bfp.cuh, or to
// FP32), and the stencil writes the caller's doubles.  Before, the fields went
// through one-column tiles: 209 us of FP64 instructions for 12 columns of 8^3x16
// between two transposes, 70 us for one column of 4^4 (a single block).
__global__ void __launch_bounds__(128) abi_to_bf_kernel(const double2 *__restrict__ in, bfc *__restrict__ v,
                                                        int *__restrict__ e, int V, int B) {
    const long i = blockIdx.x * 128l + threadIdx.x;
    if (i >= (long)V * B) return;
    const int s = (int)(i / B), j = (int)(i % B);
    const size_t base = (size_t)s * 12 * B + j;
    double2 d[12];
    bfc b[12];
    int x;
#pragma unroll
    for (int c = 0; c < 12; ++c) d[c] = in[base + (size_t)c * B];
    const int span = bf_from_double(d, b, x);
#pragma unroll
    for (int c = 0; c < 12; ++c) v[base + (size_t)c * B] = b[c];
    // not finite, or components 2^24 and more apart (3 in 10^6 sites of Gaussian
    // vectors): the sites that read it are done in FP64 without a try
    e[i] = bf_tag(span >= 24 ? BF_BAD : x, span >= 12);
}

// D_W at one site and column in FP64 (what block fixed point does not hold)
static __device__ __noinline__ void dw_site_fp64(const Geom &g, const double2 *__restrict__ U,
                                                 const double2 *__restrict__ in, double2 *__restrict__ out, int s,
                                                 int B, int dagger, double kappa) {
    double2 acc[12][1];
    if (dagger) wilson_hop<double, true, 0>(g, U, in, s, acc, B);
    else wilson_hop<double, false, 0>(g, U, in, s, acc, B);
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        const size_t o = ((size_t)s * 12 + c) * B;
        double2 v = in[o];
        v.x -= kappa * acc[c][0].x;
        v.y -= kappa * acc[c][0].y;
        out[o] = v;
    }
}

// x times 1, i, -1, -i for r = 0..3
static __device__ __forceinline__ double2 turned(double2 x, int r) {
    const double2 y = r & 1 ? make_double2(-x.y, x.x) : x;
    return r & 2 ? make_double2(-y.x, -y.y) : y;
}
// The same by a whole warp: lane 3 k + a does colour row a of hop k, then the hops
// are added in their order (the bits of dw_site_fp64).  An FP64 instruction takes a
// warp as long for one lane as for 32: 110 of them instead of 960, 4 us instead of
// 30, which every launch with one such site waited for.
static __device__ __noinline__ void dw_site_fp64_warp(const Geom &g, const double2 *__restrict__ U,
                                                      const double2 *__restrict__ in, double2 *__restrict__ out, int s,
                                                      int B, int dagger, double kappa) {
    const int lane = threadIdx.x & 31, k = min(lane / 3, 7), a = lane % 3, mu = k >> 1;
    const bool back = k & 1;
    const SiteCoords xc(g, s);
    int n = g.n[0], st = g.stride[0], c = xc.x[0];
    float bc = g.bcf[0];
#pragma unroll
    for (int m = 1; m < 4; ++m)
        if (mu == m) {
            n = g.n[m];
            st = g.stride[m];
            c = xc.x[m];
            bc = g.bcf[m];
        }
    const bool edge = c == (back ? 0 : n - 1);
    const int nb = back ? (edge ? s + (n - 1) * st : s - st) : (edge ? s - (n - 1) * st : s + st);
    const int sg = (dagger != 0) != back ? 0 : 2; // the sign of gamma, as turns
    // S_mu on the lower pair: (-i p3, -i p2), (-p3, p2), (-i p2, i p3), (p2, p3)
    const int r0 = mu == 0 || mu == 2 ? 3 : mu == 1 ? 2 : 0, r1 = mu == 0 ? 3 : mu == 2 ? 1 : 0;
    double2 w0 = make_double2(0, 0), w1 = w0;
    const double2 *q = in + (size_t)nb * 12 * B, *ul = U + ((size_t)mu * g.V + (back ? nb : s)) * 9;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const double2 p2 = q[(size_t)(6 + b) * B], p3 = q[(size_t)(9 + b) * B];
        const double2 h0 = cadd(q[(size_t)b * B], turned(mu < 2 ? p3 : p2, (r0 + sg) & 3));
        const double2 h1 = cadd(q[(size_t)(3 + b) * B], turned(mu < 2 ? p2 : p3, (r1 + sg) & 3));
        double2 u = ul[back ? b * 3 + a : a * 3 + b];
        if (back) u.y = -u.y;
        w0 = cfma(u, h0, w0);
        w1 = cfma(u, h1, w1);
    }
    if (edge && bc < 0) {
        w0 = cneg(w0);
        w1 = cneg(w1);
    }
    // S_mu^dag: (i w1, i w0), (w1, -w0), (i w0, -i w1), (w0, w1)
    const double2 t[4] = {w0, w1, turned(mu < 2 ? w1 : w0, ((mu == 0 || mu == 2 ? 1 : 0) + sg) & 3),
                          turned(mu < 2 ? w0 : w1, ((mu == 0 ? 1 : mu == 1 ? 2 : mu == 2 ? 3 : 0) + sg) & 3)};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        double2 acc = make_double2(0, 0);
#pragma unroll
        for (int h = 0; h < 8; ++h) {
            acc.x += __shfl_sync(0xffffffffu, t[i].x, 3 * h + a);
            acc.y += __shfl_sync(0xffffffffu, t[i].y, 3 * h + a);
        }
        if (lane < 3) {
            const size_t o = ((size_t)s * 12 + 3 * i + a) * B;
            double2 v = in[o];
            v.x -= kappa * acc.x;
            v.y -= kappa * acc.y;
            out[o] = v;
        }
    }
}
// most sites of a warp that it does one after the other (eight take as long as 32 threads side by side)
constexpr int FP64_WARP_MAX = 8;

// One thread per site and column; bound by the integer pipe (8^3x16: 51 us for 12
// columns, 3.9 ms for 1000; with 128 registers and four blocks an SM 57 us and 4.0 ms,
// the sizes of the terms spill).  Sites whose star holds a bad block, and those where
// bf_dw_fine finds a component too small for the common unit, are done in FP64 (`in`
// is read there: it may not overlap out).
// A warp whose sites look uneven for the most part does not try (fields of sites or
// components of very different size: 243 to 250 us a call on 12 columns of 8^3x16
// with links that do not mix them, 265 to 271 with both).
template <bool DAG>
__global__ void __launch_bounds__(128, 3)
    dslash_bf_kernel(Geom g, const int4 *__restrict__ Ubf, const double2 *__restrict__ U64, const bfc *__restrict__ v,
                     const int *__restrict__ e, const double2 *__restrict__ in, double2 *__restrict__ out, int B,
                     BfScal ks, double kappa) {
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    const bool on = i < (long)g.V * B;
    const int s = on ? (int)(i / B) : 0, j = on ? (int)(i % B) : 0;
    const BfOff<0> off{g.V, B};
    const int one = opaque_one();
    const BfStar x(g, e + j, off, s);
    const bool most = __popc(__ballot_sync(0xffffffffu, on && x.uneven)) >= 16;
    bool fp64 = on && !x.alone && (most || x.bad());
    if (on && !fp64) {
        if (x.alone) {
#pragma unroll
            for (int c = 0; c < 12; ++c) out[j + off(s, c)] = in[j + off(s, c)];
        } else {
            bfc acc[12], own[12];
            unsigned size[12];
            int ex;
            bf_hops<DAG>(x, g, Ubf, v + j, e + j, off, s, one, acc, size);
#pragma unroll
            for (int c = 0; c < 12; ++c) own[c] = v[j + off(s, c)];
            fp64 = bf_dw_fine<12>(own, x.eown, acc, size, x.eref, ks, acc, ex);
            if (!fp64)
#pragma unroll
                for (int c = 0; c < 12; ++c)
                    out[j + off(s, c)] = make_double2(bf_double(acc[c].x, ex), bf_double(acc[c].y, ex));
        }
    }
    unsigned todo = __ballot_sync(0xffffffffu, fp64);
    if (__popc(todo) > FP64_WARP_MAX) {
        if (fp64) dw_site_fp64(g, U64, in + j, out + j, s, B, DAG, kappa);
        return;
    }
    for (; todo; todo &= todo - 1) {
        const int from = __ffs(todo) - 1, sf = __shfl_sync(0xffffffffu, s, from), jf = __shfl_sync(0xffffffffu, j, from);
        dw_site_fp64_warp(g, U64, in + jf, out + jf, sf, B, DAG, kappa);
    }
}
// four threads per site and column (bf_hops_split), 32 of those per block: up to
// BF_SPLIT_MAX of them, where one thread's eight hops in a row set the time
template <bool DAG>
__global__ void __launch_bounds__(128, 4)
    dslash_bf_split_kernel(Geom g, const int4 *__restrict__ Ubf, const double2 *__restrict__ U64,
                           const bfc *__restrict__ v, const int *__restrict__ e, const double2 *__restrict__ in,
                           double2 *__restrict__ out, int B, BfScal ks, double kappa) {
    __shared__ BfSplit<32> sm;
    __shared__ int fp64[32];
    const int q = threadIdx.x / 32, t = threadIdx.x % 32;
    const long i = blockIdx.x * 32l + t;
    const bool on = i < (long)g.V * B;
    const int s = on ? (int)(i / B) : 0, j = on ? (int)(i % B) : 0;
    const BfOff<0> off{g.V, B};
    const int one = opaque_one();
    const BfStar x(g, e + j, off, s);
    const bool todo64 = on && !x.alone && x.bad(), hop = on && !x.alone && !todo64;
    if (q == 0) fp64[t] = todo64;
    bfc acc[3], own[3];
    unsigned size[3];
    int ex;
    bf_hops_split<DAG, 32>(x, g, Ubf, v + j, e + j, off, s, hop, one, sm, acc, size);
    if (hop) {
#pragma unroll
        for (int c = 0; c < 3; ++c) own[c] = v[j + off(s, 3 * q + c)];
        if (bf_dw_fine<3>(own, x.eown, acc, size, x.eref, ks, acc, ex)) fp64[t] = 1;
    }
    __syncthreads();
    if (on && !fp64[t])
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const size_t o = j + off(s, 3 * q + c);
            out[o] = x.alone ? in[o] : make_double2(bf_double(acc[c].x, ex), bf_double(acc[c].y, ex));
        }
    unsigned todo = __ballot_sync(0xffffffffu, fp64[t] != 0); // the same in every warp
    for (int k = 0; todo; todo &= todo - 1, ++k) { // the warps take turns
        const int from = __ffs(todo) - 1, sf = __shfl_sync(0xffffffffu, s, from), jf = __shfl_sync(0xffffffffu, j, from);
        if ((k & 3) == q) dw_site_fp64_warp(g, U64, in + jf, out + jf, sf, B, DAG, kappa);
    }
}

bool bf_dslash(double kappa) { return kappa >= BF_KAPPA_MIN; }
size_t bf_field_bytes(int V, int B) { return (size_t)V * B * (12 * sizeof(bfc) + sizeof(int)); }

void launch_abi_to_bf(const double *in, void *field, int V, int B, cudaStream_t st) {
    const long n = (long)V * B;
    bfc *v = (bfc *)field;
    abi_to_bf_kernel<<<(unsigned)((n + 127) / 128), 128, 0, st>>>((const double2 *)in, v, (int *)(v + 12 * n), V, B);
}
void launch_dslash_bf(const Geom &g, const void *Ubf, const void *U64, const void *field, const double *in,
                      double *out, int B, int dagger, double kappa, cudaStream_t st) {
    const long n = (long)g.V * B;
    const bool split = n <= (long)BF_SPLIT_MAX;
    const unsigned nb = (unsigned)(split ? (n + 31) / 32 : (n + 127) / 128);
    const bfc *v = (const bfc *)field;
    const int *e = (const int *)(v + 12 * n);
    const BfScal ks = bf_scal(kappa);
    auto go = [&](auto kernel) {
        kernel<<<nb, 128, 0, st>>>(g, (const int4 *)Ubf, (const double2 *)U64, v, e, (const double2 *)in,
                                   (double2 *)out, B, ks, kappa);
    };
    if (split) dagger ? go(dslash_bf_split_kernel<true>) : go(dslash_bf_split_kernel<false>);
    else dagger ? go(dslash_bf_kernel<true>) : go(dslash_bf_kernel<false>);
}

__global__ void __launch_bounds__(256) abi_to_float_kernel(const double2 *__restrict__ in, float2 *__restrict__ out,
                                                           size_t n) {
    const size_t i = blockIdx.x * (size_t)256 + threadIdx.x;
    if (i < n) {
        const double2 v = in[i];
        out[i] = make_float2((float)v.x, (float)v.y);
    }
}
template <bool DAG>
__global__ void __launch_bounds__(128, 6)
    dslash_abi_kernel(Geom g, const float2 *__restrict__ U, const float2 *__restrict__ in, double2 *__restrict__ out,
                      int B, float kappa) {
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= (long)g.V * B) return;
    const int s = (int)(i / B), j = (int)(i % B);
    float2 acc[12][1];
    wilson_hop<float, DAG, 0>(g, U, in + j, s, acc, B);
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        const size_t o = ((size_t)s * 12 + c) * B + j;
        float2 v = in[o];
        v.x -= kappa * acc[c][0].x;
        v.y -= kappa * acc[c][0].y;
        out[o] = make_double2(exact_d(v.x), exact_d(v.y));
    }
}
void launch_dslash_fp32_abi(const Geom &g, const void *U, const double *in, void *field, double *out, int B,
                            int dagger, double kappa, cudaStream_t st) {
    const long n = (long)g.V * B;
    abi_to_float_kernel<<<(unsigned)((12 * n + 255) / 256), 256, 0, st>>>((const double2 *)in, (float2 *)field,
                                                                          (size_t)12 * n);
    const int th = n < (long)GB300_SMS * 128 * 4 ? 32 : 128; // at least four blocks an SM, of one warp if need be
    const unsigned nb = (unsigned)((n + th - 1) / th);
    if (dagger)
        dslash_abi_kernel<true><<<nb, th, 0, st>>>(g, (const float2 *)U, (const float2 *)field, (double2 *)out, B,
                                                   (float)kappa);
    else
        dslash_abi_kernel<false><<<nb, th, 0, st>>>(g, (const float2 *)U, (const float2 *)field, (double2 *)out, B,
                                                    (float)kappa);
}

// ------------------------------------------------------------------ allocation-free dslash
// smpq_dslash_noalloc keeps its scratch (the tiled copies of the input and the
// output field that the kernel reads and writes) in this file-scope device
// array instead of asking for device memory.  The array is created when the
// library's device code is loaded on a GPU and stays reserved on every GPU that
// loads the library until the process exits.
#define SMPQ_NOALLOC_SCRATCH_BYTES (32u << 20)
// (the limit counts two fields; a block-fixed-point field is a 48th larger than an
// FP64 one)
static __device__ __align__(256) unsigned char
    g_noalloc_scratch[SMPQ_NOALLOC_SCRATCH_BYTES + SMPQ_NOALLOC_SCRATCH_BYTES / 96 + 256];

#include <mutex>

namespace {
constexpr int NOALLOC_MAX_DEVICES = 64;
std::mutex g_noalloc_mu;
void *g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {nullptr};

// Device address of the scratch array on the current device.  In host code
// the array's name is only a host-side handle, so the address is looked up
// once per device (with that device current) and cached.
int noalloc_scratch(smpq_ctx *ctx, int dev, void **out) {
    if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return set_err(ctx, SMPQ_EINVAL, "device index out of range");
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) return cuda_check(ctx, e != cudaSuccess ? e : cudaErrorInvalidSymbol, "scratch address");
        g_noalloc_ptr[dev] = p;
    }
    *out = g_noalloc_ptr[dev];
    return SMPQ_OK;
}
} // namespace

extern "C" int smpq_dslash_noalloc(smpq_ctx *ctx, const double *in, double *out, int B, int dagger, int precision) {
    if (!ctx) return SMPQ_EINVAL;
    if (!ctx->have_gauge) return set_err(ctx, SMPQ_ESTATE, "no gauge field loaded");
    if (!in || !out || B < 1) return set_err(ctx, SMPQ_EINVAL, "bad dslash_noalloc arguments");
    if (precision != SMPQ_FP64 && precision != SMPQ_FP32) return set_err(ctx, SMPQ_EINVAL, "bad precision");
    // in and out must be device memory of the context's GPU: a host pointer or
    // another GPU's buffer would be dereferenced by the kernels
    int rc0;
    if ((rc0 = check_device_ptr(ctx, in, "dslash_noalloc in")) || (rc0 = check_device_ptr(ctx, out, "dslash_noalloc out")))
        return rc0;
    const size_t n = (size_t)ctx->V * 12 * B;
    const size_t esz = precision == SMPQ_FP64 ? sizeof(double2) : sizeof(float2);
    const size_t half = ((n * esz + 255) / 256) * 256; // input tile, then output tile
    if (2 * half > SMPQ_NOALLOC_SCRATCH_BYTES)
        return set_err(ctx, SMPQ_EINVAL,
                       "field too large for smpq_dslash_noalloc: needs " + std::to_string(2 * half) +
                           " bytes of scratch, the limit is " + std::to_string(SMPQ_NOALLOC_SCRATCH_BYTES) +
                           " (2 * V * 12 * B * " + std::to_string(esz) + " bytes)");
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != ctx->device) cudaSetDevice(ctx->device);
    void *scratch = nullptr;
    int rc = noalloc_scratch(ctx, ctx->device, &scratch);
    if (rc == SMPQ_OK) {
        cudaStream_t st = ctx->stream;
        if (ctx->user_stream) {
            cudaEventRecord(ctx->ev0, (cudaStream_t)ctx->user_stream);
            cudaStreamWaitEvent(st, ctx->ev0, 0);
        }
        char *tin = (char *)scratch, *tout = (char *)scratch + half;
        const int BC = 1;
        const bool apart = in + 2 * n <= out || out + 2 * n <= in;
        if (precision == SMPQ_FP64 && bf_dslash(ctx->opt.kappa)) {
            const double *din = in;
            if (!apart) { // a copy of what the sites done in FP64 read
                cudaMemcpyAsync(tin, in, n * sizeof(double2), cudaMemcpyDeviceToDevice, st);
                din = (const double *)tin;
            }
            launch_abi_to_bf(din, tout, ctx->V, B, st);
            launch_dslash_bf(ctx->geom, ctx->Ubf.p, ctx->U64.p, tout, din, out, B, dagger, ctx->opt.kappa, st);
        } else if (precision == SMPQ_FP32) { // (the input is copied before anything is written)
            launch_dslash_fp32_abi(ctx->geom, ctx->U32.p, in, scratch, out, B, dagger, ctx->opt.kappa, st);
        } else {
            launch_to_tiled<double>(in, tin, ctx->V, B, BC, st);
            launch_dslash<double>(ctx->geom, ctx->U64.p, tin, tout, B, BC, dagger, ctx->opt.kappa, st);
            launch_from_tiled<double>(tout, out, ctx->V, B, BC, st);
        }
        cudaError_t e = cudaStreamSynchronize(st);
        rc = e != cudaSuccess ? cuda_check(ctx, e, "dslash_noalloc") : cuda_check(ctx, cudaGetLastError(), "dslash_noalloc launch");
    }
    if (prev >= 0 && prev != ctx->device) cudaSetDevice(prev);
    return rc;
}
