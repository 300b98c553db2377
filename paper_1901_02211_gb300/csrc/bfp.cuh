// D_W in block fixed point: FP64 accuracy on the integer pipe.
//
// GB300 executes 2 FP64 operations per clock and SM: an FP64 FMA occupies an SM
// quarter for 66 cycles a warp, a multiply-add of two 32-bit integers into a
// 64-bit sum (mad.wide) for 4.5 (both measured).  The FP64 iterations therefore keep a site's 24
// real numbers (12 complex components of one column) as 64-bit integers with
// one exponent,
//     value = v * 2^e,  |v| < 2^60, the largest at least 2^59,
// 7 bits more than a double holds for the largest component (a component that
// is smaller by 2^k keeps 60 - k bits).  Links are integers in units of 2^-60.
// A product of two such numbers, each split into a signed high and a signed
// low word, is three mad.wide into 64-bit sums (high; middle twice); low times
// low, about 2^-57 of the largest, is left out.  Sums are exact, so the hop's
// error is that of its truncations, about 2^-56 of the largest component of
// the nine sites, against 2^-53 of every partial sum in FP64.  Relative to the
// largest: a component that is smaller by 2^k and does not mix with it (unit or
// diagonal links) has k bits less.  The solver's norms, residuals and tolerances
// are those of whole vectors; the stand-alone D_W looks at every component
// (bf_dw_fine).
//   Bounds: a projected component is below 2^61, so its words are below 2^29
// and 2^31, a link's 2^28 and 2^31.  Six products in a middle sum stay below
// 6 * 2^60 + sqrt(6) * 2^59 < 2^63; the rows of a link have norm 1, so a hop's
// high sum, in units of 2^64, is below sqrt(6) * 2^(61 + 60 - 64) and eight
// hops below 2^61.3.
//
// Bound by the integer pipe: 8 hops of 228 mad.wide and about 370 cycles of
// shifts, splits, additions and loads come to 11 000 cycles a warp; the 960 FP64
// instructions that they replace took 63 000.  Measured on 8^3x16 with 72 columns:
// a solver launch of 300 us (1340 us in FP64); stand-alone with 12 columns 100 us
// a call (261).  Not kept: products of the middle words in FP32 (1.6e-16 of the
// result's norm instead of 1.2e-16), one copy of the hop for all directions (same
// time), eight copies (15 % slower: instruction cache).
#pragma once
#include "wilson.cuh"

struct __align__(16) bfc {
    long long x, y;
};
// a field of n complex values: the components, then one exponent per site and column
struct BFF {
    bfc *v;
    int *e;
};
constexpr int BF_ZERO = -(1 << 28); // exponent of a site whose components are all 0
constexpr int BF_BAD = 1 << 28;     // of one that holds an infinity or a NaN

struct bf {}; // names the format where a template takes an iteration type

// component c of site s in an RHS tile: [site][12][BC], or [12][site] for
// one-column tiles (neighbouring threads then read neighbouring sites)
template <int BC> struct BfOff {
    int V;
    __device__ __forceinline__ size_t operator()(int s, int c) const {
        if constexpr (BC == 1) return (size_t)c * V + s;
        else return ((size_t)s * 12 + c) * BC;
    }
    __device__ __forceinline__ size_t exp(int s) const { return (size_t)s * BC; }
};
// the caller's layout [site][12][B] with B only known at run time
template <> struct BfOff<0> {
    int V, B;
    __device__ __forceinline__ size_t operator()(int s, int c) const { return ((size_t)s * 12 + c) * B; }
    __device__ __forceinline__ size_t exp(int s) const { return (size_t)s * B; }
};

// c + a * b in one instruction (the compiler would turn a factor -a into a
// product and a 64-bit subtraction)
__device__ __forceinline__ long long madw(int a, int b, long long c) {
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
// 1 that the compiler does not know: high + one * middle is then one mad.wide
// instead of a sign extension and a 64-bit addition
__device__ __forceinline__ int opaque_one() {
    int v;
    asm("mov.u32 %0, 1;" : "=r"(v));
    return v;
}
// x = h * 2^32 + l with both signed
__device__ __forceinline__ void bf_split(long long x, int &h, int &l) {
    l = (int)x;
    h = (int)(x >> 32) + (int)((unsigned)l >> 31);
}
constexpr long long BF_HALF = 0x80000000ll; // rounds the middle sum

// a real factor m * 2^e, 2^61 <= |m| < 2^62 (or 0)
struct BfScal {
    int h, l, e;
};
__host__ __device__ __forceinline__ BfScal bf_scal(double s) {
    unsigned long long u;
#ifdef __CUDA_ARCH__
    u = (unsigned long long)__double_as_longlong(s);
#else
    __builtin_memcpy(&u, &s, 8);
#endif
    const int eb = (int)(u >> 52) & 0x7ff;
    long long m = eb ? (long long)((u & 0xfffffffffffffull) | 0x10000000000000ull) << 9 : 0;
    if (u >> 63) m = -m;
    BfScal r;
    r.l = (int)m;
    r.h = (int)(m >> 32) + (int)((unsigned)r.l >> 31);
    r.e = eb - 1075 - 9;
    if (eb == 0x7ff) r.e = BF_BAD; // infinity or NaN: the result is marked bad
    return r;
}
// x * s / 2^64 (the exponents add up to e_x + s.e + 64); |result| < |x| / 4
__device__ __forceinline__ long long bf_mul(long long x, const BfScal &s, int one) {
    int h, l;
    bf_split(x, h, l);
    const long long mid = madw(h, s.l, madw(l, s.h, BF_HALF));
    return madw((int)(mid >> 32), one, madw(h, s.h, 0));
}
// arithmetic right shift by any n >= 0
__device__ __forceinline__ long long bf_shr(long long x, int n) { return x >> min(n, 63); }

// v * 2^e as a double
__device__ __forceinline__ double bf_double(long long v, int e) {
    const double d = __ll2double_rn(v);
    const int hi = __double2hiint(d), eb = ((hi >> 20) & 0x7ff) + e;
    if (v == 0) return 0.0;
    if (eb < 1 || eb > 2046) return e >= BF_BAD / 2 ? __longlong_as_double(0x7ff8000000000000ll) : ldexp(d, e);
    return __hiloint2double(hi + (e << 20), __double2loint(d));
}

// 24 doubles as a block (e = BF_BAD if some are not finite); the result is the
// span of the nonzero ones, as a difference of exponents
__device__ __forceinline__ int bf_from_double(const double2 d[12], bfc v[12], int &e) {
    int top = 0, low = 0x7ff;
    bool any = false;
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        const double q[2] = {d[c].x, d[c].y};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int eb = max((__double2hiint(q[k]) >> 20) & 0x7ff, 1);
            if (q[k] != 0) {
                any = true;
                low = min(low, eb);
            }
            top = max(top, eb);
        }
    }
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        const double q[2] = {d[c].x, d[c].y};
        long long r[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const long long u = __double_as_longlong(q[k]);
            const int eb = (int)(u >> 52) & 0x7ff;
            const long long m = ((u & 0xfffffffffffffll) | (eb ? 0x10000000000000ll : 0)) << 7;
            const long long a = bf_shr(m, top - max(eb, 1));
            r[k] = u < 0 ? -a : a;
        }
        v[c] = bfc{r[0], r[1]};
    }
    e = top == 0x7ff ? BF_BAD : any ? top - 1082 : BF_ZERO;
    return any ? top - low : 0;
}

// Brings a block with |v| < 2^60 and exponent e to the normal form.
__device__ __forceinline__ void bf_normalise(bfc v[12], int &e) {
    int mx = 0, mn = -1;
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        const int a = (int)(v[c].x >> 32), b = (int)(v[c].y >> 32);
        mx = max(mx, max(a, b));
        mn = min(mn, min(a, b));
    }
    const int m = max(mx, ~mn);
    if (m == 0) { // all below 2^32: is there anything?
        int any = 0;
#pragma unroll
        for (int c = 0; c < 12; ++c) any |= (int)v[c].x | (int)v[c].y;
        if (any == 0 && e < BF_BAD / 2) e = BF_ZERO;
    }
    const int sh = max(__clz(m) - 4, 0);
#pragma unroll
    for (int c = 0; c < 12; ++c) v[c] = bfc{v[c].x << sh, v[c].y << sh};
    if (e > BF_ZERO / 2) e -= sh;
    if (e >= BF_BAD / 2) e = BF_BAD;
}

// sum of the squares of a block in normal form
__device__ __forceinline__ double bf_norm2(const bfc v[12], int e, int one) {
    if (e <= BF_ZERO / 2) return 0.0;
    if (e >= BF_BAD / 2) return __longlong_as_double(0x7ff8000000000000ll);
    long long hi = 0, lo = 0;
#pragma unroll
    for (int g = 0; g < 2; ++g) { // twelve products of 2^59 fit the middle sum
        long long mid = BF_HALF;
#pragma unroll
        for (int c = 6 * g; c < 6 * g + 6; ++c) {
            int h, l;
            bf_split(v[c].x, h, l);
            hi = madw(h, h, hi);
            mid = madw(h, l, mid);
            bf_split(v[c].y, h, l);
            hi = madw(h, h, hi);
            mid = madw(h, l, mid);
        }
        lo = madw((int)(mid >> 32), one, lo);
    }
    return bf_double(hi + 2 * lo, 64 + 2 * e);
}

// ---------------------------------------------------------------- the hop
// h = (psi_0 + G S_mu psi_lo, ...) of one colour (p0..p3: its four spin components)
template <int MU, int G> __device__ __forceinline__ void bf_project(bfc p0, bfc p1, bfc p2, bfc p3, bfc &h0, bfc &h1) {
    bfc s0, s1;
    if (MU == 0) { s0 = {p3.y, -p3.x}; s1 = {p2.y, -p2.x}; }
    else if (MU == 1) { s0 = {-p3.x, -p3.y}; s1 = {p2.x, p2.y}; }
    else if (MU == 2) { s0 = {p2.y, -p2.x}; s1 = {-p3.y, p3.x}; }
    else { s0 = p2; s1 = p3; }
    h0 = {p0.x + G * s0.x, p0.y + G * s0.y};
    h1 = {p1.x + G * s1.x, p1.y + G * s1.y};
}
// lower half += G S_mu^dag w
template <int MU, int G> __device__ __forceinline__ void bf_lower(bfc w0, bfc w1, bfc &l0, bfc &l1) {
    bfc a, b;
    if (MU == 0) { a = {-w1.y, w1.x}; b = {-w0.y, w0.x}; }
    else if (MU == 1) { a = w1; b = {-w0.x, -w0.y}; }
    else if (MU == 2) { a = {-w0.y, w0.x}; b = {w1.y, -w1.x}; }
    else { a = w0; b = w1; }
    l0 = {l0.x + G * a.x, l0.y + G * a.y};
    l1 = {l1.x + G * b.x, l1.y + G * b.y};
}

// |re| and |im| of w in units of 2^48, in the low and the high half of a word
// (one less for a negative number: bounds from below, so that a sum of eight
// terms below 2^59 stays within 16 bits)
__device__ __forceinline__ unsigned bf_size(bfc w) {
    unsigned q, m;
    asm("prmt.b32 %0, %1, %2, 0x7632;" : "=r"(q) : "r"((int)(w.x >> 32)), "r"((int)(w.y >> 32)));
    asm("prmt.b32 %0, %1, 0, 0xbb99;" : "=r"(m) : "r"(q)); // the signs, spread over each half
    return q ^ m;
}
__device__ __forceinline__ unsigned bf_swap(unsigned z) { return (z >> 16) | (z << 16); }

// acc += (1 + G g_mu) U psi(nb) (back = false, G = DAG ? 1 : -1) or (1 - G g_mu)
// U^dag psi(nb) (back = true; as the conjugate of U^T conj(h)), its sign flipped
// if flip; psi's block is shifted right by n bits to the common exponent, acc in
// units of 2^4 of that.  The orientation is a run-time value: one copy of this
// code for each direction fits the instruction cache, eight do not (measured:
// 210 against 178 ms for six classes of 8^3x16, "no instruction" the first stall).
// links: int4 {re high, re low, im high, im low} per element
// SIZES: size[c] += the leading bits of |re| (low half) and |im| (high half) of
// component c's term, in units of 2^48 (bf_dw_fine)
template <int MU, bool DAG, bool SIZES = false, typename Off>
__device__ __forceinline__ void bf_hop(bool back, const int4 *__restrict__ U, const bfc *__restrict__ in,
                                          const Off &off, int Vl, int nb, int ls, int n, bool flip, int one,
                                          bfc acc[12], unsigned *size = nullptr) {
    constexpr int GF = DAG ? 1 : -1;
    int hh[2][3][2], hl[2][3][2];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const bfc p0 = in[off(nb, a)], p1 = in[off(nb, 3 + a)], p2 = in[off(nb, 6 + a)], p3 = in[off(nb, 9 + a)];
        bfc h0, h1;
        if (back) {
            bf_project<MU, -GF>(p0, p1, p2, p3, h0, h1);
            h0.y = -h0.y;
            h1.y = -h1.y;
        } else {
            bf_project<MU, GF>(p0, p1, p2, p3, h0, h1);
        }
        if (flip) {
            h0 = {-h0.x, -h0.y};
            h1 = {-h1.x, -h1.y};
        }
        bf_split(h0.x >> n, hh[0][a][0], hl[0][a][0]);
        bf_split(h0.y >> n, hh[0][a][1], hl[0][a][1]);
        bf_split(h1.x >> n, hh[1][a][0], hl[1][a][0]);
        bf_split(h1.y >> n, hh[1][a][1], hl[1][a][1]);
    }
    const int4 *ul = U + ((size_t)MU * Vl + ls) * 9;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        int4 u[3];
        if (back) {
#pragma unroll
            for (int b = 0; b < 3; ++b) u[b] = ul[b * 3 + a];
        } else {
#pragma unroll
            for (int b = 0; b < 3; ++b) u[b] = ul[a * 3 + b];
        }
        bfc w[2];
        long long rh[2] = {0, 0}, rm[2] = {BF_HALF, BF_HALF}, ih[2] = {0, 0}, im[2] = {BF_HALF, BF_HALF};
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int ah = -u[b].z, al = -u[b].w;
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                rh[s] = madw(u[b].x, hh[s][b][0], madw(ah, hh[s][b][1], rh[s]));
                rm[s] = madw(u[b].x, hl[s][b][0], madw(u[b].y, hh[s][b][0], rm[s]));
                rm[s] = madw(ah, hl[s][b][1], madw(al, hh[s][b][1], rm[s]));
                ih[s] = madw(u[b].x, hh[s][b][1], madw(u[b].z, hh[s][b][0], ih[s]));
                im[s] = madw(u[b].x, hl[s][b][1], madw(u[b].y, hh[s][b][1], im[s]));
                im[s] = madw(u[b].z, hl[s][b][0], madw(u[b].w, hh[s][b][0], im[s]));
            }
        }
#pragma unroll
        for (int s = 0; s < 2; ++s)
            w[s] = {madw((int)(rm[s] >> 32), one, rh[s]), madw((int)(im[s] >> 32), one, ih[s])};
        if constexpr (SIZES) {
            const unsigned z0 = bf_size(w[0]), z1 = bf_size(w[1]);
            size[a] += z0;
            size[3 + a] += z1;
            // the lower half's terms (bf_lower): i w has re and im in turn
            const unsigned l0 = MU == 0 || MU == 1 ? z1 : z0, l1 = MU == 0 || MU == 1 ? z0 : z1;
            size[6 + a] += MU == 0 || MU == 2 ? bf_swap(l0) : l0;
            size[9 + a] += MU == 0 || MU == 2 ? bf_swap(l1) : l1;
        }
        if (back) {
            acc[a] = {acc[a].x + w[0].x, acc[a].y - w[0].y};
            acc[3 + a] = {acc[3 + a].x + w[1].x, acc[3 + a].y - w[1].y};
            bf_lower<MU, -GF>(bfc{w[0].x, -w[0].y}, bfc{w[1].x, -w[1].y}, acc[6 + a], acc[9 + a]);
        } else {
            acc[a] = {acc[a].x + w[0].x, acc[a].y + w[0].y};
            acc[3 + a] = {acc[3 + a].x + w[1].x, acc[3 + a].y + w[1].y};
            bf_lower<MU, GF>(w[0], w[1], acc[6 + a], acc[9 + a]);
        }
    }
}

// where a site lies at the lattice's edges, and its neighbours
struct BfSite {
    unsigned edges; // bit 2 mu: last coordinate, bit 2 mu + 1: first one
    __device__ __forceinline__ BfSite(const Geom &g, int s) {
        const SiteCoords xc(g, s);
        edges = 0;
#pragma unroll
        for (int mu = 0; mu < 4; ++mu)
            edges |= (xc.x[mu] == g.n[mu] - 1 ? 1u : 0u) << (2 * mu) | (xc.x[mu] == 0 ? 2u : 0u) << (2 * mu);
    }
    // k = 2 mu: forward in direction mu, 2 mu + 1: backward
    __device__ __forceinline__ bool edge(int k) const { return edges >> k & 1; }
    __device__ __forceinline__ int neighbour(const Geom &g, int s, int k) const {
        const int st = g.stride[k >> 1], far = (g.n[k >> 1] - 1) * st;
        return k & 1 ? (edge(k) ? s + far : s - st) : (edge(k) ? s - far : s + st);
    }
};

// acc * 2^(eref + 4) = hop(s); eref = the largest exponent of s and its neighbours
template <bool DAG, typename Off>
__device__ __forceinline__ void bf_wilson(const Geom &g, const int4 *__restrict__ U, const bfc *__restrict__ in,
                                          const int *__restrict__ ein, const Off &off, int s, int one, bfc acc[12],
                                          int &eown, int &eref) {
    const BfSite x(g, s);
    int nb[8], en[8];
    eown = eref = ein[off.exp(s)];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        nb[k] = x.neighbour(g, s, k);
        en[k] = ein[off.exp(nb[k])];
        eref = max(eref, en[k]);
    }
#pragma unroll
    for (int c = 0; c < 12; ++c) acc[c] = {0, 0};
    auto dir = [&](auto mc) {
        constexpr int MU = decltype(mc)::value;
        const bool anti = g.bcf[MU] < 0;
        // forward: (1 - g) [DAG: (1 + g)], backward: (1 + g) [DAG: (1 - g)]
#pragma unroll 1
        for (int bk = 0; bk < 2; ++bk) {
            const int n = bk ? nb[2 * MU + 1] : nb[2 * MU], e = bk ? en[2 * MU + 1] : en[2 * MU];
            bf_hop<MU, DAG>(bk != 0, U, in, off, g.V, n, bk ? n : s, min(eref - e, 63), anti && x.edge(2 * MU + bk), one,
                            acc);
        }
    };
    dir(std::integral_constant<int, 0>());
    dir(std::integral_constant<int, 1>());
    dir(std::integral_constant<int, 2>());
    dir(std::integral_constant<int, 3>());
}

// The stand-alone D_W's exponents carry in their lowest bit whether the nonzero
// components of the site span 2^12 and more.
__device__ __forceinline__ int bf_tag(int e, bool wide) { return 2 * e + wide; }
// What it knows of a site before it reads any component: its exponent and the star's
// largest, whether every neighbour is zero (D_W then changes nothing).  Neighbours and
// their exponents are formed again in each hop: kept over the eight hops they were 160
// bytes of spills.
struct BfStar : BfSite {
    int eown, eref;
    bool alone;
    bool uneven; // bf_dw_fine is likely to find a small component: tagged, or only one or two large neighbours
    template <typename Off>
    __device__ __forceinline__ BfStar(const Geom &g, const int *__restrict__ tag, const Off &off, int s) : BfSite(g, s) {
        int en[8], top = BF_ZERO, large = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            en[k] = tag[off.exp(neighbour(g, s, k))] >> 1;
            top = max(top, en[k]);
        }
        const int own = tag[off.exp(s)];
        eown = own >> 1;
        eref = max(eown, top);
#pragma unroll
        for (int k = 0; k < 8; ++k) large += en[k] >= eref - 4;
        alone = top <= BF_ZERO / 2;
        uneven = !alone && ((own & 1) || large <= 2);
    }
    // a block in the star is marked bad
    __device__ __forceinline__ bool bad() const { return eref >= BF_BAD / 2; }
};
// acc += the two hops of direction MU, size likewise (bf_hop)
template <int MU, bool DAG, typename Off>
__device__ __forceinline__ void bf_dir(const BfStar &x, const Geom &g, const int4 *__restrict__ U,
                                       const bfc *__restrict__ in, const int *__restrict__ tag, const Off &off, int s,
                                       int one, bfc acc[12], unsigned size[12]) {
    const bool anti = g.bcf[MU] < 0;
#pragma unroll 1
    for (int bk = 0; bk < 2; ++bk) {
        const int k = 2 * MU + bk, nb = x.neighbour(g, s, k);
        bf_hop<MU, DAG, true>(bk != 0, U, in, off, g.V, nb, bk ? nb : s, min(x.eref - (tag[off.exp(nb)] >> 1), 63),
                              anti && x.edge(k), one, acc, size);
    }
}
// The eight hops of the star x and their sizes, or (split) by four groups of GT
// threads (thread t of each group: the same site and column; every thread of the
// block calls it, `on` where there is something to do), for launches too small to
// hide one thread's eight hops: group q does direction q, the sums go through
// shared memory and group q keeps components 3 q .. 3 q + 2 in acc[0..2] and
// size[0..2].  Integer sums: the bits are the same.
template <bool DAG, typename Off>
__device__ __forceinline__ void bf_hops(const BfStar &x, const Geom &g, const int4 *__restrict__ U,
                                        const bfc *__restrict__ in, const int *__restrict__ tag, const Off &off, int s,
                                        int one, bfc acc[12], unsigned size[12]) {
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        acc[c] = {0, 0};
        size[c] = 0;
    }
    bf_dir<0, DAG>(x, g, U, in, tag, off, s, one, acc, size);
    bf_dir<1, DAG>(x, g, U, in, tag, off, s, one, acc, size);
    bf_dir<2, DAG>(x, g, U, in, tag, off, s, one, acc, size);
    bf_dir<3, DAG>(x, g, U, in, tag, off, s, one, acc, size);
}
template <int GT> struct BfSplit { // in shared memory
    bfc v[4][6][GT];
    unsigned z[4][6][GT];
};
template <bool DAG, int GT, typename Off>
__device__ __forceinline__ void bf_hops_split(const BfStar &x, const Geom &g, const int4 *__restrict__ U,
                                              const bfc *__restrict__ in, const int *__restrict__ tag,
                                              const Off &off, int s, bool on, int one, BfSplit<GT> &sm,
                                              bfc keep[3], unsigned zkeep[3]) {
    const int q = threadIdx.x / GT, t = threadIdx.x % GT;
    bfc acc[12];
    unsigned size[12];
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        acc[c] = {0, 0};
        size[c] = 0;
    }
    if (on) {
        if (q == 0) bf_dir<0, DAG>(x, g, U, in, tag, off, s, one, acc, size);
        else if (q == 1) bf_dir<1, DAG>(x, g, U, in, tag, off, s, one, acc, size);
        else if (q == 2) bf_dir<2, DAG>(x, g, U, in, tag, off, s, one, acc, size);
        else bf_dir<3, DAG>(x, g, U, in, tag, off, s, one, acc, size);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) { // upper half to groups 0 and 1, lower to 2 and 3
        __syncthreads();
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            sm.v[q][c][t] = acc[6 * h + c];
            sm.z[q][c][t] = size[6 * h + c];
        }
        __syncthreads();
        if ((q >> 1) == h) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int k = 3 * (q & 1) + c;
                bfc v = sm.v[0][k][t];
                unsigned z = sm.z[0][k][t];
#pragma unroll
                for (int r = 1; r < 4; ++r) {
                    v = {v.x + sm.v[r][k][t].x, v.y + sm.v[r][k][t].y};
                    z += sm.z[r][k][t];
                }
                keep[c] = v;
                zkeep[c] = z;
            }
        }
    }
}

// The stand-alone D_W: x = own - kappa acc in units of 2^ex, three bits finer than
// the solver's (bf_dw) because x goes out as doubles and needs no spare ones;
// |x| < 2^63.  kappa >= BF_KAPPA_MIN, so that kappa acc has the larger unit.
//   The error of x, about 0.3 units of 2^(ex + 3), belongs to the largest component
// of the star; FP64 arithmetic has one of about 0.4 * 2^-53 of the terms that make
// up a component.  Those are at least |own| + kappa sum |hop terms| (size): where
// that is below 2^52 units for a component, the result is true and the site is
// done in FP64.  Links that mix colours hardly ever leave such a component (2 in
// 10^5 sites of Gaussian vectors at kappa 0.21, 5 in 10^4 at the worst kappa).  At
// the line the errors are equal (root mean square 0.39 of 2^-53 of the terms in
// both, unit links and components of different size), above it block fixed point
// has the smaller one.
constexpr double BF_KAPPA_MIN = 0.0625;
constexpr int BF_FINE = 3;
template <int N>
__device__ __forceinline__ bool bf_dw_fine(const bfc own[N], int eown, const bfc acc[N], const unsigned size[N],
                                           int eref, const BfScal &k, bfc x[N], int &ex) {
    ex = eref + 4 + k.e + 64 - BF_FINE;
    const int n = ex - eown; // >= 0
    bool small = false;
    auto part = [&](long long o, long long a, unsigned z) { // z: the size in the upper half
        int h, l;
        bf_split(a, h, l);
        const long long mid = madw(h, k.l, madw(l, k.h, BF_HALF >> BF_FINE));
        o = bf_shr(o, n);
        const int oh = (int)(o >> 32);
        small |= (unsigned)(oh ^ (oh >> 31)) + (__umulhi(z, (unsigned)k.h) << BF_FINE) < 1u << (52 + BF_FINE - 32);
        return o - ((madw(h, k.h, 0) << BF_FINE) + (mid >> (32 - BF_FINE)));
    };
#pragma unroll
    for (int c = 0; c < N; ++c)
        x[c] = {part(own[c].x, acc[c].x, size[c] << 16), part(own[c].y, acc[c].y, size[c] & 0xffff0000u)};
    return small;
}
// x = own - kappa acc in units of 2^eu, eu at least `least` (>= eown + 2, the
// exponent of the block own); |x| < 2^60
template <int N>
__device__ __forceinline__ void bf_dw(const bfc own[N], int eown, const bfc acc[N], int eref, const BfScal &k,
                                      int least, int one, bfc x[N], int &eu) {
    const int eq = eref <= BF_ZERO / 2 ? BF_ZERO : eref + 4 + k.e + 64;
    eu = max(eq, least);
    const int n = eu - eown, m = eu - eq;
#pragma unroll
    for (int c = 0; c < N; ++c) {
        long long qx = bf_mul(acc[c].x, k, one), qy = bf_mul(acc[c].y, k, one);
        if (m) { // (only for a tiny kappa)
            qx = bf_shr(qx, m);
            qy = bf_shr(qy, m);
        }
        x[c] = {bf_shr(own[c].x, n) - qx, bf_shr(own[c].y, n) - qy};
    }
    if (eref >= BF_BAD / 2) eu = BF_BAD;
}

// Sites times columns up to which a stand-alone D_W is split over four threads
// each: 10 us against 20 for 256 (one vector of 4^4), 16.4 against 20.6 for 16 384,
// 24.8 against 24.5 for 24 576, 26.7 against 22.8 for 32 768 (there the SMs are
// full).  A solve's launches gained nothing from it: D_ov on 3 vectors of 8^3x16
// 13.6 against 13.2 ms.
constexpr size_t BF_SPLIT_MAX = 24000;
// thread -> (site, column) of the block-fixed-point kernels: blocks of about a
// hundred threads, so that small lattices reach every SM (24 576 sites and
// columns are 384 blocks); 128 registers a thread
template <int BC> struct BfMap {
    static constexpr int SPB = BC == 1 ? 64 : BC == 12 ? 8 : BC == 24 ? 4 : 5;
    static constexpr int THREADS = BC * SPB;
    static constexpr int BLOCKS = 512 / THREADS; // per SM
};
