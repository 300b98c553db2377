// The residual history's kernels on fields made by a test (test_gpu_history_sums.py):
// one lattice of n_sup support sites, 12 columns, every column in class 0.
#include "../paper_1901_02211_gb300/csrc/msolve.cuh"

namespace {
template <typename T> struct Dev {
    T *p = nullptr;
    size_t n;
    Dev(const T *h, size_t n_) : n(n_) {
        cudaMalloc(&p, n * sizeof(T));
        if (h) cudaMemcpy(p, h, n * sizeof(T), cudaMemcpyHostToDevice);
        else cudaMemset(p, 0, n * sizeof(T));
    }
    void get(T *h) const { cudaMemcpy(h, p, n * sizeof(T), cudaMemcpyDeviceToHost); }
    ~Dev() { cudaFree(p); }
};
} // namespace

// n iterations, nshift shifts; zn, zo [n][nshift][12], alpha, beta [n][12], c
// [nshift]; r [n][ne], ps [nshift][ne], y [ne] with ne = 144 n_sup complex numbers.
// fp32 = 0: a chunk of FP64 iterations (y and ps); 1: of FP32 ones, r and ps rounded
// to FP32 first, y by the sums that a mixed solve with this switch residual takes.
extern "C" int hist_probe(int fp32, double theta, int n, int nshift, int n_sup, const double *c, const double *zn,
                          const double *zo, const double *alpha, const double *beta, const double2 *r, double2 *ps,
                          double2 *y) {
    constexpr int B = 12;
    const size_t ne = (size_t)12 * n_sup * B, rows = (size_t)n * nshift * B;
    ShiftParams sp{};
    sp.n = nshift;
    for (int i = 0; i < nshift; ++i) sp.c[i] = c[i];
    Dev<ShiftParams> dsp(&sp, 1);
    Dev<double> hz(zn, rows), ho(zo, rows), hal(alpha, (size_t)n * B), hbe(beta, (size_t)n * B);
    Dev<double> hw(nullptr, (size_t)(n + 1) * B), v0(nullptr, nshift * B), d0(nullptr, nshift * B);
    Dev<float4> ct(nullptr, rows);
    Dev<int> cls(nullptr, B);
    Dev<double2> dy(y, ne), dps(ps, nshift * ne), dr(r, n * ne);
    std::vector<float2> r32(n * ne), p32(nshift * ne);
    for (size_t i = 0; i < n * ne; ++i) r32[i] = make_float2((float)r[i].x, (float)r[i].y);
    for (size_t i = 0; i < nshift * ne; ++i) p32[i] = make_float2((float)ps[i].x, (float)ps[i].y);
    Dev<float2> dr32(r32.data(), n * ne), dp32(p32.data(), nshift * ne);
    Scal sc{};
    sc.hz = hz.p;
    sc.ho = ho.p;
    sc.hal = hal.p;
    sc.hbe = hbe.p;
    HistLat L{};
    L.ne = ne;
    L.n_sup = n_sup;
    L.V = n_sup;
    L.nshift = nshift;
    L.B = B;
    L.rhs_class = cls.p;
    L.stride = ne;
    L.n = n;
    const dim3 grid = hist_grid<B>(L);
    const int TH = TileMap<B>::THREADS;
    if (fp32) {
        L.h = dr32.p;
        k_hist_coef<<<(unsigned)((rows + 255) / 256), 256>>>(n, nshift, B, 0, B, dsp.p, sc, ct.p);
        const bool exact = hist_exact(SMPQ_MIXED, theta);
        if (nshift == 1 && exact) k_hist_run<B, true, 1><<<grid, TH>>>(L, ho.p, ct.p, dp32.p, dy.p, true);
        else if (nshift == 1) k_hist_run<B, false, 1><<<grid, TH>>>(L, ho.p, ct.p, dp32.p, dy.p, true);
        else if (exact) k_hist_run<B, true, 14><<<grid, TH>>>(L, ho.p, ct.p, dp32.p, dy.p, true);
        else k_hist_run<B, false, 14><<<grid, TH>>>(L, ho.p, ct.p, dp32.p, dy.p, true);
    } else {
        L.h = dr.p;
        k_hist_w<<<(nshift * B + 127) / 128, 128>>>(n, nshift, B, 0, B, dsp.p, sc, v0.p, d0.p, false);
        k_hist_sum<<<(unsigned)(((size_t)(n + 1) * B + 255) / 256), 256>>>(n, nshift, B, hz.p, v0.p, hw.p);
        k_hist_y<double2, B><<<(unsigned)((ne + 255) / 256), 256>>>(L, hw.p, v0.p, dps.p, dy.p);
        if (nshift == 1) k_hist_p<double2, B, false, 1><<<grid, TH>>>(L, ho.p, d0.p, dps.p, dp32.p);
        else k_hist_p<double2, B, false, 14><<<grid, TH>>>(L, ho.p, d0.p, dps.p, dp32.p);
        dps.get(ps);
    }
    dy.get(y);
    return (int)cudaDeviceSynchronize();
}
