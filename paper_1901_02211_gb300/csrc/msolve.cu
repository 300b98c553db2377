// The multi-shift solves of the library: dispatch to the RHS tile widths (the
// solver itself is msolve.cuh, one translation unit per width), the Lanczos
// interval and the autotuner's timing.
#include <algorithm>
#include <cmath>

#include "smpq_internal.cuh"

namespace {

int dispatch_bc(const std::vector<LatIn> &lats, double tol, int max_iter, double *hist, int hist_len, int fixed) {
    switch (lats[0].spec->BC) {
    case 1: return solve_bc<1>(lats, tol, max_iter, hist, hist_len, fixed);
    case 12: return solve_bc<12>(lats, tol, max_iter, hist, hist_len, fixed);
    case 24: return solve_bc<24>(lats, tol, max_iter, hist, hist_len, fixed);
    case 48: return solve_bc<48>(lats, tol, max_iter, hist, hist_len, fixed);
    default: return set_err(lats[0].ctx, SMPQ_EINVAL, "unsupported rhs tile width");
    }
}

ShiftParams make_shifts(const smpq_ctx *ctx) {
    ShiftParams sp;
    sp.n = (int)ctx->zq.size();
    sp.s0 = *std::min_element(ctx->zq.begin(), ctx->zq.end());
    for (int i = 0; i < sp.n; ++i) {
        sp.sig[i] = ctx->zq[i] - sp.s0;
        sp.c[i] = ctx->zc[i];
    }
    return sp;
}

} // namespace

// Slots for a solve at the default tolerance on a gapped background (160 to 190
// iterations, a third of them above the mixed solve's switch, where its slots start
// anew); a longer one continues in further chunks, each of which forms the shifted
// directions at its end (two FP64 operations a shift, value and iteration).  Measured
// on 8^3x16, FP64 to 1e-14: six classes of q(x) 0.68 ms an iteration in one chunk and
// in two or three (117 ms for 173, 293 for 437); D_ov on 3 vectors, whose support is
// the lattice, 0.071 ms in one chunk and 0.086 in three (12.2 ms for 173, 37.7 for
// 437; with updates of the directions in every iteration 0.81 and 0.87).
size_t hist_bytes_wanted(int prec, int max_iter) {
    const size_t n = (size_t)std::min(max_iter, 208) + 8;
    if (prec == SMPQ_FP64) return n * sizeof(double2);
    return (prec == SMPQ_MIXED ? n * 3 / 4 : n) * sizeof(float2);
}

int multishift_solve(smpq_ctx *ctx, const SolveSpec &spec, SolveOut *out) {
    if (spec.B % spec.BC) return set_err(ctx, SMPQ_EINVAL, "rhs count must be a multiple of the tile width");
    std::vector<LatIn> lats{LatIn{ctx, &spec, spec.shifts ? *spec.shifts : make_shifts(ctx), out}};
    return dispatch_bc(lats, ctx->opt.tol, ctx->opt.max_iter, nullptr, 0, 0);
}

int multishift_solve_batch(smpq_ctx *const *ctxs, const SolveSpec *specs, SolveOut *outs, int n) {
    if (n < 1 || n > 4) return set_err(ctxs[0], SMPQ_EINVAL, "a batched solve takes 1 to 4 lattices");
    std::vector<LatIn> lats;
    for (int l = 0; l < n; ++l) {
        if (specs[l].B % specs[l].BC || specs[l].BC != specs[0].BC || specs[l].prec != specs[0].prec)
            return set_err(ctxs[0], SMPQ_EINVAL, "the lattices of a batched solve need one precision and tile width");
        lats.push_back(LatIn{ctxs[l], &specs[l], specs[l].shifts ? *specs[l].shifts : make_shifts(ctxs[l]), &outs[l]});
    }
    return dispatch_bc(lats, ctxs[0]->opt.tol, ctxs[0]->opt.max_iter, nullptr, 0, 0);
}

// ------------------------------------------------------------------ spectrum (Lanczos from CG coefficients)
__global__ void k_random_source(double2 *b, int V, unsigned long long seed) {
    long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= (long)V * 12) return;
    // splitmix64 of (seed, index): a counter-based generator
    unsigned long long z = seed + 0x9E3779B97F4A7C15ull * (unsigned long long)(i + 1);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    double u1 = ((z >> 11) + 0.5) * (1.0 / 9007199254740992.0);
    unsigned long long w = z * 0x9E3779B97F4A7C15ull + 0x632BE59BD9B4E019ull;
    w = (w ^ (w >> 30)) * 0xBF58476D1CE4E5B9ull;
    w = (w ^ (w >> 27)) * 0x94D049BB133111EBull;
    w ^= w >> 31;
    double u2 = ((w >> 11) + 0.5) * (1.0 / 9007199254740992.0);
    b[i] = make_double2(u1 - 0.5, u2 - 0.5);
}

int lanczos_extremes(smpq_ctx *ctx, int iters, double *lo, double *hi) {
    std::vector<Buf> &ws = ctx->ws;
    if (ws.size() < W_COUNT) ws.resize(W_COUNT);
    int rc;
    const int V = ctx->V;
    if ((rc = ensure(ctx, ws[W_B64], (size_t)V * 12 * sizeof(double2) + 2 * (size_t)iters * sizeof(double))))
        return rc;
    double2 *b = (double2 *)ws[W_B64].p;
    double *hist = (double *)(b + (size_t)V * 12);
    k_random_source<<<(V * 12 + 255) / 256, 256, 0, ctx->stream>>>(b, V, 0x5eed5eedull);
    cudaMemsetAsync(hist, 0, 2 * (size_t)iters * sizeof(double), ctx->stream);
    ShiftParams sp;
    sp.n = 1;
    sp.s0 = 0;
    sp.sig[0] = 0;
    sp.c[0] = 0;
    SolveSpec spec{};
    spec.B = 1;
    spec.BC = 1;
    spec.prec = SMPQ_FP64;
    spec.n_sup = 0;
    spec.d_src_field = (const double *)b;
    SolveOut out;
    // the counter lives in the scalar block; reset it through a fresh solve
    std::vector<LatIn> lats{LatIn{ctx, &spec, sp, &out}};
    rc = dispatch_bc(lats, 0.0, iters, hist, iters, iters);
    if (rc) return rc;
    std::vector<double> h(2 * (size_t)iters);
    cudaMemcpyAsync(h.data(), hist, h.size() * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream);
    cudaError_t e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) return cuda_check(ctx, e, "lanczos history");
    // CG -> Lanczos: T_kk = 1/alpha_k + beta_{k-1}/alpha_{k-1}, T_{k,k+1} = sqrt(beta_k)/alpha_k
    std::vector<double> diag, off;
    for (int k = 0; k < iters; ++k) {
        double a = h[k], bprev = k > 0 ? h[iters + k - 1] : 0.0, aprev = k > 0 ? h[k - 1] : 1.0;
        if (!(a > 0)) break;
        diag.push_back(1.0 / a + (k > 0 ? bprev / aprev : 0.0));
        double bk = h[iters + k];
        if (k + 1 < iters && h[k + 1] > 0) off.push_back(std::sqrt(bk) / a);
    }
    if (diag.size() < 2) return set_err(ctx, SMPQ_EBREAKDOWN, "Lanczos produced fewer than 2 steps");
    off.resize(diag.size() - 1);
    tridiag_extremes(diag, off, lo, hi);
    return SMPQ_OK;
}

float time_dslash_pair(smpq_ctx *ctx, int kind, int B, int BC, int tpb, int nr, int reps, void *buf, double *part,
                       double *alpha, int *err) {
    if (tpb < 1 || B % BC) return -1.f;
    switch (BC) {
    case 12: return time_kind_bc<12>(ctx, kind, B, tpb, nr, reps, buf, part, alpha, err);
    case 24: return time_kind_bc<24>(ctx, kind, B, tpb, nr, reps, buf, part, alpha, err);
    case 48: return time_kind_bc<48>(ctx, kind, B, tpb, nr, reps, buf, part, alpha, err);
    default: return -1.f;
    }
}
