"""Block fixed point (FP64 D_W and solves), the residual history's chunks and the
half-format conversion, at the sizes where their paths change."""
import numpy as np
import pytest

from conftest import KAPPA, NPOLES
from oracle import dirac, native, probing, qx, zolotarev
from synth import make_config, random_spinor
from synth.gauge import haar_su3

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_02211_gb300 import smpq
    smpq.load()
    return smpq


def _session(**kw):
    from paper_1901_02211_gb300 import Session
    return Session(**kw)


def _ref(U, psi, dims, bc, dag):
    r = native.apply_dw(U, dirac.apply_g5(psi) if dag else psi, dims, KAPPA, bc)
    return dirac.apply_g5(r) if dag else r


# 8 x 8 x 8 x 16 x 4 = 32 768 and x 5 = 40 960: either side of the 40 000 sites and
# vectors up to which four threads share one
@pytest.mark.parametrize("dims,B", [((2, 3, 5, 2), 1), ((4, 4, 4, 4), 1), ((3, 5, 4, 7), 33), ((8, 8, 8, 16), 4),
                                    ((8, 8, 8, 16), 5)])
def test_dslash_sizes(S, dims, B):
    """FP64: 60-bit blocks, within a few 2^-53 of the largest component; FP32: 2e-6 of it."""
    V = int(np.prod(dims))
    rng = np.random.default_rng(11)
    U = haar_su3(rng, 4 * V).reshape(V, 4, 3, 3)
    # sites of very different size: the exponents of neighbours are aligned
    psi = random_spinor(rng, V, B) * np.exp(rng.uniform(-12, 12, size=(V, 1, 1, B)))
    bc = (1, -1, 1, -1)
    big = np.abs(psi).max()
    with _session(bc=bc) as s:
        s.load_gauge(dims, U)
        for dag in (False, True):
            ref = _ref(U, psi, dims, bc, dag)
            assert np.abs(s.dslash(psi, dagger=dag) - ref).max() <= 16 * 2.0 ** -53 * big
            assert np.abs(s.dslash(psi, dagger=dag, precision=S.SMPQ_FP32) - ref).max() <= 2e-6 * big


def test_dslash_in_place_and_special_values(S):
    """Overlapping device buffers, zero fields, infinities, NaN and sites whose
    components are 2^40 and more apart give what FP64 arithmetic gives."""
    import torch
    cfg = make_config("flux4")
    dims, U, V = cfg["dims"], cfg["U"], 256
    psi = random_spinor(np.random.default_rng(5), V, 3)
    psi[7, 1, 2, 0] *= 1e-20
    psi[9, :, :, 1] = 0
    ref = _ref(U, psi, dims, (1, 1, 1, 1), False)
    with _session() as s:
        s.load_gauge(dims, U)
        d = torch.from_numpy(psi).cuda()
        for call in (S.smpq_dslash, S.smpq_dslash_noalloc):
            a = d.clone()
            call(s.ctx, a, a, 3)
            assert np.abs(a.cpu().numpy() - ref).max() <= 1e-13
            o = torch.empty_like(d)
            call(s.ctx, d, o, 3)
            assert np.abs(o.cpu().numpy() - ref).max() <= 1e-13
        assert not np.any(s.dslash(np.zeros_like(psi)))
        for bad in (np.nan, np.inf):
            x = psi.copy()
            x[100, 0, 0, 2] = bad
            got = s.dslash(x)
            fine = np.isfinite(_ref(U, x, dims, (1, 1, 1, 1), False))
            # sites that do not read the bad one, and the other columns, are untouched
            near = ~np.isclose(got, ref, rtol=0, atol=1e-13).all(axis=(1, 2))
            assert near[:, :2].sum() == 0 and 1 <= near[:, 2].sum() <= 9
            assert np.array_equal(np.isfinite(got), fine)
        # a range that one exponent does not hold: each spin pair on its own scale
        x = psi.copy()
        x[:, :, :, 0] *= 1e-30
        x[50, 0, 0, 0] = 1.0
        r = _ref(U, x, dims, (1, 1, 1, 1), False)
        assert np.abs(s.dslash(x) - r).max() <= 1e-13


@pytest.mark.parametrize("prec,tol,theta,bound", [("fp64", 1e-14, 1e-3, 1e-10), ("mixed", 1e-10, 1e-8, 1e-10),
                                                  ("mixed", 1e-10, 0.5, 3.4e-8)])
def test_history_chunks(S, prec, tol, theta, bound):
    """Solves that outlast the slots of the residual history: FP64 iterations beyond
    216, FP64-accurate ones of the mixed solve beyond 81, FP32 ones beyond 162.
    Bounds: the solver's 1e-10 residual; for theta = 0.5 four times the
    1.7e-8 theta by which the mixed path's q(x) follows its switch."""
    import json
    import os
    cfg = make_config("flux4x8")
    dims, U = cfg["dims"], cfg["U"]
    with open(os.path.join(os.path.dirname(__file__), "golden", "spectra.json")) as f:
        sp = json.load(f)["flux4x8"]
    a, b = 0.98 * sp["lmin2"], 1.02 * sp["lmax2"]
    c0, c, q, _ = zolotarev.zolotarev(NPOLES, a, b)
    colour, n = probing.color_sites(dims, 2, 0)
    classes = [0, 5, 9, 12, 15]  # 60 sources: a 48-column tile and 12 more
    ref, _ = qx.smp_qx(U, dims, KAPPA, (c0, c, q), colour, n, colours=classes, batch_colours=2)
    with _session(precision=getattr(S, "SMPQ_" + prec.upper()), tol=tol, switch_residual=theta) as s:
        s.load_gauge(dims, U)
        s.set_spectrum(a, b)
        s.build_sources(2, 0)
        got, _, st = s.compute_qx(classes=classes)
    mask = np.isin(colour, classes)
    assert st["n_batches"] == (1 if prec == "fp64" else 2)
    assert np.abs(got[mask] - ref[mask]).max() <= bound
    assert not np.any(got[~mask])


@pytest.mark.parametrize("fmt", ["fp16", "bf16"])
@pytest.mark.parametrize("B", [1, 16])
def test_half_conversion_range(S, fmt, B):
    """The input of the half-format D_W with norms from 1e-30 to 1e30, zeros and
    components far below the norm: the stored value is the FP64 quotient rounded to
    FP32 and the format (kappa -> 0 leaves out = in; the output is rounded again,
    to the same values)."""
    prec = S.SMPQ_FP16N if fmt == "fp16" else S.SMPQ_BF16N
    V = 256
    rng = np.random.default_rng(3)
    psi = random_spinor(rng, V, B) * 10.0 ** rng.uniform(-30, 30, size=(V, 1, 1, B))
    psi[::7, 1] *= 1e-25
    psi[3::11, 2, 1] = 0
    with _session(kappa=1e-300) as s:
        s.load_gauge(make_config("flux4")["dims"], make_config("flux4")["U"])
        got = s.dslash(psi, precision=prec)
    p = psi.reshape(V, 12, B)
    nrm = np.maximum(np.abs(p.real), np.abs(p.imag)).max(axis=1).astype(np.float32).astype(np.float64)[:, None, :]

    def rounded(x):
        f = (x / nrm).astype(np.float32)
        if fmt == "fp16":
            return f.astype(np.float16).astype(np.float64) * nrm
        import torch
        return torch.from_numpy(f).to(torch.bfloat16).to(torch.float64).numpy() * nrm

    want = rounded(p.real) + 1j * rounded(p.imag)
    # the largest stored value may be 1 - 2^-12 (its norm then changes by that and
    # the others are rounded a second time)
    unit = 2.0 ** -11 if fmt == "fp16" else 2.0 ** -8
    assert np.abs(got.reshape(V, 12, B) - want).max(axis=1, keepdims=True).__le__(unit * nrm).all()
