"""The sums over the residual history at the end of a chunk of iterations, kernel by
kernel: their rounding is FP64's."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_02211_gb300 import _build
    here = os.path.dirname(os.path.abspath(__file__))
    lib = str(tmp_path_factory.mktemp("hist") / "hist_probe.so")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    r = subprocess.run([nvcc] + _build.ARCH + ["-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", _build.INCLUDE,
                        os.path.join(here, "hist_probe.cu"), "-o", lib, "-lcudart"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    f = ctypes.CDLL(lib).hist_probe

    def call(fp32, theta, c, zn, zo, alpha, beta, r, ps, y):
        n, nshift = zn.shape[:2]
        ps, y = ps.copy(), y.copy()
        ptr = [np.ascontiguousarray(a).ctypes.data_as(ctypes.c_void_p) for a in (c, zn, zo, alpha, beta, r)]
        rc = f(int(fp32), ctypes.c_double(theta), n, nshift, r.shape[1] // 144, *ptr,
               ps.ctypes.data_as(ctypes.c_void_p), y.ctypes.data_as(ctypes.c_void_p))
        assert rc == 0
        return y, ps
    return call


def _columns(ne):
    """column of each element: [n_sup][12][12 columns]"""
    return np.arange(ne) % 12


def _fields(rng, n, nshift, ne):
    def z(*s):
        return rng.standard_normal(s) + 1j * rng.standard_normal(s)
    return z(n, ne), z(nshift, ne), z(ne)


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -130])
@pytest.mark.parametrize("nshift", [1, 14, 15])
def test_directions_after_one_iteration(probe, nshift, scale):
    """p = beta p + zeta r with zeta_{k+1} = zeta_k (the weights are then beta and zeta
    themselves): product, product and sum round once each.  scale: zeta below the FP32
    range's precision, r as much larger."""
    rng = np.random.default_rng(nshift)
    ne = 144 * 5
    r, ps, y = _fields(rng, 1, nshift, ne)
    zeta = scale * rng.uniform(0.5, 1, (1, nshift, 12))
    alpha, beta = rng.uniform(0.5, 1, (1, 12)), rng.uniform(0.5, 1, (1, 12))
    _, got = probe(False, 0, np.ones(nshift), zeta, zeta, alpha, beta, r / scale, ps, y)
    col = _columns(ne)
    b, z = beta[0, col].astype(np.longdouble), zeta[0][:, col].astype(np.longdouble)
    rl = (r / scale)[0]
    for part in ("real", "imag"):
        p, q = getattr(ps, part).astype(np.longdouble), getattr(rl, part).astype(np.longdouble)
        err = np.abs(getattr(got, part) - (b * p + z * q))
        assert (err <= 2 * U * (np.abs(b * p) + np.abs(z * q))).all()


@pytest.mark.parametrize("n,nshift", [(3, 2), (19, 14), (40, 17), (37, 1)])
def test_chunk_of_fp64_iterations(probe, n, nshift):
    """y and the directions against the recurrences in extended precision.  A weight has
    up to 5 roundings per iteration (zeta ratio twice, beta, alpha, the product) and one
    per shift; the sums one per term."""
    rng = np.random.default_rng(n)
    ne = 144 * 3
    r, ps, y = _fields(rng, n, nshift, ne)
    zn, zo = rng.uniform(0.5, 1, (2, n, nshift, 12))
    alpha, beta = rng.uniform(0.5, 1, (2, n, 12))
    if nshift > 1:
        zn[n // 2:, nshift - 1] = 0  # the last shift has converged
    c = rng.uniform(0.1, 1, nshift)
    gy, gp = probe(False, 0, c, zn, zo, alpha, beta, r, ps, y)
    col = _columns(ne)
    L = np.longdouble
    p, s = ps.astype(np.clongdouble), y.astype(np.clongdouble)
    pa, sa = np.abs(ps.real).astype(L) + 0, np.abs(y.real).astype(L)  # the same with moduli (real parts)
    for k in range(n):
        for i in range(nshift):
            z = zn[k, i, col].astype(L)
            on = z != 0
            w = np.where(on, z / zo[k, i, col].astype(L), 1)
            a = np.where(on, alpha[k, col].astype(L) * w, 0)
            b = np.where(on, beta[k, col].astype(L) * w * w, 1)
            s = s + c[i] * a * p[i]
            sa = sa + c[i] * a * pa[i]
            p[i] = np.where(on, z * r[k] + b * p[i], p[i])
            pa[i] = np.where(on, z * np.abs(r[k].real) + b * pa[i], pa[i])
    bar = (6 * n + nshift + 4) * U
    assert (np.abs(gy.real - s.real) <= bar * sa).all()
    assert (np.abs(gp.real - p.real) <= bar * pa).all()


@pytest.mark.parametrize("theta", [0.9, 0.5, 2.0 ** -7])
@pytest.mark.parametrize("nshift", [1, 15])
def test_share_of_fp32_iterations(probe, theta, nshift):
    """y after one FP32 iteration of a mixed solve with a large switch residual, where
    that iteration's share c alpha p is most of y: each term's coefficient rounds once,
    its product with the sum once."""
    rng = np.random.default_rng(5)
    ne = 144 * 5
    r, ps, _ = _fields(rng, 1, nshift, ne)
    ps = ps.astype(np.complex64).astype(complex)
    zeta = rng.uniform(0.5, 1, (1, nshift, 12))
    alpha, beta = rng.uniform(0.5, 1, (2, 1, 12))
    c = rng.uniform(0.1, 1, nshift)
    got, _ = probe(True, theta, c, zeta, zeta, alpha, beta, r, ps, np.zeros(ne, complex))
    a = c[:, None].astype(np.longdouble) * alpha[0, _columns(ne)]
    for part in ("real", "imag"):
        terms = a * getattr(ps, part)
        err = np.abs(getattr(got, part) - terms.sum(0))
        # alpha z / z rounds twice, times c once
        assert (err <= (3 + nshift) * U * np.abs(terms).sum(0)).all()


@pytest.mark.parametrize("n,nshift", [(1, 14), (7, 14), (30, 14), (30, 1)])
def test_share_below_a_small_switch_residual(probe, n, nshift):
    """At the largest switch residual with float-float sums, y of that many times the
    share: within the FP64 sums' own bound (an addition per shift and iteration)."""
    rng = np.random.default_rng(n)
    ne = 144 * 3
    r, ps, _ = _fields(rng, n, nshift, ne)
    r, ps = (x.astype(np.complex64).astype(complex) for x in (r, ps))
    zeta = np.broadcast_to(rng.uniform(0.5, 1, (1, nshift, 12)), (n, nshift, 12)).copy()
    alpha, beta = rng.uniform(0.5, 1, (2, n, 12)) / n
    c = rng.uniform(0.1, 1, nshift)
    y = 256 * (rng.choice([-1, 1], ne) + 1j * rng.choice([-1, 1], ne)) * rng.uniform(1, 2, ne)
    got, _ = probe(True, 2.0 ** -8, c, zeta, zeta, alpha, beta, r, ps, y)
    col = _columns(ne)
    s = y.astype(np.clongdouble)
    p = ps.astype(np.complex64)
    share = np.zeros(ne)
    for k in range(n):
        a = c[:, None].astype(np.longdouble) * alpha[k, col]
        s = s + (a * p).sum(0)
        share += (np.abs(a) * np.abs(p.real)).sum(0).astype(float)
        z32, b32 = zeta[k][:, col].astype(np.float32), beta[k, col].astype(np.float32)
        # the FP32 recurrence: product, then one fused multiply-add
        zr = z32 * r[k].astype(np.complex64).real, z32 * r[k].astype(np.complex64).imag
        p = ((b32.astype(float) * p.real + zr[0]).astype(np.float32)
             + 1j * (b32.astype(float) * p.imag + zr[1]).astype(np.float32)).astype(np.complex64)
    assert (np.abs(got.real - s.real) <= (n * nshift + 1) * U * (np.abs(y.real) + share)).all()
