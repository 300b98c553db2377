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

    def call(c, zn, zo, alpha, beta, r, ps, y):
        n, nshift = zn.shape[:2]
        ps, y = ps.copy(), y.copy()
        ptr = [np.ascontiguousarray(a).ctypes.data_as(ctypes.c_void_p) for a in (c, zn, zo, alpha, beta, r)]
        rc = f(n, nshift, r.shape[1] // 144, *ptr,
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
    _, got = probe(np.ones(nshift), zeta, zeta, alpha, beta, r / scale, ps, y)
    col = _columns(ne)
    b, z = beta[0, col].astype(np.longdouble), zeta[0][:, col].astype(np.longdouble)
    rl = (r / scale)[0]
    for part in ("real", "imag"):
        p, q = getattr(ps, part).astype(np.longdouble), getattr(rl, part).astype(np.longdouble)
        err = np.abs(getattr(got, part) - (b * p + z * q))
        assert (err <= 2 * U * (np.abs(b * p) + np.abs(z * q))).all()


@pytest.mark.parametrize("n,nshift", [(3, 2), (19, 14), (40, 17)])
def test_chunk_of_fp64_iterations(probe, n, nshift):
    """y and the directions against the recurrences in extended precision.  A weight has
    up to 5 roundings per iteration (zeta ratio twice, beta, alpha, the product) and one
    per shift; the sums one per term."""
    rng = np.random.default_rng(n)
    ne = 144 * 3
    r, ps, y = _fields(rng, n, nshift, ne)
    zn, zo = rng.uniform(0.5, 1, (2, n, nshift, 12))
    alpha, beta = rng.uniform(0.5, 1, (2, n, 12))
    zn[n // 2:, nshift - 1] = 0  # the last shift has converged
    c = rng.uniform(0.1, 1, nshift)
    gy, gp = probe(c, zn, zo, alpha, beta, r, ps, y)
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
