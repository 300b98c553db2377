"""The half-format conversions of the stand-alone D_W, every component against the FP64
quotient and product."""
import numpy as np
import pytest

from synth import make_config, random_spinor

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_02211_gb300 import smpq
    smpq.load()
    return smpq


def _format(f, fmt):
    """FP32 numbers rounded to the format"""
    if fmt == "fp16":
        return f.astype(np.float16).astype(np.float32)
    import torch
    return torch.from_numpy(f).to(torch.bfloat16).to(torch.float32).numpy()


@pytest.mark.parametrize("fmt", ["fp16", "bf16"])
@pytest.mark.parametrize("B", [1, 5, 16, 32])
def test_every_component(S, fmt, B):
    """kappa = 0 in FP32: out = in, with the roundings of the way: the FP64 quotient by the
    norm to FP32 and to the format, their product to FP32 in D_W, that times 1 / norm to
    the format, and the FP64 product with the norm.  Norms from 1e-30 to 1e30, components
    down to 1e-25 of the norm (either side of 2^-70, where the quotient is an FP64
    division), subnormal ones in fp16, ones below FP32's range, and zeros."""
    from paper_1901_02211_gb300 import Session
    V = 256
    rng = np.random.default_rng(B)
    psi = random_spinor(rng, V, B) * 10.0 ** rng.uniform(-30, 30, size=(V, 1, 1, B))
    psi[::3] *= 10.0 ** rng.uniform(-9, 0, size=psi[::3].shape)
    psi[1::7, 1] *= 10.0 ** rng.uniform(-25, -15, size=psi[1::7, 1].shape)
    psi[3::11, 2, 1] = 0
    cfg = make_config("flux4")
    with Session(kappa=1e-300) as s:
        s.load_gauge(cfg["dims"], cfg["U"])
        got = s.dslash(psi, precision=S.SMPQ_FP16N if fmt == "fp16" else S.SMPQ_BF16N).reshape(V, 12, B)
    p = psi.reshape(V, 12, B)
    x = np.stack([p.real, p.imag])
    nrm = np.abs(x).max(axis=(0, 2)).astype(np.float32)[None, :, None, :]
    v = _format((x / nrm.astype(np.float64)).astype(np.float32), fmt) * nrm
    nrm = np.abs(v).max(axis=(0, 2), keepdims=True)
    want = nrm.astype(np.float64) * _format(v * (np.float32(1) / nrm), fmt)
    assert np.array_equal(np.stack([got.real, got.imag]), want)


@pytest.mark.parametrize("fmt", ["FP16N", "BF16N"])
@pytest.mark.parametrize("B", [1, 16])
def test_negative_zero(S, fmt, B):
    """A negative component below the format's range is stored as -0 and comes back so."""
    from paper_1901_02211_gb300 import Session
    dims, V = (4, 4, 4, 4), 256
    U = np.broadcast_to(np.eye(3, dtype=complex), (V, 4, 3, 3)).copy()
    psi = np.zeros((V, 4, 3, B), complex)
    psi[:, :, 1] = 2.0 ** -28 * (1 + 1j)
    psi[5] = 0
    psi[5, :, 0] = 1 + 1j
    with Session(kappa=0.2) as s:  # colour 1 of site 5: -8 kappa 2^-28, the norm is 1
        s.load_gauge(dims, U)
        got = s.dslash(psi, precision=getattr(S, "SMPQ_" + fmt))[5, :, 1]
    assert np.signbit(got.real).all() and np.signbit(got.imag).all()
    assert np.abs(got).max() <= 1e-8
