"""The stand-alone FP64 D_W component by component: on links that do not mix colours
a small component stays apart from the large ones, and keeps the accuracy that FP64
arithmetic gives it."""
import numpy as np
import pytest

from oracle import dirac, native
from synth import random_spinor
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


def _links(kind, rng, V):
    if kind == "haar":
        return haar_su3(rng, 4 * V).reshape(V, 4, 3, 3)
    U = np.zeros((V, 4, 3, 3), complex)
    ph = np.zeros((V, 4, 3)) if kind == "unit" else rng.uniform(0, 2 * np.pi, (V, 4, 3))
    ph[..., 2] = -ph[..., 0] - ph[..., 1]
    U[..., range(3), range(3)] = np.exp(1j * ph)
    return U


def _terms(U, psi, dims, kappa):
    """|own| + kappa times the sum of the moduli of all products behind each real
    number of D_W psi, as re + i im."""
    nx, ny, nz, nt = dims
    V, B = psi.shape[0], psi.shape[-1]
    p = np.abs(psi.real) + 1j * np.abs(psi.imag)
    u = np.abs(U.real) + 1j * np.abs(U.imag)
    out = p.copy()

    def swap(x):
        return x.imag + 1j * x.real

    def mul(m, h):  # moduli of (re, im) of m h
        re = np.einsum("vab,vsbj->vsaj", m.real, h.real) + np.einsum("vab,vsbj->vsaj", m.imag, h.imag)
        im = np.einsum("vab,vsbj->vsaj", m.real, h.imag) + np.einsum("vab,vsbj->vsaj", m.imag, h.real)
        return re + 1j * im

    def shift(x, mu, step):
        w = np.roll(x.reshape((nt, nz, ny, nx) + x.shape[1:]), -step, axis=3 - mu)
        return w.reshape((V,) + x.shape[1:])

    for mu in range(4):
        low = p[:, 2:]
        if mu < 2:
            low = low[:, ::-1]
        h = p[:, :2] + (swap(low) if mu in (0, 2) else low)
        for w in (mul(u[:, mu], shift(h, mu, 1)), shift(mul(u[:, mu].transpose(0, 2, 1), h), mu, -1)):
            out[:, :2] += kappa * w
            w = w[:, ::-1] if mu < 2 else w
            out[:, 2:] += kappa * (swap(w) if mu in (0, 2) else w)
    return out


def _check(got, ref, terms):
    """Roundings on the longest path to a component: FP64 17 (projection 1, products
    6, hops 8, kappa and the sum 2), block fixed point 5.5 units of 2^-52 of the
    terms at its line, the oracle 17 again: 40 * 2^-53 of the terms."""
    bar = 40 * 2.0 ** -53
    assert (np.abs(got.real - ref.real) <= bar * terms.real).all()
    assert (np.abs(got.imag - ref.imag) <= bar * terms.imag).all()


def _ref(U, psi, dims, kappa, bc, dag):
    r = native.apply_dw(U, dirac.apply_g5(psi) if dag else psi, dims, kappa, bc)
    return dirac.apply_g5(r) if dag else r


# 8 x 8 x 8 x 16 x 5 lies above the number of sites and vectors up to which four
# threads share one; kappa 0.06 and 0.0625 on either side of the FP64 route
@pytest.mark.parametrize("links", ["unit", "diagonal", "haar"])
@pytest.mark.parametrize("dims,B,kappa", [((2, 3, 5, 2), 3, 0.21), ((4, 4, 4, 4), 1, 0.0625), ((3, 5, 4, 7), 2, 0.06),
                                          ((4, 6, 4, 4), 4, 0.24), ((8, 8, 8, 16), 5, 0.21)])
def test_dslash_components(S, links, dims, B, kappa):
    from paper_1901_02211_gb300 import Session
    rng = np.random.default_rng(7)
    V = int(np.prod(dims))
    U = _links(links, rng, V)
    bc = (1, -1, 1, -1)
    psi = random_spinor(rng, V, B)
    scaled = {"even": psi,
              "colours 1e-3": psi * np.array([1, 1e-3, 1e-6])[None, None, :, None],
              "colours 1e-9": psi * np.array([1e-9, 1, -1e-18])[None, None, :, None],
              "sites": psi * np.exp(rng.uniform(-12, 12, (V, 1, 1, B))),
              "constant": np.broadcast_to(random_spinor(rng, 1, B), psi.shape) * np.array([1, 1e-5, 1])[None, None, :, None]}
    point = np.zeros_like(psi)
    point[V // 2, 1, 2] = 0.3
    scaled["point"] = point
    with Session(bc=bc, kappa=kappa) as s:
        s.load_gauge(dims, U)
        for x in scaled.values():
            x = np.ascontiguousarray(x)
            terms = _terms(U, x, dims, kappa)
            for dag in (False, True):
                _check(s.dslash(x, dagger=dag), _ref(U, x, dims, kappa, bc, dag), terms)


@pytest.mark.parametrize("B", [1, 3, 6])
@pytest.mark.parametrize("shift", [0, 1, 1000])
def test_dslash_overlapping_buffers(S, shift, B):
    """out over in, or part of it: the bits of the call on two buffers, also where
    sites are done in FP64 from in."""
    import torch
    from paper_1901_02211_gb300 import Session
    rng = np.random.default_rng(19)
    dims, V = (4, 6, 4, 8), 768
    n = V * 12 * B
    psi = random_spinor(rng, V, B)
    psi[:40] *= np.array([1, 1e-7, 1])[None, None, :, None]
    psi[300, 0, 0, 0] = np.nan
    with Session() as s:
        s.load_gauge(dims, _links("diagonal", rng, V))
        for prec in (S.SMPQ_FP64, S.SMPQ_FP32):
            for call in (S.smpq_dslash, S.smpq_dslash_noalloc):
                d = torch.from_numpy(psi).cuda()
                want = torch.empty_like(d)
                call(s.ctx, d, want, B, False, prec)
                room = torch.zeros(n + shift, dtype=torch.complex128, device="cuda")
                for i, o in ((room[:n], room[shift:]), (room[shift:], room[:n])):
                    i, o = i.view(V, 4, 3, B), o.view(V, 4, 3, B)
                    i.copy_(d)
                    call(s.ctx, i, o, B, False, prec)
                    assert torch.equal(torch.view_as_real(o).view(torch.int64), torch.view_as_real(want).view(torch.int64))


def test_noalloc_in_place_at_its_limit(S):
    """The largest field that fits the scratch, in place (copy and blocks side by side)."""
    import torch
    from paper_1901_02211_gb300 import Session
    rng = np.random.default_rng(23)
    dims, V, B = (4, 4, 4, 4), 256, (32 << 20) // (2 * 256 * 12 * 16)
    psi = random_spinor(rng, V, B)
    with Session() as s:
        s.load_gauge(dims, _links("haar", rng, V))
        d = torch.from_numpy(psi).cuda()
        want = torch.empty_like(d)
        S.smpq_dslash(s.ctx, d, want, B)
        S.smpq_dslash_noalloc(s.ctx, d, d, B)
        assert torch.equal(torch.view_as_real(d), torch.view_as_real(want))


@pytest.mark.parametrize("prec,copies", [("FP64", 3.1), ("FP32", 2.0), ("FP16N", 1.6), ("BF16N", 1.6)])
def test_dslash_host_buffers_scratch(S, prec, copies):
    """Device memory that a call on host buffers takes: a copy of the vectors and the
    fields in the format's size (FP64: input, blocks and output), in copies of the
    vectors; 4 MiB for the allocator's rounding."""
    import torch
    from paper_1901_02211_gb300 import Session
    rng = np.random.default_rng(29)
    dims, V, B = (8, 8, 8, 16), 8192, 16
    psi = random_spinor(rng, V, B)
    with Session() as s:
        s.load_gauge(dims, _links("unit", rng, V))
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        s.dslash(psi, precision=getattr(S, "SMPQ_" + prec))
        assert free - torch.cuda.mem_get_info()[0] <= copies * psi.nbytes + (4 << 20)
