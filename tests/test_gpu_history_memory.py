"""Device memory of the residual history: bounded, and after what a solve cannot do
without."""
import json
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_02211_gb300 import smpq
    smpq.load()
    return torch


def _free(torch):
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()


def test_dov_holds_a_bounded_history(torch):
    """D_ov on 8 vectors of 16^3x32 (its whole history is 43.5 GB): a twelfth of the
    GPU's memory, and 353 bytes a value for the fields (3 x 16 caller side, 3 x 16.3
    vectors, 16 y, 14 x 16 directions), the partial sums and the scalars."""
    from paper_1901_02211_gb300 import Session
    dims, V, B = (16, 16, 16, 32), 131072, 8
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    u = torch.eye(3, dtype=torch.complex128, device="cuda").expand(V, 4, 3, 3).contiguous()
    psi = torch.randn(V, 4, 3, B, dtype=torch.complex128, device="cuda", generator=g)
    out = torch.empty_like(psi)
    with Session(device=0, stream=torch.cuda.current_stream().cuda_stream) as s:
        s.load_gauge(dims, u)
        s.set_spectrum(0.015, 7.3)
        from paper_1901_02211_gb300 import smpq
        free, total = _free(torch)
        smpq.smpq_apply_dov(s.ctx, psi, out, B)
        held = free - _free(torch)[0]
        # gamma_5-hermiticity of the overlap operator: |D psi|^2 = 2 Re <psi, D psi>
        n2 = (out.abs() ** 2).sum(dim=(0, 1, 2))
        re = 2 * (psi.conj() * out).real.sum(dim=(0, 1, 2))
        assert ((n2 - re).abs() <= 1e-8 * n2).all()
    assert held <= total / 12 + 353 * psi.numel() + (64 << 20)


def test_fields_come_before_the_history(torch):
    """192 sources of 8^3x16 in one mixed batch with 112 bytes a value free: the fields
    (80), y (16 on 9/256 of the lattice) and the directions (336 there) take 92.4, the
    whole history 45.6 more."""
    from paper_1901_02211_gb300 import Session, smpq
    from synth import make_config
    cfg = make_config("flux8x16")
    with open(os.path.join(os.path.dirname(__file__), "golden", "spectra.json")) as f:
        spec = json.load(f)["flux8x16"]
    classes = list(range(0, 256, 16))
    values = 12 * 8192 * 192

    def run(target):
        with Session(device=0, stream=torch.cuda.current_stream().cuda_stream, precision=smpq.SMPQ_MIXED,
                     rhs_block=192, autotune=0) as s:
            s.load_gauge(cfg["dims"], cfg["U"])
            s.set_spectrum(0.98 * spec["lmin2"], 1.02 * spec["lmax2"])
            s.build_sources(4, 0)
            block = None
            if target:
                free = _free(torch)[0]
                block = torch.empty(free - target, dtype=torch.uint8, device="cuda")
            try:
                q, Q, st = s.compute_qx(classes=classes)
                assert np.array_equal(q, s.compute_qx(classes=classes)[0])  # the same chunks again
            finally:
                del block
                torch.cuda.empty_cache()
        assert st["n_batches"] == 1
        return q

    want = run(0)
    got = run(112 * values)
    # chunks sum the same history in other portions
    assert np.abs(got - want).max() <= 1e-11 * np.abs(want).max()


def test_history_costs_no_batch(torch):
    """192 mixed sources of r = 2 on 8^3x16 cost 28.9 MB each (96 bytes a value on the
    lattice, 352 on 9/16 of it): 10.3 GB free, of which batches take 0.6, hold them in
    one batch, whatever the history would like."""
    from paper_1901_02211_gb300 import Session, smpq
    from synth import make_config
    cfg = make_config("flux8x16")
    with open(os.path.join(os.path.dirname(__file__), "golden", "spectra.json")) as f:
        spec = json.load(f)["flux8x16"]
    got = []
    for target in (0, 10300 << 20):
        with Session(device=0, stream=torch.cuda.current_stream().cuda_stream, precision=smpq.SMPQ_MIXED,
                     autotune=0) as s:
            s.load_gauge(cfg["dims"], cfg["U"])
            s.set_spectrum(0.98 * spec["lmin2"], 1.02 * spec["lmax2"])
            s.build_sources(2, 0)
            block = None
            if target:
                block = torch.empty(_free(torch)[0] - target, dtype=torch.uint8, device="cuda")
            try:
                q, Q, st = s.compute_qx()
            finally:
                del block
                torch.cuda.empty_cache()
        assert st["n_batches"] == 1
        got.append(q)
    assert np.abs(got[1] - got[0]).max() <= 1e-11 * np.abs(got[0]).max()
