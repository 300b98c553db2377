"""A last batch shorter than the others (whole 48-column tiles that hold its sources):
the results of the batches are those of one batch."""
import json
import os

import numpy as np
import pytest

from synth import make_config

pytestmark = pytest.mark.gpu

GOLD = os.path.join(os.path.dirname(__file__), "golden", "spectra.json")
# what two orders of summation may differ by, relative to the largest q(x): FP64 and
# mixed solves stop at 1e-10 (the mixed path's FP32 iterations drift by up to
# 256 u_32 theta = 1.5e-8), the FP32 ones carry directions of 6e-8
BAR = {"FP64": 1e-8, "MIXED": 1e-7, "FP32": 1e-4}


@pytest.fixture(scope="module")
def S():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_02211_gb300 import smpq
    smpq.load()
    return smpq


def _session(S, name, **kw):
    from paper_1901_02211_gb300 import Session
    cfg = make_config(name)
    with open(GOLD) as f:
        sp = json.load(f)[name]
    s = Session(**kw)
    s.load_gauge(cfg["dims"], cfg["U"])
    s.set_spectrum(0.98 * sp["lmin2"], 1.02 * sp["lmax2"])
    return s


# rhs_block 96: 108 and 120 sources leave 12 and 24 (a batch of 48); 144: 192 leave 48
@pytest.mark.parametrize("prec", sorted(BAR))
@pytest.mark.parametrize("block,n", [(96, 9), (96, 10), (144, 16)])
@pytest.mark.parametrize("extra", ["", "full_support", "low_modes"])
def test_qx(S, prec, block, n, extra):
    classes = list(range(16))[-n:]
    got = []
    for b in (block, 12 * n):
        kw = dict(full_support=1) if extra == "full_support" else {}
        with _session(S, "flux4x8", precision=getattr(S, "SMPQ_" + prec), rhs_block=b, **kw) as s:
            if extra == "low_modes":
                s.low_modes(4)
            s.build_sources(2, 0)
            q, Q, st = s.compute_qx(classes=classes)
            got.append((q, Q))
            assert st["n_batches"] == (1 if b == 12 * n else 2) and st["n_rhs"] == 12 * n
    scale = np.abs(got[1][0]).max()
    assert np.abs(got[0][0] - got[1][0]).max() <= BAR[prec] * scale
    assert abs(got[0][1] - got[1][1]) <= BAR[prec] * scale * 512


@pytest.mark.parametrize("prec", sorted(BAR))
def test_trace(S, prec):
    got = []
    for b in (144, 192):
        with _session(S, "flux4x8", precision=getattr(S, "SMPQ_" + prec), rhs_block=b) as s:
            s.build_sources(2, 0)
            t, T, st = s.trace_dwinv()
            got.append(t)
            assert st["n_batches"] == (1 if b == 192 else 2)
    assert np.abs(got[0] - got[1]).max() <= BAR[prec] * np.abs(got[1]).max()
