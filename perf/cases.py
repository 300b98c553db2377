"""The work that a user of libsmpq has it do, as cases that can be timed.

Every case goes through the public calls (the C ABI by its ctypes binding), on gauge
fields and spinors on the GPU, with the context that a program keeps: a gauge field
loaded, a Zolotarev interval set, a colouring built.  The sizes are those of the
configurations of synth/ and of bench.py (4^4, 4^3x8, 8^3x16, 16^3x32; 6^3 and 9^3 for
ragged tiles), with the probing distances of the tests and the bench.

What is listed:
  - D_W alone: the smallest call there is, FP64 on a batch of sources, FP32 on a large
    lattice, FP16 storage;
  - D_ov applied to vectors;
  - q(x): the FP64 path (the default precision) on the small lattice and on a batch, the
    mixed path (the one the bench quotes) from one colour class up to all 3072 sources,
    on a ragged lattice and on the large one, class by class as a program with
    checkpoints runs it; several lattices in one call;
  - the trace of D_W^-1.
Solves with SMPQ_FP32, SMPQ_FP16N and SMPQ_BF16N are not among them: what their shifted
systems return is the rounding of the storage format, and no two orders of summation
give the same.  Lanczos and the low modes are set-up, once for a gauge field.
"""
import math

import numpy as np
import torch

from paper_1901_02211_gb300 import Session
from paper_1901_02211_gb300 import smpq as S

KAPPA, NPOLES = 0.21, 14
# a bracket of the spectrum of H_W^2 on these backgrounds (widened by hand)
LMIN2, LMAX2 = 0.015, 7.3
PRECISION = {"fp64": S.SMPQ_FP64, "fp32": S.SMPQ_FP32, "mixed": S.SMPQ_MIXED, "fp16n": S.SMPQ_FP16N,
             "bf16n": S.SMPQ_BF16N}
# CG iterations that the smallest shift takes on these backgrounds, for work()
ITERATIONS = 180


def listed():
    return [
        # one vector on the smallest lattice, no allocation: a caller's inner loop; latency
        dict(name="dw noalloc 4^4", kind="noalloc", dims="4 4 4 4", B=1, precision="fp64", dagger=False),
        # D_W on the twelve components of a point source, the default precision
        dict(name="dw fp64 8^3x16 B12", kind="dslash", dims="8 8 8 16", B=12, precision="fp64", dagger=False),
        # D_W^dag in FP32 on the large lattice, an uneven number of vectors
        dict(name="dw fp32 16^3x32 B21", kind="dslash", dims="16 16 16 32", B=21, precision="fp32", dagger=True),
        # the half-precision storage, 16-column tiles
        dict(name="dw fp16n 8^3x16 B96", kind="dslash", dims="8 8 8 16", B=96, precision="fp16n", dagger=False),
        # D_ov on a few vectors, as an eigensolver or a check of the Ginsparg-Wilson relation applies it
        dict(name="dov 8^3x16 B3", kind="dov", dims="8 8 8 16", B=3),
        # the small parity configuration, all sources of r = 2, in the reference precision
        dict(name="q fp64 4^4 r2", kind="qx", dims="4 4 4 4", k=1, eps=0.05, r=2, mode=0, classes=0, precision="fp64",
             antiperiodic=False),
        # the reference precision on a sample of the classes of the bench's configuration
        dict(name="q fp64 8^3x16 6cl", kind="qx", dims="8 8 8 16", k=2, eps=0.1, r=4, mode=0, classes=6,
             precision="fp64", antiperiodic=True),
        # one colour class: the unit of checkpointing, and of a spot check
        dict(name="q mixed 8^3x16 1cl", kind="qx", dims="8 8 8 16", k=2, eps=0.1, r=4, mode=0, classes=1,
             precision="mixed", antiperiodic=False),
        # no power of two anywhere: 81 classes of a 9^3x12 lattice, 972 sources in one batch
        dict(name="q mixed 9^3x12 r3", kind="qx", dims="9 9 9 12", k=1, eps=0.1, r=3, mode=0, classes=0,
             precision="mixed", antiperiodic=False),
        # the large lattice, four classes at a time
        dict(name="q mixed 16^3x32 4cl", kind="qx", dims="16 16 16 32", k=-1, eps=0.15, r=4, mode=0, classes=4,
             precision="mixed", antiperiodic=False),
        # the bench's workload: every source of r = 4, 3072 of them
        dict(name="q mixed 8^3x16 r4", kind="qx", dims="8 8 8 16", k=2, eps=0.1, r=4, mode=0, classes=0,
             precision="mixed", antiperiodic=False),
        # three lattices of different sizes in one call
        dict(name="batch mixed", kind="batch", dims="4 4 4 8,6 6 6 12,8 8 8 16", k=1, eps=0.1, r=2, mode=2,
             precision="mixed"),
    ]


def draw(rng):
    def lattice(r, vmin, vmax):
        for _ in range(10000):
            v = math.exp(rng.uniform(math.log(vmin), math.log(vmax)))
            side = v ** 0.25 / r
            d = [max(1, round(side * math.exp(rng.uniform(-0.5, 0.5)))) * r for _ in range(4)]
            if min(d) >= 2 and vmin <= math.prod(d) <= vmax:
                return d
        return [4 * r // math.gcd(4, r)] * 4

    def text(d):
        return " ".join(map(str, d))

    kind = rng.choice(["noalloc", "dslash", "dslash", "dov", "qx", "qx", "qx", "qx", "batch"])
    if kind == "noalloc":
        d = lattice(1, 200, 6000)
        most = (32 << 20) // (2 * 12 * 16 * math.prod(d)) - 1
        return dict(kind=kind, dims=text(d), B=rng.randint(1, max(1, min(4, most))),
                    precision=rng.choice(["fp64", "fp32"]), dagger=rng.random() < 0.5)
    if kind == "dslash":
        d = lattice(1, 256, 131072)
        most = min(96, 3000000 // math.prod(d))
        b = max(1, round(math.exp(rng.uniform(0, math.log(most)))))
        p = rng.choice(["fp64", "fp64", "fp32", "fp16n", "bf16n"])
        if p in ("fp16n", "bf16n") and rng.random() < 0.5:
            b = max(16, b // 16 * 16) if most >= 16 else b
        return dict(kind=kind, dims=text(d), B=b, precision=p, dagger=rng.random() < 0.5)
    if kind == "dov":
        d = lattice(2, 256, 16384)
        return dict(kind=kind, dims=text(d), B=rng.randint(1, max(1, min(8, 40000 // math.prod(d)))))
    r = rng.choice([2, 2, 3, 4, 4])
    mode = rng.choice([0, 0, 0, 2]) if r % 2 == 0 else 0
    k, eps = rng.choice([1, 2, -1]), rng.choice([0.05, 0.1])
    if kind == "batch":
        r, mode = 2, 2
        ds = [lattice(2, 256, 8192) for _ in range(rng.randint(2, 4))]
        return dict(kind=kind, dims=",".join(text(d) for d in ds), k=1, eps=eps, r=r, mode=mode, precision="mixed")
    p = rng.choice(["mixed", "mixed", "mixed", "fp64"])
    d = lattice(r, 256, 131072 if p == "mixed" else 8192)
    n = r ** 4 // (2 if mode == 2 else 1)
    most = min(n, max(1, (16000000 if p == "mixed" else 900000) // (12 * math.prod(d))))
    c = max(1, round(math.exp(rng.uniform(0, math.log(most)))))
    return dict(kind=kind, dims=text(d), k=k, eps=eps, r=r, mode=mode, classes=0 if c == n else c, precision=p,
                antiperiodic=rng.random() < 0.3)


# ----------------------------------------------------------------------------- inputs


def _dims(case):
    return [tuple(int(x) for x in d.split()) for d in case["dims"].split(",")]


def _generator(seed, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + n)
    return g


def _coords(dims):
    """x, y, z, t of every site, x fastest."""
    nx, ny, nz, nt = dims
    s = torch.arange(nx * ny * nz * nt, device="cuda")
    return s % nx, s // nx % ny, s // (nx * ny) % nz, s // (nx * ny * nz)


def _cross_conj(a, b):
    return torch.linalg.cross(a, b, dim=-1).conj()


def _haar(g, n):
    """n SU(3) matrices from Gaussian rows by Gram-Schmidt; the third row is the conjugate cross product."""
    a, b = torch.randn(2, n, 3, dtype=torch.complex128, device="cuda", generator=g)
    a = a / torch.linalg.vector_norm(a, dim=-1, keepdim=True)
    b = b - (a.conj() * b).sum(-1, keepdim=True) * a
    b = b / torch.linalg.vector_norm(b, dim=-1, keepdim=True)
    return torch.stack([a, b, _cross_conj(a, b)], dim=1)


def _noise(g, n, eps):
    """exp(i eps H), H Hermitian and traceless with the weights of the Gell-Mann matrices."""
    x = torch.randn(n, 8, dtype=torch.float64, device="cuda", generator=g)
    h = torch.zeros(n, 3, 3, dtype=torch.complex128, device="cuda")
    for i, j, q in ((0, 1, 0), (0, 2, 2), (1, 2, 4)):
        h[:, i, j] = torch.complex(x[:, q], -x[:, q + 1])
        h[:, j, i] = torch.complex(x[:, q], x[:, q + 1])
    d = x[:, 7] / math.sqrt(3)
    h[:, 0, 0], h[:, 1, 1], h[:, 2, 2] = d + x[:, 6], d - x[:, 6], -2 * d
    a = 1j * eps * h / 16  # scaling and squaring of the Taylor series
    e = torch.eye(3, dtype=torch.complex128, device="cuda").expand(n, 3, 3).clone()
    term = e
    for q in range(1, 14):
        term = term @ a / q
        e = e + term
    for _ in range(4):
        e = e @ e
    return e


def gauge_field(dims, k, eps, g):
    """Quantised fluxes (k, 1), (-k, 0), (0, -1) in the x-y and z-t planes, noise, a random gauge
    transform: U[V, 4, 3, 3] on the GPU."""
    nx, ny, nz, nt = dims
    v = math.prod(dims)
    x, y, z, t = (c.double()[:, None] for c in _coords(dims))
    n12 = torch.tensor([k, -k, 0.0], dtype=torch.float64, device="cuda")
    n34 = torch.tensor([1.0, 0.0, -1.0], dtype=torch.float64, device="cuda")
    p12, p34 = 2 * math.pi * n12 / (nx * ny), 2 * math.pi * n34 / (nz * nt)
    ph = torch.stack([-p12 * y, torch.where(y == ny - 1, p12 * ny * x, 0.0), -p34 * t,
                      torch.where(t == nt - 1, p34 * nt * z, 0.0)], dim=1)
    u = torch.diag_embed(torch.exp(1j * ph))
    u = (_noise(g, 4 * v, eps) @ u.reshape(4 * v, 3, 3)).reshape(v, 4, 3, 3)
    h = _haar(g, v)
    hs = h.reshape(nt, nz, ny, nx, 3, 3)
    for mu in range(4):
        there = torch.roll(hs, -1, 3 - mu).reshape(v, 3, 3)
        u[:, mu] = h @ u[:, mu] @ there.conj().transpose(1, 2)
    return u.contiguous()


def spinors(dims, b, g):
    return torch.randn(math.prod(dims), 4, 3, b, dtype=torch.complex128, device="cuda", generator=g)


def _class_list(case, n):
    """The classes a case asks for, spread over all of them."""
    c = case.get("classes", 0)
    return list(range(n)) if not c else [i * n // c for i in range(c)]


def _inputs(case, seed):
    """[(dims, links, spinors or None)] of a case."""
    out = []
    for n, dims in enumerate(_dims(case)):
        g = _generator(seed, n)
        u = gauge_field(dims, case.get("k", 2), case.get("eps", 0.1), g)
        out.append((dims, u, spinors(dims, case["B"], g) if "B" in case else None))
    return out


def _bc(case):
    return (1, 1, 1, -1) if case.get("antiperiodic") else (1, 1, 1, 1)


def prepare(case, seed):
    state = dict(case=case, sessions=[])
    kind = case["kind"]
    for dims, u, psi in _inputs(case, seed):
        options = dict(bc=_bc(case))
        if kind in ("qx", "batch"):
            options["precision"] = PRECISION[case["precision"]]
        s = Session(device=0, stream=torch.cuda.current_stream().cuda_stream, **options)
        s.load_gauge(dims, u)
        if kind in ("dov", "qx", "batch"):
            s.set_spectrum(LMIN2, LMAX2)
        if kind in ("qx", "batch"):
            s.classes = _class_list(case, s.build_sources(case["r"], case["mode"]))
            s.q = torch.zeros(2, math.prod(dims), dtype=torch.float64, device="cuda")
        else:
            s.psi, s.out = psi, torch.empty_like(psi)
        state["sessions"].append(s)
    return state


def run(state):
    case, ss = state["case"], state["sessions"]
    kind, s = case["kind"], ss[0]
    if kind == "noalloc":
        S.smpq_dslash_noalloc(s.ctx, s.psi, s.out, case["B"], case["dagger"], PRECISION[case["precision"]])
        return s.out
    if kind == "dslash":
        S.smpq_dslash(s.ctx, s.psi, s.out, case["B"], case["dagger"], PRECISION[case["precision"]])
        return s.out
    if kind == "dov":
        S.smpq_apply_dov(s.ctx, s.psi, s.out, case["B"])
        return s.out
    if kind == "batch":
        total, _ = S.smpq_compute_qx_batch([x.ctx for x in ss], [x.q[0] for x in ss], [x.q[1] for x in ss])
        return dict(q=[x.q for x in ss], Q=total)
    if case["classes"]:
        total = S.smpq_compute_qx_classes(s.ctx, s.classes, s.q[0], s.q[1])["Q"]
    else:
        total, _ = S.smpq_compute_qx(s.ctx, s.q[0], s.q[1])
    return dict(q=s.q, Q=total)


def work(case):
    """Links and vectors once in and out; two applications of D_W (1368 flops a site and vector) per CG iteration."""
    by = {"fp64": 16, "mixed": 16, "fp32": 8, "fp16n": 4, "bf16n": 4}[case.get("precision", "fp64")]
    total = dict(bytes=0.0, flops=0.0)
    for dims in _dims(case):
        v, kind = math.prod(dims), case["kind"]
        total["bytes"] += v * 36 * by
        if kind in ("noalloc", "dslash", "dov"):
            b = case["B"]
            total["bytes"] += 2 * v * 12 * b * 16  # the caller's vectors are FP64
            total["flops"] += v * b * 1368.0 * (2 * ITERATIONS + 1 if kind == "dov" else 1)
        else:
            n = case["r"] ** 4 // (2 if case["mode"] == 2 else 1)
            total["bytes"] += 2 * v * 8
            total["flops"] += v * 12 * (case.get("classes", 0) or n) * 1368.0 * 2 * ITERATIONS
    return total


# ----------------------------------------------------------------------------- the same in 64 bits, in plain torch


def _dw(u, psi, dims, bc, dagger=False):
    """D_W psi (D_W^dag psi) on psi[V, 4, 3, B]; chiral basis, gamma_mu = [[0, S], [S^dag, 0]]."""
    nx, ny, nz, nt = dims
    v, b = psi.shape[0], psi.shape[-1]
    f = psi.reshape(nt, nz, ny, nx, 4, 3, b)
    hop = torch.zeros_like(psi)

    def shift(w, mu, step):
        axis = 3 - mu
        w = torch.roll(w.reshape((nt, nz, ny, nx) + w.shape[1:]), -step, axis)
        if bc[mu] < 0:
            w.select(axis, dims[mu] - 1 if step > 0 else 0).neg_()
        return w.reshape((v,) + w.shape[4:])

    def s_mu(mu, lo):  # S_mu on (l0, l1)
        a, c = lo[:, 0], lo[:, 1]
        return torch.stack([(-1j * c, -1j * a), (-c, a), (-1j * a, 1j * c), (a, c)][mu], dim=1)

    def s_dag(mu, up):
        a, c = up[:, 0], up[:, 1]
        return torch.stack([(1j * c, 1j * a), (c, -a), (1j * a, -1j * c), (a, c)][mu], dim=1)

    def colour(m, h):
        return sum(m[:, None, :, q, None] * h[:, :, q, None, :] for q in range(3))

    psi = f.reshape(v, 4, 3, b)
    for mu in range(4):
        for step in (1, -1):
            sign = (-1 if step > 0 else 1) * (-1 if dagger else 1)  # (1 - gamma) forward, (1 + gamma) backward
            h = psi[:, :2] + sign * s_mu(mu, psi[:, 2:])
            if step > 0:
                w = colour(u[:, mu], shift(h, mu, 1))
            else:
                w = shift(colour(u[:, mu].conj().transpose(1, 2), h), mu, -1)
            hop[:, :2] += w
            hop[:, 2:] += sign * s_dag(mu, w)
    return psi - KAPPA * hop


def _zolotarev(n, a, b):
    """c0, c, q of the rational approximation of 1/sqrt(x) on [a, b] (Zolotarev; elliptic functions by the AGM)."""
    m = 1 - a / b
    an, bn, cs = [1.0], [math.sqrt(1 - m)], [math.sqrt(m)]
    while abs(cs[-1]) > 1e-17:
        x, y = an[-1], bn[-1]
        an.append((x + y) / 2)
        bn.append(math.sqrt(x * y))
        cs.append((x - y) / 2)
        if len(an) > 40:
            break
    big = math.pi / (2 * an[-1])
    e = []
    for j in range(1, 2 * n + 1):
        phi = 2.0 ** (len(an) - 1) * an[-1] * j * big / (2 * n + 1)
        for q in range(len(an) - 1, 0, -1):
            phi = (phi + math.asin(cs[q] * math.sin(phi) / an[q])) / 2
        e.append(math.tan(phi) ** 2)
    poles, zeros = np.array(e[0::2]), np.array(e[1::2])

    def ends(y):
        return math.sqrt(y) * np.prod((y + zeros) / (y + poles))

    d0 = 2 / (ends(1.0) + ends(b / a))
    res = [d0 * np.prod(zeros - poles[i]) / np.prod(np.delete(poles, i) - poles[i]) for i in range(n)]
    return d0 / math.sqrt(a), np.array(res) * math.sqrt(a), poles * a


def _shifted_sum(u, b, dims, bc, shifts, weights, tol=1e-14):
    """sum_i w_i (D_W^dag D_W + s_i)^-1 b by multi-shift CG, every shift to `tol`."""
    base = min(shifts)
    sig = [x - base for x in shifts]
    dot = lambda x: (x.real.square() + x.imag.square()).sum((0, 1, 2))  # noqa: E731
    y, r, p = torch.zeros_like(b), b.clone(), b.clone()
    ps = [b.clone() for _ in shifts]
    live = [True] * len(shifts)
    rr = dot(r)
    bb = rr.clone()
    one = torch.ones_like(rr)
    z, zp = [one.clone() for _ in shifts], [one.clone() for _ in shifts]
    ap, bp = one.clone(), torch.zeros_like(rr)
    for _ in range(1500):
        t = _dw(u, p, dims, bc)
        pap = dot(t) + base * dot(p)
        a = torch.where(pap > 0, rr / pap, 0.0)
        r = r - a * (_dw(u, t, dims, bc, True) + base * p)
        new = dot(r)
        beta = torch.where(rr > 0, new / rr, 0.0)
        for i, s in enumerate(sig):
            if not live[i]:
                continue
            den = a * bp * (zp[i] - z[i]) + zp[i] * ap * (1 + s * a)
            zn = torch.where(den != 0, z[i] * zp[i] * ap / den, 0.0)
            ratio = torch.where(z[i] != 0, zn / z[i], 0.0)
            y += weights[i] * (a * ratio) * ps[i]
            ps[i].mul_(beta * ratio * ratio).addcmul_(r, zn.to(r.dtype).expand_as(r))
            zp[i], z[i] = z[i], zn
            live[i] = bool((zn * zn * new > tol * tol * bb).any())
        if not any(live):
            break
        p = r + beta * p
        ap, bp, rr = a, beta, new
    return y


def _colours(dims, r, mode):
    """Colour of every site: Normal (0) or Combine (2)."""
    x = [c % r for c in _coords(dims)]
    if mode == 0:
        return x[0] + r * (x[1] + r * (x[2] + r * x[3]))
    h = r // 2
    e, d = [c % h for c in x], [c // h for c in x]
    d = [torch.where(d[0] == 1, 1 - c, c) for c in d]
    return 8 * (e[0] + h * (e[1] + h * (e[2] + h * e[3]))) + d[1] + 2 * d[2] + 4 * d[3]


def exact(case, seed):
    kind = case["kind"]
    volume = sum(math.prod(d) for d in _dims(case))
    c0, c, q = _zolotarev(NPOLES, LMIN2, LMAX2)
    bc = _bc(case)
    if kind in ("noalloc", "dslash"):
        dims, u, psi = _inputs(case, seed)[0]
        return torch.cat([_dw(u, x, dims, bc, case["dagger"]) for x in psi.split(16, dim=-1)], dim=-1)
    if kind == "dov":
        dims, u, psi = _inputs(case, seed)[0]
        return psi + _dw(u, c0 * psi + _shifted_sum(u, psi, dims, bc, list(q), list(c)), dims, bc)
    n = case["r"] ** 4 // (2 if case["mode"] == 2 else 1)
    if 12 * (case.get("classes", 0) or n) * volume > 3000000:
        return None
    qs, totals = [], []
    for dims, u, _ in _inputs(case, seed):
        v = math.prod(dims)
        colour = _colours(dims, case["r"], case["mode"])
        got = torch.zeros(v, dtype=torch.complex128, device="cuda")
        todo = _class_list(case, n)
        for cl in [todo[i:i + max(1, 50000 // v)] for i in range(0, len(todo), max(1, 50000 // v))]:
            b = torch.zeros(v, 4, 3, 12 * len(cl), dtype=torch.complex128, device="cuda")
            for m, x in enumerate(cl):
                for comp in range(12):
                    b[colour == x, comp // 3, comp % 3, 12 * m + comp] = 1
            w = _dw(u, c0 * b + _shifted_sum(u, b, dims, bc, list(q), list(c)), dims, bc)
            for m, x in enumerate(cl):
                for comp in range(12):
                    here = colour == x
                    got[here] += (0.5 if comp < 6 else -0.5) * w[here, comp // 3, comp % 3, 12 * m + comp]
        qs.append(torch.stack([got.real, got.imag]).contiguous())
        totals.append(float(got.real.sum()))
    return dict(q=qs, Q=totals) if kind == "batch" else dict(q=qs[0], Q=totals[0])
