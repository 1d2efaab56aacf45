"""Performance cases: the work a user of the library has it do, through ``Model``, ``Batch`` and
``FaberFWI``, with the sizes of the workloads in ``paper_2401_16322_gb300/workloads.py`` and
generic ragged ones.

``listed`` names the cases, ``draw`` makes further ones of the same ranges, ``prepare`` builds
what a user's program holds before the call (models, initial wavefields, vectors), ``run`` makes
one pass and returns its outputs, ``work`` counts what a pass cannot do without, and ``exact``
gives the same outputs in FP64 from plain torch operations that share nothing with the library.

Kinds: "apply" (H x and H^T x on device vectors), "step" (time steps of one 2D or 3D model from a
given wavefield, or of a batch of models of uneven sizes) and "fwi" (seismograms and the gradient
with respect to c^2).  A time step is ``k`` leap-frog stability steps.
"""
import math
from fractions import Fraction

import numpy as np
import torch
import torch.nn.functional as F

from paper_2401_16322_gb300.ewave import (LEAPFROG_AVERAGED, LEAPFROG_DIFFERENCE, Batch, Model)
from paper_2401_16322_gb300.fwi import FaberFWI

DX = 10.0
C_MIN, C_MAX = 1500.0, 4500.0
F_PEAK, T0, AMP = 10.0, 0.27, 1e5
TAYLOR_P = 12
T_START = 0.22            # the source is near its peak in the first steps of a pass
REC_EVERY = 4             # receivers on every 4th column of the top row


# ---------------------------------------------------------------- the cases
def _case(name, kind, **kw):
    c = {"name": name, "kind": kind, "dims": 2, "nx": 101, "ny": 101, "nz": 1, "shots": 1, "small": 0,
         "order": 8, "pml": 40, "free_surface": True, "precision": "f32", "method": "hork-horner", "m": 0,
         "k": 1.0, "steps": 1, "dense": False}
    c.update(kw)
    return c


def listed():
    return [
        # a user's own iterative solver: one product each with H and H^T on device vectors
        _case("apply-2d-f32", "apply", nx=601, ny=301, method="apply"),
        # the paper's small test case: 101 x 101, 4th order, no free surface, FP64; latency counts
        _case("hork12-2d-o4-f64-small", "step", order=4, pml=20, free_surface=False, precision="f64", method="hork",
              m=12, k=2.0, steps=4),
        # one shot of the layered 601 x 301 model: every vector fits the L2 cache
        _case("horner20-2d-f32-single", "step", nx=601, ny=301, m=20, k=4.0, steps=4),
        # FP64 reference seismograms of the same model (every error measure starts from them)
        _case("faber60-2d-f64-single", "step", nx=601, ny=301, precision="f64", method="faber", m=60, k=8.0),
        # the headline: 64 shots on 1001 x 501 and eight smaller models in the same launches
        _case("horner20-2d-f32-batch", "step", nx=1001, ny=501, shots=64, small=8, m=20, k=4.0),
        # the library's default evaluation of HORK, with an accumulator; ragged sizes
        _case("hork20-2d-f32-shots", "step", nx=803, ny=397, shots=16, method="hork", m=20, k=4.0),
        # the paper's exponential integrator with the largest steps, many shots
        _case("faber80-2d-f32-shots", "step", nx=1001, ny=501, shots=16, method="faber", m=80, k=16.0),
        # Krylov steps on vectors far larger than the L2 cache
        _case("krylov20-2d-f32-shots", "step", nx=1001, ny=501, shots=16, method="krylov", m=20, k=4.0),
        # the low-order baseline in the form that reaches 1e-4 in FP32
        _case("leapfrog-2d-f32-shots", "step", nx=1001, ny=501, shots=16, method="leapfrog-difference", k=0.0625,
              steps=16),
        # inversion: seismograms and gradient of 16 shots, exact discrete adjoint
        _case("fwi-horner20-2d-f32", "fwi", nx=401, ny=201, shots=16, m=20, k=4.0, steps=8),
        # inversion with Krylov steps and the adjoint of their exponential from dense states
        _case("fwi-krylov20-2d-f32", "fwi", nx=401, ny=201, shots=16, method="krylov", m=20, k=8.0, steps=4,
              dense=True),
        # three dimensions: large Faber steps on a ragged box
        _case("faber40-3d-f32", "step", dims=3, nx=251, ny=229, nz=197, pml=30, method="faber", m=40, k=8.0),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: kind, method, precision, grid, shots, layer and step drawn over the ranges
    of the listed ones, no dearer than the dearest of them."""
    most = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["apply", "step", "step", "step", "step3", "step3", "batch", "fwi"])
        prec = "f64" if kind in ("apply", "step") and rng.random() < 0.25 else "f32"
        order = 4 if kind in ("apply", "step") and rng.random() < 0.2 else 8
        fs = order == 8 and rng.random() < 0.75
        c = _case("", "step" if kind in ("step3", "batch") else kind, order=order, free_surface=fs, precision=prec,
                  pml=rng.choice([10, 20, 30, 40]))
        del c["name"]
        c["nx"], c["ny"] = _size(rng, 101, 1201), _size(rng, 91, 601)
        if kind == "apply":
            c["method"] = "apply"
        elif kind == "step3":
            c.update(dims=3, nx=_size(rng, 90, 260), ny=_size(rng, 90, 260), nz=_size(rng, 90, 260), pml=30)
            c["method"], c["m"], c["k"] = rng.choice([("faber", 20, 3.0), ("faber", 60, 12.0), ("hork-horner", 12, 2.0),
                                                      ("hork", 16, 2.0), ("leapfrog", 0, 0.5)])
            c["steps"] = 8 if c["method"] == "leapfrog" else 1
        else:
            c["shots"] = _size(rng, 1, 20)
            pick = [("hork-horner", 20, 4.0), ("hork-horner", 12, 2.0), ("hork", 20, 4.0), ("hork", 16, 3.0),
                    ("faber", 30, 5.0), ("faber", 60, 11.0), ("krylov", 20, 4.0), ("krylov", 10, 2.0)]
            if kind == "step":
                pick += [("leapfrog-difference", 0, 0.0625), ("leapfrog", 0, 0.25)]
            if kind == "fwi":
                c["nx"], c["ny"] = _size(rng, 151, 501), _size(rng, 121, 251)
                pick = [("hork-horner", 20, 4.0), ("hork", 12, 2.0), ("faber", 40, 7.0), ("krylov", 20, 8.0)]
            c["method"], c["m"], c["k"] = rng.choice(pick)
            c["steps"] = rng.choice([8, 16]) if c["method"].startswith("leapfrog") else rng.choice([1, 2, 3])
            if kind == "batch":
                c.update(small=rng.randint(2, 8), steps=1)
            if kind == "fwi":
                c.update(steps=rng.randint(3, 6), dense=c["method"] == "krylov", pml=min(c["pml"], 30))
        c["pml"] = min(c["pml"], min(c["nx"], c["ny"]) // 3)
        if _cost(c) <= 0.7 * most:
            return c


# ---------------------------------------------------------------- sizes and counts
def _grids(c):
    """(nx, ny, nz, shots) of every model of the case: the main one, then the smaller ones with
    one shot each, from a fifth to four fifths of its size."""
    out = [(c["nx"], c["ny"], c["nz"], c["shots"])]
    for q in range(c["small"]):
        s = 0.2 + 0.6 * q / max(1, c["small"] - 1)
        out.append((int(round(s * c["nx"])), int(round(s * c["ny"])), 1, 1))
    return out


def _points(c):
    return sum(nx * ny * nz * ns for nx, ny, nz, ns in _grids(c))


def work(case):
    """Words per grid point of one pass over the grid, every operand read once and every result
    written once; a product with H has to read its whole operand before the next one starts, so
    the products of a step are counted one by one.  F fields a vector, one word of c^2."""
    nf = 4 if case["dims"] == 2 else 6
    m, meth = case["m"], case["method"]
    word = 8 if case["precision"] == "f64" else 4
    prod = 2 * nf + 1                                    # y = H x
    flop = (90 if case["order"] == 8 else 55) if case["dims"] == 2 else 140
    if case["kind"] == "apply":
        words, flops = 2 * prod, 2 * flop
    elif meth == "hork-horner":                          # V_j = V_0 + (dt/j) H V_{j+1}
        words, flops = m * (prod + nf), m * (flop + 2 * nf)
    elif meth == "hork":                                 # k_i and the accumulator
        words, flops = m * (prod + 2 * nf), m * (flop + 4 * nf)
    elif meth == "faber":                                # p_j, p_{j-2} and the accumulator
        words, flops = m * (prod + 3 * nf), m * (flop + 6 * nf)
    elif meth == "krylov":                               # products, basis reads, combination
        words = m * prod + nf * m * (m + 1) // 2 + nf * (m + 1)
        flops = m * flop + 4 * nf * m * (m + 1) // 2 + 2 * nf * m
    else:                                                # leap-frog
        words = {"leapfrog-difference": 11}.get(meth, 10) if case["dims"] == 2 else 15
        flops = flop
    if case["kind"] == "fwi":
        # the forward step and its stored states, then H^T products and gradient terms
        if meth == "krylov":
            words = 2 * words + 8 * nf + 4 * (nf + 3)
            flops = 2 * flops + 4 * 40
        else:
            words = words + 2 * nf + m * prod + m * (prod + nf) + m * (nf + 3)
            flops = 3 * flops + m * 40
    n = _points(case) * case["steps"]
    return {"bytes": float(n * words * word), "flops": float(n * flops)}


def _cost(c):
    """What bounds a drawn case: bytes at FP32 bandwidth, FP64 arithmetic at its own low rate."""
    w = work(c)
    return max(w["bytes"], w["flops"] * (20.0 if c["precision"] == "f64" else 0.3))


def _dt(c):
    s2 = {8: 6.501587301587302, 4: 16.0 / 3.0}[c["order"]]   # |minimum symbol| of the second derivative
    return c["k"] * 2.0 * DX / (C_MAX * math.sqrt(c["dims"] * s2))


def _beta0(c):
    return 3.0 * C_MAX / (2.0 * c["pml"] * DX) * math.log(1e3)


# ---------------------------------------------------------------- inputs
_DEV = "cuda" if torch.cuda.is_available() else "cpu"


def _smooth(gen, lead, shape, cells, mode):
    """Smooth random fields [*lead, *shape] of unit size: coarse normal values, interpolated."""
    coarse = [max(4, s // cells + 2) for s in shape]
    n = int(np.prod(lead))
    a = torch.randn(n, 1, *coarse, generator=gen, dtype=torch.float32).to(_DEV)
    return F.interpolate(a, size=list(shape), mode=mode, align_corners=True).view(*lead, *shape)


def _inputs(c, seed):
    """Per model: c^2 [(nz,) ny, nx] (FP64, values exact in FP32), and wavefield
    [shots, fields, (nz,) ny, nx] with values exact in FP32 and zeros in the padding entries."""
    gen = torch.Generator().manual_seed(1000003 * int(seed) + 17)
    mode = "bicubic" if c["dims"] == 2 else "trilinear"
    nf = 4 if c["dims"] == 2 else 6
    out = []
    for nx, ny, nz, ns in _grids(c):
        shape = (ny, nx) if c["dims"] == 2 else (nz, ny, nx)
        # layers of rising velocity with sharp interfaces and a smooth perturbation
        depths = torch.sort(torch.rand(8, generator=gen) * shape[0])[0]
        base = torch.linspace(C_MIN, C_MAX, 9) * (1.0 + 0.05 * (2.0 * torch.rand(9, generator=gen) - 1.0))
        layer = torch.searchsorted(depths, torch.arange(shape[0]) + 0.5)
        vel = base[layer].to(_DEV).view(-1, *([1] * (len(shape) - 1)))
        vel = (vel * (1.0 + 0.05 * _smooth(gen, (1,), shape, 16, mode)[0])).clamp(C_MIN, C_MAX)
        vel.view(-1)[-1] = C_MAX                        # the Faber ellipse follows the largest velocity
        c2 = vel.square().float().double()
        u = None
        if c["kind"] != "fwi":                          # an inversion starts from rest
            u = _smooth(gen, (ns, nf), shape, 8, mode)
            # sizes of a 10 Hz field of unit amplitude: v ~ omega u, w ~ d_x u, psi ~ u / omega
            for f, s in enumerate([1.0, 60.0, 0.02, 0.02] if nf == 4 else [1.0, 60.0, 0.02, 0.02, 0.02, 0.016]):
                u[:, f] *= s
            for a in range(c["dims"]):                  # w_x has no last column, w_y no last row, ...
                u[:, 2 + a].select(-1 - a, -1).zero_()
        out.append((c2, u))
    return out


def _sources(nx, shots):
    """Source columns, evenly along the line."""
    return [int(round(v)) for v in np.linspace(0.2 * nx, 0.8 * nx, shots)] if shots > 1 else [nx // 2]


def _src_row(c):
    """Two rows below a free surface, else the middle of the grid."""
    rows = c["ny"] if c["dims"] == 2 else c["nz"]
    return 2 if c["free_surface"] else rows // 2


def _rec_cols(nx):
    return list(range(0, nx, REC_EVERY))


def _fields(md):
    """The padded state [shots, fields, (nz,) ny, pitch] as a view."""
    shape = (md.ny, md.layout.pitch) if md.dims == 2 else (md.nz, md.ny, md.layout.pitch)
    return md.state.view(md.nshots, 4 if md.dims == 2 else 6, *shape)


def _model(c, grid, c2, u, capacity):
    nx, ny, nz, ns = grid
    cols = _rec_cols(nx)
    md = Model(nx, ny, DX, c["order"], c["pml"], _beta0(c), c["free_surface"], precision=c["precision"],
               nshots=ns, p=TAYLOR_P, max_receivers=len(cols), nz=nz if c["dims"] == 3 else None)
    md.set_velocity(c2.sqrt().cpu().numpy())
    row = min(_src_row(c), (ny if c["dims"] == 2 else nz) - 1)
    for s, i in enumerate(_sources(nx, ns)):
        if c["dims"] == 2:
            md.set_source_receivers(s, i * DX, row * DX, F_PEAK, T0, AMP, np.array([[r * DX, 0.0] for r in cols]))
        else:
            mid = (ny // 2) * DX
            md.set_source_receivers3d(s, i * DX, mid, row * DX, F_PEAK, T0, AMP,
                                      np.array([[r * DX, mid, 0.0] for r in cols]))
    md.bind_seismogram(capacity)
    if c["method"] == "hork-horner":
        md.set_hork_form("horner")
    if u is not None:
        _fields(md)[..., :nx].copy_(u)
    return md


def prepare(case, seed):
    c = case
    models = [_model(c, g, c2, u, c["steps"]) for g, (c2, u) in zip(_grids(c), _inputs(c, seed))]
    st = {"case": c, "models": models, "t": T_START, "dt": _dt(c)}
    md = models[0]
    if c["kind"] == "apply":
        st["x"] = md.state.clone()
        st["y"], st["z"] = md.new_vector(), md.new_vector()
    elif c["kind"] == "fwi":
        if c["method"] == "krylov":
            md.set_krylov_adjoint("exponential")
        st["fwi"] = FaberFWI(md, st["dt"], c["m"], c["steps"], len(_rec_cols(c["nx"])), t0=T_START,
                             method="hork" if c["method"] == "hork-horner" else c["method"],
                             dense_states=c["dense"])
        st["c2"] = _inputs(c, seed)[0][0]
        st["data"] = _observed(c, seed)
    elif len(models) > 1:
        st["batch"] = Batch(models)
    return st


def _observed(c, seed):
    gen = torch.Generator().manual_seed(7919 * int(seed) + 5)
    return 0.1 * torch.randn(c["shots"], c["steps"], len(_rec_cols(c["nx"])), generator=gen).to(_DEV)


# ---------------------------------------------------------------- one pass
def run(state):
    c, models = state["case"], state["models"]
    md, dt = models[0], state["dt"]
    if c["kind"] == "apply":
        md.apply_device(state["x"], state["y"])
        md.apply_device(state["x"], state["z"], transpose=True)
        return {"hx": state["y"], "htx": state["z"]}
    if c["kind"] == "fwi":
        seis = state["fwi"].forward(state["c2"])
        grad = state["fwi"].backward(seis - state["data"])
        return {"seis": seis, "grad": grad}
    # time steps: the wavefield goes on from where the last pass left it
    t, steps = state["t"], c["steps"]
    state["t"] = t + steps * dt
    for x in models:
        x.reset_recording()
    meth = "hork" if c["method"] == "hork-horner" else c["method"]
    if meth.startswith("leapfrog"):
        md.step_leapfrog(t, dt, steps, LEAPFROG_DIFFERENCE if meth == "leapfrog-difference" else LEAPFROG_AVERAGED)
        # v is not a field of the leap-frog scheme
        s = _fields(md)
        return {"seis": md.seismo, "u": s[:, 0], "w": s[:, 2:]}
    if "batch" in state:
        state["batch"].step(meth, t, dt, c["m"], steps)
    else:
        md.step(meth, t, dt, c["m"], steps)
    return {"state": [x.state for x in models], "seis": [x.seismo for x in models]}


# ---------------------------------------------------------------- FP64 values
_STAG = {8: (1225.0 / 1024.0, -245.0 / 3072.0, 49.0 / 5120.0, -5.0 / 7168.0), 4: (9.0 / 8.0, -1.0 / 24.0)}
_CENT = {8: (-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0), 4: (-5.0 / 2.0, 4.0 / 3.0, -1.0 / 12.0)}


def _one_sided(points, at, powers, deriv):
    """Weights on ``points`` whose sum over s^p is the ``deriv``-th derivative of s^p at ``at``
    (rational elimination: the weights are exact before they are rounded)."""
    rows = []
    for p in powers:
        d = 0 if p < deriv else (p if deriv == 1 else p * (p - 1)) * Fraction(at) ** (p - deriv)
        rows.append([Fraction(s) ** p for s in points] + [Fraction(d)])
    n = len(rows)
    for i in range(n):
        piv = next(r for r in range(i, n) if rows[r][i] != 0)
        rows[i], rows[piv] = rows[piv], rows[i]
        rows[i] = [v / rows[i][i] for v in rows[i]]
        for r in range(n):
            if r != i and rows[r][i] != 0:
                rows[r] = [v - rows[r][i] * q for v, q in zip(rows[r], rows[i])]
    return [float(r[-1]) for r in rows]


def _surface_rows():
    """Free-surface rows by depth (s = -y in cells): u_yy at nodes 0..3 and u_y at half rows
    0..2, exact for the powers without a slope at the surface; d_y w_y at nodes 0..3 from w_y(0) = 0
    and the eight nearest half rows.  y points up, so first derivatives change sign."""
    uyy = [_one_sided(range(9), j, [0, 2, 3, 4, 5, 6, 7, 8, 9], 2) for j in range(4)]
    uy = [[-w for w in _one_sided(range(8), j + 0.5, [0, 2, 3, 4, 5, 6, 7, 8], 1)] for j in range(3)]
    half = [0.0] + [q + 0.5 for q in range(8)]
    dwy = [[-w for w in _one_sided(half, j, range(9), 1)[1:]] for j in range(4)]
    return uyy, uy, dwy


class _Operator:
    """H of one model in FP64: fields [shots, field, (nz,) ny, nx], padding entries zero."""

    def __init__(self, c, c2, columns=()):
        self.c2, self.dims, self.columns = c2, c["dims"], columns   # columns: the shots' source columns
        self.shape = tuple(c2.shape)
        self.stag, self.cent = _STAG[c["order"]], _CENT[c["order"]]
        self.fs = _surface_rows() if c["free_surface"] else None
        self.node, self.half, self.mask = [], [], []
        for a in range(self.dims):                      # axis a counts from x; the last is vertical
            n = self.shape[-1 - a]
            i = torch.arange(n, dtype=torch.float64, device=c2.device)
            surface = c["free_surface"] and a == self.dims - 1

            def beta(lo, hi):
                d = hi if surface else torch.minimum(lo, hi)
                b = _beta0(c) * (1.0 - d / c["pml"]).square()
                return torch.where(d <= c["pml"], b, torch.zeros_like(b)).view([n] + [1] * a)
            keep = torch.ones(n, dtype=torch.float64, device=c2.device)
            keep[-1] = 0.0
            self.node.append(beta(i + 1.0, n - i))
            self.mask.append(keep.view([n] + [1] * a))
            self.half.append(beta(i + 1.5, n - i - 0.5) * self.mask[-1])

    def _at(self, x, a, off):
        """x shifted by ``off`` along axis a, zero beyond the grid."""
        d, n = x.dim() - 1 - a, x.shape[-1 - a]
        if abs(off) >= n:
            return torch.zeros_like(x)
        pad = [0, 0] * a + ([0, off] if off >= 0 else [-off, 0])
        return F.pad(x.narrow(d, max(0, off), n - abs(off)), pad)

    def _rows(self, x, out, rows):
        """The first rows of ``out`` along the vertical axis replaced by one-sided sums."""
        a = self.dims - 1
        d = x.dim() - 1 - a
        new = [sum(float(w) * x.select(d, q) for q, w in enumerate(r) if q < x.shape[d]) for r in rows]
        return torch.cat([torch.stack(new, d), out.narrow(d, len(rows), out.shape[d] - len(rows))], d)

    def d_half(self, u, a):
        up = a == self.dims - 1
        out = 0
        for k, s in enumerate(self.stag):
            d = self._at(u, a, 1 + k) - self._at(u, a, -k)
            out = out + (-s if up else s) * d
        if up and self.fs:
            out = self._rows(u, out, self.fs[1])
        return out * self.mask[a] / DX

    def d_node(self, w, a):
        up = a == self.dims - 1
        out = 0
        for k, s in enumerate(self.stag):
            d = self._at(w, a, k) - self._at(w, a, -1 - k)
            out = out + (-s if up else s) * d
        if up and self.fs:
            out = self._rows(w, out, self.fs[2])
        return out / DX

    def d_second(self, u, a):
        out = self.cent[0] * u
        for k in range(1, len(self.cent)):
            out = out + self.cent[k] * (self._at(u, a, k) + self._at(u, a, -k))
        if a == self.dims - 1 and self.fs:
            out = self._rows(u, out, self.fs[0])
        return out / (DX * DX)

    def force(self, u, w, psi):
        """The v row without its own damping term, and the gradients' part of the w rows."""
        n, ax = self.node, range(self.dims)
        pair = sum(n[a] * n[b] for a in ax for b in ax if a < b)
        acc = sum(self.d_second(u, a) + self.d_node(w[a], a) for a in ax)
        hv = -pair * u + self.c2 * acc
        if psi is not None:
            hv = hv - n[0] * n[1] * n[2] * psi
        gw = []
        for a in ax:
            others = [n[b] for b in ax if b != a]
            g = (sum(others) - self.half[a]) * self.d_half(u, a)
            if psi is not None:
                g = g + others[0] * others[1] * self.d_half(psi, a)
            gw.append(g)
        return hv, gw

    def __call__(self, x):
        u, v = x[:, 0], x[:, 1]
        w = [x[:, 2 + a] * self.mask[a] for a in range(self.dims)]
        psi = x[:, 5] if self.dims == 3 else None
        hv, gw = self.force(u, w, psi)
        hv = hv - sum(self.node) * v
        rows = [v, hv] + [gw[a] - self.half[a] * w[a] for a in range(self.dims)]
        return torch.stack(rows + ([u] if psi is not None else []), 1)


def _ricker_derivatives(t, count):
    """r and its derivatives at t: r = -g''/(2a), g a Gaussian, g^(k) = -2a tau g^(k-1) - 2a (k-1) g^(k-2)."""
    a, tau = (math.pi * F_PEAK) ** 2, t - T0
    g = [math.exp(-a * tau * tau)]
    for k in range(1, count + 2):
        g.append(-2.0 * a * tau * g[k - 1] - (2.0 * a * (k - 1) * g[k - 2] if k > 1 else 0.0))
    return [-g[k + 2] / (2.0 * a) for k in range(count)]


class _Augmented:
    """dt H~ on (fields, tail): the source enters the v row through W, the tail is shifted."""

    def __init__(self, c, op, grid, t, dt):
        self.op, self.dt = op, dt
        row = min(_src_row(c), op.shape[0] - 1)
        at = [row] if c["dims"] == 2 else [row, grid[1] // 2]
        self.spot = torch.zeros(len(op.columns), *op.shape, dtype=torch.float64, device=op.c2.device)
        for s, i in enumerate(op.columns):
            self.spot[(s, *at, i)] = AMP / (DX * DX)
        r = _ricker_derivatives(t, TAYLOR_P)
        self.W = torch.tensor([dt ** (TAYLOR_P - 1 - q) * r[TAYLOR_P - 1 - q] for q in range(TAYLOR_P)],
                              dtype=torch.float64, device=op.c2.device)
        self.tail = torch.zeros(TAYLOR_P, dtype=torch.float64, device=op.c2.device)
        self.tail[-1] = 1.0

    def __call__(self, x, y):
        hx = self.op(x)
        src = torch.stack([self.spot if f == 1 else torch.zeros_like(self.spot) for f in range(hx.shape[1])], 1)
        return self.dt * (hx + torch.dot(self.W, y) * src), F.pad(y[1:], (0, 1))


def _taylor(A, x, m):
    y, term, out = A.tail, x, x
    for k in range(1, m + 1):
        term, y = A(term, y)
        term, y = term / k, y / k
        out = out + term
    return out


def _faber(c, A, x, dt, m):
    """Faber recurrence on the ellipse through the corners of the rectangle
    [-dims beta0, 0] x [-omega, omega], and the coefficients of exp by the trapezoid rule."""
    th = np.linspace(0.0, math.pi, 20001)
    cent = _CENT[c["order"]]
    s2 = (cent[0] + 2.0 * sum(cent[k] * np.cos(k * th) for k in range(1, len(cent)))).min()
    omega = (1.30 if c["free_surface"] else 1.05) * float(A.op.c2.max().sqrt()) * math.sqrt(c["dims"] * abs(s2)) / DX
    b = c["dims"] * _beta0(c)
    ar, ai = math.sqrt(2.0) * 0.5 * b, math.sqrt(2.0) * omega
    g = 0.5 * (ar + ai)
    c0, c1 = -0.5 * b / g, (ar - ai) / (ar + ai)
    n = max(4 * m, 64)
    w = np.exp(2j * math.pi * np.arange(n) / n)
    f = np.exp(dt * g * (w + c0 + c1 / w))
    a = [float((f * w ** -j).sum().real / n) for j in range(m + 1)]

    def B(x, y):
        hx, hy = A(x, y)
        return hx / (dt * g) - c0 * x, hy / (dt * g) - c0 * y
    p, py = x, A.tail
    q, qy = B(p, py)
    out = a[0] * p + a[1] * q
    for j in range(2, m + 1):
        r, ry = B(q, qy)
        cj = 2.0 * c1 if j == 2 else c1
        r, ry = r - cj * p, ry - cj * py
        out = out + a[j] * r
        p, py, q, qy = q, qy, r, ry
    return out


def _krylov(A, x, m):
    """Arnoldi with modified Gram-Schmidt on [x; eta e_p], eta = |x|, one shot at a time."""
    res, spot = [], A.spot
    for s in range(x.shape[0]):
        A.spot = spot[s:s + 1]
        xs = x[s:s + 1]
        eta = float(xs.norm()) or 1.0
        W, A.W = A.W, A.W / eta
        beta = math.sqrt(float(xs.square().sum()) + eta * eta)
        V, T = [xs / beta], [A.tail * eta / beta]
        H = torch.zeros(m, m, dtype=torch.float64)
        for j in range(m):
            q, y = A(V[j], T[j])
            for k in range(j + 1):
                h = (q * V[k]).sum() + torch.dot(y, T[k])
                H[k, j] = h
                q, y = q - h * V[k], y - h * T[k]
            if j + 1 < m:
                h = torch.sqrt(q.square().sum() + y.square().sum())
                H[j + 1, j] = h
                V.append(q / h)
                T.append(y / h)
        e = torch.matrix_exp(H)[:, 0]
        res.append(sum(beta * float(e[k]) * V[k] for k in range(m)))
        A.W = W
    A.spot = spot
    return torch.cat(res, 0)


def _leapfrog(c, op, grid, x, t, dt, steps):
    """Two-step scheme with time-averaged damping, from x as both levels; psi by the trapezoid rule."""
    ax = range(op.dims)
    u = um = x[:, 0]
    w = wm = [x[:, 2 + a] for a in ax]
    psi = x[:, 5] if op.dims == 3 else None
    b = sum(op.node)
    seis = []
    for n in range(steps):
        A = _Augmented(c, op, grid, t + n * dt, dt)
        hv, gw = op.force(u, w, psi)
        hv = hv + A.W[-1] * A.spot
        un = ((2.0 * u - um) / dt ** 2 + b * um / (2.0 * dt) + hv) / (1.0 / dt ** 2 + b / (2.0 * dt))
        wn = [((1.0 - op.half[a] * dt) * wm[a] + 2.0 * dt * gw[a]) / (1.0 + op.half[a] * dt) for a in ax]
        if psi is not None:
            psi = psi + 0.5 * dt * (u + un)
        u, um, w, wm = un, u, wn, w
        seis.append(_record(c, grid, u))
    return u, w + ([psi] if psi is not None else []), torch.stack(seis, 1)


def _record(c, grid, u):
    cols = torch.tensor(_rec_cols(grid[0]), device=u.device)
    return (u[:, 0] if c["dims"] == 2 else u[:, 0, grid[1] // 2])[:, cols]


def _advance(c, op, grid, x, t, dt, steps):
    """Time steps of a one-step method: the state and the samples [shots, steps, receivers]."""
    seis = []
    for n in range(steps):
        A = _Augmented(c, op, grid, t + n * dt, dt)
        if c["method"] == "faber":
            x = _faber(c, A, x, dt, c["m"])
        elif c["method"] == "krylov":
            x = _krylov(A, x, c["m"])
        else:
            x = _taylor(A, x, c["m"])
        seis.append(_record(c, grid, x[:, 0]))
    return x, torch.stack(seis, 1)


def _padded(c, x):
    """Rows of the library's pitch: a whole number of 128 bytes."""
    per = 32 if c["precision"] == "f32" else 16
    nx = x.shape[-1]
    return F.pad(x, (0, -(-nx // per) * per - nx))


def exact(case, seed):
    c = case
    dt = _dt(c)
    made = _inputs(c, seed)
    grids = _grids(c)
    cols = _sources(c["nx"], c["shots"])
    if c["kind"] == "apply":
        op, x = _Operator(c, made[0][0]), made[0][1].double()
        xg = torch.zeros_like(x, requires_grad=True)
        y = op(x)
        ht, = torch.autograd.grad(op(xg), xg, x)
        return {"hx": _padded(c, y).flatten(), "htx": _padded(c, ht).flatten()}
    if c["kind"] == "fwi":
        c2 = made[0][0].clone().requires_grad_(c["method"] != "krylov")
        x = torch.zeros(c["shots"], 4, *c2.shape, dtype=torch.float64, device=c2.device)
        _, seis = _advance(c, _Operator(c, c2, cols), grids[0], x, T_START, dt, c["steps"])
        if c["method"] == "krylov":
            # its gradient is a quadrature of the exponential's adjoint, not a derivative of the step
            return {"seis": seis, "grad": None}
        res = (seis - _observed(c, seed).double()).detach()
        g, = torch.autograd.grad(seis, c2, res)
        return {"seis": seis.detach(), "grad": g}
    if c["method"].startswith("leapfrog"):
        op = _Operator(c, made[0][0], cols)
        u, w, seis = _leapfrog(c, op, grids[0], made[0][1].double(), T_START, dt, c["steps"])
        return {"seis": seis.flatten(), "u": _padded(c, u), "w": _padded(c, torch.stack(w, 1))}
    out = {"state": [], "seis": []}
    with torch.no_grad():
        for (c2, x), g in zip(made, grids):
            state, seis = [], []
            for s in range(0, g[3], 8):                 # a few shots at a time bounds the memory
                op = _Operator(c, c2, _sources(g[0], g[3])[s:s + 8])
                y, r = _advance(c, op, g, x[s:s + 8].double(), T_START, dt, c["steps"])
                state.append(_padded(c, y).flatten())
                seis.append(r.flatten())
            out["state"].append(torch.cat(state))
            out["seis"].append(torch.cat(seis))
    return out

