"""FP32 sets of more chunks than one co-resident grid holds take their Arnoldi columns in two
passes over the basis; besides the plain Krylov step that serves the exponential adjoint (Arnoldi
on H and, without tails, on H^T; from a checkpoint and from dense states) and the adaptive step.
Against the oracle: the error is at most the acceptance tolerance of such a step, or four times
the error that one shot of the same model makes, which takes modified Gram-Schmidt on the column
kernel or in flat passes (four times covers the spread of two independent roundings)."""
import numpy as np
import pytest

from _helpers import TOL, flatten, gpu_model, oracle_model, rel_l2
from oracle.adjoint import krylov_adjoint_step
from oracle.krylov_adaptive import krylov_adaptive_step
from oracle.model import unflatten
from oracle.source import PointSource
from paper_2401_16322_gb300.workloads import layered, random_state, smooth_random_state

pytestmark = pytest.mark.gpu

NSHOTS = 500                       # 2 chunks of 8192 elements a shot; 912 chunks fit a grid
PICK = (0, 1, 250, NSHOTS - 1)
TOL_ADJ = 3e-5                     # an FP32 adjoint step against the oracle's


def _src(om, s):
    return (20 + s % 30) * om.dx, 2 * om.dx, 30.0, 0.04, 1e3


def _start(om, s):
    return flatten(smooth_random_state([f.shape for f in om.zeros_state()], 50 + s % 97))


@pytest.mark.parametrize("m", [8, 20, 40])
@pytest.mark.parametrize("route", ["checkpoint", "dense states"])
def test_exponential_adjoint_step(route, m):
    import torch
    nx, ny, dt, t = 70, 39, 1.2e-3, 0.02
    om = oracle_model(nx, ny, layered(nx, ny, 12, vmin=1500, vmax=3000), pml=9, fs=True)

    def adjoint(shots):
        g = gpu_model(om, "f32", nshots=len(shots), p=8)
        nv, fe = g.vector_elems, g.layout.field_elems
        lam = torch.zeros(len(shots) * nv, device="cuda")
        grad = torch.zeros(len(shots) * fe, device="cuda")
        for k, s in enumerate(shots):
            g.set_source_receivers(k, *_src(om, s))
            g.set_state(k, _start(om, s))
            g.pack(random_state([(om.n,)], 60 + s % 97)[0], lam[k * nv:(k + 1) * nv])
        ck = g.state.clone()
        g.set_krylov_adjoint("exponential")
        xd = torch.zeros(4 * len(shots) * nv, device="cuda")
        g.step_krylov_dense(t, dt, m, xd)          # (tunes the passes, too)
        if route == "checkpoint":
            g.adjoint_step(t, dt, m, ck, lam, grad, method="krylov")
        else:
            g.adjoint_step_krylov_dense(t, dt, m, xd, lam, grad)
        g.sync()
        out = {s: (g.unpack(lam[k * nv:(k + 1) * nv]),
                   grad[k * fe:(k + 1) * fe].view(ny, g.layout.pitch)[:, :nx].double().cpu().numpy())
               for k, s in enumerate(shots) if s in PICK}
        g.close()
        return out

    many = adjoint(range(NSHOTS))
    for s in PICK:
        src = PointSource(om, *_src(om, s)[:4], amp=1e3, p=8)
        Ub, gr = krylov_adjoint_step(om, _start(om, s), random_state([(om.n,)], 60 + s % 97)[0], src, t, dt, m)
        one = adjoint([s])[s]
        for got, alone, want in zip(many[s], one, (Ub, gr.reshape(ny, nx))):
            bound = max(TOL_ADJ, 4 * rel_l2(alone, want))
            assert rel_l2(got, want) < bound, (s, rel_l2(got, want), bound)


@pytest.mark.parametrize("window", [0, 4])
@pytest.mark.parametrize("dt,m_max", [(2e-3, 30), (6e-3, 10)])
def test_adaptive_step(window, dt, m_max):
    """m_max 10 at 6 ms takes substeps, whose Arnoldi processes start from the tail the last one
    left; a loose tolerance of the step itself (1e-7, relative to the state) is part of the error
    of both."""
    nx, ny, t0, tol = 70, 39, 0.03, 1e-7
    om = oracle_model(nx, ny, layered(nx, ny, 4), pml=6, fs=True)

    def step(shots):
        g = gpu_model(om, "f32", nshots=len(shots), p=8)
        g.set_krylov_window(window)
        for k, s in enumerate(shots):
            g.set_source_receivers(k, *_src(om, s))
            g.set_state(k, _start(om, s))
        st = g.step_krylov_adaptive(t0, dt, tol, 1, m_max, 1)
        g.sync()
        out = {s: g.get_state(k) for k, s in enumerate(shots) if s in PICK}
        g.close()
        return out, st

    many, st = step(range(NSHOTS))
    assert st["max_dim"] <= m_max and (m_max == 30 or st["substeps"] > NSHOTS)
    for s in PICK:
        src = PointSource(om, *_src(om, s)[:4], amp=1e3, p=8)
        ref, _ = krylov_adaptive_step(om, unflatten(om, _start(om, s)), src, t0, dt, tol, 1, m_max, window=window or None)
        one = step([s])[0][s]
        bound = max(TOL["f32"], 4 * rel_l2(one, flatten(ref)))
        assert rel_l2(many[s], flatten(ref)) < bound, (s, rel_l2(many[s], flatten(ref)), bound)
