"""The two-pass Gram-Schmidt of an FP32 Arnoldi column (one pass of dots and a triangular solve,
one update pass), taken by problem sets of more chunks than one co-resident grid holds (here
many shots of a small model), where it can go wrong: one chunk a vector and a ragged last chunk,
more than 32 basis vectors (two rows a lane in the solve), reduction batches that do not come
out even, a window, 3D, a tail that ends the Krylov space early and a non-finite state.

The bound: the error against the oracle (FP64, modified Gram-Schmidt) is at most the acceptance
tolerance of an FP32 step, or four times the error that the library's modified Gram-Schmidt
(the column kernel, which one shot of the same model takes) makes on the same state.  The
exponential of a small or windowed Hessenberg matrix of norm h carries FP32 rounding as h eps
exp-conditioned noise, above the plain tolerance for both; four times covers the spread of two
independent roundings."""
import numpy as np
import pytest

from _helpers import TOL, flatten, gpu_model, oracle_model, rel_l2
from oracle.krylov import krylov_step
from oracle.model import unflatten
from oracle.source import PointSource
from paper_2401_16322_gb300.workloads import layered, smooth_random_state

pytestmark = pytest.mark.gpu


CHUNK = 8192                  # elements of a problem's padded vector per block


def _shots(nx, ny):
    """Enough shots for 1000 chunks (a co-resident grid holds at most 912)."""
    pitch = (nx + 31) // 32 * 32
    return -(-1000 // -(-4 * ny * pitch // CHUNK))


@pytest.mark.parametrize("nx,ny,m,window", [
    (20, 9, 1, 0), (20, 9, 2, 0), (33, 17, 5, 0), (64, 32, 12, 0), (97, 41, 34, 0), (150, 70, 48, 0), (97, 41, 20, 1),
    (97, 41, 21, 3), (137, 53, 44, 37)])
def test_fp32_krylov_step_matches_the_oracle(nx, ny, m, window):
    om = oracle_model(nx, ny, layered(nx, ny, 4), pml=3, fs=True)
    nshots = _shots(nx, ny)
    g = gpu_model(om, "f32", nshots=nshots, p=10, max_receivers=1)
    pick = [0, 1, nshots // 2, nshots - 1]
    dt, t0 = 1e-3, 0.03
    base = flatten(smooth_random_state([f.shape for f in om.zeros_state()], 50))
    states = {}
    for s in range(nshots):
        g.set_source_receivers(s, (5 + s % 7) * om.dx, 2 * om.dx, 25.0, 0.05, 1e3)
        states[s] = base if s not in pick else flatten(
            smooth_random_state([f.shape for f in om.zeros_state()], 51 + s))
        g.set_state(s, states[s])
    if window:
        g.set_krylov_window(window)
    assert g.step_krylov(t0, dt, m, 1) <= m
    one = gpu_model(om, "f32", p=10, max_receivers=1)
    if window:
        one.set_krylov_window(window)
    for s in pick:
        src = PointSource(om, (5 + s % 7) * om.dx, 2 * om.dx, 25.0, 0.05, amp=1e3, p=10)
        U = krylov_step(om, unflatten(om, states[s]), src, t0, dt, m, window=window or None)
        one.set_source_receivers(0, (5 + s % 7) * om.dx, 2 * om.dx, 25.0, 0.05, 1e3)
        one.set_state(0, states[s])
        one.step_krylov(t0, dt, m, 1)
        bound = max(TOL["f32"], 4 * rel_l2(one.get_state(0), flatten(U)))
        assert rel_l2(g.get_state(s), flatten(U)) < bound, (s, rel_l2(g.get_state(s), flatten(U)), bound)
    one.close()
    g.close()


def test_3d_krylov_step_matches_the_oracle():
    from oracle.model import default_beta0
    from oracle.wave3d_pml import Model3DPML
    from paper_2401_16322_gb300 import Model
    from paper_2401_16322_gb300.workloads import layered3d
    n, nshots = 12, 1000
    c = layered3d(n, n, n, 3)
    om = Model3DPML(n, n, n, 10.0, 8, 3, default_beta0(float(c.max()), 3, 10.0), True, c)
    g = Model(n, n, 10.0, 8, 3, om.beta0, True, precision="f32", nshots=nshots, nz=n)
    g.set_velocity(c)
    U0 = flatten(smooth_random_state([f.shape for f in om.zeros_state()], 7))
    for s in range(nshots):
        g.set_state(s, U0 * (1.0 + s))
    g.step_krylov(0.0, 1e-3, 10, 1)
    U = krylov_step(om, unflatten(om, U0), None, 0.0, 1e-3, 10)
    one = Model(n, n, 10.0, 8, 3, om.beta0, True, precision="f32", nz=n)
    one.set_velocity(c)
    for s in (0, 500, nshots - 1):
        one.set_state(0, U0 * (1.0 + s))
        one.step_krylov(0.0, 1e-3, 10, 1)
        bound = max(TOL["f32"], 4 * rel_l2(one.get_state(0) / (1.0 + s), flatten(U)))
        assert rel_l2(g.get_state(s) / (1.0 + s), flatten(U)) < bound
    one.close()
    g.close()


def test_zero_state_and_a_non_finite_state_beside_it():
    """From U = 0 with a silent source the Krylov space is the tail's (4 entries) and the state
    stays zero; a shot with an infinity is reported."""
    from paper_2401_16322_gb300.ewave import EwaveError
    om = oracle_model(40, 20, layered(40, 20, 4), pml=3, fs=True)
    g = gpu_model(om, "f32", nshots=_shots(40, 20), p=4)
    assert g.step_krylov(0.0, 1e-3, 12, 2) <= 12
    assert not g.state.any()
    x = np.ones(om.n)
    x[7] = np.inf
    g.set_state(3, x)
    with pytest.raises(EwaveError, match="NONFINITE"):
        g.step_krylov(0.0, 1e-3, 6, 1)
    g.close()
