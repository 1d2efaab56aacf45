"""The one-thread-per-point passes (FP64, and H x on a caller's vectors in both precisions) at
the sizes where their blocks (32 x 4 points cut out of 64 x 16 tiles), their edge taps and their
free-surface rows can go wrong: grids narrower than a block, one point past a block or a tile,
lower than the stencil, and layers that meet in the middle.  Against the oracle's assembled
operator and its integrators, with the acceptance tolerances."""
import numpy as np
import pytest

from _helpers import TOL, flatten, gpu_model, oracle_ellipse, oracle_model, rel_l2
from oracle.model import unflatten
from oracle.operator import assemble_H
from oracle.simulate import run
from oracle.source import PointSource
from paper_2401_16322_gb300.workloads import layered, smooth_random_state

pytestmark = pytest.mark.gpu

# (nx, ny, order, free surface, layer width)
GRIDS = [(7, 5, 8, False, 2), (9, 12, 8, True, 3), (31, 9, 8, True, 4), (32, 16, 8, False, 8), (33, 17, 8, True, 20),
         (64, 4, 4, False, 2), (65, 33, 4, False, 5), (97, 20, 8, True, 1), (130, 35, 8, True, 0)]


def _model(nx, ny, order, fs, pml, seed):
    return oracle_model(nx, ny, layered(nx, ny, seed), order=order, pml=pml, fs=fs)


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("grid", GRIDS)
def test_operator_and_transpose_on_caller_vectors(grid, prec):
    om = _model(*grid, seed=3)
    g = gpu_model(om, prec)
    x = flatten(smooth_random_state([f.shape for f in om.zeros_state()], 11, sigma_cells=1.0))
    H = assemble_H(om)
    for transpose, ref in ((False, H @ x), (True, H.T @ x)):
        got = g.apply(x, transpose)
        assert rel_l2(got, ref) < TOL[prec], (transpose, rel_l2(got, ref))
    g.close()


def test_operator_on_another_stream_is_complete_on_return():
    """A model bound to a stream of its own: the caller may read y on the current stream."""
    import torch
    from paper_2401_16322_gb300 import Model
    om = _model(97, 65, 8, True, 10, seed=3)
    g = Model(om.nx, om.ny, om.dx, om.order, om.pml, om.beta0, True, precision="f64", stream=torch.cuda.Stream())
    g.set_velocity(om.c)
    x = flatten(smooth_random_state([f.shape for f in om.zeros_state()], 11))
    dx, dy = g.new_vector(), g.new_vector()
    g.pack(x, dx)
    torch.cuda.synchronize()
    g.apply_device(dx, dy)
    y = dy.clone()
    assert rel_l2(g.unpack(y), assemble_H(om) @ x) < TOL["f64"]
    g.close()


@pytest.mark.parametrize("method,m", [("faber", 1), ("faber", 9), ("hork", 5), ("hork-horner", 5), ("rk44", 0),
                                      ("krylov", 6), ("leapfrog", 0)])
@pytest.mark.parametrize("grid", [GRIDS[1], GRIDS[4], GRIDS[6], GRIDS[8]])
def test_fp64_steps(grid, method, m):
    om = _model(*grid, seed=5)
    g = gpu_model(om, "f64", p=8, max_receivers=2)
    rec = np.array([[0.0, 0.0], [(om.nx - 1) * om.dx, 0.0]])
    sx, sy = (om.nx // 2) * om.dx, min(2, om.ny - 1) * om.dx
    g.set_source_receivers(0, sx, sy, 20.0, 0.05, 1e3, rec)
    g.set_faber_ellipse(*oracle_ellipse(om))
    g.bind_seismogram(3)
    U0 = flatten(smooth_random_state([f.shape for f in om.zeros_state()], 13))
    g.set_state(0, U0)
    name = "hork" if method == "hork-horner" else method
    if method == "hork-horner":
        g.set_hork_form("horner")
    dt = 5e-4
    g.step(name, 0.03, dt, m, 3)
    src = PointSource(om, sx, sy, 20.0, 0.05, amp=1e3, p=8)
    U, _ = run(om, name, dt, 3, src=src, m=m, U0=unflatten(om, U0), t0=0.03)
    got, ref = unflatten(om, g.get_state(0)), U
    for f in range(4):
        if not (name == "leapfrog" and f == 1):       # v is not a field of the leap-frog scheme
            assert rel_l2(got[f], ref[f]) < 3 * TOL["f64"], (f, rel_l2(got[f], ref[f]))
    g.close()
