"""Every shape that a 2D FP32 pass may run on does the same arithmetic per point: the variants that
choose a shape by the pass's operands (U and A, A alone, U alone, neither) give the bits of one
that runs every pass on the same tiles.  Grids just past a tile edge and ragged, both orders, with
and without the free surface."""
import numpy as np
import pytest

from _helpers import flatten, gpu_model, oracle_ellipse, oracle_model
from paper_2401_16322_gb300.workloads import layered, smooth_random_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,order,fs", [(65, 31, 8, True), (130, 61, 8, False), (83, 37, 4, False)])
@pytest.mark.parametrize("method,m", [("faber", 9), ("hork", 6), ("horner", 6), ("rk32", 0), ("rk44", 0)])
def test_shapes_by_operands_agree_bitwise(nx, ny, order, fs, method, m):
    om = oracle_model(nx, ny, layered(nx, ny, 17), order=order, pml=10, fs=fs)
    U0 = tuple(smooth_random_state([f.shape for f in om.zeros_state()], 13))
    out = []
    for variant in (7, 10, 11, 13, 14, -1):
        g = gpu_model(om, "f32", p=8, max_receivers=1)
        g.set_source_receivers(0, (nx // 2) * om.dx, 5 * om.dx, 25.0, 0.05, 1e3, np.array([[0.0, 0.0]]))
        g.set_faber_ellipse(*oracle_ellipse(om))
        g.set_kernel_variant(variant)
        if method == "horner":
            g.set_hork_form("horner")
        g.set_state(0, flatten(U0))
        g.step("hork" if method == "horner" else method, 0.03, 1.1e-3, m, 3)
        out.append(g.get_state(0))
        g.close()
    assert np.isfinite(out[0]).all()
    for o in out[1:]:
        assert np.array_equal(out[0], o)
