"""The testing switch between the Gram-Schmidt forms reaches every problem set: off, a set too
large for the column kernel takes a flat pass per step, which gives each shot the bits that one
shot alone has (FP32, one pass shape)."""
import numpy as np
import pytest

from _helpers import flatten, gpu_model, oracle_model
from paper_2401_16322_gb300.workloads import layered, smooth_random_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("window", [0, 3])
def test_flat_passes_on_a_large_set_equal_one_shot_alone(window):
    from paper_2401_16322_gb300.ewave import debug_set_column_kernel
    nx, ny, m, dt, t0 = 137, 53, 14, 1e-3, 0.03
    om = oracle_model(nx, ny, layered(nx, ny, 4), pml=8, fs=True)
    nshots = 250                                      # 5 chunks a shot, 912 fit a grid
    U = flatten(smooth_random_state([f.shape for f in om.zeros_state()], 21))

    def step(ns, first):
        g = gpu_model(om, "f32", nshots=ns, p=8)
        g.set_kernel_variant(14)
        if window:
            g.set_krylov_window(window)
        for s in range(ns):
            g.set_source_receivers(s, (5 + (first + s) % 7) * om.dx, 2 * om.dx, 25.0, 0.05, 1e3)
            g.set_state(s, U)
        g.step_krylov(t0, dt, m, 1)
        out = [g.get_state(s) for s in (0, ns - 1)]
        g.close()
        return out

    debug_set_column_kernel(False)
    try:
        many = step(nshots, 0)
        for got, first in zip(many, (0, nshots - 1)):
            assert np.array_equal(got, step(1, first)[0])
    finally:
        debug_set_column_kernel(True)
