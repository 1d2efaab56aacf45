"""The range of the FP32 Krylov step's inner products: a state is taken up to the size at which
the sum of four products still fits FP32, however many elements are summed.  All of a step scales
with its state by a power of two without rounding (the start vector is balanced by |U|), so the
step of 2^62 U is 2^62 times the step of U, up to the order of the sums: an FP64 sum against the
pair sums differs in the 14th digit or so, which can move an FP32 coefficient by one rounding
(6e-8), and with it the state by that much a basis vector: 12 of them stay below 1e-6."""
import numpy as np
import pytest

from _helpers import flatten, gpu_model, oracle_model, rel_l2
from paper_2401_16322_gb300.workloads import layered, smooth_random_state

pytestmark = pytest.mark.gpu

SCALE = 2.0 ** 62              # four squares of it: 8.5e37


@pytest.mark.parametrize("form", ["column kernel", "flat passes", "two passes"])
def test_a_large_state_gives_the_scaled_step(form):
    from paper_2401_16322_gb300.ewave import debug_set_column_kernel
    nx, ny, m, dt = 137, 53, 12, 1e-3
    om = oracle_model(nx, ny, layered(nx, ny, 4), pml=8, fs=True)
    nshots = 250 if form == "two passes" else 2       # 5 chunks of 8192 elements a shot, 912 fit a grid
    U = flatten(smooth_random_state([f.shape for f in om.zeros_state()], 21))
    U /= np.abs(U).max()
    debug_set_column_kernel(form != "flat passes")
    try:
        got = []
        for scale in (1.0, SCALE):
            g = gpu_model(om, "f32", nshots=nshots, p=8)
            g.set_kernel_variant(14)
            for s in range(nshots):
                g.set_state(s, U * scale)
            g.step_krylov(0.0, dt, m, 1)
            got.append([g.get_state(s) / scale for s in (0, nshots - 1)])
            g.close()
    finally:
        debug_set_column_kernel(True)
    for a, b in zip(*got):
        assert rel_l2(b, a) < 1e-6, rel_l2(b, a)
