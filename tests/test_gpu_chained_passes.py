"""FP64 steps whose passes go out as one cooperative launch (small 2D grids) against the same steps
launched pass by pass (as they are while passes are timed): bit for bit, since both do the same
arithmetic per point.  Grids below, at and above the number of blocks that fit a launch, several
problems in one launch, more passes than one launch holds, steps captured in a graph; and a
barrier wait that gives up is reported and leaves the handle usable."""
import numpy as np
import pytest

from _helpers import flatten, gpu_model, oracle_ellipse, oracle_model
from paper_2401_16322_gb300.workloads import layered, smooth_random_state

pytestmark = pytest.mark.gpu


def _model(nx, ny, order, fs):
    om = oracle_model(nx, ny, layered(nx, ny, 17), order=order, pml=10, fs=fs)
    rec = np.array([[x * om.dx, 3 * om.dx] for x in range(2, nx - 2, 9)])
    g = gpu_model(om, "f64", p=8, max_receivers=len(rec))
    g.set_source_receivers(0, (nx // 2) * om.dx, 5 * om.dx, 25.0, 0.05, 1e3, rec)
    g.set_faber_ellipse(*oracle_ellipse(om))
    U0 = tuple(smooth_random_state([f.shape for f in om.zeros_state()], 13))
    return g, rec, U0


# 64 x 16 tiles of 8 blocks: 76 tiles are four blocks on each of 152 SMs
@pytest.mark.parametrize("nx,ny", [(41, 33), (65, 37), (256, 301), (256, 305)])
@pytest.mark.parametrize("order,fs", [(8, True), (4, False)])
@pytest.mark.parametrize("method,m", [("faber", 12), ("horner", 140), ("hork", 5), ("horner", 5), ("rk32", 0), ("rk44", 0)])
def test_chained_passes_equal_separate_passes(nx, ny, order, fs, method, m):
    if m == 140 and nx > 65:
        pytest.skip("the split of a long chain does not depend on the size")
    out = []
    for separate in (False, True):
        g, rec, U0 = _model(nx, ny, order, fs)
        g.bind_seismogram(4)
        if method == "horner":
            g.set_hork_form("horner")
        g.set_state(0, flatten(U0))
        g.enable_kernel_timing(separate)
        g.step("hork" if method == "horner" else method, 0.03, 1.1e-3, m, 4)
        out.append((g.get_state(0), g.seismogram(0, len(rec), 4)))
        g.close()
    assert np.isfinite(out[0][0]).all()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


def test_chained_batch_equals_single_models():
    from paper_2401_16322_gb300 import Batch
    sizes = [(41, 33), (130, 61), (65, 20)]
    alone, both = [], []
    for nx, ny in sizes:
        g, _, U0 = _model(nx, ny, 8, True)
        g.set_state(0, flatten(U0))
        g.step("hork", 0.03, 1.1e-3, 6, 3)
        alone.append(g.get_state(0))
        g.close()
        g, _, U0 = _model(nx, ny, 8, True)
        g.set_state(0, flatten(U0))
        both.append(g)
    Batch(both).step("hork", 0.03, 1.1e-3, 6, 3)
    for g, want in zip(both, alone):
        assert np.array_equal(g.get_state(0), want)


def test_barrier_wait_timeout_is_reported_and_the_next_call_recovers():
    from paper_2401_16322_gb300.ewave import EwaveError, debug_set_wait_limit
    g, _, U0 = _model(83, 37, 8, True)
    g.set_state(0, flatten(U0))
    g.step("hork", 0.03, 1.1e-3, 6, 2)
    want = g.get_state(0)
    try:
        debug_set_wait_limit(0)
        g.step("hork", 0.03, 1.1e-3, 6, 2)
        with pytest.raises(EwaveError, match="TIMEOUT"):
            g.sync()
    finally:
        debug_set_wait_limit(1_000_000_000)
    g.set_state(0, flatten(U0))
    g.step("hork", 0.03, 1.1e-3, 6, 2)
    g.sync()
    assert np.array_equal(g.get_state(0), want)
    g.close()
