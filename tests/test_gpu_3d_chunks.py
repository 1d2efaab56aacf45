"""The FP32 3D pass cuts a column into chunks of planes by the number of tasks the chip can run at
once: one or several chunks, even and ragged last chunks, columns just past a tile edge, with and
without the free-surface planes, against the oracle and with the same tolerance as the operator
and integrator tests."""
import numpy as np
import pytest

from _helpers import TOL, flatten, rel_l2, rel_l2_fields
from oracle import faber
from oracle import wave3d as W
from test_gpu_3d import _models
from paper_2401_16322_gb300.workloads import smooth_random_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz,fs", [(15, True), (31, False), (32, True), (33, False), (65, True)])
@pytest.mark.parametrize("nx,ny", [(64, 17), (65, 24)])
def test_chunked_columns_match_oracle(nx, ny, nz, fs):
    om, g = _models(nx, ny, nz, "f32", fs=fs, p=10, max_receivers=1)
    at = (30 * 10.0, 8 * 10.0, (nz // 2) * 10.0)
    src = W.PointSource3D(om, *at, 25.0, 0.05, amp=1e3, p=10)
    g.set_source_receivers3d(0, *at, 25.0, 0.05, 1e3, np.array([[0.0, 0.0, 0.0]]))
    params = faber.ellipse_params(om.c_max, om.beta0, om.dx, om.order, dims=3, free_surface=fs)
    g.set_faber_ellipse(*params)
    U0 = tuple(smooth_random_state(om.field_shapes(), 8))
    g.set_state(0, flatten(U0))
    g.step("faber", 0.03, 1.0e-3, 8, 1)
    U = faber.faber_step(om, U0, src, 0.03, 1.0e-3, 8, params)
    got = g.get_state(0)
    g.close()
    assert rel_l2(got, flatten(U)) < 3 * TOL["f32"]
    assert max(rel_l2_fields(got, flatten(U), om.field_shapes())) < 3 * TOL["f32"]
