"""FP32 Faber and HORK adjoint steps on both sides of the degree from which the recompute pass
stores the gradient's factor instead of the vectors, where the tape's fields fill up (four to a
vector) and at a degree past that, against the oracle with the tolerance of the FP32 adjoint step
tests; and the injection of receivers that share nodes."""
import numpy as np
import pytest

from _helpers import flatten, rel_l2
from oracle.adjoint import faber_adjoint_step, hork_adjoint_step
from oracle.faber import ellipse_params
from oracle.model import Model as OModel
from oracle.model import default_beta0
from oracle.source import PointSource
from paper_2401_16322_gb300.workloads import layered, random_state, smooth_random_state

pytestmark = pytest.mark.gpu

DX = 10.0


@pytest.mark.parametrize("m", [2, 3, 4, 5, 9])
@pytest.mark.parametrize("method", ["faber", "hork", "horner"])
def test_adjoint_step_around_the_tape_degree(method, m):
    import torch
    from paper_2401_16322_gb300 import Model
    nx, ny, order, fs, pml = 130, 49, 8, True, 9
    c = layered(nx, ny, 12, vmin=1500, vmax=3000)
    beta0 = default_beta0(3000.0, pml, DX)
    om = OModel(nx, ny, DX, order, pml, beta0, fs, c)
    ell = ellipse_params(3000.0, beta0, DX, order, free_surface=fs)
    g = Model(nx, ny, DX, order, pml, beta0, fs, precision="f32", nshots=2, p=8)
    g.set_velocity(c)
    for k in range(2):
        g.set_source_receivers(k, (40 + 30 * k) * DX, 2 * DX, 30.0, 0.04, 1e3, np.zeros((0, 2)))
    g.set_faber_ellipse(*ell)
    if method == "horner":
        g.set_hork_form("horner")
    name = "faber" if method == "faber" else "hork"
    dt, t = 1.2e-3, 0.02
    g.step(name, t, dt, m, 1)
    nv, fe = g.vector_elems, g.layout.field_elems
    Us = [flatten(smooth_random_state([f.shape for f in om.zeros_state()], 50 + k)) for k in range(2)]
    ybars = [random_state([(om.n,)], 60 + k)[0] for k in range(2)]
    ck = torch.zeros(2 * nv, dtype=torch.float32, device="cuda")
    lam = torch.zeros(2 * nv, dtype=torch.float32, device="cuda")
    for k in range(2):
        g.pack(Us[k], ck[k * nv:(k + 1) * nv])
        g.pack(ybars[k], lam[k * nv:(k + 1) * nv])
    grad = torch.zeros(2 * fe, dtype=torch.float32, device="cuda")
    g.adjoint_step(t, dt, m, ck, lam, grad, method=name)
    g.sync()
    for k in range(2):
        src = PointSource(om, (40 + 30 * k) * DX, 2 * DX, 30.0, 0.04, amp=1e3, p=8)
        if name == "faber":
            Ub, gr = faber_adjoint_step(om, Us[k], ybars[k], src, t, dt, m, ell)
        else:
            Ub, gr = hork_adjoint_step(om, Us[k], ybars[k], src, t, dt, m)
        assert rel_l2(g.unpack(lam[k * nv:(k + 1) * nv]), Ub) < 3e-5
        got = grad[k * fe:(k + 1) * fe].view(ny, g.layout.pitch)[:, :nx].double().cpu().numpy()
        assert rel_l2(got, gr.reshape(ny, nx)) < 3e-5
    g.close()


@pytest.mark.parametrize("nrec", [1, 5, 300])
def test_injection_adds_coincident_receivers(nrec):
    import torch
    from paper_2401_16322_gb300 import Model
    nx, ny = 40, 33
    g = Model(nx, ny, DX, 8, 8, 10.0, True, precision="f32", nshots=2, p=8, max_receivers=nrec)
    g.set_velocity(np.full((ny, nx), 2000.0))
    rng = np.random.default_rng(5)
    nodes = [np.stack([rng.integers(0, nx, nrec), rng.integers(0, 6, nrec)], 1) for _ in range(2)]
    for k in range(2):
        g.set_source_receivers(k, 20 * DX, 2 * DX, 30.0, 0.04, 1e3, nodes[k] * DX)
    nv = g.vector_elems
    x = rng.standard_normal((2, nx * ny)).astype(np.float32)
    vals = rng.standard_normal((2, nrec)).astype(np.float32)
    lam = torch.zeros(2, nv, dtype=torch.float32, device="cuda")
    u = lam[:, :g.layout.field_elems].view(2, ny, g.layout.pitch)[:, :, :nx]
    u.copy_(torch.from_numpy(x).view(2, ny, nx))
    g.adjoint_inject(lam.view(-1), torch.from_numpy(vals).cuda().contiguous())
    g.sync()
    want = x.astype(np.float64).reshape(2, ny, nx)
    size = np.abs(want)
    for k in range(2):
        np.add.at(want[k], (nodes[k][:, 1], nodes[k][:, 0]), vals[k])
        np.add.at(size[k], (nodes[k][:, 1], nodes[k][:, 0]), np.abs(vals[k]))
    # a node's sum of n FP32 terms is off by at most (n - 1) roundings of the terms' magnitudes
    n = 1 + max(np.unique(nodes[k], axis=0, return_counts=True)[1].max() for k in range(2))
    assert (np.abs(u.double().cpu().numpy() - want) <= n * 2.0 ** -24 * size).all()
    assert (lam[:, g.layout.field_elems:] == 0).all()
    g.close()
