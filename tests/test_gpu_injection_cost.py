"""Injecting the residual of many receivers: the work grows with their number, not with its
square, and receivers that share a node are summed in their order whatever their number."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DX = 10.0


def _model(nx, ny, nrec, prec="f32", nodes=None):
    from paper_2401_16322_gb300 import Model
    g = Model(nx, ny, DX, 8, 8, 10.0, True, precision=prec, nshots=2, p=8, max_receivers=nrec)
    g.set_velocity(np.full((ny, nx), 2000.0))
    for k in range(2):
        g.set_source_receivers(k, 20 * DX, 2 * DX, 30.0, 0.04, 1e3, nodes[k] * DX)
    return g


def test_time_grows_with_the_number_of_receivers():
    """8 times the receivers: 8 times the time at most where it is linear, 64 where it is
    quadratic; the line is drawn between."""
    import torch
    nx, ny, best = 300, 200, []
    rng = np.random.default_rng(3)
    for nrec in (4096, 32768):
        nodes = [np.stack([rng.integers(0, nx, nrec), rng.integers(0, ny, nrec)], 1) for _ in range(2)]
        g = _model(nx, ny, nrec, nodes=nodes)
        lam = torch.zeros(2 * g.vector_elems, dtype=torch.float32, device="cuda")
        vals = torch.ones(2, nrec, dtype=torch.float32, device="cuda")
        t = []
        for _ in range(8):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            g.adjoint_inject(lam, vals)
            e[1].record()
            e[1].synchronize()
            t.append(e[0].elapsed_time(e[1]))
        best.append(min(t[3:]))
        g.close()
    assert best[1] < 20 * best[0], best


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("nrec,nn", [(1, 1), (255, 1), (256, 3), (257, 257), (5000, 7), (5000, 60000)])
def test_sums_run_in_the_receivers_order(prec, nrec, nn):
    """Bit for bit: lam + v_0 + v_1 + ..., in the arithmetic of the model's precision."""
    import torch
    nx, ny = 300, 200
    rng = np.random.default_rng(nrec + nn)
    where = rng.permutation(nx * ny)[:nn]
    pick = [where[rng.integers(0, nn, nrec)] for _ in range(2)]
    g = _model(nx, ny, nrec, prec, [np.stack([p % nx, p // nx], 1) for p in pick])
    dt = np.float32 if prec == "f32" else np.float64
    want = rng.standard_normal((2, ny, nx)).astype(dt)
    vals = rng.standard_normal((2, nrec)).astype(dt)
    lam = torch.zeros(2, g.vector_elems, dtype=g.dtype, device="cuda")
    u = lam[:, :g.layout.field_elems].view(2, ny, g.layout.pitch)[:, :, :nx]
    u.copy_(torch.from_numpy(want))
    g.adjoint_inject(lam.view(-1), torch.from_numpy(vals).cuda())
    g.sync()
    for k in range(2):
        flat = want[k].reshape(-1)
        for r in range(nrec):
            flat[pick[k][r]] += vals[k, r]
    assert np.array_equal(u.cpu().numpy(), want)
    g.close()
