"""The FP32 adjoint step under every pass shape a user can select: the recompute that stores the
gradient's factor and the reverse passes do the same arithmetic per point whatever the shape, so
cotangents and gradients have the bits of the default's -- which the oracle checks elsewhere."""
import numpy as np
import pytest

from paper_2401_16322_gb300.workloads import layered

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method,m", [("faber", 9), ("hork", 6)])
@pytest.mark.parametrize("nx,ny,order", [(130, 49, 8), (75, 39, 4)])
def test_adjoint_step_does_not_depend_on_the_variant(method, m, nx, ny, order):
    import torch
    from paper_2401_16322_gb300 import Model
    from paper_2401_16322_gb300.ewave import NUM_KERNEL_VARIANTS
    c = layered(nx, ny, 12, vmin=1500, vmax=3000)
    gen = torch.Generator(device="cuda").manual_seed(5)
    out = {}
    for v in [14] + [v for v in range(NUM_KERNEL_VARIANTS) if v != 14]:
        g = Model(nx, ny, 10.0, order, 9, 100.0, order == 8, precision="f32", nshots=2, p=8)
        g.set_velocity(c)
        for k in range(2):
            g.set_source_receivers(k, (30 + 20 * k) * 10.0, 20.0, 30.0, 0.04, 1e3)
        g.set_kernel_variant(v)
        nv, fe = g.vector_elems, g.layout.field_elems
        if not out:
            # random values on the grid's own points, zeros in the padding
            inside = torch.zeros(2, 4, ny, g.layout.pitch, device="cuda")
            inside[..., :nx] = 1.0
            inside[:, 2, :, nx - 1] = 0.0
            inside[:, 3, ny - 1] = 0.0
            pad = torch.zeros(2, nv, device="cuda")
            pad[:, :4 * fe].view(2, 4, fe)[..., :ny * g.layout.pitch] = inside.view(2, 4, -1)
            ck, ybar = (torch.randn(2, nv, generator=gen, device="cuda") * pad for _ in range(2))
        lam, grad = ybar.clone().view(-1), torch.zeros(2 * fe, device="cuda")
        g.adjoint_step(0.02, 1.2e-3, m, ck.view(-1), lam, grad, method=method)
        g.sync()
        out[v] = (lam, grad)
        g.close()
    assert bool(torch.isfinite(out[14][1]).all()) and bool(out[14][1].any())
    for v, (lam, grad) in out.items():
        assert torch.equal(lam, out[14][0]), v
        assert torch.equal(grad, out[14][1]), v
    assert np.isfinite(float(out[14][0].norm()))
