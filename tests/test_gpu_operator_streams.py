"""H x on a caller's vectors when other work is queued: a model whose stream is not the caller's
takes x when the caller's stream has written it and overwrites y when the caller's stream has
read it; and vectors that come from another stream's memory outlive the product; and the
C entry returns with y complete."""
import numpy as np
import pytest

from _helpers import TOL, flatten, oracle_model, rel_l2
from oracle.operator import assemble_H
from paper_2401_16322_gb300.workloads import layered, smooth_random_state

pytestmark = pytest.mark.gpu


def _busy():
    """Some tens of milliseconds of work on the current stream."""
    import torch
    a = torch.full((4096, 4096), 1e-4, device="cuda")
    b = a
    for _ in range(30):
        b = b @ a
    return b


def _case(stream):
    import torch
    from paper_2401_16322_gb300 import Model
    om = oracle_model(97, 65, layered(97, 65, 3), pml=10, fs=True)
    g = Model(om.nx, om.ny, om.dx, om.order, om.pml, om.beta0, True, precision="f64", stream=stream)
    g.set_velocity(om.c)
    x = flatten(smooth_random_state([f.shape for f in om.zeros_state()], 11))
    src, dx, dy = g.new_vector(), g.new_vector(), g.new_vector()
    g.pack(x, src)
    _busy()                                        # (loads the library's kernels)
    g.apply_device(src, dy)
    dy.fill_(3.0)
    torch.cuda.synchronize()
    return om, g, x, src, dx, dy


@pytest.mark.parametrize("model_on", ["own stream", "current stream"])
@pytest.mark.parametrize("transpose", [False, True])
def test_operands_are_ordered_against_the_callers_stream(model_on, transpose):
    """No synchronisation between the caller's work and the product, on either side."""
    import torch
    om, g, x, src, dx, dy = _case(torch.cuda.Stream() if model_on == "own stream" else None)
    caller = torch.cuda.current_stream() if model_on == "own stream" else torch.cuda.Stream()
    with torch.cuda.stream(caller):
        _busy()
        old = dy.clone()                           # reads y before the product
        dx.copy_(src)                              # writes x before the product
        g.apply_device(dx, dy, transpose)
        new = dy.clone()                           # reads y after it
    torch.cuda.synchronize()
    H = assemble_H(om)
    assert bool((old == 3.0).all())
    assert rel_l2(g.unpack(new), (H.T if transpose else H) @ x) < TOL["f64"]
    g.close()


@pytest.mark.parametrize("which", ["x", "y"])
def test_vectors_of_another_stream_may_be_freed_after_the_call(which):
    """The vector is allocated on a side stream, whose next allocation would take its place while
    the product waits behind other work."""
    import torch
    om, g, x, src, dx, dy = _case(None)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        v = torch.empty_like(src)
        if which == "x":
            v.copy_(src)
    torch.cuda.synchronize()
    _busy()
    if which == "x":
        g.apply_device(v, dy)
        del v
    else:
        g.apply_device(src, v)
        del v
    with torch.cuda.stream(side):
        other = [torch.full_like(src, 5.0) for _ in range(4)]
    torch.cuda.synchronize()
    if which == "x":
        assert rel_l2(g.unpack(dy), assemble_H(om) @ x) < TOL["f64"]
    assert all(bool((o == 5.0).all()) for o in other)     # (y: written by nobody else)
    g.close()


@pytest.mark.parametrize("transpose", [0, 1])
def test_c_entry_returns_with_y_complete(transpose):
    """The model's stream is busy when the product is asked for; on return y can be read on any
    stream."""
    import torch
    s = torch.cuda.Stream()
    om, g, x, src, dx, dy = _case(s)
    with torch.cuda.stream(s):
        _busy()
        dx.copy_(src)
    assert g.lib.ewv_apply_operator(g.h, transpose, dx.data_ptr(), dy.data_ptr()) == 0
    assert s.query()
    y = dy.clone()
    H = assemble_H(om)
    assert rel_l2(g.unpack(y), (H.T if transpose else H) @ x) < TOL["f64"]
    g.close()
