"""A lost tile hand-over in the tensor-core field kernel: the bounded wait for it
runs out, the whole launch ends after that one wait, the call reports
SC_ERR_TIMEOUT, and the next call on the context is bitwise equal to one made
before.  Each class of the kernel, alone (descriptor in the launch's parameters)
and in a batch (work queue, and the launch's abort word); the lost tile is the
first of its run, inside one, the last, and of a later run.  The direct kernel's
many-thread layouts, which these omega counts take when it is pinned, likewise."""
import time

import numpy as np
import pytest

from paper_1609_08146_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1609_08146_gb300 as sc  # noqa: E402


def _request(ctx, n_omega, n_points):
    w = wl.sweep(1e4, 128, n_points=n_points)
    mc = w["mirror"]
    m = ctx.mirror(mc["f"], 0.0, mc["r_max"], mc["n_r"], mc["n_theta"])
    om = wl.uniform_omegas(n_omega)
    inc = ctx.incident(profile="gauss", w0=w["beam"]["w0"],
                       spectrum=dict(kind="sampled", omega=om, amp=np.ones(om.size)))
    return m, inc, om, torch.tensor(w["points"], device="cuda")


def _lose(ctx, tile, run):
    before = run()
    ctx.set_option(sc.SC_OPT_FAIL_COPY, tile)
    try:
        t0 = time.time()
        with pytest.raises(sc.ScError) as e:
            run()
        dt = time.time() - t0
    finally:
        ctx.set_option(sc.SC_OPT_FAIL_COPY, -1)
    assert e.value.status == sc.SC_ERR_TIMEOUT
    assert 0.5 < dt < 5.0, dt
    for a, b in zip(before, run()):
        assert torch.equal(a, b)


@pytest.mark.parametrize("n_omega", [40, 100, 200])
@pytest.mark.parametrize("tile", [0, 2, 4, 9])
@pytest.mark.parametrize("batch", [False, True])
def test_lost_tile(n_omega, tile, batch):
    ctx = sc.Context(0)
    try:
        reqs = [_request(ctx, n_omega, 700), _request(ctx, n_omega + 1, 300)]
        if batch:
            _lose(ctx, tile, lambda: [t for o in ctx.eval_batch(reqs, stats=True)[0] for t in o])
        else:
            _lose(ctx, tile, lambda: ctx.eval(*reqs[0], stats=True)[:2])
    finally:
        ctx.close()


@pytest.mark.parametrize("n_omega", [128, 256])
@pytest.mark.parametrize("tile", [0, 7])
def test_lost_copy_in_the_pinned_direct_kernel(n_omega, tile):
    ctx = sc.Context(0)
    try:
        ctx.set_option(sc.SC_OPT_TILE_LAYOUT, 0)
        req = _request(ctx, n_omega, 700)
        _lose(ctx, tile, lambda: ctx.eval(*req, stats=True)[:2])
    finally:
        ctx.close()
