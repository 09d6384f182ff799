"""The tensor-core kernel's plain loop, which takes the points whose operands do not
fit fp16: every point within a sixteenth of the mirror's smallest distance of it, or
beyond.  Omega counts on either side of each change of its layout (4, 8, 16 and 32
lanes per node, 5 to 8 omegas a lane), tables of fewer node tiles than warps
(several warps share a tile), of one more, and of several rounds, a rim and none,
flushes after every tile, focal points in between.

It does the direct kernel's operations in shorter runs and adds at most three more
FP32 sums, so its error against the oracle, as a relative norm over all points, is
held to twice that of the direct kernel on the same input."""
import numpy as np
import pytest

import oracle
from paper_1609_08146_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1609_08146_gb300 as sc  # noqa: E402

F = 20.0


@pytest.fixture(scope="module")
def ctx():
    c = sc.Context(0)
    yield c
    c.close()


def _points(seed):
    """Off the focus, up to twice the focal length away but not closer than 1 to the mirror; the last ones near it."""
    rng = np.random.default_rng(seed)
    u = rng.normal(size=(40, 3))
    p = u / np.linalg.norm(u, axis=1)[:, None] * rng.uniform(0.95, 2.0, size=(40, 1)) * F
    z_mirror = (p[:, 0] ** 2 + p[:, 1] ** 2) / (4 * F) - F
    p = p[np.abs(p[:, 2] - z_mirror) > 1.0][:13]
    return np.vstack([p, rng.uniform(-1.0, 1.0, size=(3, 3))])


def _compare(ctx, mirror, n_omega, seed):
    m = ctx.mirror(F, mirror.get("r_min", 0.0), 2 * F, mirror["n_r"], mirror["n_theta"], rim=mirror["rim"])
    om = wl.uniform_omegas(n_omega)
    beam = dict(profile="gauss", w0=0.6 * F, pol="radial")
    inc = ctx.incident(spectrum=dict(kind="sampled", omega=om, amp=np.ones(om.size)), **beam)
    pts = _points(seed)
    ref = oracle.field(dict(mirror, f=F, r_max=2 * F, rim=int(mirror["rim"])), dict(beam, r_norm=2 * F), om, pts)
    err = []
    for layout in (-1, 0):
        ctx.set_option(sc.SC_OPT_TILE_LAYOUT, layout)
        out = ctx.eval(m, inc, om, torch.tensor(pts, device="cuda"))
        err.append([np.linalg.norm(x.cpu().numpy()[:, :13] - r[:, :13]) / np.linalg.norm(r[:, :13])
                    for x, r in zip(out, ref)])
    ctx.set_option(sc.SC_OPT_TILE_LAYOUT, -1)
    for new, old in zip(*err):
        assert new <= 2 * old, (new, old)


@pytest.mark.parametrize("n_omega", [25, 28, 29, 32, 33, 40, 41, 48, 57, 64, 65, 80, 81, 112, 128, 129, 160, 193, 256])
def test_layouts(ctx, n_omega):
    _compare(ctx, dict(n_r=23, n_theta=24, rim=True), n_omega, n_omega)


@pytest.mark.parametrize("n_r,n_theta,rim", [(4, 8, False), (3, 40, True), (15, 32, True), (16, 32, False), (17, 32, True),
                                             (64, 33, True)])
@pytest.mark.parametrize("n_omega", [30, 50, 100, 200])
def test_tables(ctx, n_r, n_theta, rim, n_omega):
    mirror = dict(n_r=n_r, n_theta=n_theta, rim=rim, r_min=4.0)
    try:
        for flush in (2048, 32):
            ctx.set_option(sc.SC_OPT_FLUSH_NODES, flush)
            _compare(ctx, mirror, n_omega, n_r)
    finally:
        ctx.set_option(sc.SC_OPT_FLUSH_NODES, 2048)
