"""The tensor-core field kernel (25 to 256 omegas a chunk) against the FP64
oracle and against the direct kernel that SC_OPT_TILE_LAYOUT = 0 pins.

Sizes at its edges: the smallest and largest counts of either class (128 / 129
omegas), a rest of one omega (257) and of a tensor chunk (300), row phasors that
end inside a segment of eight, one node tile, runs of five tiles and one more
or fewer, a ragged last tile, runs cut by SC_OPT_FLUSH_NODES, several splits,
no rim.  The bound is the FP32 path's gate, 1e-5 of the peak field, and three
times the direct kernel's own error where that is larger than 3e-6: points far
off the focus, whose phase FP32 cannot hold on either kernel.  Among them are
points near and beyond the mirror, which do not qualify for fp16 operands and
take the kernel's plain FP32 loop.
"""
import numpy as np
import pytest

import oracle
from paper_1609_08146_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1609_08146_gb300 as sc  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    c = sc.Context(0)
    yield c
    c.close()


def _err(F, R):
    """Per point: worst omega of |F - R| over the peak |R| of that omega."""
    d = np.sqrt(np.sum(np.abs(F - R) ** 2, axis=2))
    return np.max(d / np.max(np.sqrt(np.sum(np.abs(R) ** 2, axis=2)), axis=1, keepdims=True), axis=0)


def _both(ctx, mirror, om, pts, pol="linear", **opts):
    m = ctx.mirror(mirror["f"], mirror.get("r_min", 0.0), mirror["r_max"], mirror["n_r"], mirror["n_theta"],
                   rim=mirror.get("rim", True))
    beam = dict(profile="gauss", w0=0.6 * mirror["f"], pol=pol, zernike=[0.05, -0.1])
    inc = ctx.incident(spectrum=dict(kind="sampled", omega=om, amp=np.ones(om.size)), **beam)
    P = torch.tensor(pts, device="cuda")
    out = []
    for layout in (-1, 0):
        ctx.set_option(sc.SC_OPT_TILE_LAYOUT, layout)
        E, B, st = ctx.eval(m, inc, om, P, stats=True)
        assert (st["kernel_class"] >= 30) == (layout == -1)
        out.append((E.cpu().numpy().astype(complex), B.cpu().numpy().astype(complex)))
    ctx.set_option(sc.SC_OPT_TILE_LAYOUT, -1)
    ref = oracle.field(dict(mirror, rim=int(mirror.get("rim", True))), dict(beam, r_norm=mirror["r_max"]), om, pts)
    for new, old, want in zip(out[0], out[1], ref):
        assert np.all(_err(new, want) <= np.maximum(1e-5, 3 * _err(old, want)))


@pytest.mark.parametrize("n_omega", [25, 32, 63, 64, 65, 127, 128, 129, 192, 255, 256, 257, 300])
def test_omega_counts(ctx, n_omega):
    mirror = dict(f=1000.0, r_max=2000.0, n_r=37, n_theta=33)
    pts = np.vstack([np.zeros((1, 3)), wl.random_cube(20, 2.0, seed=n_omega)])
    _both(ctx, mirror, wl.uniform_omegas(n_omega), pts)


@pytest.mark.parametrize("n_r,n_theta,rim", [(1, 3, True), (4, 8, True), (5, 32, False), (6, 32, True), (11, 32, True),
                                             (7, 23, False)])
def test_short_runs(ctx, n_r, n_theta, rim):
    mirror = dict(f=300.0, r_min=40.0, r_max=600.0, n_r=n_r, n_theta=n_theta, rim=rim)
    for n in (40, 200):
        _both(ctx, mirror, wl.uniform_omegas(n), wl.random_cube(9, 1.5, seed=n_r), pol="radial")


def test_splits_and_flush(ctx):
    mirror = dict(f=5e4, r_max=1e5, n_r=48, n_theta=40)
    try:
        ctx.set_option(sc.SC_OPT_NODES_PER_SPLIT, 32 * 7)
        for flush in (32, 96, 2048):
            ctx.set_option(sc.SC_OPT_FLUSH_NODES, flush)
            _both(ctx, mirror, wl.uniform_omegas(150), wl.random_cube(11, 2.0, seed=flush), pol="azimuthal")
    finally:
        ctx.set_option(sc.SC_OPT_NODES_PER_SPLIT, 0)
        ctx.set_option(sc.SC_OPT_FLUSH_NODES, 2048)


@pytest.mark.parametrize("n_omega", [40, 130])
def test_points_off_the_focus(ctx, n_omega):
    rng = np.random.default_rng(n_omega)
    near = rng.uniform(-1.0, 1.0, size=(6, 3))
    far = np.vstack([near, 15 * rng.uniform(-1.0, 1.0, size=(8, 3)), [[0.1, 0.2, -19.5], [3.0, 0.0, -19.0]],
                     200 * rng.uniform(-1.0, 1.0, size=(4, 3)), near + 0.3])
    _both(ctx, dict(f=20.0, r_max=40.0, n_r=40, n_theta=44), wl.uniform_omegas(n_omega), far)
