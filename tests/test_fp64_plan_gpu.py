"""The FP64 field sum at the edges of its plan, against the FP64 oracle at the
FP64 path's gate: omegas at and beside 6, 12, 24, ... per point (threads per
point and omegas per thread change there, 193 and more take several groups),
grids uniform to rounding (rotated phasors) and not (a sincos per omega), node
counts below and above one round of a point's threads, point counts that leave
lanes idle, node splits and none (an exhausted budget), several node tables."""
import math

import numpy as np
import pytest

import oracle
from paper_1609_08146_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1609_08146_gb300 as sc  # noqa: E402


def _check(ctx, mirror, om, pts, order=0, tol=None):
    beam = dict(profile="gauss", w0=0.6 * mirror["f"], pol="radial", order=order)
    m = ctx.mirror(mirror["f"], mirror.get("r_min", 0.0), mirror["r_max"], mirror["n_r"], mirror["n_theta"],
                   rim=bool(mirror.get("rim", 1)))
    inc = ctx.incident(spectrum=dict(kind="sampled", omega=om, amp=np.exp(1j * np.arange(om.size))), **beam)
    E, B = ctx.eval(m, inc, om, torch.tensor(pts, device="cuda"), precision="fp64")
    ref = oracle.field(mirror, dict(beam, r_norm=mirror["r_max"]), om, pts, amp=np.exp(1j * np.arange(om.size)))
    tol = tol or 1e-12 + 2e-16 * 2 * math.pi * max(om) * mirror["r_max"]
    for F, R in zip((E, B), ref):
        d = np.sqrt(np.sum(np.abs(F.cpu().numpy() - R) ** 2, axis=2))
        assert np.all(d <= tol * np.max(np.sqrt(np.sum(np.abs(R) ** 2, axis=2)), axis=1, keepdims=True))


@pytest.mark.parametrize("n_omega", [1, 2, 5, 6, 7, 11, 13, 24, 25, 47, 49, 97, 192, 193, 200])
def test_omega_counts(n_omega):
    ctx = sc.Context(0)
    mirror = dict(f=30.0, r_min=4.0, r_max=60.0, n_r=9, n_theta=15, rim=1)
    pts = wl.random_cube(21, 1.5, seed=n_omega)
    _check(ctx, mirror, wl.uniform_omegas(n_omega), pts)
    if n_omega > 1:
        # any grid: not uniform, then uniform but for one omega
        rng = np.random.default_rng(n_omega)
        _check(ctx, mirror, np.sort(rng.uniform(0.5, 1.5, n_omega)), pts)
        om = np.linspace(0.7, 1.3, n_omega)
        om[n_omega // 2] *= 1 + 1e-13
        _check(ctx, mirror, om, pts)
    ctx.close()


@pytest.mark.parametrize("n_r,n_theta,rim,n_points", [(1, 1, 1, 1), (1, 7, 0, 3), (4, 8, 1, 128), (40, 40, 1, 129),
                                                      (40, 40, 0, 3000)])
def test_sizes_and_splits(n_r, n_theta, rim, n_points):
    mirror = dict(f=30.0, r_max=60.0, n_r=n_r, n_theta=n_theta, rim=rim)
    pts = wl.random_cube(n_points, 1.5, seed=n_points)
    for budget in (0, 2 << 20):  # node splits' workspace, and no room for one
        ctx = sc.Context(0, budget_bytes=budget)
        for n in (1, 20):
            _check(ctx, mirror, wl.uniform_omegas(n), pts)
        ctx.close()


def test_several_node_tables():
    ctx = sc.Context(0)
    mirror = dict(f=30.0, r_max=60.0, n_r=24, n_theta=24, rim=1)
    # (the oracle takes the first-order terms by finite differences: 1e-11)
    for pts in (wl.random_cube(5, 1.0, seed=1), wl.random_cube(4000, 1.0, seed=2)):
        _check(ctx, mirror, wl.uniform_omegas(9), pts, order=1, tol=2e-11)
    ctx.close()
