"""The FP64 field sum under device budgets: its node splits' workspace is scratch.
Without room for it the call runs all the same and gives the same bits (threads per
point and omegas per thread at their edges, uniform grids and others, several node
tables, host outputs), and a call's workspace, held, does not refuse a larger call
that fits without it."""
import numpy as np
import pytest

from paper_1609_08146_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1609_08146_gb300 as sc  # noqa: E402

MB = 1 << 20


def _beam(ctx, n, om, order=0):
    return ctx.mirror(30.0, 3.0, 60.0, n, n), ctx.incident(
        profile="gauss", w0=18.0, pol="radial", order=order,
        spectrum=dict(kind="sampled", omega=om, amp=np.exp(1j * np.arange(om.size))))


def _eval(ctx, m, inc, om, pts, host=False):
    out = ctx.eval(m, inc, om, pts if host else torch.tensor(pts, device="cuda"), precision="fp64")
    return out if host else [x.cpu().numpy() for x in out]


@pytest.mark.parametrize("n_omega,n_points", [(1, 700), (2, 129), (5, 300), (7, 90), (24, 33), (47, 60), (193, 9)])
@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("uniform", [True, False])
def test_same_bits_without_room(n_omega, n_points, order, uniform):
    om = wl.uniform_omegas(n_omega)
    if not uniform:
        om = np.sort(om * (1 + 1e-3 * np.random.default_rng(n_omega).uniform(-1, 1, n_omega)))
    pts = wl.random_cube(n_points, 1.5, seed=n_omega)
    tables = (48 * 48 + 96) * 120 * (2 if order else 1)  # FP32 and FP64 records, tiles rounded up
    out = []
    for budget in (0, tables + 64 * 1024):
        ctx = sc.Context(0, budget_bytes=budget)
        out.append(_eval(ctx, *_beam(ctx, 48, om, order), om, pts))
        ctx.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("mb", [4, 6])
def test_workspace_is_given_back(mb):
    om = np.ones(1)
    small, large = wl.random_cube(200, 1.0, seed=1), wl.random_cube(30000, 1.0, seed=2)
    out = []
    for budget in (0, mb * MB):
        ctx = sc.Context(0, budget_bytes=budget)
        beam = _beam(ctx, 64, om)  # one node table: 0.5 MB, and 3.6 MB of points and outputs
        out.append([x for p in (small, large, small) for x in _eval(ctx, *beam, om, p, host=True)])
        ctx.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
