"""The cross-split reduction at the edges of its thread counts: 1, 2, 4 and 8
threads per (point, omega) for up to 4, 8, 16 and more splits, whole and ragged
last shares, with and without B and the rim, one and several node tables, against
the FP64 oracle at the FP32 path's gate."""
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
    c.set_option(sc.SC_OPT_NODES_PER_SPLIT, 0)
    c.close()


@pytest.mark.parametrize("splits", [1, 2, 4, 5, 8, 9, 16, 17, 24, 33, 64, 66])
@pytest.mark.parametrize("n_omega,order,rim", [(1, 0, True), (7, 1, True), (30, 0, False)])
def test_split_counts(ctx, splits, n_omega, order, rim):
    tiles = 66
    mirror = dict(f=200.0, r_max=400.0, n_r=tiles, n_theta=32, rim=rim)
    per = -(-tiles // splits)
    ctx.set_option(sc.SC_OPT_NODES_PER_SPLIT, 32 * per)
    om = wl.uniform_omegas(n_omega)
    pts = wl.random_cube(37, 1.5, seed=splits)
    m = ctx.mirror(200.0, 0.0, 400.0, tiles, 32, rim=rim)
    inc = ctx.incident(profile="gauss", w0=120.0, pol="radial", order=order,
                       spectrum=dict(kind="sampled", omega=om, amp=np.ones(n_omega)))
    E, B, st = ctx.eval(m, inc, om, torch.tensor(pts, device="cuda"), stats=True)
    assert st["splits"] == -(-tiles // per)
    E2 = torch.empty_like(E)
    ctx.eval(m, inc, om, torch.tensor(pts, device="cuda"), out=(E2, None))
    assert torch.equal(E, E2)
    ref = oracle.field(dict(mirror, rim=int(rim)), dict(profile="gauss", w0=120.0, pol="radial", order=order,
                                                        r_norm=400.0), om, pts)
    for F, R in zip((E, B), ref):
        d = np.sqrt(np.sum(np.abs(F.cpu().numpy() - R) ** 2, axis=2))
        assert np.all(d <= 1e-5 * np.max(np.sqrt(np.sum(np.abs(R) ** 2, axis=2)), axis=1, keepdims=True))
