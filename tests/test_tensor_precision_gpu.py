"""The tensor-core field kernel's error near the focus as a relative norm over points
and omegas, against the FP64 path: at 1e-6 a class that lost one of its operands' low
halves fails (2^-12 of every term, some 6e-6 of a sum of a thousand), which the
FP32 path's gate of 1e-5 of the peak field would let pass.

The bound: two operands of 22 bits with the product of their low halves left out,
3 units of 2^-23; what a run of five tiles loses to truncation beyond its give-back,
2.5 units; a phase rounded to FP32 and the seed's and rotations' errors, 2 units:
8.9e-7 if all of them added up.

Coherent sums (an unaberrated beam at the focus) and sums of all but random phase (an
aberrated one), one node tile to hundreds, and a beam of many node tables whose weights
alternate in sign (Laguerre-Gauss)."""
import numpy as np
import pytest

from paper_1609_08146_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1609_08146_gb300 as sc  # noqa: E402

BEAMS = {
    "coherent": dict(profile="gauss", pol="linear", pol_angle=0.4),
    "aberrated": dict(profile="supergauss", pol="radial", zernike=[float(v) for v in 0.7 * np.cos(np.arange(14.0))]),
    "vortex": dict(profile="laguerre_gauss", lg_p=0, lg_l=1, omega_band=(0.5, 1.5)),
}


@pytest.fixture(scope="module")
def ctx():
    c = sc.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n_omega", [25, 64, 65, 128, 129, 256])
@pytest.mark.parametrize("beam", list(BEAMS))
@pytest.mark.parametrize("n_r,n_theta", [(4, 8), (37, 33), (96, 80)])
def test_relative_norm(ctx, n_omega, beam, n_r, n_theta):
    f = 1000.0
    b = dict(BEAMS[beam], w0=0.6 * f)
    if beam == "vortex":
        b["z_waist"] = -0.5 * f
    om = wl.uniform_omegas(n_omega, 0.5, 1.5) if beam == "vortex" else wl.uniform_omegas(n_omega)
    m = ctx.mirror(f, 0.0, 2 * f, n_r, n_theta)
    inc = ctx.incident(spectrum=dict(kind="sampled", omega=om, amp=np.ones(om.size)), **b)
    pts = torch.tensor(wl.random_cube(60, 1.0, seed=n_omega), device="cuda")
    *got, st = ctx.eval(m, inc, om, pts, stats=True)
    assert st["kernel_class"] >= 30
    for x, ref in zip(got, ctx.eval(m, inc, om, pts, precision="fp64")):
        assert (x.to(torch.complex128) - ref).norm() <= 1e-6 * ref.norm()
