"""Values with an infinity or a NaN in the tensor-core inverse transform: each is
what the plain sum gives (an infinity with the sign of its phase, NaN where the phase
is zero), also at times where a cosine or sine is all but zero, and many of them cost
a bounded multiple of a finite transform (one sincos per phase and value made it
1800 times)."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("n_omega,n_t", [(65, 200), (96, 128), (130, 300)])
@pytest.mark.parametrize("dtype", [np.complex64, np.complex128])
def test_one_infinity_in_every_value(ctx, n_omega, n_t, dtype):
    """Value v has its infinity at omega v: in the real part (E), in the imaginary part (B)."""
    om = np.linspace(0.5, 1.5, n_omega)  # with the times below: whole and half turns among the phases
    t = np.arange(n_t) / 8.0 - 4.0
    n_pts = (n_omega + 2) // 3
    F = np.zeros((2, n_omega, n_pts, 3), dtype=dtype)
    ph = 2 * np.pi * om[:, None] * t
    want = np.zeros((2, n_t, n_pts * 3))
    for v in range(n_omega):
        sign = 1.0 if v % 2 else -1.0
        F[0, v, v // 3, v % 3] = complex(sign * np.inf, 0.0)
        F[1, v, v // 3, v % 3] = complex(0.0, sign * np.inf)
        with np.errstate(invalid="ignore"):
            want[0, :, v] = sign * np.inf * np.cos(ph[v])
            want[1, :, v] = sign * np.inf * np.sin(ph[v])
    out = ctx.time_domain(torch.tensor(F[0], device="cuda"), torch.tensor(F[1], device="cuda"), om, t,
                          precision="fp32" if dtype == np.complex64 else "fp64")
    for got, ref in zip(out, want):
        np.testing.assert_array_equal(got.cpu().numpy().reshape(n_t, -1), ref)


def test_many_cost_no_sincos_each(ctx):
    g = torch.Generator(device="cuda").manual_seed(1)
    E = torch.view_as_complex(torch.randn((256, 2000, 3, 2), generator=g, device="cuda"))
    om, t = np.linspace(0.5, 1.5, 256), np.arange(512) / 8.0 - 32.0

    def ms():
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        out = []
        for _ in range(4):
            a.record()
            ctx.time_domain(E, None, om, t)
            b.record()
            b.synchronize()
            out.append(a.elapsed_time(b))
        return min(out[1:])

    finite = ms()
    E[7] = float("nan")
    assert ms() < 150 * finite
