"""The inverse transform at the edges of its kernels' tiles, against numpy in 64
bits: one stage of 16 omegas and one more, runs of three stages and parts of one,
128 and 256 times and one more, values at and beside a tile's 128 columns, counts
on either side of the line between the FP32 and the tensor kernel; both
precisions' spectra, E alone, grids uniform to rounding and only to 1e-9, values
of very different size side by side, infinities and NaN.

The bound, 2^-19 of 2 dk sum |F| per value: two operands in 22 bits each (4 units
of 2^-23 together), up to ten accumulations that drop up to one unit of 2^-23 of the
sum each, and the additions of the runs."""
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


def _spectra(n, npts, seed):
    rng = np.random.default_rng(seed)
    size = 10.0 ** rng.uniform(-12, 12, size=(1, npts, 3))  # values of very different size
    return [((rng.normal(size=(n, npts, 3)) + 1j * rng.normal(size=(n, npts, 3))) * size).astype(np.complex64)
            for _ in range(2)]


def _check(ctx, F, om, t, out):
    dk = 2 * np.pi * (om[-1] - om[0]) / (om.size - 1) if om.size > 1 else 1.0
    ref = 2 * dk * np.einsum("npc,nt->tpc", F.astype(complex), np.exp(-2j * np.pi * np.outer(om, t))).real
    bound = 2.0 ** -19 * 2 * dk * np.sum(np.abs(F.astype(complex)), axis=0)
    assert np.all(np.abs(out.cpu().numpy() - ref) <= bound)


@pytest.mark.parametrize("n_omega", [1, 15, 16, 17, 48, 80, 81, 96, 160, 250])
@pytest.mark.parametrize("n_t,npts", [(1, 1), (127, 42), (128, 43), (129, 85), (256, 86), (257, 300), (400, 43)])
def test_sizes(ctx, n_omega, n_t, npts):
    E, B = _spectra(n_omega, npts, n_omega + n_t)
    om = np.array([1.0]) if n_omega == 1 else np.linspace(0.5, 1.5, n_omega)
    if n_omega % 2 and n_omega > 2:  # uniform to 1e-9 only
        om = om * (1 + 1e-10 * np.random.default_rng(n_t).uniform(-1, 1, n_omega))
    t = np.random.default_rng(npts).uniform(-30, 30, n_t)
    Et, Bt = ctx.time_domain(torch.tensor(E, device="cuda"), torch.tensor(B, device="cuda"), om, t)
    _check(ctx, E, om, t, Et)
    _check(ctx, B, om, t, Bt)
    E64 = torch.tensor(E, device="cuda").to(torch.complex128)
    Et, none = ctx.time_domain(E64, None, om, t, precision="fp64")
    assert none is None
    _check(ctx, E, om, t, Et)


def test_infinities_and_nan_stay_in_their_value(ctx):
    E, B = _spectra(96, 60, 5)
    om, t = np.linspace(0.5, 1.5, 96), np.linspace(-5, 5, 140)
    clean = [x.cpu().numpy() for x in ctx.time_domain(torch.tensor(E, device="cuda"), torch.tensor(B, device="cuda"), om, t)]
    E[3, 10, 1] = np.inf
    E[70, 50, 2] = np.nan
    B[20, 0, 0] = complex(0.0, -np.inf)
    dirty = [x.cpu().numpy() for x in ctx.time_domain(torch.tensor(E, device="cuda"), torch.tensor(B, device="cuda"), om, t)]
    bad = [{(10, 1), (50, 2)}, {(0, 0)}]
    for c, d, b in zip(clean, dirty, bad):
        for p in range(60):
            for k in range(3):
                if (p, k) in b:
                    assert not np.any(np.isfinite(d[:, p, k]))
                else:
                    assert np.array_equal(c[:, p, k], d[:, p, k])
    # the sign of an infinity is the sign of its cosine
    assert np.array_equal(np.sign(dirty[0][:, 10, 1]), np.sign(np.cos(2 * np.pi * om[3] * t)))
