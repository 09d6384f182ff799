"""Calls under a device budget that holds what they need and nothing besides:
scratch that only makes a call faster costs speed there, not the call, and what one
call keeps of it does not refuse the next."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1609_08146_gb300 as sc  # noqa: E402


def _spectra(n_omega, n_points):
    rng = np.random.default_rng(n_omega)
    return [(rng.normal(size=(n_omega, n_points, 3)) + 1j * rng.normal(size=(n_omega, n_points, 3))).astype(np.complex64)
            for _ in range(2)]


@pytest.mark.parametrize("n_omega,n_points,n_t", [(64, 2000, 512), (16, 3000, 400), (250, 40, 129)])
@pytest.mark.parametrize("host", [False, True])
def test_transform_without_room_for_the_tensor_kernel(n_omega, n_points, n_t, host):
    """The FP32 kernel's buffers exactly: wavenumbers, times, its phase table, and a host call's staging."""
    need = 8 * (n_omega + n_t) + 8 * n_omega * n_t
    if host:
        need += 2 * (8 * n_omega + 4 * n_t) * 3 * n_points
    F = _spectra(n_omega, n_points)
    om, t = np.linspace(0.5, 1.5, n_omega), np.arange(n_t) / 8.0
    ctx = sc.Context(0, budget_bytes=need)
    try:
        got = ctx.time_domain(*(F if host else [torch.tensor(x, device="cuda") for x in F]), om, t)
    finally:
        ctx.close()
    dk = 2 * np.pi / (n_omega - 1)
    for x, out in zip(F, got):
        ref = 2 * dk * np.einsum("npc,nt->tpc", x.astype(complex), np.exp(-2j * np.pi * np.outer(om, t))).real
        # test_idft_gpu.py's bound; the FP32 kernel's n_omega additions lie within it too
        bound = 2.0 ** -19 * 2 * dk * np.sum(np.abs(x.astype(complex)), axis=0)
        assert np.all(np.abs((out if host else out.cpu().numpy()) - ref) <= bound)


def test_transform_scratch_is_given_back():
    """A transform's scratch, held, does not refuse an evaluation that fits without it."""
    n_omega, n_points, n_t = 64, 20000, 512
    F = [torch.tensor(x, device="cuda") for x in _spectra(n_omega, n_points)]
    om, t = np.linspace(0.5, 1.5, n_omega), np.arange(n_t) / 8.0
    pts = np.random.default_rng(1).uniform(-1, 1, (600, 3))

    def evaluate(ctx):
        m = ctx.mirror(30.0, 0.0, 60.0, 32, 32)
        inc = ctx.incident(profile="gauss", w0=18.0, spectrum=dict(kind="sampled", omega=np.ones(1), amp=np.ones(1)))
        return ctx.eval(m, inc, [1.0], pts)

    def fits(budget, transform):
        ctx = sc.Context(0, budget_bytes=budget)
        try:
            if transform:
                ctx.time_domain(*F, om, t)
            evaluate(ctx)
            return True
        except sc.ScError as e:
            assert e.status == sc.SC_ERR_OOM
            return False
        finally:
            ctx.close()

    lo, hi = 1 << 14, 64 << 20  # the smallest budget of the evaluation alone
    while hi - lo > 1024:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if fits(mid, False) else (mid, hi)
    # a kilobyte for the bisection and what a transform keeps beside its scratch (wavenumbers, times)
    assert fits(max(hi + 1024 + 8 * (n_omega + n_t), 8 * (n_omega + n_t) + 8 * n_omega * n_t), True)
