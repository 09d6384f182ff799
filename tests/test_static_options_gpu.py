"""sc_eval_fp32_static takes the kernel that the context's options leave it, as
sc_eval does: with one node split and the same options both give the same bits (the
grids' steps and wavenumbers are exact).  It never cuts its omegas, so sc_eval, which
cuts 100 of them when the tensor kernel is off, is asked not to."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1609_08146_gb300 as sc  # noqa: E402


@pytest.mark.parametrize("n_omega", [24, 25, 64, 100, 256])
@pytest.mark.parametrize("options", [{}, {sc.SC_OPT_TILE_LAYOUT: 0}, {sc.SC_OPT_OMEGA_CHUNKS: 0}])
def test_same_kernel_as_sc_eval(n_omega, options):
    ctx = sc.Context(0)
    try:
        for k, v in {sc.SC_OPT_AUTOTUNE: 0, sc.SC_OPT_NODES_PER_SPLIT: 32 * 32, **options}.items():
            ctx.set_option(k, v)
        om = 0.5 + np.arange(n_omega) / 256.0
        amp = np.exp(1j * np.arange(n_omega))
        m = ctx.mirror(100.0, 0.0, 200.0, 32, 32)
        inc = ctx.incident(profile="gauss", w0=60.0, spectrum=dict(kind="sampled", omega=om, amp=amp))
        P = torch.tensor(np.random.default_rng(n_omega).uniform(-1, 1, (37, 3)), device="cuda")
        if options:
            ctx.set_option(sc.SC_OPT_OMEGA_CHUNKS, 0)
        E, B, st = ctx.eval(m, inc, om, P, stats=True)
        ctx.set_option(sc.SC_OPT_OMEGA_CHUNKS, options.get(sc.SC_OPT_OMEGA_CHUNKS, 1))
        assert (st["kernel_class"] >= 30) == (n_omega >= 25 and not options)
        Es, Bs = torch.empty_like(E), torch.empty_like(B)
        a = torch.tensor(ctx.spectrum(inc, om), device="cuda")
        ctx._check(ctx._lib.sc_eval_fp32_static(ctx._h, m._h, inc._h, om[0], om[1] - om[0], n_omega,
                                                ctypes.cast(a.data_ptr(), sc._DP), P.data_ptr(), P.shape[0],
                                                Es.data_ptr(), Bs.data_ptr()))
        torch.cuda.synchronize()
        assert torch.equal(E, Es) and torch.equal(B, Bs)
    finally:
        ctx.close()
