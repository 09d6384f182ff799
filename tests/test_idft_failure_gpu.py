"""A lost copy in the tensor-core inverse transform: its bounded wait runs out, a
call with host outputs reports SC_ERR_TIMEOUT instead of returning whatever its
buffers hold, one with device outputs through the next call that synchronizes, and
the next transform equals one made before."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1609_08146_gb300 as sc  # noqa: E402


@pytest.mark.parametrize("n_t", [100, 300])
@pytest.mark.parametrize("stage", [0, 2, 3, 5])
@pytest.mark.parametrize("host", [True, False])
def test_lost_table_stage(n_t, stage, host):
    ctx = sc.Context(0)
    try:
        rng = np.random.default_rng(stage)
        F = [(rng.normal(size=(96, 100, 3)) + 1j * rng.normal(size=(96, 100, 3))).astype(np.complex64) for _ in range(2)]
        om, t = np.linspace(0.5, 1.5, 96), np.arange(n_t) / 8.0
        if not host:
            F = [torch.tensor(x, device="cuda") for x in F]
        before = [x.copy() if host else x.clone() for x in ctx.time_domain(*F, om, t)]
        ctx.set_option(sc.SC_OPT_FAIL_COPY, stage)
        t0 = time.time()
        with pytest.raises(sc.ScError) as e:
            ctx.time_domain(*F, om, t)
            if not host:
                ctx.counters()
        assert e.value.status == sc.SC_ERR_TIMEOUT
        assert 0.5 < time.time() - t0 < 5.0
        ctx.set_option(sc.SC_OPT_FAIL_COPY, -1)
        for a, b in zip(before, ctx.time_domain(*F, om, t)):
            assert np.array_equal(a, b) if host else torch.equal(a, b)
    finally:
        ctx.close()
