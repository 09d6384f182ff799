"""The tensor-core inverse transform over the whole range of FP32: values next to
ordinary ones whose entries are the largest and smallest that FP32 holds.  (The FP32
kernel of small transforms adds subnormal values on FP32's own grid of 2^-149, with a
rounding per addition.)

The bound is that of test_idft_gpu.py, 2^-19 of 2 dk sum |F| per value, and for
subnormal results 2^-149: half of that for the rounding of the sum, which 2 dk < 1
makes no larger, and half for that of the product."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1609_08146_gb300 as sc  # noqa: E402

SIZES = [1.0, 1e-30, 1e-33, 1e-35, 1e-37, 1e-40, 3e-44, 1e30, 7e34, 9e34, 1e35, 1e36]


@pytest.fixture(scope="module")
def ctx():
    c = sc.Context(0)
    yield c
    c.close()


def _check(F, om, t, out):
    dk = 2 * np.pi * (om[-1] - om[0]) / (om.size - 1)
    ref = 2 * dk * np.einsum("npc,nt->tpc", F.astype(complex), np.exp(-2j * np.pi * np.outer(om, t))).real
    bound = 2.0 ** -19 * 2 * dk * np.sum(np.abs(F.astype(complex)), axis=0) + 2.0 ** -149
    assert np.all(np.abs(out.cpu().numpy() - ref) <= bound)


@pytest.mark.parametrize("n_t", [200, 512])
@pytest.mark.parametrize("dtype", [np.complex64, np.complex128])
def test_values_of_every_size(ctx, n_t, dtype):
    rng = np.random.default_rng(n_t)
    size = np.array(SIZES * 2, dtype=np.float32)[None, :, None]
    r = rng.normal(size=(64, size.size, 3, 2)).astype(np.float32) * size[..., None]
    F = (r[..., 0] + 1j * r[..., 1]).astype(np.complex64)
    om, t = np.linspace(0.5, 1.5, 64), np.arange(n_t) / 8.0 - 4.0
    out, _ = ctx.time_domain(torch.tensor(F.astype(dtype), device="cuda"), None, om, t,
                             precision="fp32" if dtype == np.complex64 else "fp64")
    _check(F, om, t, out)


@pytest.mark.parametrize("n_t", [33, 512])
def test_largest_entry(ctx, n_t):
    """One entry of the largest binade: the sum and its product with 2 dk stay finite."""
    F = np.ones((64, 2, 3), dtype=np.complex64)
    F[17, 0] = 3e38
    om, t = np.linspace(0.5, 1.5, 64), np.arange(n_t) / 8.0 - 4.0
    out, _ = ctx.time_domain(torch.tensor(F, device="cuda"), None, om, t)
    _check(F, om, t, out)
