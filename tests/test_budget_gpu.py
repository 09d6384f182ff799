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


def _smallest(run, lo=1 << 14, hi=64 << 20):
    """Smallest budget (to 2 KB) with which run(ctx) is not refused."""
    def fits(budget):
        ctx = sc.Context(0, budget_bytes=budget)
        try:
            run(ctx)
            return True
        except sc.ScError as e:
            assert e.status == sc.SC_ERR_OOM
            return False
        finally:
            ctx.close()

    while hi - lo > 2048:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if fits(mid) else (mid, hi)
    return hi


def _request(ctx, n_omega, n_points, n=64):
    om = np.ones(1) if n_omega == 1 else np.linspace(0.5, 1.5, n_omega)
    m = ctx.mirror(30.0, 0.0, 60.0, n, n)
    inc = ctx.incident(profile="gauss", w0=18.0, spectrum=dict(kind="sampled", omega=om, amp=np.ones(n_omega)))
    return m, inc, om, torch.tensor(np.random.default_rng(n_points).uniform(-1, 1, (n_points, 3)), device="cuda")


def _needs(n_omega, n_points, n=64):
    """Node table (40 and 80 bytes a node, whole tiles, one rim) and the workspace of one split and the rim, and a
    launch's descriptors, spectrum and slack."""
    return (n * n + -(-n // 32) * 32) * 120 + 2 * n_points * n_omega * 96 + (80 << 10)


@pytest.mark.parametrize("n_omega,n_points", [(1, 1024), (3, 300), (8, 1024), (24, 100), (25, 16), (64, 1024), (256, 100)])
def test_splits_never_refuse_a_request(n_omega, n_points):
    """More node splits are faster but need more workspace: a request runs where one split fits, and with room
    for no more than that its result is that of any other split count to the FP32 path's rounding."""
    assert _smallest(lambda ctx: ctx.eval(*_request(ctx, n_omega, n_points))) <= _needs(n_omega, n_points)
    out = []
    for budget in (0, _needs(n_omega, n_points)):
        ctx = sc.Context(0, budget_bytes=budget)
        out.append(ctx.eval(*_request(ctx, n_omega, n_points)))
        ctx.close()
    for a, b in zip(*out):
        # two FP32 sums, each within the path's 1e-5 of the peak
        assert (a - b).abs().max() <= 2e-5 * b.abs().max()


def test_batch_runs_where_its_requests_do():
    """A batch's launches are cut to what the budget holds."""
    shapes = [(1 + 7 * i % 50, 40 + 13 * i) for i in range(12)]
    tables = 12 * _needs(1, 0)
    largest = max(_needs(*s) - _needs(1, 0) for s in shapes)
    # (and every request's spectrum and descriptors)
    assert _smallest(lambda ctx: ctx.eval_batch([_request(ctx, *s) for s in shapes])) <= tables + largest + (64 << 10)


def test_workspace_is_given_back():
    """The workspace that one call leaves does not refuse a call that fits without it."""
    n_points = 40000
    pts = np.random.default_rng(1).uniform(-1, 1, (n_points, 3))

    def both(ctx):
        r = _request(ctx, 8, 1024)
        ctx.eval(*r)  # the most splits that fit
        ctx.eval(r[0], r[1], r[2][:1], pts)  # host points and outputs: 24 + 48 bytes a point
    assert _smallest(both) <= _needs(1, n_points) + 72 * n_points
