"""Adaptive weights where a chain is near singular or grows: the weights do not depend on whether the errors are asked for,
and both follow the FP64 oracle's sequential filters."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sal():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_06174_gb300 as s
    s.load()
    return s


def _run(sal, S3, D, **kw):
    shape = S3.shape[1:]
    eng = sal.Saliency(shape, sal.Params(n=2))
    try:
        nblk = -(-shape[2] // kw["sections"]) if kw.get("sections") else 1
        W, W_only = (torch.empty((nblk, 3), device="cuda") for _ in range(2))
        err2 = torch.empty(int(np.prod(shape)), device="cuda")
        S3d, Dd = torch.from_numpy(S3).cuda(), torch.from_numpy(D).cuda()
        sal.sal_adapt_weights(eng.h, S3d, Dd, W, err2=err2, **kw)
        sal.sal_adapt_weights(eng.h, S3d, Dd, W_only, **kw)
        return W.cpu().numpy(), W_only.cpu().numpy(), err2.cpu().numpy().astype(np.float64)
    finally:
        eng.close()


def _filter(S3, D, sections=0, **kw):
    """The oracle's filters on maps normalised as FP32 features are, y blocks of `sections`."""
    lo, hi = S3.reshape(3, -1).min(1).astype(np.float64), S3.reshape(3, -1).max(1).astype(np.float64)
    x = (S3.astype(np.float64) - lo[:, None, None, None]) / (hi - lo)[:, None, None, None]
    sec = sections or S3.shape[3]
    out = [oracle.adapt_weights(x[..., y:y + sec], D[..., y:y + sec], return_trace=True, **kw)
           for y in range(0, S3.shape[3], sec)]
    return np.array([w for w, _ in out]), np.concatenate([e for _, e in out])


@pytest.mark.parametrize("seed", range(4))
def test_weights_do_not_depend_on_the_errors_being_asked_for(sal, seed):
    """RLS whose maps are one map in the first sections (near singular there) and almost one behind them (pivots of 1e-6 of
    the trace, above the level of 1e-7 where the regrouped sums are left alone)."""
    r = np.random.RandomState(seed)
    shape = (32, 32, 24)
    S3 = np.repeat(r.rand(1, *shape).astype(np.float32), 3, 0)
    S3[1:, :, :, 12:] += (3e-3 * r.randn(2, 32, 32, 12)).astype(np.float32)
    S3[:, 0, 0, 0], S3[:, 1, 0, 0] = -0.05, 1.05   # the same bounds for all
    D = (S3[0] + 0.1 * r.randn(*shape)).astype(np.float32)
    W, W_only, err2 = _run(sal, S3, D, method="rls")
    assert np.array_equal(W, W_only)
    _, want = _filter(S3, D, method="rls")
    assert np.linalg.norm(err2 - want) <= 1e-4 * np.linalg.norm(want)


@pytest.mark.parametrize("sections", [0, 3])
def test_a_chain_that_grows_follows_the_filter(sal, sections):
    """LMS a little beyond its stability limit: finite weights that have grown by orders of magnitude."""
    r = np.random.RandomState(7)
    S3, D = r.rand(3, 6, 5, 9).astype(np.float32), r.rand(6, 5, 9).astype(np.float32)
    W, W_only, err2 = _run(sal, S3, D, method="lms", sections=sections, mu=2.2)
    want, want_e = _filter(S3, D, sections, method="lms", mu=2.2)
    assert np.isfinite(want).all() and np.abs(want).max() > 1e3
    assert np.array_equal(W, W_only, equal_nan=True)
    # x carries the 1e-7 of an FP32 reciprocal, up to 270 steps of it
    assert np.abs(W - want).max() <= 270 * 1e-6 * np.abs(want).max()
    assert np.linalg.norm(err2 - want_e) <= 2 * 270 * 1e-6 * np.linalg.norm(want_e)


@pytest.mark.parametrize("method,shape,regrouped", [
    ("lms", (16, 17, 3), True), ("lms", (15, 18, 3), False), ("lms", (12, 16, 20), False),
    ("nlms", (8, 17, 5), True), ("nlms", (9, 15, 5), False), ("rls", (8, 8, 9), True), ("rls", (7, 9, 9), False),
])
def test_short_chains_run_step_by_step(sal, method, shape, regrouped):
    """On both sides of the chain length from which the regrouped form's launches cost less than the filter's steps (two
    launches, the bounds and the filter): the same values."""
    r = np.random.RandomState(3)
    S3 = (np.abs(r.randn(3, *shape)) * 0.2 + 0.05).astype(np.float32)
    D = (S3[0] * 1.5 + 0.1 * r.randn(*shape)).astype(np.float32)
    before = sal.sal_launch_count()
    W, W_only, err2 = _run(sal, S3, D, method=method, sections=1)
    assert sal.sal_launch_count() - before == (5 + 4 if regrouped else 2 + 2)
    want, want_e = _filter(S3, D, 1, method=method)
    assert np.array_equal(W, W_only)
    assert np.abs(W - want).max() <= 1e-5 * max(1.0, np.abs(want).max())
    assert np.linalg.norm(err2 - want_e) <= 1e-5 * np.linalg.norm(want_e)
