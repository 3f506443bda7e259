"""What one extreme value may touch in the FP32 forms that slide along y: an output (forward) or a sample (adjoint) whose
windows do not hold it keeps the accuracy it has without it."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# volumes large enough for the forward's long runs; brick corners (xb, yb) of the second brick along x and along y
FORWARD = {8: ((20, 48, 96), (8, 32)), 16: ((9, 36, 96), (12, 32)), 32: ((4, 30, 64), (6, 32))}
RUN = {8: 8, 16: 16, 32: 8}   # outputs along y that share one recursion: a value leaves a rounding error to those after it


@pytest.fixture(scope="module")
def sal():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_06174_gb300 as s
    s.load()
    return s


def _features(sal, V, n, boundary="zero"):
    eng = sal.Saliency(V.shape, sal.Params(n=n, boundary=boundary))
    try:
        E = torch.empty((3,) + V.shape, device="cuda")
        sal.sal_local_spectra_project(eng.h, torch.from_numpy(V).cuda(), E)
        return E.cpu().numpy().astype(np.float64)
    finally:
        eng.close()


def _held(shape, p, n, more=0):
    """Outputs whose window holds sample p, or which lie up to `more` outputs behind such a one along y."""
    t, x, y = (np.arange(L) for L in shape)
    a, b, c = (t - n // 2 <= p[0]) & (p[0] < t + n // 2), (x - n // 2 <= p[1]) & (p[1] < x + n // 2), \
        (y - n // 2 - more <= p[2]) & (p[2] < y + n // 2)
    return a[:, None, None] & b[None, :, None] & c[None, None, :]


@pytest.mark.parametrize("value", [1e6, -1e30])
@pytest.mark.parametrize("at", ["corner", "inner", "both"])
@pytest.mark.parametrize("n", [8, 16])   # (32: every window of a brick holds all of its voxels)
def test_an_outlier_costs_other_windows_no_precision(sal, n, at, value):
    """Outliers at a brick's first voxel and at one in its middle: a few dozen FP32 roundings per feature elsewhere."""
    shape, (xb, yb) = FORWARD[n]
    r = np.random.RandomState(n)
    V = r.randn(*shape).astype(np.float32)
    t0 = shape[0] // 2
    spots = {"corner": [(t0, xb, yb)], "inner": [(t0, xb + n // 2 - 1, yb + n // 2 - 1)]}
    spots["both"] = spots["corner"] + spots["inner"]
    held = np.zeros(shape, bool)
    for p in spots[at]:
        V[p] = value
        held |= _held(shape, p, n, 15)
    near = np.zeros(shape, bool)   # the bricks that hold the spots, and those that begin behind them
    near[t0, xb - 4:xb + 14, yb - 4:yb + 36] = True
    pts = np.argwhere(near & ~held)
    pts = pts[r.permutation(len(pts))[:{8: 600, 16: 300}[n]]]
    got = _features(sal, V, n)[:, pts[:, 0], pts[:, 1], pts[:, 2]].T
    want = oracle.features_at(V, pts, n, boundary="zero")
    assert np.abs(got - want).max(initial=0) <= 32 * 2.0 ** -24 * np.abs(want).min()


ADJOINT_RUN = {8: 4, 16: 8}   # outputs along y whose gradients are formed from one run of sums


def _adjoint(sal, V, gE, n):
    eng = sal.Saliency(V.shape, sal.Params(n=n, boundary="zero"))
    try:
        gV = torch.empty(V.shape, device="cuda")
        sal.sal_local_spectra_project_backward(eng.h, torch.from_numpy(V).cuda(), torch.from_numpy(gE).cuda(), gV)
        return gV.cpu().numpy().astype(np.float64)
    finally:
        eng.close()


def _reached(shape, p, n, more=0):
    """Samples in the window of output p, or of one of the `more` outputs behind it along y."""
    a, b, c = ((np.arange(L) >= q - n // 2) & (np.arange(L) < q + n // 2 + m) for L, q, m in zip(shape, p, (0, 0, more)))
    return a[:, None, None] & b[None, :, None] & c[None, None, :]


@pytest.mark.parametrize("value", [1e5, 1e30])
@pytest.mark.parametrize("n,shape,p", [(8, (9, 30, 60), (4, 14, 16)), (8, (9, 30, 60), (4, 14, 21)),
                                       (16, (17, 40, 70), (8, 18, 16)), (16, (17, 40, 70), (8, 18, 34))])
def test_a_strong_gradient_costs_other_samples_no_precision(sal, n, shape, p, value):
    """One output's gradient far above the others': samples outside its window and those of the rest of its run keep the
    adjoint's bar of 1e-5 relative to what they are."""
    r = np.random.RandomState(n)
    V, gE = r.randn(*shape).astype(np.float32), r.randn(3, *shape).astype(np.float32)
    clean = _adjoint(sal, V, gE, n)
    gE[(slice(None),) + p] = value
    got, want = _adjoint(sal, V, gE, n), oracle.features_adjoint(V, gE, n, boundary="zero")
    far = ~_reached(shape, p, n, ADJOINT_RUN[n] - 1)
    rms = np.sqrt(np.mean(want[far] ** 2))
    assert np.abs(got - want)[far].max() <= 1e-5 * rms
    assert np.abs(got - clean)[far].max() <= 1e-5 * rms


@pytest.mark.parametrize("n,shape,p", [(8, (9, 30, 60), (4, 14, 16)), (16, (17, 40, 70), (8, 18, 16))])
def test_the_adjoint_keeps_a_nan_to_its_runs(sal, n, shape, p):
    """In a gradient: the samples of its run's windows.  In the volume: those of the runs of every output that holds it."""
    r = np.random.RandomState(n)
    V, gE = r.randn(*shape).astype(np.float32), r.randn(3, *shape).astype(np.float32)
    more = ADJOINT_RUN[n] - 1
    gE[(1,) + p] = np.nan
    bad = np.isnan(_adjoint(sal, V, gE, n))
    assert bad[_reached(shape, p, n)].all() and not bad[~_reached(shape, p, n, more)].any()
    gE[(1,) + p] = 1.0
    V[p] = np.nan
    bad = np.isnan(_adjoint(sal, V, gE, n))
    t, x, y = np.nonzero(bad)
    assert abs(t - p[0]).max() <= n and abs(x - p[1]).max() < n
    assert y.min() >= p[2] - n + 1 and y.max() <= p[2] + n - 1 + more


@pytest.mark.parametrize("value", [1e6, np.nan])
@pytest.mark.parametrize("n", [8, 16, 32])
def test_the_forward_keeps_an_extreme_value_to_its_runs(sal, n, value):
    """An outlier anywhere reaches the outputs of its windows and those of their runs; the others are what they are
    without it."""
    shape, (xb, yb) = FORWARD[n]
    r = np.random.RandomState(n)
    V = r.randn(*shape).astype(np.float32)
    p = (shape[0] // 2, xb + 2, yb + 3 - n // 2)   # in the windows of a brick's first outputs alone, so most of its run is free
    V[p] = 0.0
    clean = _features(sal, V, n)
    V[p] = value
    E = _features(sal, V, n)
    own, free = _held(shape, p, n), ~_held(shape, p, n, RUN[n] - 1)
    if np.isnan(value):
        assert np.isnan(E[:, own]).all()
    # two roundings of a feature, a few dozen 2^-24 each (another value may be taken from a brick at staging)
    assert np.abs(E - clean)[:, free].max() <= 64 * 2.0 ** -24 * clean[:, free].min()


@pytest.mark.parametrize("n", [8, 16])
def test_windows_of_zeros_have_no_gradient(sal, n):
    """A muted volume: zeros behind the samples along y, and beside them.  Outputs whose windows hold nothing else get no
    gradient through |F| = 0, wherever in a run they lie."""
    r = np.random.RandomState(n)
    shape = (5, 20, 3 * n + 21)
    for end in range(n // 2, n // 2 + 9):
        V, gE = np.zeros(shape, np.float32), r.randn(3, *shape).astype(np.float32)
        V[:, 4:9, :end] = r.randn(5, 5, end)
        got = _adjoint(sal, V, gE, n)
        assert (got[:, :, end + 2 * n - 1:] == 0).all()
        want = oracle.features_adjoint(V, gE, n, boundary="zero")
        assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
