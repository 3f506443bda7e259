"""The FP32 adjoint's bricks with more small bins than they list (constant regions: every bin but DC), n = 8 and 16: values
against the FP64 oracle over ragged bricks, border extensions, lattice planes and several slabs, and what they cost."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
RTOL = 1e-5   # the bar of the FP32 adjoint
BRICK = {8: (16, 23, 23), 16: (12, 27, 31)}   # x0 of a brick, extents of its block along x and y; 16 outputs along y


@pytest.fixture(scope="module")
def sal():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_06174_gb300 as s
    s.load()
    return s


def _half_constant(shape, seed=3):
    """A seismic volume whose far half along y is one value."""
    V, _ = synth.volume(synth.small_spec(shape, seed=seed, faults=1))
    V = np.ascontiguousarray(V, np.float32)
    V[:, :, shape[2] // 2:] = 0.375
    return V


def _adjoint(sal, V, gE, **params):
    eng = sal.Saliency(V.shape, sal.Params(**params))
    try:
        gV = torch.empty(V.shape, dtype=torch.float32, device="cuda")
        sal.sal_local_spectra_project_backward(eng.h, torch.from_numpy(V).cuda(), torch.from_numpy(gE).cuda(), gV)
        torch.cuda.synchronize()
        return gV.cpu().numpy().astype(np.float64)
    finally:
        eng.close()


@pytest.mark.parametrize("n,shape,boundary,stride,planes", [
    (8, (9, 18, 70), "symmetric", 1, 0), (8, (10, 5, 52), "periodic", 1, 0), (8, (9, 37, 45), "zero", 1, 0),
    (8, (11, 17, 50), "symmetric", 2, 0), (8, (9, 18, 50), "symmetric", 1, 2),
    (16, (18, 13, 50), "zero", 1, 0), (16, (17, 25, 48), "periodic", 2, 0), (16, (18, 14, 40), "symmetric", 1, 3),
])
def test_dense_bricks_match_oracle(sal, n, shape, boundary, stride, planes):
    """planes > 0: a budget that holds that many planes of bricks at a time."""
    V = _half_constant(shape)
    inside = shape[2] - shape[2] // 2 - n   # outputs along y of every (t0, x0) whose window holds nothing else
    assert max(0, inside // stride) * (n // 2 + 1) * n * n > 1024
    assert oracle.band_count(V, n, boundary, lo=2.0 ** -40, hi=2.0 ** -36).sum() == 0
    gE = synth.random_volume((3,) + shape, seed=n + 9)
    budget = 0
    if planes:
        base = sal.Saliency(shape, sal.Params(n=n, boundary=boundary))
        created = sal.sal_workspace_size(base.h)
        base.close()
        bx, xh, yh = BRICK[n]
        per_ext = -(-shape[1] // bx) * -(-shape[2] // 16) * -(-xh * yh // 4) * 16
        budget = created + 12 * int(np.prod(shape)) + 1216 * 64 * 8 + (n - 1) * per_ext + (n + 1) * per_ext * planes
    got = _adjoint(sal, V, gE, n=n, boundary=boundary, stride=stride, hbm_budget_bytes=budget)
    want = oracle.features_adjoint(V, gE, n, boundary=boundary, stride=stride)
    assert np.linalg.norm(got - want) <= RTOL * np.linalg.norm(want)


@pytest.mark.parametrize("n", [8, 16])
def test_dense_bricks_are_spread_over_the_device(sal, n):
    """A few constant bricks against a textured volume of the same size: 3 (n = 8) and 8 (n = 16) times as long with separable
    float-float spectra, 23 and 430 with a direct sum per bin, 100 and 2900 with those by one CTA per brick.  And bricks
    with a few hundred to a thousand small bins (a lone sample): 2 and 7 times as long, 6 and 150 with a CTA per x position,
    20 and 700 with one per brick."""
    shape = (6, 8, 10)
    gE = torch.from_numpy(synth.random_volume((3,) + shape, seed=1)).cuda()
    gV = torch.empty(shape, device="cuda")
    eng = sal.Saliency(shape, sal.Params(n=n))

    def run(V):
        times = []
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            sal.sal_local_spectra_project_backward(eng.h, V, gE, gV)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)
    try:
        textured = run(torch.from_numpy(synth.random_volume(shape, seed=2)).cuda())
        constant = run(torch.full(shape, 0.375, device="cuda"))
        lone = torch.zeros(shape, device="cuda")
        lone[0, 0, 0] = 1.0
        lone = run(lone)
    finally:
        eng.close()
    assert constant <= 50 * textured
    assert lone <= (5 if n == 8 else 50) * textured


@pytest.mark.parametrize("n,shape,boundary,share", [(8, (12, 16, 20), "symmetric", 0.05), (8, (12, 16, 20), "zero", 0.01),
                                                    (8, (9, 18, 40), "periodic", 0.02), (16, (12, 16, 20), "symmetric", 0.01),
                                                    (16, (18, 13, 35), "zero", 0.002)])
def test_bricks_of_sparse_volumes_match_oracle(sal, n, shape, boundary, share):
    """Isolated samples: cubes that hold few of them have many bins that are zero, of which some bricks list up to the
    limit and others more."""
    r = np.random.RandomState(n)
    V = (r.randn(*shape) * (r.rand(*shape) < share)).astype(np.float32)
    V[0, 0, 0] = 1.0
    assert oracle.band_count(V, n, boundary, lo=2.0 ** -40, hi=2.0 ** -36).sum() == 0
    gE = synth.random_volume((3,) + shape, seed=n + 9)
    got, want = _adjoint(sal, V, gE, n=n, boundary=boundary), oracle.features_adjoint(V, gE, n, boundary=boundary)
    assert np.linalg.norm(got - want) <= RTOL * np.linalg.norm(want)
