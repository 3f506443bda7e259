"""hbm_budget_bytes: what once held a handle still does, forward and backward, whatever tables the faster forms have since
brought."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SHAPE = (4, 5, 6)


@pytest.fixture(scope="module")
def sal():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_06174_gb300 as s
    s.load()
    return s


# the scratch of a 4 x 5 x 6 handle when the direct forms were all there was: 24 bytes a voxel, 195,072 bytes for the
# reductions and each precision's tables
@pytest.mark.parametrize("prec,n,held", [("fp32", 8, 200352), ("fp32", 16, 213504), ("fp32", 32, 197952),
                                         ("bf16", 8, 234880), ("fp16", 16, 253472), ("bf16", 32, 197952)])
@pytest.mark.parametrize("short", [0, 1])
def test_a_budget_that_held_a_handle_still_does(sal, prec, n, held, short):
    V, _ = synth.volume(synth.small_spec(SHAPE, seed=n, faults=1))
    budget = held
    if n < 32:   # the gradient's scratch on top: three maps, partial sums, and one plane of bricks of the direct form
        by = 16 if n == 16 or prec != "fp32" else 32
        bx = 1 if prec == "fp32" else 128 // n
        xh, yh = bx + n - 1, by + n - 1
        per_ext = -(-SHAPE[1] // bx) * -(-xh * yh // 4) * 16
        budget += 12 * int(np.prod(SHAPE)) + 1216 * 64 * 8 + 2 * n * per_ext
    eng = sal.Saliency(SHAPE, sal.Params(n=n, prec=prec, hbm_budget_bytes=budget if not short else held))
    try:
        tol = 1e-5 if prec == "fp32" else 1e-2
        E = eng.local_spectra_project(torch.from_numpy(V)).cpu().numpy()
        want = oracle.features(V, n)
        assert np.linalg.norm(E - want) <= tol * np.linalg.norm(want)
        assert sal.sal_workspace_size(eng.h) <= held
        if n < 32 and not short:
            gE = synth.random_volume((3,) + SHAPE, seed=2)
            gV = torch.empty(SHAPE, device="cuda")
            sal.sal_local_spectra_project_backward(eng.h, torch.from_numpy(V).cuda(), torch.from_numpy(gE).cuda(), gV)
            want = oracle.features_adjoint(V, gE, n)
            assert np.linalg.norm(gV.cpu().numpy() - want) <= (tol if prec == "fp32" else 5e-2) * np.linalg.norm(want)
            assert sal.sal_workspace_size(eng.h) <= budget
    finally:
        eng.close()
