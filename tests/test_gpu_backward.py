"""GPU parity of the backward (differentiation form) against the FP64 oracle adjoint, through the
C ABI, plus central finite differences of the GPU forward and a weight-fitting run.

Tolerances (FP32 path): relative L2 <= 1e-5 for each step's adjoint.  The sign of each
center-surround difference (a kink of |.|) is an integer-valued decision: the step tests feed
both sides the same FP32 features and FP32 weights, so both take it on identical numbers.

The oracle takes the zero subgradient of |F| only where F = 0 up to FP64 rounding (2^-40 of the
window L1 norm).  The inputs below hold, by construction of the border extension and by chance,
many cubes with bins between that level and 2^-17 L1, where FP32 has no usable direction F/|F|:
the FP32 adjoint resolves those bins exactly (integer test for the bins that vanish for every
input, FP64 recompute for the rest), and the tests assert from the oracle that such bins are
present, so the 1e-5 bar is met on ill-conditioned cubes, not around them.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
RTOL = 1e-5


def rel_l2(a, b):
    a = np.asarray(a, np.float64)
    b = np.asarray(b, np.float64)
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


@pytest.fixture(scope="module")
def sal():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_06174_gb300 as s
    s.load()
    return s


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()


# brick sizes along y of the spectral adjoint (used to force several t-slabs through the budget)
_BY = {2: 32, 4: 32, 8: 32, 16: 16}


@pytest.mark.parametrize("n,shape,boundary,slabs", [
    (2, (5, 6, 40), "symmetric", 1),
    (4, (7, 5, 37), "periodic", 1),
    (4, (6, 9, 20), "zero", 3),
    (8, (10, 9, 45), "symmetric", 1),
    (8, (9, 7, 33), "symmetric", 4),
    (16, (6, 5, 21), "symmetric", 1),
    (16, (5, 4, 17), "periodic", 2),
])
def test_spectral_adjoint_matches_oracle(sal, n, shape, boundary, slabs):
    V, _ = synth.volume(synth.small_spec(shape, seed=n + 100, faults=1))
    gE = synth.random_volume((3,) + shape, seed=n + 7)
    budget = 0
    if slabs > 1:
        # gE (3 planes), the reduction partials, n - 1 fixed overlap-add planes, and per t-plane of a slab
        # the brick blocks (n slices of n x (BY + n - 1) floats, padded to 4) plus one overlap-add plane
        nseg = -(-shape[2] // _BY[n])
        per_ext = shape[1] * nseg * (-(-n * (_BY[n] + n - 1) // 4) * 4) * 4
        per_t = n * per_ext
        base = sal.Saliency(shape, sal.Params(n=n, boundary=boundary))
        created = sal.sal_workspace_size(base.h)
        base.close()
        N = int(np.prod(shape))
        budget = (created + 3 * N * 4 + 1216 * 64 * 8 + (n - 1) * per_ext
                  + (per_t + per_ext) * max(1, shape[0] // slabs))
    eng = sal.Saliency(shape, sal.Params(n=n, boundary=boundary, hbm_budget_bytes=budget))
    try:
        gV = torch.empty(shape, dtype=torch.float32, device="cuda")
        sal.sal_local_spectra_project_backward(eng.h, _cuda(V), _cuda(gE), gV)
        torch.cuda.synchronize()
        got = gV.cpu().numpy()
    finally:
        eng.close()
    ref = oracle.features_adjoint(V, gE, n, boundary=boundary)
    assert rel_l2(got, ref) <= RTOL, rel_l2(got, ref)


@pytest.mark.parametrize("n,shape,boundary,source", [
    (8, (9, 7, 33), "symmetric", "seismic"),
    (8, (16, 16, 40), "symmetric", "seismic"),
    (16, (6, 5, 21), "symmetric", "seismic"),
    (16, (20, 20, 40), "symmetric", "seismic"),
    (16, (9, 8, 24), "symmetric", "random"),
    (16, (17, 18, 40), "periodic", "seismic"),
    (16, (20, 20, 40), "symmetric", "half-constant"),
])
def test_spectral_adjoint_ill_conditioned_cubes(sal, n, shape, boundary, source):
    """Inputs the oracle shows to hold cubes with small non-zero bins (2^-40 < |F| / L1 <= 2^-17) and,
    under the symmetric extension, bins that vanish for every input: the whole gradient at 1e-5.  The
    half-constant volume (a seismic volume whose far half along y is one value) adds cubes whose every
    non-DC bin is zero, many more small bins per brick than the per-brick list of the listed-bin pass holds,
    so those bricks resolve their bins themselves."""
    if source == "seismic":
        V, _ = synth.volume(synth.small_spec(shape, seed=3, faults=1))
    elif source == "half-constant":
        V, _ = synth.volume(synth.small_spec(shape, seed=3, faults=1))
        V = np.ascontiguousarray(V, np.float32)
        V[:, :, shape[2] // 2:] = 0.375
    else:
        V = synth.random_volume(shape, seed=0)
    small = oracle.band_count(V, n, boundary)
    assert small.sum() > 0, "the input holds no ill-conditioned cube"
    # the kernel takes F = 0 at 2^-36 of the L1 norm after its float-float recompute, the oracle at 2^-40:
    # the two decisions can differ only for bins between the two levels, and the input holds none
    assert oracle.band_count(V, n, boundary, lo=2.0 ** -40, hi=2.0 ** -36).sum() == 0
    gE = synth.random_volume((3,) + shape, seed=n + 9)
    eng = sal.Saliency(shape, sal.Params(n=n, boundary=boundary))
    try:
        gV = torch.empty(shape, dtype=torch.float32, device="cuda")
        sal.sal_local_spectra_project_backward(eng.h, _cuda(V), _cuda(gE), gV)
        torch.cuda.synchronize()
        got = gV.cpu().numpy()
    finally:
        eng.close()
    ref = oracle.features_adjoint(V, gE, n, boundary=boundary)
    assert rel_l2(got, ref) <= RTOL, (rel_l2(got, ref), int((small > 0).sum()))


@pytest.mark.parametrize("n,shape,taper,prec,tol", [
    (8, (6, 7, 70), "hann", "fp32", RTOL),
    (16, (5, 6, 40), "hann", "fp32", RTOL),
    (16, (5, 6, 40), "hann", "bf16", 1e-2),
    (8, (4, 5, 150), "rect", "fp32", RTOL),
    (16, (3, 4, 100), "rect", "fp32", RTOL),
])
def test_spectral_adjoint_taper_and_long_rows(sal, n, shape, taper, prec, tol):
    """The Hann taper (the FP32 adjoint recomputes the forward stage 3 by the direct sum there) and rows of
    many y bricks (the sliding recomputation restarts from a direct sum for every run of outputs)."""
    V, _ = synth.volume(synth.small_spec(shape, seed=n + 31, faults=2))
    gE = synth.random_volume((3,) + shape, seed=n + 32)
    eng = sal.Saliency(shape, sal.Params(n=n, taper=taper, prec=prec))
    try:
        gV = torch.empty(shape, dtype=torch.float32, device="cuda")
        sal.sal_local_spectra_project_backward(eng.h, _cuda(V), _cuda(gE), gV)
        torch.cuda.synchronize()
        got = gV.cpu().numpy()
    finally:
        eng.close()
    ref = oracle.features_adjoint(V, gE, n, taper=taper)
    assert rel_l2(got, ref) <= tol, rel_l2(got, ref)


# the sliding adjoint's bricks (n = 8: 16 x0 by 16 y0; 16: 12 by 16, two to a CTA) past their edges, an odd brick over,
# cubes larger than the volume, every border extension, lattice planes
@pytest.mark.parametrize("feature", ["abs", "energy"])
@pytest.mark.parametrize("n,shape,boundary,stride", [
    (8, (3, 17, 17), "symmetric", 1), (8, (2, 33, 40), "zero", 1), (8, (9, 5, 3), "periodic", 1),
    (8, (7, 18, 33), "symmetric", 3), (16, (3, 13, 17), "zero", 1), (16, (2, 25, 33), "symmetric", 1),
    (16, (17, 3, 5), "periodic", 1), (16, (5, 12, 19), "periodic", 2), (16, (1, 1, 16), "zero", 1),
])
def test_sliding_adjoint_bricks_match_oracle(sal, n, shape, boundary, stride, feature):
    r = np.random.RandomState(n + sum(shape))
    V, gE = r.randn(*shape).astype(np.float32) + 0.3, r.randn(3, *shape).astype(np.float32)
    eng = sal.Saliency(shape, sal.Params(n=n, boundary=boundary, stride=stride, feature=feature))
    try:
        gV = torch.empty(shape, dtype=torch.float32, device="cuda")
        sal.sal_local_spectra_project_backward(eng.h, _cuda(V), _cuda(gE), gV)
        torch.cuda.synchronize()
        got = gV.cpu().numpy()
    finally:
        eng.close()
    want = oracle.features_adjoint(V, gE, n, boundary=boundary, feature=feature, stride=stride)
    assert rel_l2(got, want) <= RTOL


def test_adjoint_within_a_budget_the_sliding_form_exceeds(sal):
    """One x position: the sliding form's bricks take more scratch than the direct form's, which then runs."""
    shape, n = (6, 1, 40), 16
    V, gE = synth.random_volume(shape, seed=1), synth.random_volume((3,) + shape, seed=2)
    base = sal.Saliency(shape, sal.Params(n=n))
    created = sal.sal_workspace_size(base.h)
    base.close()
    per_ext = 3 * 496 * 4   # three y segments of 16 x 31 floats; a block holds n of them
    budget = created + 3 * int(np.prod(shape)) * 4 + 1216 * 64 * 8 + (n - 1) * per_ext + n * per_ext + per_ext
    eng = sal.Saliency(shape, sal.Params(n=n, hbm_budget_bytes=budget))
    try:
        gV = torch.empty(shape, dtype=torch.float32, device="cuda")
        sal.sal_local_spectra_project_backward(eng.h, _cuda(V), _cuda(gE), gV)
        torch.cuda.synchronize()
        assert rel_l2(gV.cpu().numpy(), oracle.features_adjoint(V, gE, n)) <= RTOL
    finally:
        eng.close()


@pytest.mark.parametrize("boundary,shape", [("symmetric", (9, 8, 35)), ("periodic", (9, 8, 35)), ("zero", (9, 8, 35)),
                                            ("symmetric", (20, 24, 70)), ("periodic", (20, 24, 70)),
                                            ("zero", (19, 27, 66))])
def test_center_surround_adjoint_matches_oracle(sal, boundary, shape):
    """Volumes too small to fill the GPU with tiles: the row kernel, interior and border voxels."""
    _check_center_surround_adjoint(sal, boundary, shape, sal.Params(n=4, boundary=boundary, alpha=[1.0, 0.7, 1.3]))


@pytest.mark.parametrize("boundary", ["symmetric", "periodic", "zero"])
def test_center_surround_adjoint_tiled_kernel(sal, boundary):
    """A volume whose 16 x 16 x 8 tiles fill two waves of the GPU (smaller ones take the row kernel), with
    ragged tiles on every axis; E and gS random (the adjoint takes any E).  gE and the direction gradients
    together: the tiled kernel also sums the weight-gradient terms (one pass over E and gS)."""
    shape = (100, 130, 150)
    E32 = np.abs(synth.random_volume((3,) + shape, seed=21)).astype(np.float32)
    gS3 = synth.random_volume((3,) + shape, seed=22)
    alpha = [1.0, 0.7, 1.3]
    params = sal.Params(n=4, boundary=boundary, alpha=alpha)
    offs, g, did, _ = oracle.dcs_stencil(params.directions, params.R, params.sigma, alpha)
    w32 = (np.asarray(alpha, np.float32)[did] * g.astype(np.float32)).astype(np.float64)
    eng = sal.Saliency(shape, params)
    try:
        gE = torch.empty((3,) + shape, dtype=torch.float32, device="cuda")
        ga = torch.empty(3, dtype=torch.float32, device="cuda")
        sal.sal_center_surround_backward(eng.h, _cuda(E32), _cuda(gS3), gE, ga)
        torch.cuda.synchronize()
    finally:
        eng.close()
    refE, gw = oracle.center_surround_adjoint(E32, gS3, offs, w32, boundary)
    ref_ga = oracle.direction_gradient(gw, g.astype(np.float32), did)
    assert rel_l2(gE.cpu().numpy(), refE) <= RTOL
    assert rel_l2(ga.cpu().numpy(), ref_ga) <= RTOL


@pytest.mark.parametrize("boundary", ["symmetric", "zero"])
def test_center_surround_adjoint_wide_in_plane_window(sal, boundary):
    """An in-plane window of 8 steps each way (the largest offset the library takes) on a volume the tiled
    kernel takes: its planes (32 x 32 with the halo) are larger than what it prefetches into registers, so
    the rest of each plane is loaded at store time."""
    params = sal.Params(n=4, boundary=boundary, directions=((0, 1, 0), (0, 0, 1)), R=8, alpha=[1.1, 0.9])
    _check_center_surround_adjoint(sal, boundary, (8, 520, 440), params, random_e=True)


def _check_center_surround_adjoint(sal, boundary, shape, params, random_e=False):
    if random_e:
        E32 = np.abs(synth.random_volume((3,) + shape, seed=5)).astype(np.float32)
    else:
        V, _ = synth.volume(synth.small_spec(shape, seed=5, faults=1))
        E32 = oracle.features(V, 4, boundary=boundary).astype(np.float32)
    gS3 = synth.random_volume((3,) + shape, seed=11)
    alpha = params.alpha
    offs, g, did, w = oracle.dcs_stencil(params.directions, params.R, params.sigma, alpha)
    w32 = (np.asarray(alpha, np.float32)[did] * g.astype(np.float32)).astype(np.float64)  # the kernel's weights
    eng = sal.Saliency(shape, params)
    try:
        gE = torch.empty((3,) + shape, dtype=torch.float32, device="cuda")
        ga = torch.empty(len(alpha), dtype=torch.float32, device="cuda")
        sal.sal_center_surround_backward(eng.h, _cuda(E32), _cuda(gS3), gE, ga)
        torch.cuda.synchronize()
    finally:
        eng.close()
    refE, gw = oracle.center_surround_adjoint(E32, gS3, offs, w32, boundary)
    ref_ga = oracle.direction_gradient(gw, g.astype(np.float32), did)
    assert rel_l2(gE.cpu().numpy(), refE) <= RTOL
    assert rel_l2(ga.cpu().numpy(), ref_ga) <= RTOL


def test_combine_adjoint_matches_oracle(sal):
    shape = (11, 10, 30)
    rng = np.random.default_rng(3)
    S3 = rng.random((3,) + shape).astype(np.float32)
    gS = rng.standard_normal(shape).astype(np.float32)
    W = np.array([0.5, 0.2, 0.3], np.float32)
    eng = sal.Saliency(shape, sal.Params(n=4))
    try:
        gS3 = torch.empty((3,) + shape, dtype=torch.float32, device="cuda")
        gW = torch.empty(3, dtype=torch.float32, device="cuda")
        sal.sal_combine_backward(eng.h, _cuda(S3), _cuda(W), _cuda(gS), gS3, gW)
        torch.cuda.synchronize()
    finally:
        eng.close()
    fwd = oracle.combine(S3, W.astype(np.float64))
    ref3, refW = oracle.combine_backward(fwd, W.astype(np.float64), gS)
    assert rel_l2(gS3.cpu().numpy(), ref3) <= RTOL
    assert rel_l2(gW.cpu().numpy(), refW) <= RTOL


@pytest.mark.parametrize("n,shape", [(4, (10, 9, 33)), (8, (12, 10, 40)), (16, (6, 6, 18))])
def test_fused_backward_matches_oracle(sal, n, shape):
    """sal_saliency_backward end to end (forward recomputed inside) against the FP64 adjoint."""
    V, D = synth.volume(synth.small_spec(shape, seed=n, faults=2))
    W = np.array([0.45, 0.35, 0.2])
    alpha = [1.0, 0.8, 1.2]
    params = sal.Params(n=n, alpha=alpha)
    st = oracle.dcs_stencil(params.directions, params.R, params.sigma, alpha)
    fwd = oracle.saliency(V, n, stencil=st, weights=W)
    gS = (fwd["S"] - D).astype(np.float32)
    ref = oracle.saliency_backward(V, n, W, gS, stencil=st, fwd=fwd)
    eng = sal.Saliency(shape, params)
    try:
        gV, gW, ga = eng.backward(_cuda(V), _cuda(W), _cuda(gS))
        torch.cuda.synchronize()
    finally:
        eng.close()
    assert rel_l2(gV.cpu().numpy(), ref["gV"]) <= RTOL, rel_l2(gV.cpu().numpy(), ref["gV"])
    assert rel_l2(gW.cpu().numpy(), ref["gW"]) <= RTOL
    assert rel_l2(ga.cpu().numpy(), ref["galpha"]) <= RTOL


def test_finite_differences_of_gpu_forward(sal):
    """Central differences (eps = 1e-3, 64 seeded entries) of L = sum gS * S on the FP32 GPU
    forward with the forward's min-max bounds held fixed, against sal_saliency_backward."""
    V, D = synth.volume(synth.small_spec((24, 20, 40), seed=0, faults=1))
    n = 8
    W = torch.tensor([0.5, 0.3, 0.2], device="cuda")
    eng = sal.Saliency(V.shape, sal.Params(n=n))
    try:
        Vt = _cuda(V)
        S3 = eng.center_surround(eng.local_spectra_project(Vt)).double()
        lo = S3.amin(dim=(1, 2, 3), keepdim=True)
        hi = S3.amax(dim=(1, 2, 3), keepdim=True)
        C = (W.double()[:, None, None, None] * (S3 - lo) / (hi - lo)).sum(0)
        loC, hiC = C.min(), C.max()
        gS = _cuda(((C - loC) / (hiC - loC)).cpu().numpy() - D)

        def L(Vx):
            S3x = eng.center_surround(eng.local_spectra_project(Vx)).double()
            Cx = (W.double()[:, None, None, None] * (S3x - lo) / (hi - lo)).sum(0)
            return float(((Cx - loC) / (hiC - loC) * gS.double()).sum())

        gV, _, _ = eng.backward(Vt, W, gS)
        idx = synth.sample_points(V.shape, 64, seed=1234)
        eps = 1e-3
        fd = []
        for p in idx:
            Vp = Vt.clone(); Vp[tuple(p)] += eps
            Vm = Vt.clone(); Vm[tuple(p)] -= eps
            fd.append((L(Vp) - L(Vm)) / (2 * eps))
        an = gV.cpu().numpy()[idx[:, 0], idx[:, 1], idx[:, 2]]
    finally:
        eng.close()
    fd = np.array(fd)
    # FP32 forward noise and the kinks of |.| bound the agreement of single entries; the
    # 64-vector agrees to about 1e-2.
    assert rel_l2(an, fd) <= 2e-2, rel_l2(an, fd)


@pytest.mark.parametrize("n", [8, 16])
def test_finite_differences_differentiation_workload_128(sal, n):
    """The differentiation-form workload at full size: the 128^3 single-fault volume, the L2 loss to
    its fault mask (gS = S - D), central differences (eps = 1e-3) of the FP32 GPU forward at 64 seeded
    entries with the forward's min-max bounds held fixed, against sal_saliency_backward."""
    V, D = synth.volume("fault128")
    W = torch.tensor([0.5, 0.3, 0.2], device="cuda")
    eng = sal.Saliency(V.shape, sal.Params(n=n))
    try:
        Vt = _cuda(V)
        S3 = eng.center_surround(eng.local_spectra_project(Vt)).double()
        lo = S3.amin(dim=(1, 2, 3), keepdim=True)
        hi = S3.amax(dim=(1, 2, 3), keepdim=True)
        C = (W.double()[:, None, None, None] * (S3 - lo) / (hi - lo)).sum(0)
        loC, hiC = C.min(), C.max()
        gS = _cuda(((C - loC) / (hiC - loC)).cpu().numpy() - D)

        def L(Vx):
            S3x = eng.center_surround(eng.local_spectra_project(Vx)).double()
            Cx = (W.double()[:, None, None, None] * (S3x - lo) / (hi - lo)).sum(0)
            return float(((Cx - loC) / (hiC - loC) * gS.double()).sum())

        gV, _, _ = eng.backward(Vt, W, gS)
        idx = synth.sample_points(V.shape, 64, seed=1234)
        eps = 1e-3
        fd = []
        for p in idx:
            Vp = Vt.clone(); Vp[tuple(p)] += eps
            Vm = Vt.clone(); Vm[tuple(p)] -= eps
            fd.append((L(Vp) - L(Vm)) / (2 * eps))
        an = gV.cpu().numpy()[idx[:, 0], idx[:, 1], idx[:, 2]]
    finally:
        eng.close()
    fd = np.array(fd)
    print("n", n, "FD vs analytic rel-L2", f"{rel_l2(an, fd):.2e}")
    assert rel_l2(an, fd) <= 2e-2, rel_l2(an, fd)


def test_autograd_matches_abi_and_descends(sal):
    """The autograd Function returns exactly the C-ABI per-step adjoint calls on the forward's E and
    S3 (and the fused backward call to rounding: it applies the combination coefficients at another
    point), and a small step of V along the negative gradient lowers the L2 distance of S to a
    fault mask."""
    from paper_2201_06174_gb300.autograd import saliency
    V, D = synth.volume(synth.small_spec((20, 18, 36), seed=2, faults=2))
    eng = sal.Saliency(V.shape, sal.Params(n=8))
    try:
        Vt = _cuda(V)
        Dt = _cuda(D)
        Vr = Vt.clone().requires_grad_(True)
        Wr = torch.tensor([0.5, 0.3, 0.2], device="cuda", requires_grad=True)
        ar = torch.tensor([1.0, 0.9, 1.1], device="cuda", requires_grad=True)
        S = saliency(Vr, Wr, ar, eng)
        loss0 = 0.5 * ((S - Dt) ** 2).sum()
        loss0.backward()
        gS = (S.detach() - Dt).contiguous()
        eng.set_alpha(ar.detach().cpu().numpy())
        # the per-step calls on the forward's intermediates
        E = torch.empty((3,) + V.shape, device="cuda")
        S3 = torch.empty_like(E)
        Sx = torch.empty(V.shape, device="cuda")
        sal.sal_saliency(eng.h, Vt, None, Wr.detach(), Sx, S3, E)
        gS3, gE = torch.empty_like(E), torch.empty_like(E)
        gW1, ga1, gV1 = torch.empty(3, device="cuda"), torch.empty(3, device="cuda"), torch.empty_like(Vt)
        sal.sal_combine_backward(eng.h, S3, Wr.detach(), gS, gS3, gW1)
        sal.sal_center_surround_backward(eng.h, E, gS3, gE, ga1)
        sal.sal_local_spectra_project_backward(eng.h, Vt, gE, gV1)
        assert torch.equal(Vr.grad, gV1) and torch.equal(Wr.grad, gW1) and torch.equal(ar.grad, ga1)
        gV, gW, ga = eng.backward(Vt, Wr.detach(), gS)
        for a, b in ((Vr.grad, gV), (Wr.grad, gW), (ar.grad, ga)):
            assert float((a - b).norm()) <= 1e-6 * float(b.norm())
        eta = 1e-3 * float(Vt.norm()) / float(gV.norm())
        with torch.no_grad():
            S1 = saliency(Vt - eta * gV, Wr.detach(), ar.detach(), eng)
            loss1 = 0.5 * ((S1 - Dt) ** 2).sum()
        assert float(loss1) < float(loss0)
    finally:
        eng.close()


@pytest.mark.parametrize("wanted", [(True, False, False), (False, True, False), (False, False, True), (True, False, True)])
def test_autograd_of_some_inputs_matches_that_of_all(wanted):
    """What a caller does not differentiate by is not computed, and the rest is the same: the FP64 sums of the alpha
    gradient are taken in another order without the features' gradient, and rounded once to FP32."""
    import torch
    from paper_2201_06174_gb300 import autograd as sal_autograd, sal as capi
    shape = (11, 9, 14)
    g = torch.Generator().manual_seed(3)
    V, gS = (torch.randn(shape, generator=g).cuda() for _ in range(2))
    W, alpha = torch.tensor([0.2, 0.5, 0.4]).cuda(), torch.tensor([1.0, 0.9, 1.1]).cuda()
    eng = capi.Saliency(shape, capi.Params(n=8, directions=((1, 0, 0), (0, 1, 0), (1, 1, 0))))
    try:
        def grads(need):
            x = [t.clone().requires_grad_(r) for t, r in zip((V, W, alpha), need)]
            eng.set_alpha([3.0, 3.0, 3.0])   # not the one of this call
            S = sal_autograd.saliency(*x, eng)
            eng.set_alpha([2.0, 2.0, 2.0])   # nor in its backward
            return torch.autograd.grad(S, [t for t, r in zip(x, need) if r], gS)
        full = grads((True, True, True))
        for got, want in zip(grads(wanted), [f for f, r in zip(full, wanted) if r]):
            assert torch.allclose(got, want, rtol=2.0 ** -22, atol=0)
    finally:
        eng.close()
