"""The reductions that the last block of a launch finishes (bounds, weights, template fit, combination bounds, gradient of
the weights), at grids of one block, of a few, and at the largest, against the entry point that keeps a separate launch for
each; and repeated, since the blocks are counted in memory that outlives the call."""
import contextlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

from paper_2201_06174_gb300 import sal  # noqa: E402

# voxels of one thread, one block and one over; a few blocks; the largest grid (1216 blocks of 256) and one voxel over it
SHAPES = [(1, 1, 1), (1, 1, 256), (1, 1, 257), (5, 7, 11), (76, 64, 64), (1, 1, 311297)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("mode", ["equal", "given", "fit"])
def test_combine_bounds_and_weights_match_separate_launches(shape, mode):
    g = torch.Generator().manual_seed(5)
    p = sal.Params(n=8, directions=((1, 0, 0), (0, 1, 0)), R=1)
    S3 = torch.rand((3,) + shape, generator=g).cuda()
    D = torch.rand(shape, generator=g).cuda() if mode == "fit" else None
    W = torch.tensor([0.2, 0.5, 0.4]).cuda() if mode == "given" else None
    S_ref, W_ref = torch.empty(shape, device="cuda"), torch.empty(3, device="cuda")
    sal.sal_combine_noalloc(S3, D, W, W_ref, S_ref)
    with contextlib.closing(sal.Saliency(shape, p)) as eng:
        for _ in range(3):
            S, Wo = torch.empty(shape, device="cuda"), torch.empty(3, device="cuda")
            sal.sal_combine(eng.h, S3, D, W, Wo, S)
            if mode == "fit":   # FP64 sums in another order, rounded to FP32 after a solve whose pivots are >= 1e-6 of N
                assert torch.allclose(Wo, W_ref, rtol=1e-5, atol=1e-6)
                assert torch.allclose(S, S_ref, rtol=1e-5, atol=1e-5)
            else:               # minima and maxima do not depend on the order
                assert torch.equal(Wo, W_ref) and torch.equal(S, S_ref)


@pytest.mark.parametrize("shape", [(1, 1, 1), (4, 8, 9), (40, 41, 43), (80, 64, 64)])
def test_fused_bounds_of_a_whole_call_match_the_staged_calls(shape):
    g = torch.Generator().manual_seed(6)
    V = torch.randn(shape, generator=g).cuda()
    p = sal.Params(n=8, directions=((1, 0, 0), (0, 1, 0)), R=1)
    W = torch.tensor([0.2, 0.5, 0.4]).cuda()
    gS = torch.randn(shape, generator=g).cuda()
    with contextlib.closing(sal.Saliency(shape, p)) as eng:
        first = None
        for _ in range(2):
            r = eng.saliency(V, W=W, intermediates=True)
            S, Wo = torch.empty(shape, device="cuda"), torch.empty(3, device="cuda")
            sal.sal_combine(eng.h, r["S3"], None, W, Wo, S)
            assert torch.equal(r["S"], S)
            gS3, gW = torch.empty_like(r["S3"]), torch.empty(3, device="cuda")
            sal.sal_combine_backward(eng.h, r["S3"], W, gS, gS3, gW)
            if first is None:
                first = gW.clone()
            assert torch.equal(gW, first)
            s3, gs = r["S3"].double().flatten(1), gS.double().flatten()
            lo, hi = s3.amin(1), s3.amax(1)
            inv = torch.where(hi > lo, 1.0 / (hi - lo), torch.zeros_like(lo))
            c = ((s3 - lo[:, None]) * inv[:, None] * W.double()[:, None]).sum(0)
            span = float(c.max() - c.min())
            terms = (s3 - lo[:, None]) * inv[:, None] / (span if span > 0 else np.inf)
            ref = (terms * gs).sum(1)
            # every term carries a few roundings of 2^-24: the scales inv and invC, the difference S3 - lo, the product
            assert float((gW.double() - ref).abs().max()) <= 16 * 2.0 ** -24 * float((terms * gs).abs().sum(1).max()) + 1e-30
