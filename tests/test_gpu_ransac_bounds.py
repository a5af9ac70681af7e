"""RANSAC's FP32 inlier decision with its error bound, on the GPU against the
FP64 oracle: scores, winner and inliers are identical whatever the scale of
the coordinates and the threshold (far below, at and far above the errors),
with points that are not finite or not valid, and with more points than one
staged block (1024) or one turn of the cluster (2048)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from workloads import planted_correspondences, ransac_samples  # noqa: E402


@pytest.fixture(scope="module")
def b():
    import paper_2202_13347_gb300 as pkg
    pkg.build()
    return pkg.load()


@pytest.fixture(scope="module")
def ctx(b):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return b.Context(0)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("projective", [True, False])
@pytest.mark.parametrize("n,scale,tau", [(7, 1.0, 1.5), (1024, 1.0, 1.5), (1025, 50.0, 75.0), (2049, 1e-3, 1.5e-3),
                                         (300, 1.0, 0.01), (300, 1.0, 1e9), (500, 1e6, 1.5)])
def test_decisions_are_the_fp64_ones(b, ctx, orc, projective, n, scale, tau):
    src, dst, _, _ = planted_correspondences(n + 11, n, projective, 0.3, noise=0.3)
    src, dst = src * scale, dst * scale
    k = 4 if projective else 3
    samp = ransac_samples(n + 12, n, 200, k)
    valid = np.ones(n, bool)
    if n > 100:
        src[3], dst[5], src[8] = np.nan, np.inf, 1e300
        valid[[3, 5, 8]] = False
        valid[20:40] = False
        samp[np.isin(samp, [3, 5, 8])] = 50
    g = ctx.fastncc_ransac(dev(src), dev(dst), dev(samp.astype(np.int32)), valid=dev(valid.astype(np.uint8)),
                           model=b.MODEL_PROJECTIVE if projective else b.MODEL_AFFINE, threshold=tau, want_scores=True)
    ctx.sync()
    with np.errstate(all="ignore"):
        o = orc.ransac(src, dst, samp, valid=valid, model=orc.PROJECTIVE if projective else orc.AFFINE, tau=tau)
    np.testing.assert_array_equal(g["scores"].cpu().numpy(), o["scores"])
    assert [int(v) for v in g["info"].cpu()] == [o["best"], o["count"]]
    np.testing.assert_array_equal(g["inlier"].cpu().numpy(), o["inlier"])


def test_no_points(b, ctx):
    e = torch.zeros((0, 2), dtype=torch.float64, device="cuda")
    g = ctx.fastncc_ransac(e, e, torch.zeros((5, 4), dtype=torch.int32, device="cuda"), want_scores=True)
    ctx.sync()
    assert (g["scores"].cpu() == -1).all() and [int(v) for v in g["info"].cpu()] == [-1, 0]
