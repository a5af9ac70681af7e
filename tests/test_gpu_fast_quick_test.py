"""The FAST kernel's quick test and pixel list on the GPU against the oracle:
images where it turns everything away, nothing away, or only by one side of a
pair; exact ties at the threshold; sub-tile edges.  FP32 differences of the
stored values on both sides: points and scores are identical."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    import paper_2202_13347_gb300 as pkg
    pkg.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return pkg.load().Context(0)


def image(kind, H, W):
    rng = np.random.default_rng(H * 1000 + W)
    y, x = np.mgrid[0:H, 0:W]
    if kind == "noise":          # most pixels pass the quick test
        return rng.random((H, W)).astype(np.float32)
    if kind == "steps":          # plateaus of 1/8: differences exactly at the threshold
        return (rng.integers(0, 9, (H // 3 + 1, W // 3 + 1)).repeat(3, 0).repeat(3, 1)[:H, :W] / 8).astype(np.float32)
    if kind == "lines":          # edges: opposite pairs straddle them
        return (((x // 7) % 2) * 0.6 + ((y // 11) % 2) * 0.3).astype(np.float32)
    img = np.zeros((H, W), np.float32)   # isolated dots, one bright and one dark
    img[::13, ::17] = 1.0
    img[5::13, 8::17] = -1.0
    return img


@pytest.mark.parametrize("kind", ["noise", "steps", "lines", "dots"])
@pytest.mark.parametrize("H,W,gy,gx,t", [(64, 64, 1, 1, 0.125), (65, 129, 1, 2, 0.0), (66, 63, 3, 1, 0.125),
                                         (7, 9, 1, 3, 0.05), (200, 130, 200, 13, 0.125)])
def test_points_and_scores_match_the_oracle(ctx, orc, kind, H, W, gy, gx, t):
    img = image(kind, H, W)
    p, s = ctx.fast_blocks(torch.from_numpy(img).cuda(), t, gy, gx, 0)
    ctx.sync()
    op, os_ = orc.fast_blocks(img, t, gy, gx, 0)
    np.testing.assert_array_equal(p.cpu().numpy(), op)
    np.testing.assert_array_equal(s.cpu().numpy(), os_)
