"""Block FAST with a threshold of 0, where every pixel is scored without the quick
test, against the oracle: sub-tile edges, blocks smaller and larger than a
sub-tile, flat and fully textured images.  FP32 differences of the stored values
on both sides: points and scores are identical."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("kind", ["noise", "ramp", "flat"])
@pytest.mark.parametrize("H,W,gy,gx,margin", [(64, 64, 1, 1, 0), (66, 131, 1, 1, 3), (200, 130, 3, 50, 0), (7, 7, 1, 1, 0),
                                              (140, 140, 1, 2, 20)])
def test_points_and_scores_match_the_oracle(orc, kind, H, W, gy, gx, margin):
    import paper_2202_13347_gb300 as pkg
    pkg.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = pkg.load().Context(0)
    rng = np.random.default_rng(H + W)
    y, x = np.mgrid[0:H, 0:W]
    img = {"noise": rng.random((H, W)), "ramp": ((x * x + 3 * y) % 17) / 16.0, "flat": np.full((H, W), 0.5)}[kind]
    img = img.astype(np.float32)
    p, s = ctx.fast_blocks(torch.from_numpy(img).cuda(), 0.0, gy, gx, margin)
    ctx.sync()
    op, os_ = orc.fast_blocks(img, 0.0, gy, gx, margin)
    np.testing.assert_array_equal(p.cpu().numpy(), op)
    np.testing.assert_array_equal(s.cpu().numpy(), os_)
