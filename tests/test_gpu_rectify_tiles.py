"""The rectification's per-tile mapping on the GPU against the oracle (which
maps and blends in double): tile edges, one and four tiles a warp, images of
one to three pixels a side, models whose border lines run through pixel
centres, strong scale and perspective (the FP64 route).  Fill positions are
identical; a value differs by the blend's FP32 roundings (4 x 2^-24 of the
largest sample) and the position's 2^-22 px of the steepest pixel step."""
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


def rotation(a, tx=0.0, ty=0.0, s=1.0):
    return np.array([[s * np.cos(a), -s * np.sin(a), tx], [s * np.sin(a), s * np.cos(a), ty], [0, 0, 1.0]])


MODELS = {
    "identity": np.eye(3),
    "integer": np.array([[1, 0, 31.0], [0, 1, -9.0], [0, 0, 1]]),
    "half": np.array([[1, 0, 0.5], [0, 1, -0.25], [0, 0, 1]]),
    "mirror": np.array([[-1, 0, 62.0], [0, 1, 0], [0, 0, 1]]),
    "quarter": np.array([[0, -1, 40.0], [1, 0, 0], [0, 0, 1]]),
    "rotated": rotation(0.3, 20, -5),
    "near": np.array([[1.01, 0.013, 3.3], [-0.011, 0.99, -7.7], [1.5e-5, -2e-5, 1]]),
    "shrink": rotation(0.1, s=0.2),
    "perspective": np.array([[1, 0, 0], [0, 1, 0], [4e-3, 1e-3, 1]]),
}


@pytest.mark.parametrize("model", sorted(MODELS))
@pytest.mark.parametrize("shape,out_shape", [((63, 65), (63, 65)), ((1, 1), (9, 40)), ((2, 3), (70, 33)),
                                             ((64, 256), (65, 257)), ((700, 2100), (1100, 2200))])
def test_matches_oracle(ctx, orc, model, shape, out_shape):
    rng = np.random.default_rng(shape[0] + len(model))
    img = rng.random(shape).astype(np.float32)
    H = MODELS[model]
    g = ctx.rectify(torch.from_numpy(img).cuda(), torch.from_numpy(H).cuda(), out_shape=out_shape, fill=-1.0)
    ctx.sync()
    g = g.cpu().numpy()
    o = orc.rectify(img, H, out_shape=out_shape, fill=-1.0)
    np.testing.assert_array_equal(g == -1.0, o == -1.0)
    assert np.abs(g - o).max() <= 4 * 2.0 ** -24 + 2 * 2.0 ** -22
