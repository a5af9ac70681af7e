"""Precision of the rectified values against float64 on white noise, where a
position's error shows most (neighbouring samples differ by up to 1).

Bound: FP32 blend of samples in [0, 1]: each of the two row blends rounds a
difference and a sum (2 x 2^-25), the column blend the same on top: 2^-23.
Position: the fraction's rounding (2^-25 px) and what the mapping may be off
before it (9 x 2^-24 of the perspective term, which is below 0.03 px on these
models, and 40 x 2^-33 px: below 2^-25), per axis, times a step of at most 1."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BOUND = 2.0 ** -23 + 2 * (2.0 ** -25 + 2.0 ** -25)
MODELS = {
    "rotation": [[0.98, -0.17, 200.3], [0.17, 0.98, -120.7], [0, 0, 1]],
    "projective": [[1.011, 0.013, 21.3], [-0.017, 0.991, -33.1], [1.3e-5, -0.9e-5, 1]],
    "projective_strong": [[0.99, 0.02, -14.6], [0.02, 1.01, 38.2], [-2e-5, 2e-5, 1]],
    "shrink": [[0.27, 0.01, 3.3], [-0.02, 0.31, 40.7], [0, 0, 1]],
}


@pytest.mark.parametrize("shape", [(2048, 2048), (331, 4801)])
@pytest.mark.parametrize("model", sorted(MODELS))
def test_values_match_float64(model, shape):
    import paper_2202_13347_gb300 as pkg
    pkg.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = pkg.load().Context(0)
    H, W = shape
    img = torch.from_numpy(np.random.default_rng(H).random(shape).astype(np.float32)).cuda()
    M = torch.tensor(MODELS[model], dtype=torch.float64, device="cuda")
    got = ctx.rectify(img, M, fill=-1.0)
    ctx.sync()
    a = np.linalg.inv(np.array(MODELS[model]))
    a /= a[2, 2]
    y, x = torch.meshgrid(torch.arange(H, device="cuda").double(), torch.arange(W, device="cuda").double(),
                          indexing="ij")
    w = a[2, 0] * x + a[2, 1] * y + 1.0
    u, v = (a[0, 0] * x + a[0, 1] * y + a[0, 2]) / w, (a[1, 0] * x + a[1, 1] * y + a[1, 2]) / w
    inside = (u > 1e-6) & (v > 1e-6) & (u < W - 1 - 1e-6) & (v < H - 1 - 1e-6)
    assert int(inside.sum()) > H * W // 20
    u, v = u[inside], v[inside]
    i, j = v.floor().long(), u.floor().long()
    fy, fx, s = v - i, u - j, img.double()
    want = (s[i, j] * (1 - fx) + s[i, j + 1] * fx) * (1 - fy) + (s[i + 1, j] * (1 - fx) + s[i + 1, j + 1] * fx) * fy
    assert float((got[inside].double() - want).abs().max()) <= BOUND
