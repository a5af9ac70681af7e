"""The integral images' tile kernels on the GPU (tiles of 128 columns x 64
rows, eight rows a warp) at sizes around their edges: exact 64-bit sums, so every
exported entry equals the FP64 prefix of the pixels rounded to 2^-28 (exact in
FP64 here: below 2^53 units), alone and through the batched launch; and the
template sums take the same rounding."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SIZES = [(1, 1), (1, 130), (130, 1), (63, 127), (64, 128), (65, 129), (66, 260), (129, 257), (200, 384), (191, 33)]


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


def image(H, W, seed):
    return torch.from_numpy(np.random.default_rng(seed + 1000 * H + W).random((H, W)).astype(np.float32)).cuda()


@pytest.mark.parametrize("H,W", SIZES)
def test_planes_are_exact_sums(b, ctx, H, W):
    cube = ctx.sfoc_build(image(H, W, 1))
    g = cube.export()
    # the per-pixel sums as the kernels form them: channel after channel in FP32
    s1 = torch.zeros((H, W), device="cuda")
    s2 = torch.zeros((H, W), dtype=torch.float64, device="cuda")
    for c in range(g.shape[0]):
        s1 = s1 + g[c]
        s2 = (g[c].double() * g[c].double() + s2).float().double()   # one rounding, as a fused multiply-add
    P = cube.export_integral()
    for k, s in enumerate((s1.double(), s2)):
        units = torch.round(s * 2.0 ** 28)
        want = torch.nn.functional.pad(units.cumsum(0).cumsum(1), (1, 0, 1, 0)) / 2.0 ** 28
        assert torch.equal(P[k], want)


def test_batched_matches_equal_single_ones(b, ctx):
    m, R = 11, 4
    refs, sens, pts = [], [], []
    for H, W in [(40, 40), (64, 128), (65, 129), (130, 70), (129, 300)]:
        refs.append(ctx.sfoc_build(image(H, W, 2)))
        sens.append(ctx.sfoc_build(image(H, W, 3)))
        y, x = np.mgrid[9:H - 9:7, 9:W - 9:9]
        pts.append(torch.from_numpy(np.stack([x.ravel(), y.ravel()], 1).astype(np.int32)).cuda())
    one = [ctx.fastncc_match(r, s, p, m, R, corr_path=b.CORR_DIRECT_F32)["raw"] for r, s, p in zip(refs, sens, pts)]
    refs2 = [ctx.sfoc_build(image(H, W, 2)) for H, W in [(40, 40), (64, 128), (65, 129), (130, 70), (129, 300)]]
    outs = ctx.fastncc_match_batch(refs2, sens, pts, [m] * 5, [R] * 5, corr_path=b.CORR_DIRECT_F32)
    ctx.sync()
    for a, o in zip(one, outs):
        assert torch.equal(a, o)
