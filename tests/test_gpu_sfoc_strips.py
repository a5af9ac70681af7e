"""The streaming SFOC kernels (strips of 32 and 64 columns, rows in blocks of
4 and 8, segments per image) on the GPU against the oracle at sizes around
their edges, in both cube types, alone and batched.  FP32: 2e-5 absolute (FP32
filtering of [0, 1] images, values normalised to at most 1), and where a group's
norm is small 1e-6 / (norm + eps) on top: the FP32 error of a pre-normalisation
value is divided by the norm (the bound the descriptor variants are held to;
images of one row or column have no gradient across it).  BF16: one bf16 ulp of
the FP32 value (2^-8 relative) on top.  A batch gives bit for bit what
single builds give; a rebuild in place gives the same again."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from workloads import optical_like  # noqa: E402

from test_gpu_parity import _group_norm_tol  # noqa: E402

SIZES = [(1, 1), (1, 200), (200, 1), (7, 63), (8, 64), (9, 65), (17, 128), (31, 33), (40, 97), (64, 129), (70, 191),
         (257, 66), (300, 256)]


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


def image(H, W):
    rng = np.random.default_rng(100 * H + W)
    return optical_like(rng, H, W) if min(H, W) > 30 else rng.random((H, W)).astype(np.float32)


@pytest.mark.parametrize("dt", ["f32", "bf16"])
@pytest.mark.parametrize("H,W", SIZES)
def test_cube_matches_oracle(b, ctx, orc, H, W, dt):
    img = image(H, W)
    p = b.params(dtype=b.DTYPE_BF16 if dt == "bf16" else b.DTYPE_F32)
    cube = ctx.sfoc_build(torch.from_numpy(img).cuda(), p=p)
    got = cube.export().cpu().numpy().astype(np.float64)
    want = orc.sfoc_roi(img).data
    tol = _group_norm_tol(orc, img, {}) + (np.abs(want) * 2.0 ** -8 if dt == "bf16" else 0.0)
    assert np.all(np.abs(got - want) <= tol), np.abs(got - want).max()
    again = ctx.sfoc_build(torch.from_numpy(img).cuda(), p=p, out=cube).export().cpu().numpy()
    np.testing.assert_array_equal(again, got.astype(np.float32))
    # the sum planes, through the integral images: each entry within one unit of
    # 2^-28 per pixel plus the cube's own error summed over the channels
    P = cube.export_integral().cpu().numpy()
    g = got.sum(0), (got * got).sum(0)
    for k in range(2):
        ref = np.pad(g[k].cumsum(0).cumsum(1), ((1, 0), (1, 0)))
        n = np.outer(np.arange(H + 1), np.arange(W + 1))
        assert np.all(np.abs(P[k] - ref) <= n * (2.0 ** -28 + 12 * 6 * 2.0 ** -24))


@pytest.mark.parametrize("dt", ["f32", "bf16"])
def test_batch_and_u16_equal_single(b, ctx, dt):
    p = b.params(dtype=b.DTYPE_BF16 if dt == "bf16" else b.DTYPE_F32)
    imgs = [torch.from_numpy(image(H, W)).cuda() for H, W in SIZES + [(530, 700)]]
    outs = ctx.sfoc_build_batch(imgs, p=p)
    for im, o in zip(imgs, outs):
        one = ctx.sfoc_build(im, p=p)
        assert torch.equal(one.export(), o.export())
    v = (imgs[-1] * 65535.0).round()
    u = torch.where(v >= 32768, v - 65536, v).to(torch.int16)
    # correctly rounded v / 65535, by NumPy: torch divides a CUDA tensor by a
    # scalar as a product with the rounded reciprocal
    f = torch.from_numpy(v.cpu().numpy() / np.float32(65535.0)).cuda()
    assert torch.equal(ctx.sfoc_build_u16(u, p=p).export(), ctx.sfoc_build(f, p=p).export())


def test_every_16_bit_value_is_correctly_rounded(b, ctx):
    v = torch.arange(65536, dtype=torch.int32).reshape(256, 256)
    u = torch.where(v >= 32768, v - 65536, v).to(torch.int16).cuda()
    f = torch.from_numpy(v.numpy().astype(np.float32) / np.float32(65535.0)).cuda()
    assert torch.equal(ctx.sfoc_build_u16(u).export(), ctx.sfoc_build(f).export())
