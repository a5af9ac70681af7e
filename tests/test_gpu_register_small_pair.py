"""Both cubes of a small pair built in one launch per kernel
(fastncc_register_pair): bit for bit what two builds and a match give, in both
cube types, for images of uneven and tiny sizes, again after a change of shape
and of type on the same context, where the workspace was made by a single build,
and replayed from a captured graph on new images."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def b():
    import paper_2202_13347_gb300 as pkg
    pkg.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return pkg.load()


def image(H, W, seed):
    return torch.from_numpy(np.random.default_rng(seed + 1000 * H + W).random((H, W)).astype(np.float32)).cuda()


def points(H, W, m, R):
    lo = m // 2 + R + 1
    y, x = np.mgrid[lo:H - lo:9, lo:W - lo:11]
    return torch.from_numpy(np.stack([x.ravel(), y.ravel()], 1).astype(np.int32)).cuda()


SIZES = [((60, 70), (61, 67)), ((64, 64), (64, 64)), ((130, 257), (300, 191)), ((512, 500), (40, 40)),
         ((1000, 1000), (1024, 1024)), ((1200, 1100), (1100, 1200))]  # the last: above the size of a joint launch


@pytest.mark.parametrize("dt", ["f32", "bf16"])
def test_equals_builds_and_match(b, dt):
    m, R = 15, 4
    p = b.params(dtype=b.DTYPE_BF16 if dt == "bf16" else b.DTYPE_F32)
    ctx, ctx2 = b.Context(0), b.Context(0)
    path = b.CORR_FFT
    for (hr, wr), (hs, ws) in SIZES + SIZES[:2]:
        ref, sen = image(hr, wr, 1), image(hs, ws, 2)
        pts = points(min(hr, hs), min(wr, ws), m, R)
        one = ctx.register_pair(ref, sen, pts, m, R, p=p, corr_path=path)
        two = ctx2.fastncc_match(ctx2.sfoc_build(ref, p=p), ctx2.sfoc_build(sen, p=p), pts, m, R, corr_path=path)["raw"]
        ctx.sync()
        ctx2.sync()
        assert torch.equal(one, two)


def test_after_single_build_and_in_a_graph(b):
    m, R, H, W = 15, 4, 300, 280
    stream = torch.cuda.Stream()
    ctx = b.Context(0, stream)
    with torch.cuda.stream(stream):
        ref, sen, pts = image(H, W, 1), image(H, W, 2), points(H, W, m, R)
        ctx.sfoc_build(ref)  # the workspace of one image: a joint build would need two
        a = ctx.register_pair(ref, sen, pts, m, R, corr_path=b.CORR_FFT).clone()
        ctx.reserve(64 << 20)
        c = ctx.register_pair(ref, sen, pts, m, R, corr_path=b.CORR_FFT).clone()
    stream.synchronize()
    assert torch.equal(a, c)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        out = ctx.register_pair(ref, sen, pts, m, R, corr_path=b.CORR_FFT)
    with torch.cuda.stream(stream):
        ref.copy_(image(H, W, 3))
        sen.copy_(image(H, W, 4))
        g.replay()
        got = out.clone()
        want = ctx.register_pair(ref, sen, pts, m, R, corr_path=b.CORR_FFT)
    stream.synchronize()
    assert torch.equal(got, want)
