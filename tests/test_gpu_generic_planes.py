"""The bf16 planes of a cube built with parameters other than the paper's: the
Fourier correlation, which reads them, against Eq. 8 in float64 from the exported
cube (which reads the chunks), at widths around the tile of 32 columns and an odd
one.  Tolerance 1e-5, the bound of these transforms' NCC on textured windows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from workloads import optical_like  # noqa: E402


@pytest.mark.parametrize("kw", [dict(dil=(1, 2)), dict(radius_mult=2.0), dict(sigma_d1=0.0, sigma_d2=0.0)])
@pytest.mark.parametrize("H,W", [(96, 96), (131, 97), (65, 127)])
def test_planes_hold_the_chunks_values(kw, H, W):
    import paper_2202_13347_gb300 as pkg
    pkg.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    b = pkg.load()
    ctx = b.Context(0)
    p = b.params(dtype=b.DTYPE_BF16, **kw)
    ref = optical_like(np.random.default_rng(H + W), H, W)
    sen = (1.0 - np.roll(ref, (1, -2), (0, 1))).astype(np.float32)
    rc, sc = (ctx.sfoc_build(torch.from_numpy(np.ascontiguousarray(v)).cuda(), p=p) for v in (ref, sen))
    m, R = 17, 4
    h, P = m // 2, 2 * R + 1
    pts = torch.tensor([[h + R, h + R], [W - h - R - 1, H - h - R - 1], [W // 2, H // 2], [W - h - R - 1, h + R]],
                       dtype=torch.int32, device="cuda")
    got = ctx.fastncc_match(rc, sc, pts, m, R, corr_path=b.CORR_FFT, want_maps=True)
    ctx.sync()
    vr, vs = rc.export().double(), sc.export().double()
    for k, (x, y) in enumerate(pts.tolist()):
        t = vs[:, y - h:y + h + 1, x - h:x + h + 1]
        t = t - t.mean()
        w = vr[:, y - h - R:y + h + R + 1, x - h - R:x + h + R + 1].unfold(1, m, 1).unfold(2, m, 1)
        w = w - w.mean((0, 3, 4), keepdim=True)
        want = (w * t[:, None, None]).sum((0, 3, 4)) / (w.square().sum((0, 3, 4)) * t.square().sum()).sqrt()
        assert want.shape == (P, P)
        assert float((got["maps"][k].double() - want).abs().max()) <= 1e-5
