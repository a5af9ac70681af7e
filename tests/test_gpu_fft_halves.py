"""The Fourier correlation by halves of the spectrum (sides 96, 160, 192, 224)
on the GPU, both cube types, at the edges of every side, for one point and for
more points than CTAs, against Eq. 8 evaluated in float64 by torch from the
exported cubes.

Tolerance: a transform of length L adds at most ~5 log2(L) 2^-24 of the input's
norm (below 2.4e-6 for L <= 224; window, template and inverse transforms in
both directions), which reaches NCC multiplied by |S| / |S - mean S| (at most
4 on these textured windows): 1e-5 bounds it.  A template of one pixel has a
window of up to 96^2 pixels around it and |S| measured over the window instead:
m = 9 is the smallest here."""
import json

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from workloads import optical_like  # noqa: E402


@pytest.fixture(scope="module")
def b():
    import paper_2202_13347_gb300 as pkg
    pkg.build()
    return pkg.load()


@pytest.fixture()
def ctx(b):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return b.Context(0)


def side(m, R):
    return (m + 2 * R + 31) // 32 * 32


def force(ctx, dt, m, R, option):
    ctx.autotune_import(json.dumps({"sfoc_autotune": 1, "entries": [
        {"dtype": dt, "family": 0, "m": m, "R": R, "path": 6, "option": option, "sample": 1, "candidates": []}]}))


def cubes(b, ctx, dt, H, W, seed, nan_at=None):
    rng = np.random.default_rng(seed)
    ref = optical_like(rng, H, W)
    sen = (1.0 - np.roll(ref, (2, -3), (0, 1))).astype(np.float32)
    if nan_at is not None:
        ref[nan_at] = np.nan
    p = b.params(dtype=dt)
    return [ctx.sfoc_build(torch.from_numpy(np.ascontiguousarray(v)).cuda(), p=p) for v in (ref, sen)]


def points(H, W, m, R, n, seed):
    g = torch.Generator().manual_seed(seed)
    lo = ((m - 1) // 2 if m % 2 else m // 2) + R
    x = torch.randint(lo, W - m - 2 * R + lo + 1, (n,), generator=g)
    y = torch.randint(lo, H - m - 2 * R + lo + 1, (n,), generator=g)
    return torch.stack([x, y], 1).to(torch.int32).cuda()


def ncc_maps(ref, sen, pts, m, R):
    """Eq. 8 in float64, (n, 2R+1, 2R+1)."""
    ref, sen = ref.double(), sen.double()
    h, L, P = ((m - 1) // 2 if m % 2 else m // 2), m + 2 * R, 2 * R + 1
    out = []
    for x, y in pts.tolist():
        t = sen[:, y - h:y - h + m, x - h:x - h + m]
        w = ref[:, y - h - R:y - h - R + L, x - h - R:x - h - R + L]
        t = t - t.mean()
        num = torch.fft.irfft2((torch.fft.rfft2(w) * torch.fft.rfft2(t, s=(L, L)).conj()).sum(0), s=(L, L))[:P, :P]
        pre = [torch.nn.functional.pad(v.cumsum(0).cumsum(1), (1, 0, 1, 0)) for v in (w.sum(0), w.square().sum(0))]
        s1, s2 = (q[m:, m:] - q[:P, m:] - q[m:, :P] + q[:P, :P] for q in pre)
        out.append(num / ((s2 - s1 * s1 / t.numel()) * t.square().sum()).sqrt())
    return torch.stack(out)


EDGES = [(9, 28), (41, 12), (44, 26), (96, 0), (66, 32), (127, 1), (97, 32), (34, 63), (128, 32), (67, 63), (80, 60),
         (92, 63), (98, 63)]


@pytest.mark.parametrize("dt", [0, 1], ids=["f32", "bf16"])
@pytest.mark.parametrize("m,R", EDGES)
@pytest.mark.parametrize("n", [1, 5])
def test_maps_match_float64(b, ctx, dt, m, R, n):
    assert side(m, R) in (96, 160, 192, 224)
    if dt == 0 and (m, R) == (98, 63):
        pytest.skip("no form serves F32 cubes there")
    H, W = m + 2 * R + 11, m + 2 * R + 38
    rc, sc = cubes(b, ctx, dt, H, W, m + R)
    pts = points(H, W, m, R, n, 3)
    force(ctx, dt, m, R, side(m, R))
    g = ctx.fastncc_match(rc, sc, pts, m, R, want_maps=True)
    ctx.sync()
    assert (g["status"] != b.PT_OUT_OF_BOUNDS).all()
    want = ncc_maps(rc.export(), sc.export(), pts, m, R)
    assert float((g["maps"].double() - want).abs().max()) <= 1e-5


def test_more_points_than_ctas_and_the_batch(b, ctx):
    """Every point of a launch that wraps its CTAs; the batch's results are the
    single call's, bit for bit, with pairs of several sides in one plan."""
    jobs = [(61, 16, 1300), (61, 40, 320), (81, 40, 320), (80, 60, 160)]
    rc, sc = cubes(b, ctx, 0, 420, 400, 9)
    pts = [points(420, 400, m, R, n, 5) for m, R, n in jobs]
    for m, R, _ in jobs:
        force(ctx, 0, m, R, side(m, R))
    one = [ctx.fastncc_match(rc, sc, p, m, R, want_maps=True) for (m, R, _), p in zip(jobs, pts)]
    ctx.sync()
    for (m, R, _), p, g in zip(jobs, pts, one):
        want = ncc_maps(rc.export(), sc.export(), p[::37], m, R)
        assert float((g["maps"][::37].double() - want).abs().max()) <= 1e-5
    outs = ctx.fastncc_match_batch([rc] * 4, [sc] * 4, pts, [j[0] for j in jobs], [j[1] for j in jobs])
    ctx.sync()
    for g, o in zip(one, outs):
        assert torch.equal(g["raw"], o)


@pytest.mark.parametrize("dt", [0, 1], ids=["f32", "bf16"])
def test_offsets_clear_of_a_nan_keep_their_score(b, ctx, dt):
    """Beyond m + 2R = 128 a non-finite value stays with the offsets whose windows
    hold it, as in the direct and tensor-core forms."""
    m, R = 81, 40
    rc, sc = cubes(b, ctx, dt, 250, 240, 4, nan_at=(60, 70))
    pts = points(250, 240, m, R, 12, 6)
    a = ctx.fastncc_match(rc, sc, pts, m, R, corr_path=b.CORR_TC_BAND if dt else b.CORR_DIRECT_F32, want_maps=True)
    force(ctx, dt, m, R, side(m, R))
    g = ctx.fastncc_match(rc, sc, pts, m, R, want_maps=True)
    ctx.sync()
    assert torch.equal(torch.isnan(a["maps"]), torch.isnan(g["maps"])) and torch.isnan(g["maps"]).any()
    assert torch.equal(a["status"], g["status"])
    ok = ~torch.isnan(g["maps"])
    assert float((a["maps"][ok] - g["maps"][ok]).abs().max()) <= 2e-4   # two forms, each within 1e-4


def test_what_is_refused_stays_refused(b, ctx):
    rc, sc = cubes(b, ctx, 0, 300, 300, 2)
    p = points(300, 300, 9, 60, 2, 1)
    with pytest.raises(b.SfocError):
        ctx.fastncc_match(rc, sc, p, 9, 60, corr_path=b.CORR_FFT)     # m + 2R = 129
    for m, R, opt in ((101, 40, 128), (101, 40, 160), (101, 40, 224), (41, 10, 96), (81, 20, 96), (128, 63, 256),
                      (128, 48, 224)):
        with pytest.raises(b.SfocError):
            force(ctx, 0, m, R, opt)
    for m, R, opt in ((41, 10, 64), (41, 10, 128), (61, 16, 128), (61, 16, 96), (81, 20, 128), (101, 40, 192)):
        force(ctx, 0, m, R, opt)
        assert ctx.autotune_entry(0, m, R)["option"] == opt
