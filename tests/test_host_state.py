"""Host-side state of the C ABI on the CPU: the library's host sources over a fake
CUDA runtime (host_fake.cpp), where allocations are counted and limited, launches
counted and timed by a table."""
import ctypes as C
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2202_13347_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")
F32, BF16 = 0, 1
AUTO, DIRECT, BAND, FFT = 0, 1, 5, 6


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("host")
    fake = os.path.join(HERE, "host_fake.cpp")
    flags = ["-std=c++17", "-O1", "-w", "-Wno-psabi", "-fPIC", "-I", os.path.join(CUDA, "include"), "-I", os.path.join(ROOT, "include"),
             "-I", CSRC, "-x", "c++"]
    objs = []
    for src in (os.path.join(CSRC, "sfoc_api.cu"), os.path.join(CSRC, "batch.cu"), fake):
        objs.append(str(d / (os.path.basename(src) + ".o")))
        shim = [] if src == fake else ["-DHOST_SHIM", "-include", fake]
        subprocess.run(["g++"] + flags + shim + ["-c", src, "-o", objs[-1]], check=True)
    so = str(d / "host.so")
    subprocess.run(["g++", "-shared", "-o", so, "-Wl,-z,lazy", "-Wl,-Bsymbolic"] + objs, check=True)   # the rest is bound when called
    L = C.CDLL(so, mode=os.RTLD_LAZY)
    L.fk_live.restype = L.fk_bytes.restype = C.c_size_t
    L.fk_limit.argtypes = [C.c_size_t]
    L.fk_cost.argtypes = [C.c_int, C.c_int, C.c_double]
    L.sfoc_last_error_string.restype = C.c_char_p
    L.sfoc_last_error_string.argtypes = [C.c_void_p]
    L.sfoc_ctx_launch_count.restype = C.c_int64
    L.sfoc_ctx_launch_count.argtypes = [C.c_void_p]
    return L


class Ctx:
    """A context of the faked library; points and images are addresses nothing reads."""

    def __init__(self, lib):
        self.L, self.h = lib, C.c_void_p()
        lib.fk_limit(C.c_size_t(-1).value)
        lib.fk_capturing(0)
        assert lib.sfoc_ctx_create(C.byref(self.h), 0, None) == 0
        lib.fk_reset()

    def ok(self, rc):
        assert rc == 0, self.L.sfoc_last_error_string(self.h).decode()

    def close(self):
        assert self.L.sfoc_ctx_destroy(self.h) == 0

    def pair(self, ref, sen, n=10, m=41, R=10, p=None):
        a = C.c_void_p(4096)
        return self.L.fastncc_register_pair(self.h, a, ref[0], ref[1], a, sen[0], sen[1], a, n, m, R, p, None, a)

    def build(self, H, W, p=None, out=None):
        c = C.c_void_p(out)
        assert self.L.sfoc_build(self.h, C.c_void_p(4096), H, W, C.c_size_t(W), None, 0, 0, p, C.byref(c)) == 0
        return c

    def match(self, a, b, n, m, R):
        p = C.c_void_p(4096)
        assert self.L.fastncc_match(self.h, a, b, p, n, m, R, None, p) == 0
        return self.L.fk_last_form()

    def launches(self):
        return self.L.sfoc_ctx_launch_count(self.h)


@pytest.fixture()
def ctx(lib):
    c = Ctx(lib)
    yield c
    c.close()


def test_ransac_counts_the_launches_its_launcher_reports(ctx):
    a, before = C.c_void_p(4096), ctx.launches()
    for hyps, want in ((16, 4), (0, 2)):
        assert ctx.L.fastncc_ransac(ctx.h, a, a, None, 8, 1, a, hyps, C.c_double(1.5), 1, a, a, a, None) == 0
        assert ctx.launches() - before == want
        before = ctx.launches()


def params(ctx, dtype):
    from paper_2202_13347_gb300.binding import Params
    p = Params()
    assert ctx.L.sfoc_params_default(C.byref(p)) == 0
    p.cube_dtype = dtype
    return C.byref(p)


def plans_built(ctx):
    n = C.c_size_t()
    assert ctx.L.sfoc_ctx_plan_info(ctx.h, None, 0, C.byref(n)) == 0
    buf = C.create_string_buffer(n.value)
    assert ctx.L.sfoc_ctx_plan_info(ctx.h, buf, n.value, C.byref(n)) == 0
    return int(buf.value.decode().split('"plans_built": ')[1].split(",")[0].split("}")[0])


def test_a_batch_plan_is_not_kept_for_a_cube_whose_planes_moved(ctx):
    """A cube freed and built again may come back at the same addresses but for one
    buffer: a plan holds that buffer's address in its tables."""
    H, W = 300, 320
    plane = 2 * 12 * 320 * H      # the BF16 planes: rows of 32 elements' multiples
    p = params(ctx, BF16)
    arr = lambda t, v: (t * 1)(v)  # noqa: E731
    sen = ctx.build(H, W, p)

    def match(ref):
        ctx.ok(ctx.L.fastncc_match_batch(ctx.h, 1, arr(C.c_void_p, ref.value), arr(C.c_void_p, sen.value),
                                         arr(C.c_void_p, 4096), arr(C.c_int, 50), arr(C.c_int, 41), arr(C.c_int, 10),
                                         None, arr(C.c_void_p, 4096)))
        return plans_built(ctx)

    ref = ctx.build(H, W, p)
    n = match(ref)
    assert match(ref) == n
    assert ctx.L.sfoc_cube_free(ref) == 0
    held = C.c_void_p()
    assert ctx.L.cudaMalloc(C.byref(held), C.c_size_t(plane)) == 0   # takes the freed planes' place
    again = ctx.build(H, W, p)
    if again.value != ref.value:
        pytest.skip("the host allocator moved the cube itself")
    assert match(again) == n + 1
    for c in (again, sen):
        assert ctx.L.sfoc_cube_free(c) == 0
    assert ctx.L.cudaFree(held) == 0


def test_pair_cubes_of_changing_shapes_do_not_pile_up(lib):
    """fastncc_register_pair keeps one pair of cubes: those a change of shape or type
    replaces are freed, but for cubes that a captured graph may read, which live
    as long as the context."""
    shapes = [((300, 280), (310, 290)), ((500, 400), (300, 280)), ((1500, 1400), (1400, 1500))]   # joint and single builds
    live = lib.fk_live()
    ctx = Ctx(lib)
    for dt in (F32, BF16, F32):
        for ref, sen in shapes * 2:
            ctx.ok(ctx.pair(ref, sen, p=params(ctx, dt)))
    seen = set()
    for _ in range(3):
        for dt in (F32, BF16):
            for ref, sen in shapes:
                ctx.ok(ctx.pair(ref, sen, p=params(ctx, dt)))
                seen.add((dt, ref, lib.fk_bytes()))
    assert len(seen) == 2 * len(shapes)          # the same memory in use each time a shape comes back
    ref, sen = shapes[0]
    ctx.ok(ctx.pair(ref, sen))
    lib.fk_capturing(1)
    ctx.ok(ctx.pair(ref, sen))                   # into a graph: these cubes stay
    lib.fk_capturing(0)
    held = lib.fk_live()
    ctx.ok(ctx.pair(*shapes[1]))
    ctx.ok(ctx.pair(ref, sen))
    ctx.ok(ctx.pair(*shapes[1]))
    assert lib.fk_live() > held
    ctx.close()
    assert lib.fk_live() == live


def test_a_pair_whose_joint_workspace_does_not_fit_is_built_one_by_one(ctx):
    """Both cubes of a small pair are built together with a workspace for two; where
    the device has no room for that, the two builds of one workspace still run."""
    H, W = 512, 480
    one = 4 * 12 * 480 * H
    room = 2 * (4 * 480 * H * 14 + 16 * (H + 1) * (W + 1)) + one + (3 << 20)   # two cubes, one workspace
    ctx.L.fk_limit(C.c_size_t(ctx.L.fk_bytes() + room))
    ctx.L.fk_reset()
    ctx.ok(ctx.pair((H, W), (H, W)))
    assert (ctx.L.fk_count(b"steer_two"), ctx.L.fk_count(b"steer")) == (0, 2)
    ctx.L.fk_limit(C.c_size_t(-1).value)
    again = Ctx(ctx.L)
    again.ok(again.pair((H, W), (H, W)))
    assert (ctx.L.fk_count(b"steer_two"), ctx.L.fk_count(b"steer")) == (1, 0)
    again.close()


def test_stage_timing_times_the_launches_that_run_without_it(ctx):
    """Both cubes of a small pair come from one launch per kernel, with stage timing
    as without: one steering and two smoothing launches."""
    shape = (512, 480)
    for timing in (0, 1):
        assert ctx.L.sfoc_ctx_enable_timing(ctx.h, timing) == 0
        ctx.L.fk_reset()
        before = ctx.launches()
        ctx.ok(ctx.pair(shape, shape))
        made = [ctx.L.fk_count(k) for k in (b"steer_two", b"smooth_two", b"steer", b"smooth")]
        assert made == [1, 1, 0, 0]
        if timing:
            ms, n = (C.c_double * 7)(), (C.c_int64 * 7)()
            assert ctx.L.sfoc_ctx_stage_times(ctx.h, ms, n) == 0
            assert list(n)[:2] == [1, 2] and sum(n) == ctx.launches() - before


# milliseconds of a form for 1 .. period points per SM (fk_cost; more points repeat the period), after
# measurements: one CTA per SM, four (side 96), two (side 160)
COSTS = {"f32_96": {(FFT, 128): {1: 0.088}, (FFT, 96): {1: 0.123, 2: 0.155, 3: 0.215, 4: 0.253}, (DIRECT, 0): {1: 5.0}},
         "bf16_96": {(BAND, 0): {1: 0.080}, (FFT, 128): {1: 0.100}, (FFT, 96): {1: 0.145, 2: 0.182, 3: 0.248, 4: 0.290}},
         "bf16_160": {(BAND, 0): {1: 0.196}, (FFT, 160): {1: 0.288, 2: 0.380}}}


@pytest.mark.parametrize("case,dtype,m,R", [("f32_96", F32, 41, 25), ("bf16_96", BF16, 41, 25), ("bf16_160", BF16, 81, 30)])
@pytest.mark.parametrize("first", [100, 304, 456, 2000])
def test_few_points_and_many_take_the_form_that_is_faster_for_them(lib, case, dtype, m, R, first):
    """One measurement per (dtype, m, R), on the first call's points, serves calls of any
    number of points: none takes a form that is over 10 % slower than the best for
    it (a first call of up to a point per SM knows only that and keeps its choice)."""
    ctx = Ctx(lib)
    forms = COSTS[case]
    lib.fk_no_costs()
    for (path, side), by_waves in forms.items():
        for w, ms in by_waves.items():
            lib.fk_cost(1000 * path + side, w, ms)

    def cost(path, side, n):
        by, k = forms[path, side], (n + 151) // 152
        period = max(by)
        return k // period * by[period] + (by[k % period] if k % period else 0.0)

    cubes = [ctx.build(700, 700, params(ctx, dtype)) for _ in range(2)]
    other = Ctx(lib)
    ctx.match(*cubes, first, m, R)
    counted = ctx.launches()
    n = C.c_size_t()
    ctx.ok(lib.sfoc_ctx_autotune_export(ctx.h, None, 0, C.byref(n)))
    text = C.create_string_buffer(n.value)
    ctx.ok(lib.sfoc_ctx_autotune_export(ctx.h, text, n, C.byref(n)))
    other.ok(lib.sfoc_ctx_autotune_import(other.h, text))
    for points in (1, 100, 152, 153, 304, 400, 456, 608, 1216, 5000):
        form = ctx.match(*cubes, points, m, R)
        assert other.match(*cubes, points, m, R) == form        # and after a round trip through the text
        if first > 152 or points <= 152:
            best = min(cost(p, s, points) for p, s in forms)
            assert cost(*divmod(form, 1000), points) <= 1.1 * best, (points, form)
    assert ctx.launches() - counted < 10 * 8                   # nothing is measured again
    # text without the numbers of points: its form for every call
    path, side = list(forms)[-1]
    plain = ('{"entries": [{"dtype": %d, "family": 0, "m": %d, "R": %d, "path": %d, "option": %d, "sample": 1, '
             '"candidates": []}]}' % (dtype, m, R, path, side)).encode()
    ctx.ok(lib.sfoc_ctx_autotune_import(ctx.h, plain))
    assert {ctx.match(*cubes, k, m, R) for k in (1, 500, 5000)} == {1000 * path + side}
    bad = plain.replace(b'"candidates"', b'"waves": [%d, %d, 7, 0, 6, 64, 6, 64], "candidates"' % (path, side))
    assert lib.sfoc_ctx_autotune_import(ctx.h, bad) != 0
    for c in cubes:
        assert lib.sfoc_cube_free(c) == 0
    other.close()
    ctx.close()


def test_a_sample_that_leaves_the_chip_idle_promises_nothing_for_more_points(lib):
    """The direct kernel runs three points of m = 15, R = 1 on an SM at a time: 304
    points take no longer than 152, which says nothing about 608."""
    ctx = Ctx(lib)
    lib.fk_no_costs()
    for (path, side), by_waves in {(FFT, 64): (0.028, 0.038), (FFT, 128): (0.075,), (DIRECT, 0): (0.0567, 0.0568, 0.0589)}.items():
        for w, ms in enumerate(by_waves):
            lib.fk_cost(1000 * path + side, w + 1, ms)
    cubes = [ctx.build(400, 400) for _ in range(2)]
    assert [ctx.match(*cubes, n, 15, 1) for n in (304, 100, 608, 1216, 5000)] == [1000 * FFT + 64] * 5
    for c in cubes:
        assert lib.sfoc_cube_free(c) == 0
    ctx.close()


def test_the_sm_count_is_asked_once(ctx):
    """Not on every call: small calls wait for the host."""
    cubes = [ctx.build(300, 300) for _ in range(2)]
    ctx.match(*cubes, 200, 41, 10)
    ctx.L.fk_reset()
    for n in (10, 200, 1000):
        ctx.match(*cubes, n, 41, 10)
        ctx.ok(ctx.pair((300, 300), (300, 300)))
    assert ctx.L.fk_count(b"attribute") == 0
    for c in cubes:
        assert ctx.L.sfoc_cube_free(c) == 0


def test_launch_plans_ask_the_device_for_its_sms():
    """Segment heights and grids that fill the chip follow the device's SM count."""
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            code = [line.split("//")[0] for line in f]
        assert not [c for c in code if "152" in c], name
