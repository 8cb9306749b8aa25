"""What the entry points do on the host, on the CPU with a runtime that only
writes down its calls."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
import fake_api  # noqa: E402
from paper_2212_00488_gb300 import _lib  # noqa: E402

pytestmark = pytest.mark.skipif(not fake_api.available(), reason="needs the CUDA headers and g++")

CALLER = 0x77       # the caller's stream


@pytest.fixture(scope="module")
def fake_lib(tmp_path_factory):
    return fake_api.build(tmp_path_factory.mktemp("fake"))


@pytest.fixture
def fake(fake_lib, monkeypatch):
    monkeypatch.setattr(_lib, "_lib", fake_lib)      # the binding's functions call the fake
    fake_lib.fake_reset()
    return fake_lib


def _lines(fake):
    return [ln.split() for ln in fake.fake_log().decode().splitlines()]


def _context(**params):
    p = _lib.stereo_default_params()
    for k, v in params.items():
        setattr(p, k, v)
    return _lib.stereo_create(0, p)


def _jobs(widths):
    return [_lib.stereo_job(1, 1, w, 60, 16, 1, None, None, None) for w in widths]


def _caller_waits_for_all(lines):
    """The last launch is followed by an event of its stream that the caller's stream waits for."""
    last = max(i for i, ln in enumerate(lines) if ln[0] in ("launch", "graph"))
    own = lines[last][-1]
    after = lines[last + 1:]
    return any(a[0] == "record" and a[2] == own and ["wait", f"{CALLER:x}", a[1]] in after[i + 1:]
               for i, a in enumerate(after))


@pytest.mark.parametrize("fail", [None, 0, 1, 2, 3])
@pytest.mark.parametrize("what", ["batch", "forward", "backward"])
def test_caller_waits_for_what_was_queued_also_after_an_error(fake, what, fail):
    # the kernels run on the context's stream; those queued before one fails still
    # read the caller's inputs, so the caller's stream has to come after them
    ctx = _context()
    _lib.stereo_set_tile(ctx, 1)
    fake.fake_reset()
    if fail is not None:
        fake.fake_fail_at(fail)

    def call():
        if what == "batch":
            _lib.stereo_compute_batch(ctx, _jobs([80, 80]), CALLER)
        elif what == "forward":
            _lib.stereo_diff_forward(ctx, 1, 8, 8, 4, 1, 1, 1, 1, 1, 0.1, 1, 1, CALLER)
        else:
            _lib.stereo_diff_backward(ctx, 1, 8, 8, 4, 1, 1, 1, 1, 1, 0.1, 1, 1, 1, 1, 1, 1, CALLER)
    if fail is None:
        call()
    else:
        with pytest.raises(_lib.StereoError) as e:
            call()
        assert e.value.code == _lib.STEREO_ECUDA and "a call failed" in str(e.value)
    assert _caller_waits_for_all(_lines(fake))
    _lib.stereo_destroy(ctx)


def _tile_of(ctx, jobs):
    _lib.stereo_compute_batch(ctx, jobs, CALLER)
    return _lib.stereo_batch_tile(ctx)[0]


def test_a_remembered_tile_holds_for_its_matching_costs_only(fake, tmp_path):
    # at wx 33 the 16-bit tile fits the default costs (67 P < 2^16) and not those
    # of lambda_ad 0.2: the other context's choice must not be taken for its own
    path = str(tmp_path / "tune.txt")
    a, b = _context(wx=33), _context(wx=33, lambda_ad=0.2)
    jobs = _jobs([80])
    assert _tile_of(a, jobs) == 0
    assert _lib.stereo_tune_save(a, path) == 1
    assert _lib.stereo_tune_load(b, path) == 1
    assert _tile_of(b, jobs) == 1
    # each finds its own choice again, without tuning, from one file
    assert _lib.stereo_tune_save(b, path) == 2
    for params, tile in ((dict(wx=33), 0), (dict(wx=33, lambda_ad=0.2), 1)):
        c = _context(**params)
        assert _lib.stereo_tune_load(c, path) == 2
        fake.fake_reset()
        assert _tile_of(c, jobs) == tile
        assert sum(ln[:2] == ["launch", "batch"] for ln in _lines(fake)) == 1
        _lib.stereo_destroy(c)
    _lib.stereo_destroy(a)
    _lib.stereo_destroy(b)


def test_a_remembered_tile_that_does_not_fit_is_tuned_again(fake, tmp_path):
    path = tmp_path / "tune.txt"
    a = _context(wx=40)                     # 81 P > 2^16: not the 16-bit tile
    jobs = _jobs([80])
    assert _tile_of(a, jobs) == 1
    _lib.stereo_tune_save(a, str(path))
    sig = path.read_text().split("\t")[0]
    path.write_text(f"{sig}\t0\n")
    c = _context(wx=40)
    assert _lib.stereo_tune_load(c, str(path)) == 1
    assert _tile_of(c, jobs) == 1
    _lib.stereo_destroy(a)
    _lib.stereo_destroy(c)


def test_batches_of_aligned_and_of_mixed_frames_keep_a_graph_each(fake):
    # frames whose rows are word-aligned and others take a grey launch each, so
    # batches of one size come in two topologies; taking them in turn must not
    # instantiate a graph again on every call
    ctx = _context()
    _lib.stereo_set_tile(ctx, 1)
    fake.fake_reset()
    for _ in range(3):
        for widths in ([80] * 6, [80] * 3 + [81] * 3, [81] * 6):
            _lib.stereo_compute_batch(ctx, _jobs(widths), CALLER)
    lines = _lines(fake)
    assert sum(ln[0] == "graph" for ln in lines) == 9
    assert sum(ln[0] == "instantiate" for ln in lines) == 2
    _lib.stereo_destroy(ctx)


@pytest.mark.parametrize("downscale", [0, 1])
def test_a_frame_takes_the_planes_it_uses(fake, downscale):
    p = _lib.stereo_default_params()
    p.downscale = downscale
    W, H = 642, 481
    X, Y = (W // 2, H // 2) if downscale else (W, H)
    n = X * Y
    # full-res grey of the left image beside both processed ones, or the processed ones alone; pixel and arm
    # words, the fused kernel's arm words (whole row quads), keys; medians and filled map
    planes = [W * H] * downscale + [n] * 2 + [4 * n] * 6 + [4 * X * ((Y + p.wy + 3) // 4 * 4)] * 2 + [n, 4 * n]
    assert _lib.stereo_job_bytes(p, W, H, 64) == sum((b + 255) // 256 * 256 for b in planes) + 256


@pytest.mark.parametrize("what", ["query", "launch"])
def test_a_call_after_one_that_failed_is_not_refused_for_it(fake, what):
    # the runtime keeps a failed call's error until it is asked for, and the grey
    # conversion's launch reports what it is then told
    ctx = _context(downscale=0)
    _lib.stereo_set_tile(ctx, 1)
    fake.fake_reset()
    if what == "query":
        fake.fake_fail_query(1)
    else:
        fake.fake_fail_at(3)
    with pytest.raises(_lib.StereoError):
        _lib.stereo_compute_batch(ctx, _jobs([80, 80]), CALLER)
    fake.fake_fail_query(0)
    fake.fake_fail_at(-1)
    _lib.stereo_compute(ctx, 1, 1, 80, 60, 16, 1, 0, 0, 0, CALLER)
    _lib.stereo_destroy(ctx)
