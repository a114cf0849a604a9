"""Which launches a run's periods are made of: what the rules on sizes choose,
seen from outside (launch counts and the buffer parities in a saved state)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2105_13276_gb300 import dmr as D  # noqa: E402
from paper_2105_13276_gb300 import workloads as W  # noqa: E402

FIELDS = ("Ex", "Ey", "Hz", "vx", "vy", "n", "S2", "erms")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2105_13276_gb300 import build as B
    B.build()
    D.load()


def _centre(nx, ny, w, h):
    i, j = (nx - w) // 2, (ny - h) // 2
    return (i, j, i + w, j + h)


def _run(nx, ny, r, rect, NT=64, strips=False, seed=3, **kw):
    run = D.Run(W.base_cfg(nx=nx, ny=ny, r=r, n_lambda=NT // 2, steps_per_period=NT, precision=1, growth=0, **kw))
    if r > 1:
        run.set_patch(rect)
    if strips:
        run.set_launch_shape(48)
    scale = dict(Ex=1e5, Ey=1e5, Hz=3e2, vx=1e4, vy=1e4)
    for level in range(2 if r > 1 else 1):
        for k, f in enumerate(scale):
            run.write(f, level, W.random_fields(run.shape(f, level)[0], seed + 10 * level + k, scale[f]))
    run.seed_gaussian(1e14, 0.5 * nx * run.dxc, 0.5 * ny * run.dxc, 0.1 * run.lam, 0.1 * run.lam)
    return run


def _equal(a, b, r):
    for level in range(2 if r > 1 else 1):
        for f in FIELDS:
            assert np.array_equal(a.read(f, level), b.read(f, level)), (f, level)


def _parities(run):
    """Buffer parities of the coarse and the fine fields (header of a saved state)."""
    h = run.save_state()[:40].cpu().numpy().view(np.int32)
    return int(h[8]), int(h[9])


def _launches(run, steps):
    n = run.launch_count()
    run.advance(steps)
    return run.launch_count() - n


SHAPES = [(100, 70, 1, 0), (96, 90, 2, 20), (160, 150, 2, 12), (170, 130, 3, 12)]


@pytest.mark.parametrize("nx,ny,r,w,NT", [s + (NT,) for s in SHAPES for NT in (20, 36, 60, 63, 64, 100, 120)] +
                         [(96, 90, 3, 40, 64), (96, 90, 3, 40, 36)])
def test_a_period_ends_in_the_parity_it_started_with(nx, ny, r, w, NT):
    """A captured period is replayed only then; each period takes the same
    launches, fewer than one per step and sub-step, with the same bits."""
    rect = _centre(nx, ny, w, w) if r > 1 else None
    a, b = _run(nx, ny, r, rect, NT), _run(nx, ny, r, rect, NT, strips=True)
    a.set_graphs(True)
    a.advance(NT)
    b.advance(NT)
    par = _parities(a)
    counts = set()
    for _ in range(3):
        counts.add(_launches(a, NT))
        assert _parities(a) == par
    assert len(counts) == 1
    assert counts.pop() < _launches(b, NT)
    b.advance(2 * NT)
    _equal(a, b, r)


@pytest.mark.parametrize("calls", [(7, 9, 16, 32), (32, 32), (1, 63), (3, 13, 48), (64,), (5, 27, 100, 60)])
def test_a_period_in_parts(calls):
    """Calls that stop inside a period and go on between its groups."""
    for nx, ny, r, w in [(100, 70, 1, 0), (160, 150, 2, 12), (96, 90, 3, 20)]:
        rect = _centre(nx, ny, w, w) if r > 1 else None
        a, b = _run(nx, ny, r, rect), _run(nx, ny, r, rect, strips=True)
        for n in calls:
            a.advance(n)
            b.advance(n)
        _equal(a, b, r)


@pytest.mark.parametrize("nx,ny,r,w", [(320, 310, 2, 58), (110, 100, 3, 41), (110, 100, 4, 31), (160, 150, 6, 18)])
def test_a_rectangle_that_fits_for_fewer_steps_only(nx, ny, r, w):
    """Too large a window for 8 steps per launch, not for 3 to 7."""
    rect = _centre(nx, ny, w, w)
    a, b = _run(nx, ny, r, rect), _run(nx, ny, r, rect, strips=True)
    assert _launches(a, 64) < 64        # one per coarse step at least otherwise
    b.advance(64)
    _equal(a, b, r)
    a.autotune()
    a.set_graphs(True)
    a.advance(128)
    b.advance(128)
    _equal(a, b, r)


def test_strips_where_a_shorter_group_is_slower():
    """r = 2 on a small mesh."""
    nx, ny, w = 160, 140, 58
    rect = _centre(nx, ny, w, w)
    a, b = _run(nx, ny, 2, rect), _run(nx, ny, 2, rect, strips=True)
    assert _launches(a, 64) == _launches(b, 64)
    _equal(a, b, 2)


@pytest.mark.parametrize("nx,ny,w,strips", [(120, 110, 16, (2, 3)), (70, 64, 16, (2,)), (40, 32, 8, ()),
                                             (200, 150, 54, (2, 3, 4))])
def test_calls_of_few_steps(nx, ny, w, strips):
    """r = 2: two to four steps in one launch only where the near region is small."""
    rect = _centre(nx, ny, w, w)
    a, b = _run(nx, ny, 2, rect), _run(nx, ny, 2, rect, strips=True)
    for k in (2, 3, 4, 2, 5):
        n, m = _launches(a, k), _launches(b, k)
        assert m == 2 * k
        assert n == m if k in strips else n < m, k
    _equal(a, b, 2)


@pytest.mark.parametrize("nx,ny,w,h,strips", [
    (150, 150, 49, 8, True), (400, 100, 49, 8, True), (400, 100, 8, 49, False), (300, 50, 49, 8, True),
    (150, 150, 32, 32, True), (512, 512, 32, 32, False), (512, 512, 50, 50, True), (973, 51, 16, 16, False)])
def test_calls_of_two_steps_by_the_rectangles_shape(nx, ny, w, h, strips):
    """r = 2: the rows that the near region's warps step, not its nodes."""
    rect = _centre(nx, ny, w, h)
    a, b = _run(nx, ny, 2, rect), _run(nx, ny, 2, rect, strips=True)
    for _ in range(3):
        n, m = _launches(a, 2), _launches(b, 2)
        assert (n == m) if strips else (n < m)
    _equal(a, b, 2)


@pytest.mark.parametrize("nx,ny,r,w,h,captured,direct", [
    (200, 150, 4, 40, 40, 4, 2), (200, 150, 4, 80, 60, 2, 2), (200, 150, 3, 50, 50, 3, 2), (200, 150, 2, 70, 60, 2, 2),
    (512, 400, 4, 40, 40, 4, 4), (512, 400, 4, 60, 50, 4, 2), (200, 150, 5, 30, 30, 2, 2), (100, 96, 4, 40, 36, 2, 2)])
def test_fine_sub_steps_of_a_small_fine_mesh(nx, ny, r, w, h, captured, direct):
    """Launches per coarse step of a rectangle too large for the near region:
    r strips, or the coarse step's and one of fine tiles."""
    NT, rect = 64, _centre(nx, ny, w, h)
    a, b = _run(nx, ny, r, rect), _run(nx, ny, r, rect, strips=True)
    assert _launches(a, 8) == 8 * direct
    a.advance(NT - 8)
    a.set_graphs(True)
    a.advance(NT)
    b.advance(2 * NT)
    _equal(a, b, r)
    end = _launches(b, NT) - r * NT      # the period end's launches
    assert _launches(a, NT) == captured * NT + end
    _equal(a, b, r)


@pytest.mark.parametrize("nx,ny,r,w,h,direct", [(51, 973, 4, 20, 20, 4), (51, 973, 3, 30, 30, 3), (51, 973, 4, 40, 24, 2),
                                                (60, 2000, 4, 20, 20, 2)])
def test_fine_sub_steps_in_a_narrow_domain(nx, ny, r, w, h, direct):
    """Too narrow for the near region, launched one by one."""
    rect = _centre(nx, ny, w, h)
    a, b = _run(nx, ny, r, rect), _run(nx, ny, r, rect, strips=True)
    assert _launches(a, 8) == 8 * direct
    b.advance(8)
    _equal(a, b, r)


@pytest.mark.parametrize("nx,ny,r,w,h,kw,captured,direct", [
    (64, 183, 4, 16, 54, {}, 4, 2), (40, 212, 4, 40, 9, {}, 2, 2), (64, 183, 4, 30, 54, dict(coupling=1), 4, 2), (150, 120, 3, 50, 50, {}, 3, 2), (232, 87, 3, 115, 4, {}, 3, 2),
    (89, 705, 3, 76, 95, dict(coupling=1), 3, 3), (301, 187, 3, 90, 90, dict(coupling=1), 3, 3),
    (301, 187, 3, 90, 90, dict(coupling=1, boundary=1), 3, 3), (301, 187, 3, 90, 90, {}, 2, 2),
    (600, 300, 4, 50, 50, {}, 2, 2), (200, 150, 4, 76, 95, {}, 2, 2), (200, 150, 3, 120, 120, dict(coupling=1), 2, 2)])
def test_fine_sub_steps_by_the_sizes_of_both_meshes(nx, ny, r, w, h, kw, captured, direct):
    NT, rect = 64, _centre(nx, ny, w, h)
    a, b = _run(nx, ny, r, rect, **kw), _run(nx, ny, r, rect, strips=True, **kw)
    assert _launches(a, 8) == 8 * direct
    a.advance(NT - 8)
    a.set_graphs(True)
    a.advance(NT)
    b.advance(2 * NT)
    end = _launches(b, NT) - r * NT
    assert _launches(a, NT) == captured * NT + end
    _equal(a, b, r)


def test_the_autotuner_compares_like_with_like():
    """Groups of 6 or 7 steps, 15 % faster here than the tuned form of one step
    (timed without its E^2 sample that form was chosen); the run is as before."""
    nx, ny, r, w = 110, 100, 4, 31
    rect = _centre(nx, ny, w, w)
    a, b = _run(nx, ny, r, rect), _run(nx, ny, r, rect, strips=True)
    a.set_graphs(True)
    a.autotune()
    _equal(a, b, r)
    assert _launches(a, 64) < 64
    b.advance(64)
    _equal(a, b, r)


@pytest.mark.parametrize("force", [lambda run: run.set_launch_shape(48), lambda run: run.set_strip_columns(2)])
def test_the_autotuner_replaces_a_forced_shape(force):
    nx, ny, r, w = 200, 150, 3, 20
    rect = _centre(nx, ny, w, w)
    a, b = _run(nx, ny, r, rect), _run(nx, ny, r, rect, strips=True)
    force(a)
    assert _launches(a, 64) == _launches(b, 64)
    a.autotune()
    assert _launches(a, 64) < 64
    b.advance(64)
    _equal(a, b, r)
