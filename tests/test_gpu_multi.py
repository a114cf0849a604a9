"""Several coarse steps per launch (FP32, Mur sides): the same bits as one
launch per EM step and sub-step, in every field of both meshes, the running
E^2 sums, E_rms and the mask, after each call of a sequence of step counts.

A run whose launch shape is set takes the one-step launches, so it is the
reference.  Sizes at the tiles' edges (64 columns, rows of a tile), odd and
ragged ones, rectangles inside, at sides and in corners, thin and one coarse
cell wide, r = 2..5, both coupling readings, step counts that split a period,
graphs, and a domain that the near region steps whole."""
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


def _pair(nx, ny, r, rect, seed=3, **kw):
    cfg = W.base_cfg(nx=nx, ny=ny, r=r, n_lambda=16, steps_per_period=32, precision=1, growth=0, **kw)
    runs = []
    for one_step in (False, True):
        run = D.Run(cfg)
        if r > 1:
            run.set_patch(rect)
        if one_step:
            run.set_launch_shape(48)
        scale = dict(Ex=1e5, Ey=1e5, Hz=3e2, vx=1e4, vy=1e4)
        for level in range(2 if r > 1 else 1):
            for k, f in enumerate(scale):
                run.write(f, level, W.random_fields(run.shape(f, level)[0], seed + 10 * level + k, scale[f]))
        run.seed_gaussian(3e17, 0.5 * nx * run.dxc, 0.5 * ny * run.dxc, 0.1 * run.lam, 0.1 * run.lam)
        runs.append(run)
    return runs


def _same(a, b, r, steps):
    for n in steps:
        a.advance(n)
        b.advance(n)
        for level in range(2 if r > 1 else 1):
            for f in FIELDS:
                assert np.array_equal(a.read(f, level), b.read(f, level)), (n, f, level)
    if r > 1:
        assert np.array_equal(a.read("mask"), b.read("mask"))
    assert a.launch_count() < b.launch_count()


@pytest.mark.parametrize("nx,ny", [(63, 40), (64, 33), (127, 64), (129, 97), (200, 31), (301, 187)])
def test_uniform_mesh(nx, ny):
    a, b = _pair(nx, ny, 1, None)
    _same(a, b, 1, [2, 3, 7, 4, 32])


@pytest.mark.parametrize("nx,ny,r,rect", [
    (200, 151, 2, (90, 70, 102, 80)), (301, 187, 2, (290, 1, 299, 7)), (200, 150, 3, (0, 70, 15, 90)),
    (200, 150, 4, (188, 140, 200, 150)), (200, 150, 2, (0, 0, 9, 3)), (211, 143, 2, (100, 71, 101, 73)),
    (160, 129, 5, (70, 60, 76, 66))])
def test_rectangle_with_tiles_around_it(nx, ny, r, rect):
    a, b = _pair(nx, ny, r, rect)
    _same(a, b, r, [2, 3, 4, 7, 16, 32])


@pytest.mark.parametrize("nx,ny,r,rect", [
    (96, 96, 2, (73, 40, 89, 56)), (40, 32, 2, (12, 10, 24, 20)), (33, 41, 3, (0, 10, 12, 41)), (64, 20, 2, (3, 2, 33, 18)),
    (20, 90, 4, (8, 40, 12, 44))])
@pytest.mark.parametrize("coupling", [0, 1])
def test_whole_domain_in_the_near_region(nx, ny, r, rect, coupling):
    a, b = _pair(nx, ny, r, rect, coupling=coupling)
    _same(a, b, r, [8, 24, 5, 59])


@pytest.mark.parametrize("nx,ny,r,rect", [(200, 151, 2, (90, 70, 102, 80)), (96, 96, 2, (73, 40, 89, 56)), (129, 97, 1, None)])
def test_graphs_and_autotuner(nx, ny, r, rect):
    a, b = _pair(nx, ny, r, rect)
    a.set_graphs(True)
    _same(a, b, r, [32, 64, 5, 27])
    a.autotune()
    before = {f: a.read(f, level) for f in FIELDS for level in range(1)}
    assert all(np.array_equal(before[f], b.read(f)) for f in FIELDS)
    for n in (32, 64):
        a.advance(n)
        b.advance(n)
    for level in range(2 if r > 1 else 1):
        for f in FIELDS:
            assert np.array_equal(a.read(f, level), b.read(f, level)), (f, level)


def test_growth_in_free_running_mode():
    """The rectangle grows out of the near region's first plan; same log, same bits."""
    w = W.small_dmr(nx=180, ny=130, rect=(70, 60, 82, 70), precision=1)
    runs = [D.run_from_workload(w) for _ in range(2)]
    runs[1].set_launch_shape(48)
    grown = {tuple(w["rect"])}
    for _ in range(8):
        for run in runs:
            run.advance(32)
        assert runs[0].get_patch() == runs[1].get_patch()
        grown.add(runs[0].get_patch())
        for level in (0, 1):
            for f in FIELDS:
                assert np.array_equal(runs[0].read(f, level), runs[1].read(f, level)), (f, level)
    assert len(grown) > 1


def test_batch_of_more_runs_than_one_launch_takes():
    """43 runs of uneven sizes (40 per launch): each has the bits of its own run
    with one launch per step; whole periods in groups, the rest step by step."""
    rng = np.random.default_rng(5)
    sizes = [(int(rng.integers(63, 170)), int(rng.integers(60, 150))) for _ in range(43)]
    cfgs, rects = [], []
    for nx, ny in sizes:
        cfgs.append(W.base_cfg(nx=nx, ny=ny, r=2, n_lambda=16, steps_per_period=32, precision=1, growth=0,
                               E0=float(rng.uniform(3e6, 6e6)), coupling=int(rng.integers(0, 2))))
        i0, j0 = int(rng.integers(0, nx - 12)), int(rng.integers(0, ny - 9))
        rects.append((i0, j0, i0 + 12, j0 + 9))
    batch = D.Batch(cfgs)
    for run, rect in zip(batch.runs, rects):
        run.set_patch(rect)
        run.seed_gaussian(3e17, rect[0] * run.dxc, rect[1] * run.dxc, 0.1 * run.lam, 0.1 * run.lam)
    batch.advance(64)
    batch.advance(5)
    for q in (0, 17, 39, 40, 42):
        one = D.Run(cfgs[q])
        one.set_launch_shape(48)
        one.set_patch(rects[q])
        one.seed_gaussian(3e17, rects[q][0] * one.dxc, rects[q][1] * one.dxc, 0.1 * one.lam, 0.1 * one.lam)
        one.advance(69)
        for level in (0, 1):
            for f in FIELDS:
                assert np.array_equal(batch.runs[q].read(f, level), one.read(f, level)), (q, f, level)


@pytest.mark.parametrize("nx,ny,r,rect,kw", [
    (120, 90, 3, (20, 11, 61, 44), {}), (120, 90, 4, (20, 11, 37, 28), {}), (120, 90, 4, (0, 0, 50, 33), {}),
    (120, 90, 3, (70, 50, 120, 90), {}), (100, 90, 5, (3, 2, 16, 81), {}), (100, 90, 8, (30, 40, 38, 47), {}),
    (100, 80, 4, (0, 7, 100, 70), dict(coupling=1)), (121, 97, 3, (30, 31, 75, 62), dict(boundary=1)),
    (33, 20, 16, (4, 3, 9, 9), {}), (130, 70, 3, (10, 10, 32, 26), {})])
def test_fine_sub_steps_in_one_launch(nx, ny, r, rect, kw):
    """Fine meshes of a tile and more (64 columns): one column past a tile's,
    ragged, at sides and corners, r that divides neither the columns nor the
    rows of a tile, both couplings, CPML outside."""
    a, b = _pair(nx, ny, r, rect, **kw)
    _same(a, b, r, [1, 2, 13, 16, 5])


@pytest.mark.parametrize("r", [2, 3])
def test_fine_tiles_after_the_autotuner(r):
    a, b = _pair(150, 140, r, (10, 20, 131, 122))
    a.autotune()
    a.set_graphs(True)
    for n in (32, 64, 7):
        a.advance(n)
        b.advance(n)
        for level in (0, 1):
            for f in FIELDS:
                assert np.array_equal(a.read(f, level), b.read(f, level)), (n, f, level)
