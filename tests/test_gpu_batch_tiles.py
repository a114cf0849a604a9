"""Batches whose whole periods take several coarse steps per launch: runs with
tiles (more than 20000 cells) among runs that the near region steps whole, on
both sides of the 40 runs that one launch takes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2105_13276_gb300 import dmr as D  # noqa: E402
from paper_2105_13276_gb300 import workloads as W  # noqa: E402

FIELDS = ("Ex", "Ey", "Hz", "vx", "vy", "n", "S2", "erms")
NT = 32
# run of the batch: size and rectangle (inside, at sides, in corners)
TILED = {0: (201, 151, (189, 142, 201, 151)), 1: (173, 260, (0, 250, 9, 260)), 13: (311, 97, (150, 0, 162, 9)),
         38: (160, 129, (70, 60, 76, 66)), 39: (173, 260, (80, 128, 92, 137)), 40: (201, 151, (0, 0, 12, 9)),
         41: (311, 97, (299, 40, 311, 49)), 43: (64, 400, (3, 193, 14, 200))}
# the same with more than a million nodes in all
LARGE = {**TILED, 2: (700, 611, (300, 301, 312, 310)), 42: (613, 1100, (601, 0, 613, 9))}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2105_13276_gb300 import build as B
    B.build()
    D.load()


def _start(run, rect, k):
    run.set_patch(rect)
    scale = dict(Ex=1e5, Ey=1e5, Hz=3e2, vx=1e4, vy=1e4)
    for level in (0, 1):
        for q, f in enumerate(scale):
            run.write(f, level, W.random_fields(run.shape(f, level)[0], 100 * k + 10 * level + q, scale[f]))
    run.seed_gaussian(1e14, rect[0] * run.dxc, rect[1] * run.dxc, 0.1 * run.lam, 0.1 * run.lam)


@pytest.mark.parametrize("r,tiled", [(2, TILED), (2, LARGE), (4, TILED), (6, TILED)])
def test_tiled_runs_in_a_batch(r, tiled):
    rng = np.random.default_rng(7)
    cfgs, rects = [], []
    for k in range(45):
        nx, ny, rect = tiled.get(k, (int(rng.integers(63, 130)), int(rng.integers(63, 120)), None))
        if rect is None:
            i0, j0 = int(rng.integers(0, nx - 12)), int(rng.integers(0, ny - 9))
            rect = (i0, j0, i0 + 12, j0 + 9)
        assert (k in tiled) == (nx * ny > 20000)
        cfgs.append(W.base_cfg(nx=nx, ny=ny, r=r, n_lambda=NT // 2, steps_per_period=NT, precision=1, growth=0,
                               E0=float(rng.uniform(3e6, 6e6)), coupling=int(rng.integers(0, 2))))
        rects.append(rect)
    a, b = D.Batch(cfgs), D.Batch(cfgs)          # whole periods; graphs off: step by step
    b.set_graphs(False)
    for batch in (a, b):
        for k, (run, rect) in enumerate(zip(batch.runs, rects)):
            _start(run, rect, k)
    counts = []
    for batch in (a, b):
        batch.advance(NT)
        n = batch.launch_count()
        batch.advance(NT)
        counts.append(batch.launch_count() - n)
    ends = counts[1] - r * NT                     # the period end's launches
    assert counts[0] - ends <= NT < r * NT, counts
    for k in range(45):
        for level in (0, 1):
            for f in FIELDS:
                assert np.array_equal(a.runs[k].read(f, level), b.runs[k].read(f, level)), (k, f, level)
    # one step per launch of a single run, over a period's end and into the next
    a.advance(NT + 5)
    for k in tiled:
        one = D.Run(cfgs[k])
        one.set_launch_shape(48)
        _start(one, rects[k], k)
        one.advance(3 * NT + 5)
        for level in (0, 1):
            for f in FIELDS:
                assert np.array_equal(a.runs[k].read(f, level), one.read(f, level)), (k, f, level)


@pytest.mark.parametrize("n,size,r,w,grouped", [
    (8, 100, 2, 10, True), (24, 100, 2, 24, True), (100, 70, 2, 24, False), (100, 100, 2, 24, False),
    (64, 128, 2, 10, True), (64, 70, 4, 10, False), (15, 70, 2, 50, True)])
def test_many_small_runs(n, size, r, w, grouped):
    """Groups of steps only while the near regions' turns are shorter than the strips."""
    i = (size - w) // 2
    cfgs = [W.base_cfg(nx=size, ny=size - q % 3, r=r, n_lambda=NT // 2, steps_per_period=NT, precision=1, growth=0,
                       patch_cap_cells=(r * w) ** 2) for q in range(n)]
    a, b = D.Batch(cfgs), D.Batch(cfgs)
    b.set_graphs(False)
    counts = []
    for batch in (a, b):
        for k, run in enumerate(batch.runs):
            _start(run, (i, i, i + w, i + w), k)
        batch.advance(NT)
        c = batch.launch_count()
        batch.advance(NT)
        counts.append(batch.launch_count() - c)
    assert (counts[0] < counts[1]) == grouped and counts[0] <= counts[1], counts
    for k in (0, n // 2, n - 1):
        for level in (0, 1):
            for f in FIELDS:
                assert np.array_equal(a.runs[k].read(f, level), b.runs[k].read(f, level)), (k, f, level)
