"""Flags of the period end (Sec. III.A-III.D): each block reduces its nodes'
flags and adds them to the control block once.  Mesh sizes around the blocks of
32 x 8 nodes; a density that is nowhere zero, one that is flagged everywhere,
one that is flagged nowhere, and a NaN at a block's edge."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2105_13276_gb300 import dmr as D  # noqa: E402
from paper_2105_13276_gb300 import workloads as W  # noqa: E402


def _run(nx, ny, precision, n):
    cfg = W.base_cfg(nx=nx, ny=ny, r=2, n_lambda=16, steps_per_period=32, growth=0, precision=precision)
    run = D.Run(cfg)
    run.set_patch((nx // 4, ny // 4, nx // 4 + 2, ny // 4 + 2))
    run.write("n", 1, np.full(run.shape("n", 1)[0], n.flat[0]))
    run.write("n", 0, n)
    return run, cfg


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx,ny", [(30, 6), (31, 7), (32, 8), (63, 33), (95, 17)])
@pytest.mark.parametrize("level", [1e-11, 1e16, 1e19])
def test_flag_sums_equal_the_mask(nx, ny, precision, level):
    rng = np.random.default_rng(nx * 100 + ny)
    n = level * (1.0 + rng.random((ny + 1, nx + 1)))
    run, cfg = _run(nx, ny, precision, n)
    run.advance(cfg["steps_per_period"])
    st, mask, now = run.stats(), run.read("mask"), run.read("n")
    assert st["n_max"] == float(now.max()) > 0.0
    assert st["flags"] == int(mask.sum())
    assert (mask.sum() > 0) == (level > 1e16) and (level < 1e18 or mask.all())


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("at", [(0, 0), (7, 31), (8, 32), (17, 40)])
def test_a_nan_node_stops_the_run(precision, at):
    n = np.full((18, 41), 1e15)
    n[at] = np.nan
    run, cfg = _run(40, 17, precision, n)
    with pytest.raises(D.DMRError) as e:
        run.advance(cfg["steps_per_period"])
    assert e.value.code == D.EUNSTABLE
