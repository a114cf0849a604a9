"""Period end with several node rows per thread (meshes of many blocks) against
the oracle: mesh sizes at the change-over, with whole and ragged last blocks, on
the coarse and on the fine mesh."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import dmr_oracle as O  # noqa: E402
from paper_2105_13276_gb300 import dmr as D  # noqa: E402
from paper_2105_13276_gb300 import workloads as W  # noqa: E402
from tests.test_gpu_parity import TOL32, TOL64, compare  # noqa: E402


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("r,nx,ny,rect", [(1, 1023, 599, None), (1, 1023, 607, None), (1, 1024, 608, None),
                                          (1, 1000, 640, None), (2, 550, 330, (10, 9, 523, 323))])
def test_period_end_matches_the_oracle(r, nx, ny, rect, precision):
    w = W.small_dmr(nx=nx, ny=ny, r=r, rect=rect, precision=precision, growth=0)
    steps = w["cfg"]["steps_per_period"]
    sim, run = O.sim_from_workload(w), D.run_from_workload(w)
    sim.advance(steps)
    run.advance(steps)
    tol = TOL64 if precision == 0 else TOL32
    compare(run, sim, tol, fields=("n",), levels=(0, 1) if r > 1 else (0,), s2=False)
    st = run.stats()
    assert abs(st["N_e"] / sim.N_e - 1) < tol
    assert abs(st["P_abs"] / sim.P_abs - 1) < tol
