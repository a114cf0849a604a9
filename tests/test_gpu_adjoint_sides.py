"""FP64 adjoint against complex-step derivatives where the reversed step's node
formulas meet: mesh sizes around its blocks of 32 x 8 nodes, rectangles in the
middle, at domain sides and in corners (fine meshes with Mur sides), one coarse
cell wide (a Mur row and column next to both sides), r = 2 and 3."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import dmr_oracle as O  # noqa: E402
from paper_2105_13276_gb300 import workloads as W  # noqa: E402
from tests.test_gpu_adjoint import TOL_ADJ64, cs_grads, gpu_grads, oracle_run  # noqa: E402


@pytest.mark.parametrize("nx,ny,r,rect", [(31, 15, 1, None), (32, 16, 1, None), (33, 8, 1, None),
                                          (32, 17, 2, (8, 4, 23, 12)), (33, 16, 2, (0, 0, 16, 8)),
                                          (40, 15, 2, (25, 7, 40, 15)), (31, 20, 3, (10, 9, 11, 10)),
                                          (36, 12, 2, (0, 5, 36, 6))])
def test_gradients_match_complex_step(nx, ny, r, rect):
    w = W.small_dmr(nx=nx, ny=ny, r=r, rect=rect, growth=0)
    sim = O.sim_from_workload(w)
    seed = (sim.fine if r > 1 else sim.coarse).n.copy()
    NT = w["cfg"]["steps_per_period"]
    steps, K = 2 * NT, NT
    ref = oracle_run(w, w["cfg"]["E0"], 1.0, seed, steps)
    rng = np.random.default_rng(nx * ny + r)
    target = ref.coarse.n * (1 + 0.05 * rng.standard_normal(ref.coarse.n.shape))
    u = rng.standard_normal(seed.shape)
    n_end, gE0, gnu, gseed = gpu_grads(w, seed, steps, K, target)
    cE0, cnu, cseed = cs_grads(w, seed, steps, ref.log, target, u)
    errs = (abs(gE0 / cE0 - 1), abs(gnu / cnu - 1), abs(float(np.sum(gseed * u)) / cseed - 1))
    assert max(errs) <= TOL_ADJ64, errs
