"""The run's state after a backward pass: the recompute of a segment keeps E and v
in the records it writes, and the workspace gets them back at the segment's end.
The state is then that of the first segment's end, bit for bit, and the run goes
on from it.  Both parities of the fine buffers (r odd and even), a rectangle that
grows, a uniform mesh."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2105_13276_gb300 import dmr as D  # noqa: E402
from paper_2105_13276_gb300 import workloads as W  # noqa: E402


def _same(a, b, levels):
    for level in levels:
        for name in ("Ex", "Ey", "Hz", "vx", "vy", "n"):
            np.testing.assert_array_equal(a.read(name, level), b.read(name, level), err_msg="%s %d" % (name, level))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("r,periods,keep", [(1, 2, 1), (2, 4, 2), (3, 3, 3), (2, 5, 1)])
def test_state_after_backward_is_the_first_segments_end(r, periods, keep, precision):
    w = W.small_dmr(r=r, rect=(12, 10, 24, 20) if r > 1 else None, precision=precision)
    T = w["cfg"]["steps_per_period"]
    a, b = D.run_from_workload(w), D.run_from_workload(w)
    ck = a.adjoint_record(periods * T, keep * T)
    shape = (w["cfg"]["ny"] + 1, w["cfg"]["nx"] + 1)
    g = torch.ones(shape, dtype=torch.float64 if precision == 0 else torch.float32, device="cuda")
    a.adjoint_backward(g, ck, None)
    b.advance(keep * T)
    levels = (0, 1) if r > 1 else (0,)
    _same(a, b, levels)
    a.advance(T)
    b.advance(T)
    _same(a, b, levels)
