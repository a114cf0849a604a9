"""Device-to-device reads and writes of fields: the copy kernel against the
runtime's host copies, and which buffers it may be given."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2105_13276_gb300 import dmr as D  # noqa: E402
from paper_2105_13276_gb300 import workloads as W  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2105_13276_gb300 import build as B
    B.build()
    D.load()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx,ny", [(5, 4), (16, 262138), (16, 262139), (4, 262201), (513, 37)])
def test_rows_and_columns(nx, ny, precision):
    """Up to a grid's last block in y, one past it, and the edges of a block."""
    run = D.Run(W.base_cfg(nx=nx, ny=ny, r=1, n_lambda=16, steps_per_period=32, precision=precision, growth=0))
    for k, f in enumerate(("Ex", "n")):
        shape = run.shape(f)[0]
        a = np.random.default_rng(k).random(shape).astype(run.fdtype)
        src = torch.from_numpy(a).to(run.device)
        out = torch.empty_like(src)
        torch.cuda.synchronize()
        run.write_from(f, 0, src)
        run.read_into(f, 0, out)
        run.sync()
        assert np.array_equal(run.read(f), a)
        assert np.array_equal(out.cpu().numpy(), a)
