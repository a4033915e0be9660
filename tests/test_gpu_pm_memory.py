"""Device memory of a PM force call: 28 bytes of scratch a grid point beside the Green's table of
(n/2+1)^3 floats (a mesh of 256^3, whose transforms ask for no work area to speak of)."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0910_0121_gb300 import build as _build  # noqa: E402

_build.build()
from paper_0910_0121_gb300 import greem  # noqa: E402


def test_pm_scratch():
    n = 256
    P = torch.rand((1000, 3), dtype=torch.float64, device="cuda")
    M = torch.ones(1000, dtype=torch.float32, device="cuda")
    acc = torch.empty((1000, 3), dtype=torch.float32, device="cuda")
    ctx = greem.Context()
    ctx.pm_force(P, M, 1.0, 16, 0.1, greem.ASSIGN_TSC, acc)  # loads the transforms' library
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    ctx.pm_force(P, M, 1.0, n, 0.1, greem.ASSIGN_TSC, acc)
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    ctx.close()
    # buffers grow by an eighth beyond what is asked for
    assert used <= 1.125 * (28 * n**3 + 4 * (n // 2 + 1)**3) + (32 << 20)
