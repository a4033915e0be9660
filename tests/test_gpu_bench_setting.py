"""bench.settle: both arms time one setting unless the autotuner's pick is clearly faster."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0910_0121_gb300 import build as _build  # noqa: E402

_build.build()
import bench  # noqa: E402
from paper_0910_0121_gb300 import greem  # noqa: E402


class Clock:
    """A context whose calls take the given GPU cycles per n_crit."""

    def __init__(self, cycles):
        self.cycles = cycles

    def short_force(self, P, M, p, acc):
        torch.cuda._sleep(self.cycles[p.n_crit])


@pytest.mark.parametrize("ratio,fixed", [(1.0, True), (0.9, True), (1.2, False)])
def test_settle(ratio, fixed):
    nc = bench.SETTING["n_crit"]
    pick = greem.params(L=2.0, r_cut=0.01, theta=0.4, n_crit=96, n_leaf=7, list_chunk=512, block_shape=8)
    base = 2_000_000
    got = bench.settle(Clock({96: base, nc: int(ratio * base)}), None, None, None, pick)
    want = dict(bench.SETTING) if fixed else dict(n_crit=96, list_chunk=512, block_shape=8)
    assert {k: getattr(got, k) for k in want} == want
    assert (got.L, got.r_cut, got.theta, got.n_leaf) == (2.0, 0.01, 0.4, 7)
