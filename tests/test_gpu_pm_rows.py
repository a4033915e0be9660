"""Rows of grid points added by vector atomics (particles out of order, n_pm a multiple of 4)
or scalar ones (particles in grid order, rows that wrap, other n_pm), and the interleaved
field read back: PM accelerations against the FP64 oracle for both orders."""
import numpy as np
import pytest

from oracle import pm as pmo

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0910_0121_gb300 import build as _build  # noqa: E402

_build.build()
from paper_0910_0121_gb300 import greem  # noqa: E402


@pytest.mark.parametrize("n", [8, 10, 34, 36])
@pytest.mark.parametrize("scheme", [pmo.CIC, pmo.TSC])
@pytest.mark.parametrize("order", ["grid", "shuffled", "one row"])
def test_pm_orders(n, scheme, order):
    rng = np.random.default_rng(n)
    k = 13
    q = (np.arange(k) + 0.5) / k
    pos = np.stack(np.meshgrid(q, q, q, indexing="ij"), axis=-1).reshape(-1, 3) + 0.01 * rng.standard_normal((k ** 3, 3))
    if order == "shuffled":
        pos = pos[rng.permutation(len(pos))]
    if order == "one row":  # a dense row across the end of the box
        pos[:500] = np.array([0.5, 0.5, 0.0]) + 0.1 * rng.standard_normal((500, 3)) * [0.01, 0.01, 1.0]
    pos = np.mod(pos, 1.0)
    mass = rng.uniform(0.5, 1.5, len(pos)).astype(np.float32) / len(pos)
    rc = min(0.4, 3.0 / n)
    ref = pmo.pm_accel(pos, mass, 1.0, n, rc, scheme)
    ctx = greem.Context()
    got = ctx.pm_force(torch.from_numpy(pos).cuda(), torch.from_numpy(mass).cuda(), 1.0, n, rc, scheme)
    got = got.cpu().numpy().astype(np.float64)
    ctx.close()
    rms = np.sqrt(np.mean(np.sum(ref * ref, axis=1)))
    assert np.linalg.norm(got - ref, axis=1).max() <= 2e-4 * rms
