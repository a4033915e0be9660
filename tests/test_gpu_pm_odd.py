"""Meshes with an odd number of points a side, which have no Nyquist mode: PM accelerations
against the FP64 oracle, alone and added to the short-range force."""
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


@pytest.mark.parametrize("n", [8, 9, 25, 26, 33, 45])
@pytest.mark.parametrize("scheme", [pmo.CIC, pmo.TSC])
def test_odd_and_even_meshes(n, scheme):
    rng = np.random.default_rng(n)
    pos = rng.random((3000, 3))
    mass = rng.uniform(0.5, 1.5, len(pos)).astype(np.float32) / len(pos)
    rc = min(0.4, 3.0 / n)
    ref = pmo.pm_accel(pos, mass, 1.0, n, rc, scheme)
    rms = np.sqrt(np.mean(np.sum(ref * ref, axis=1)))
    P, M = torch.from_numpy(pos).cuda(), torch.from_numpy(mass).cuda()
    ctx = greem.Context()
    got = ctx.pm_force(P, M, 1.0, n, rc, scheme).double()
    # FP32 mesh against FP64: the bound of the other mesh tests
    assert np.linalg.norm(got.cpu().numpy() - ref, axis=1).max() <= 2e-4 * rms
    kw = dict(L=1.0, r_cut=rc, theta=0.5, n_crit=32)
    pp = ctx.short_force(P, M, greem.params(**kw))
    both = ctx.short_force(P, M, greem.params(flags=greem.FLAG_ADD_PM, n_pm=n, assign=scheme, **kw))
    # one rounding of the sum, and the order of the assignment's atomics
    assert float((both.double() - pp.double() - got).norm(dim=1).max()) <= 2e-4 * rms + 1e-6 * float(pp.norm(dim=1).max())
    ctx.close()
