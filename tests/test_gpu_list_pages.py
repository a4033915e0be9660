"""Pages of the list pool: lists that fill a page, outgrow one, or meet an empty pool give
the accelerations of an unconstrained call bit for bit, and the same list lengths."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0910_0121_gb300 import build as _build  # noqa: E402

_build.build()
from paper_0910_0121_gb300 import greem  # noqa: E402


@pytest.mark.parametrize("n,theta,cap", [(300, 0.5, 1), (6000, 0.5, 4096), (6000, 0.0, 8192), (40000, 0.3, 3 * 4096)])
def test_small_pools_and_long_lists(n, theta, cap):
    rng = np.random.default_rng(n)
    pos = rng.random((n, 3))
    pos[: n // 2] = np.mod(0.3 + 0.01 * rng.standard_normal((n // 2, 3)), 1.0)  # lists beyond a page at theta = 0
    P = torch.from_numpy(pos).cuda()
    M = torch.from_numpy(rng.uniform(0.5, 1.5, n).astype(np.float32)).cuda()
    p = greem.params(L=1.0, r_cut=0.1, theta=theta, n_crit=32)
    a, b = greem.Context(), greem.Context()
    ref = a.short_force(P, M, p)
    b.debug_set(greem.DEBUG_LIST_CAP, cap)
    got = b.short_force(P, M, p)
    sa, sb = a.stats(), b.stats()
    assert sb["retries"] >= 1
    assert torch.equal(ref, got)
    assert all(sa[k] == sb[k] for k in ("n_groups", "n_list_entries", "n_interactions"))
    a.close()
    b.close()
