"""Lists longer than a page of the pool: a warp takes the whole pages of a mean list before it
walks the next one, so each list of one and a half pages takes two (after the page that a warp
takes before its first), and a pool of that size needs no retry; one that starts from nothing
needs one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0910_0121_gb300 import build as _build  # noqa: E402

_build.build()
from paper_0910_0121_gb300 import greem  # noqa: E402

PAGE = 4096


@pytest.mark.parametrize("flags", [0, greem.FLAG_INDEX_LISTS])
def test_pool_of_lists_beyond_a_page(flags):
    # one group per particle, theta = 0: a list holds the particles within r_cut, 31% of 20000
    n = 20000
    rng = np.random.default_rng(2)
    P = torch.from_numpy(rng.random((n, 3))).cuda()
    M = torch.ones(n, dtype=torch.float32, device="cuda")
    p = greem.params(L=1.0, r_cut=0.42, theta=0.0, n_crit=1, n_leaf=2, flags=flags)
    ctx = greem.Context()
    ref = ctx.short_force(P, M, p)
    st = ctx.stats()
    assert st["n_groups"] == n and 1.4 * PAGE * n < st["n_list_entries"] < 1.6 * PAGE * n
    warps = 32 * torch.cuda.get_device_properties(0).multi_processor_count
    for pages, retries in ((warps + 2 * n, 0), (1, 1)):
        c = greem.Context()
        c.debug_set(greem.DEBUG_LIST_CAP, pages * PAGE)
        c.debug_set(greem.DEBUG_NODE_CAP, 4 * n)  # (the usual first guess is below 2 nodes a particle)
        assert torch.equal(c.short_force(P, M, p), ref)
        assert c.stats()["retries"] == retries
        c.close()
    ctx.close()
