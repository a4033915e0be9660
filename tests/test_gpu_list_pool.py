"""The list pool of small calls: no page for every warp of the GPU, but at least half of one where
lists of that many particles can fill it, and no retry; a larger call of the same context grows
it."""
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


def _set(n, clustered):
    rng = np.random.default_rng(n)
    pos = rng.random((n, 3))
    if clustered:
        pos[: n // 2] = np.mod(0.2 + 0.01 * rng.standard_normal((n // 2, 3)), 1.0)
    return torch.from_numpy(pos).cuda(), torch.ones(n, dtype=torch.float32, device="cuda")


@pytest.mark.parametrize("clustered", [False, True])
@pytest.mark.parametrize("n,n_crit,theta", [(1, 64, 0.5), (1000, 1, 0.5), (4096, 64, 0.5), (4096, 64, 0.0), (8192, 64, 0.5)])
def test_pool_of_small_calls(n, n_crit, theta, clustered):
    warps = 32 * torch.cuda.get_device_properties(0).multi_processor_count
    p = greem.params(L=1.0, r_cut=0.15, theta=theta, n_crit=n_crit)
    ctx = greem.Context()
    ref = ctx.short_force(*_set(n, clustered), p)
    st = ctx.stats()
    assert st["retries"] == 0
    assert st["list_capacity"] <= 32 * n + PAGE // 2 * warps
    assert st["list_capacity"] >= 32 * n + min(PAGE // 2 * warps, n * n)
    if n == 1:
        assert st["list_capacity"] <= 2 * PAGE
    big = _set(100000, clustered)
    acc = ctx.short_force(*big, p)
    assert ctx.stats()["list_capacity"] >= 32 * 100000 + PAGE * warps
    assert torch.equal(ctx.short_force(*_set(n, clustered), p), ref)
    other = greem.Context()
    assert torch.equal(other.short_force(*big, p), acc)
    other.close()
    ctx.close()
