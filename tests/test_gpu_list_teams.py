"""Lists walked by teams of 4 and 2 warps (few groups) and by single warps (many): a box
alone and the same box beside a large one, whose groups put the call past both lines, give
the same accelerations bit for bit, also with second moments and from a small stack."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0910_0121_gb300 import build as _build  # noqa: E402

_build.build()
from paper_0910_0121_gb300 import greem  # noqa: E402


def box(n, seed):
    rng = np.random.default_rng(seed)
    pos = rng.random((n, 3))
    k = n // 2
    pos[:k] = np.mod(0.6 + 0.02 * rng.standard_normal((k, 3)), 1.0)
    return pos, rng.uniform(0.5, 1.5, n).astype(np.float32)


@pytest.mark.parametrize("n,r_cut,quad,stack", [(1, 0.1, False, 0), (33, 0.45, False, 0), (5000, 0.1, False, 0),
                                                (5000, 0.1, True, 0), (9000, 0.05, False, 64), (40000, 0.05, False, 0),
                                                (40000, 0.03, True, 64)])
def test_teams_build_the_lists_of_one_warp(n, r_cut, quad, stack):
    flags = greem.FLAG_QUADRUPOLE if quad else 0
    p = greem.params(L=1.0, r_cut=r_cut, theta=0.5, n_crit=64, flags=flags)
    big = greem.params(L=1.0, r_cut=0.02, theta=0.5, n_crit=16, flags=flags)
    pos, mass = box(n, n)
    fill, fmass = box(150000, 7)
    P = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    a, b = greem.Context(), greem.Context()
    if stack:
        a.debug_set(greem.DEBUG_STACK_CAP, stack)
    alone = a.short_force(P(pos), P(mass), p)
    groups = a.stats()["n_groups"]
    if stack:
        assert a.stats()["retries"] >= 1
    both = b.short_force_batched(P(np.concatenate([pos, fill])), P(np.concatenate([mass, fmass])),
                                 np.array([0, n, n + 150000]), [p, big])
    warps = 32 * torch.cuda.get_device_properties(0).multi_processor_count
    assert 3 * b.stats()["n_groups"] > 2 * warps
    assert 3 * groups <= 2 * warps
    assert torch.equal(alone, both[:n])
    a.close()
    b.close()
