"""Moments and second moments of every level in one climb from the deepest nodes: shallow and
deep trees of all sizes, on both sides of the line between the leaf pass's tiles, against
sums over each node's particles."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0910_0121_gb300 import build as _build  # noqa: E402

_build.build()
from paper_0910_0121_gb300 import greem  # noqa: E402


@pytest.mark.parametrize("n,depth", [(1, 0.1), (9, 1e-6), (257, 0.1), (4096, 0.1), (50000, 1e-6), (311296, 1e-3),
                                     (311297, 1e-3), (700001, 1e-4)])
def test_moments_of_every_node(n, depth):
    rng = np.random.default_rng(n)
    pos = rng.random((n, 3))
    k = n // 2  # half the particles around one point, down to the finest levels for small depths
    pos[:k] = np.mod(0.3 + depth * rng.standard_normal((k, 3)) ** 3, 1.0)
    mass = rng.uniform(0.5, 1.5, n).astype(np.float32)
    ctx = greem.Context()
    ctx.short_force(torch.from_numpy(pos).cuda(), torch.from_numpy(mass).cuda(),
                    greem.params(L=1.0, r_cut=0.01, theta=0.5, n_crit=64, flags=greem.FLAG_QUADRUPOLE))
    nodes, mom, quad = (ctx.dump(w) for w in (greem.DUMP_NODES, greem.DUMP_MOMENTS, greem.DUMP_QUADRUPOLES))
    perm = ctx.dump(greem.DUMP_PERM)
    ctx.close()
    x, m = pos[perm], mass[perm].astype(np.float64)
    big = np.argsort(nodes[:, 5] - nodes[:, 4])[-300:]  # the upper tree, every level of the dense point
    for i in np.unique(np.concatenate([big, rng.integers(0, len(nodes), 300)])):
        b, e = nodes[i, 4], nodes[i, 5]
        M = m[b:e].sum()
        c = (m[b:e, None] * x[b:e]).sum(0) / M
        assert abs(mom[i, 0] - M) <= 1e-13 * M
        assert np.abs(mom[i, 1:] - c).max() <= 1e-13
        d = x[b:e] - c
        q = np.einsum("j,ja,jb->ab", m[b:e], d, d)
        side = 0.5 ** nodes[i, 0]
        got = quad[i]
        ref = np.array([q[0, 0], q[1, 1], q[2, 2], q[0, 1], q[0, 2], q[1, 2]])
        assert np.abs(got - ref).max() <= 2e-5 * M * side * side
