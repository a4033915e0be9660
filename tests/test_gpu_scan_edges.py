"""The single-pass scans at the edges of their tiles (4096 counts, 1024 nodes), the sort on
both sides of its two tile sizes (768 and 3072 pairs, the line at 200000) and the key
kernel's digit counts: trees and groups against the oracle's, bit for bit, for particle
numbers around the tile sizes, one box and several."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from paper_0910_0121_gb300 import build as _build  # noqa: E402

_build.build()
from paper_0910_0121_gb300 import greem  # noqa: E402


def _check(ctx, pos, mass, n_crit, n_leaf):
    t = oracle.Tree(pos, mass, 1.0, 0.05, n_crit=n_crit, n_leaf=n_leaf)
    key, perm = t.sorted()[:2]
    assert np.array_equal(ctx.dump(greem.DUMP_KEYS), key) and np.array_equal(ctx.dump(greem.DUMP_PERM), perm)
    assert np.array_equal(ctx.dump(greem.DUMP_NODES)[:, :8], t.nodes()[:, :8])
    assert np.array_equal(ctx.dump(greem.DUMP_GROUPS), t.groups())


@pytest.mark.parametrize("n", [1, 31, 255, 257, 767, 769, 4095, 4096, 4097, 65537, 200000, 200001, 204287, 204289])
@pytest.mark.parametrize("n_crit,n_leaf", [(1, 1), (64, 10)])
def test_tree_and_groups(n, n_crit, n_leaf):
    rng = np.random.default_rng(n)
    pos, mass = rng.random((n, 3)), np.ones(n, np.float32)
    pos[: n // 2] = np.mod(0.9 + 1e-4 * rng.standard_normal((n // 2, 3)), 1.0)
    ctx = greem.Context()
    ctx.build_tree(torch.from_numpy(pos).cuda(), torch.from_numpy(mass).cuda(),
                   greem.params(L=1.0, r_cut=0.05, n_crit=n_crit, n_leaf=n_leaf))
    _check(ctx, pos, mass, n_crit, n_leaf)
    ctx.close()


@pytest.mark.parametrize("nbox", [2, 5, 300])
def test_boxes_sort_apart(nbox):
    rng = np.random.default_rng(nbox)
    off = np.concatenate([[0], np.cumsum(rng.integers(1, 3000 // min(nbox, 100), nbox))])
    pos, mass = rng.random((off[-1], 3)), np.ones(off[-1], np.float32)
    P, M = torch.from_numpy(pos).cuda(), torch.from_numpy(mass).cuda()
    p = greem.params(L=1.0, r_cut=0.05, n_crit=16)
    ctx = greem.Context()
    acc = ctx.short_force_batched(P, M, off, [p] * nbox)
    for b in (0, nbox // 2, nbox - 1):
        one = ctx.short_force(P[off[b]:off[b + 1]].contiguous(), M[off[b]:off[b + 1]].contiguous(), p)
        assert torch.equal(one, acc[off[b]:off[b + 1]])
    ctx.close()
