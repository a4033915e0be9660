"""Prefix sums whose wait on earlier tiles gives up (each of them made to, after a larger call
has left its numbers in the context's buffers): the call returns TIMEOUT, what follows the
sum touches nothing, and the next call gives the bits of an undisturbed one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0910_0121_gb300 import build as _build  # noqa: E402

_build.build()
from paper_0910_0121_gb300 import greem  # noqa: E402


def _set(n, seed):
    rng = np.random.default_rng(seed)
    pos = rng.random((n, 3))
    pos[: n // 2] = np.mod(0.4 + 0.02 * rng.standard_normal((n // 2, 3)), 1.0)
    return torch.from_numpy(pos).cuda(), torch.from_numpy(rng.uniform(0.5, 1.5, n).astype(np.float32)).cuda()


def _timeout(f):
    with pytest.raises(greem.GreemError) as e:
        f()
    assert e.value.code == greem.ERR_TIMEOUT


# n: small and large sort tiles; more than one tile of each sum (4096 counts, 1024 nodes)
@pytest.mark.parametrize("n,n_crit", [(60000, 8), (220000, 32)])
@pytest.mark.parametrize("which", [greem.LOOK_SORT, greem.LOOK_NODES, greem.LOOK_GROUPS, greem.LOOK_SECOND,
                                   greem.LOOK_SORT | greem.LOOK_NODES | greem.LOOK_GROUPS])
def test_a_look_back_that_gives_up(n, n_crit, which):
    P, M = _set(n, n)
    big = _set(3 * n, 1)
    kw = dict(L=1.0, r_cut=0.04, theta=0.5, n_crit=n_crit)
    kinds = [dict(flags=greem.FLAG_QUADRUPOLE)]
    if which != greem.LOOK_SECOND:
        kinds += [dict(), dict(precision=greem.F64)]
    ctx = greem.Context()
    for k in kinds:
        p = greem.params(**kw, **k)
        ref = ctx.short_force(P, M, p)
        ctx.short_force(*big, p)
        ctx.debug_set(greem.DEBUG_LOOK_BACK, which)
        _timeout(lambda: ctx.short_force(P, M, p))
        _timeout(lambda: ctx.short_force_batched(P, M, [0, n // 3, n], [p, p]))
        if which != greem.LOOK_SECOND:
            _timeout(lambda: ctx.build_tree(P, M, p))
        ctx.debug_set(greem.DEBUG_LOOK_BACK, 0)
        assert torch.equal(ctx.short_force(P, M, p), ref)
    ctx.close()


@pytest.mark.parametrize("grid", [(2, 1, 1), (5, 2, 2)])  # one and two chunks of receiving boxes
def test_domain_calls_report_a_sum_that_gave_up(grid):
    n = 600000  # more than one tile of counts per call
    P, M = _set(n, 5)
    ctx = greem.Context()
    cells = ctx.cell_index(P[:2000].contiguous(), 1.0).cpu().numpy()
    boxes = greem.domain_boxes(cells, grid)
    pack = lambda: ctx.domain_pack(P, M, None, 1.0, boxes)  # noqa: E731
    let = lambda: ctx.let_export(boxes, 0, with_refs=True)  # noqa: E731
    ctx.build_tree(P, M, greem.params(L=1.0, r_cut=0.04, theta=0.5))
    ref_let = let()
    ctx.debug_set(greem.DEBUG_LOOK_BACK, greem.LOOK_LET)
    _timeout(let)
    ctx.debug_set(greem.DEBUG_LOOK_BACK, greem.LOOK_DOMAIN)
    again = let()
    _timeout(pack)
    ctx.debug_set(greem.DEBUG_LOOK_BACK, 0)
    assert all(torch.equal(a, b) for a, b in zip(ref_let[:3], again[:3])) and np.array_equal(ref_let[3], again[3])
    po, mo, io, counts = pack()
    assert counts.sum() == n and torch.equal(io.sort().values, torch.arange(n, device="cuda"))
    assert torch.equal(po, P[io]) and torch.equal(mo, M[io])
    ctx.close()


def test_bad_masks_are_refused():
    ctx = greem.Context()
    with pytest.raises(greem.GreemError) as e:
        ctx.debug_set(greem.DEBUG_LOOK_BACK, 1 << 10)
    assert e.value.code == greem.ERR_INVALID_ARG
    ctx.close()
