"""Passes of the force kernels capped by the box's size and dealt out to several work items:
boxes on both sides of every line give the FP64 form's accelerations to FP32 accuracy, and
the same bits alone and in a batched call, at several block shapes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0910_0121_gb300 import build as _build  # noqa: E402

_build.build()
from paper_0910_0121_gb300 import greem  # noqa: E402


def _box(n, seed):
    rng = np.random.default_rng(seed)
    pos = rng.random((n, 3))
    pos[: n // 3] = np.mod(0.7 + 0.02 * rng.standard_normal((n // 3, 3)), 1.0)
    return pos, rng.uniform(0.5, 1.5, n).astype(np.float32) / n


# groups per reference warp (4 n / n_crit / 2432): below 0.5, 0.5 to 3, 3 to 14, above; one
# particle, n_crit of one, and groups beyond the widest pass
@pytest.mark.parametrize("n,n_crit", [(1, 64), (700, 1), (19000, 64), (20000, 64), (30000, 512), (150000, 128),
                                      (900000, 128)])
@pytest.mark.parametrize("eps", [0.0, 1e-3])
def test_capped_passes(n, n_crit, eps):
    pos, mass = _box(n, n)
    P, M = torch.from_numpy(pos).cuda(), torch.from_numpy(mass).cuda()
    kw = dict(L=1.0, r_cut=0.6 * max(n, 8) ** (-1.0 / 3.0), theta=0.6, n_crit=n_crit, eps=eps)
    ctx = greem.Context()
    acc = ctx.short_force(P, M, greem.params(**kw))
    st = ctx.stats()
    assert st["n_evaluated"] >= st["n_interactions"]
    for shape in (1, 5):
        assert torch.equal(ctx.short_force(P, M, greem.params(block_shape=shape, **kw)), acc)
    small = _box(2500, 3)
    pb = torch.cat([P, torch.from_numpy(small[0]).cuda()])
    mb = torch.cat([M, torch.from_numpy(small[1]).cuda()])
    both = ctx.short_force_batched(pb, mb, [0, n, n + 2500], [greem.params(**kw), greem.params(**dict(kw, n_crit=32))])
    assert torch.equal(both[:n], acc)
    if n <= 200000:
        k64 = dict(kw, precision=greem.F64)
        ref = ctx.short_force(P, M, greem.params(**k64))
        both = ctx.short_force_batched(pb, mb, [0, n, n + 2500],
                                       [greem.params(**k64), greem.params(**dict(k64, n_crit=32, eps=1e-4))])
        assert torch.equal(both[:n], ref)
        nr = ref.norm(dim=1)
        err = ((acc.double() - ref).norm(dim=1) / nr)[nr > 1e-6 * nr.median()]
        if err.numel():
            assert float(err.median()) <= 1e-5 and float(err.quantile(0.999)) <= 1e-4
    ctx.close()
