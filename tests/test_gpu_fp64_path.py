"""The FP64 path's kernels (precision = 1: split pair sums, split-K GEMM) at the sizes where their
splits have edges: a single source chunk, chunk boundaries inside bodies, ragged 64-row GEMM tiles
(1, 64 and 65 columns), uneven suspensions, 1 to 4 right-hand sides.  Bar: 1e-11 of the oracle, the
FP64 path's (both sides round in FP64; the 64-bit sums of a few thousand terms stay below 1e-13)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from mfs_inputs.workloads import batched_suspensions, sphere_suspension  # noqa: E402
from oracle import Problem  # noqa: E402

from test_gpu_parity import _ctx, _rel, _seg  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("kind,count,m,n,nrhs", [
    ("stokes", 1, 40, 13, 1), ("stokes", 2, 90, 41, 3), ("stokes", 16, 70, 33, 4), ("stokes", 13, 61, 30, 2),
    ("laplace", 1, 40, 13, 1), ("laplace", 65, 47, 22, 1), ("laplace", 16, 47, 22, 4),
])
def test_fp64_operator_sizes(kind, count, m, n, nrhs):
    wl = sphere_suspension(count=count, m=m, n=n, kind=kind, seed=31 + count)
    ctx = _ctx(wl, precision=1, autotune=0)
    pr, d = Problem(wl), ctx.d
    rng = np.random.default_rng(count)
    g = rng.standard_normal((nrhs, ctx.sum_M, d))
    s = rng.standard_normal((nrhs, ctx.sum_N, d))
    y = ctx.matvec(torch.tensor(g, device="cuda")).cpu().numpy()
    u = ctx.pair_sum(torch.tensor(s, device="cuda"), include_self=True).cpu().numpy()
    bodies = list(range(count))
    for h in range(nrhs):
        assert _rel(y[h].reshape(-1), pr.matvec(bodies, g[h].reshape(-1))) < 1e-11
        parts = [s[h][k * n:(k + 1) * n].reshape(-1) for k in bodies]
        assert _rel(u[h].reshape(-1), np.concatenate(pr.pair_sum(bodies, parts, include_self=True))) < 1e-11
    ctx.close()


def test_fp64_uneven_suspensions():
    wl = batched_suspensions(num_suspensions=3, p_lo=2, p_hi=9, m=75, n=34, nrhs=2, seed=8)
    ctx = _ctx(wl, precision=1, autotune=0)
    pr = Problem(wl)
    g = np.random.default_rng(3).standard_normal((2, ctx.sum_M, 3))
    y = ctx.matvec(torch.tensor(g, device="cuda")).cpu().numpy()
    yt = ctx.matvec_transposed(torch.tensor(g, device="cuda")).cpu().numpy()
    for h in range(2):
        for out, op in ((y, pr.matvec), (yt, pr.matvec_T)):
            ref = [op(list(pr.suspension_bodies(s)), g[h].reshape(-1)[_seg(pr, list(pr.suspension_bodies(s)), "colloc")])
                   for s in range(wl.num_suspensions)]
            assert _rel(out[h].reshape(-1), np.concatenate(ref)) < 1e-11
    ctx.close()
