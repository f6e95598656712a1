"""The GMRES kernels where their forms change: lanes just short enough for the one-launch (cluster) step
and just too long, lanes of very different length in one solve, more columns than one round of the dot
kernel takes (64), a full basis, a zero right-hand side.  Bars: 1e-5 of the oracle for FP32 solves, 1e-9 for FP64 ones at tolerance 1e-12."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from mfs_inputs.workloads import batched_suspensions, sphere_suspension, spheroid_cluster  # noqa: E402
from oracle import Problem  # noqa: E402

from test_gpu_parity import _ctx, _rel  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("count", [1, 60, 61])  # 273 entries a body: 16380 and 16653 around the 16384 of a cluster
def test_lane_lengths(count):
    wl = sphere_suspension(count=count, m=91, n=45, seed=count)
    ctx = _ctx(wl, autotune=0)
    U, W, info = ctx.solve_mobility(wl.F, wl.T)
    Ur, Wr, _ = Problem(wl).solve_mobility(wl.F[0], wl.T[0], tol=1e-12)
    assert _rel(np.concatenate([U[0], W[0]]), np.concatenate([Ur, Wr])) < 1e-5
    U2, W2, info2 = ctx.solve_mobility(wl.F, wl.T)  # the whole loop as one graph
    assert torch.equal(U, U2) and torch.equal(W, W2) and info2.iters == info.iters and info2.matvecs == info.matvecs
    ctx.close()


def test_uneven_lanes():
    wl = batched_suspensions(num_suspensions=5, p_lo=1, p_hi=70, m=91, n=45, nrhs=2, seed=8)  # short and long lanes
    assert np.diff(wl.body_offsets).max() > 60 > 20 > np.diff(wl.body_offsets).min()
    ctx = _ctx(wl, autotune=0)
    pr = Problem(wl)
    U, W, _ = ctx.solve_mobility(wl.F, wl.T)
    for h in range(2):
        Ur, Wr, _ = pr.solve_mobility(wl.F[h], wl.T[h], tol=1e-12)
        assert _rel(np.concatenate([U[h], W[h]]), np.concatenate([Ur, Wr])) < 1e-5
    ctx.close()


@pytest.mark.parametrize("count,columns", [(14, 48), (40, 64)])  # one and two rounds of the dot kernel
def test_many_columns(count, columns):
    wl = spheroid_cluster(count=count, m=160, n=80, seed=5)
    V = np.random.default_rng(2).standard_normal((2, 1, count, 3))
    ctx = _ctx(wl, autotune=0, precision=1, gmres_tol=1e-12)
    F, T, info = ctx.solve_resistance(V[0], V[1])
    Fr, Tr, _ = Problem(wl).solve_resistance(V[0][0], V[1][0], tol=1e-13)
    assert info.iters > columns
    assert _rel(np.concatenate([F[0], T[0]]), np.concatenate([Fr, Tr])) < 1e-9
    ctx.close()


def test_full_basis_and_zero_rhs():
    wl = spheroid_cluster(count=14, m=160, n=80, seed=5)
    out = []
    for graphs in (0, 1):  # the basis fills up: the last iterate comes back either way
        ctx = _ctx(wl, autotune=0, max_iter=3, restart=3, graphs=graphs)
        for _ in range(2):
            U, W, info = ctx.solve_mobility(np.ones((1, 14, 3)), np.ones((1, 14, 3)), allow_not_converged=True)
            assert info.iters == 3 and info.matvecs == 3 and not info.converged and torch.isfinite(U).all()
            out.append(U)
        z, _, info = ctx.solve_mobility(np.zeros((1, 14, 3)), np.zeros((1, 14, 3)))  # b = 0: no lane runs
        assert info.converged and info.iters == 0 and not z.any()
        ctx.close()
    assert all(torch.equal(out[0], u) for u in out[1:])
