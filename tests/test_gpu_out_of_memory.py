"""A refused buffer leaves the context usable (mfs_selftest_fail_alloc).

Every buffer that a call allocates is refused in turn.  The call reports MFS_ERR_OOM, and the next
call, of the sizes solved before, gives what it gave before bit for bit: no half-built set of buffers
is taken for a whole one.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from mfs_inputs.workloads import sphere_suspension  # noqa: E402

from test_gpu_parity import _ctx  # noqa: E402

OOM = 3


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


def _refuse_in_turn(ctx, call, after, want):
    """`call` with its 1st, 2nd, ... buffer refused, until it asks for no more; `after` in between."""
    from paper_2409_04215_gb300.api import MFSError

    for nth in range(1, 100):
        assert ctx._lib.mfs_selftest_fail_alloc(ctx._ctx, nth) == 0
        try:
            call()
        except MFSError as e:
            assert e.status == OOM, str(e)
        else:
            assert ctx._lib.mfs_selftest_fail_alloc(ctx._ctx, 0) == 0
            return nth - 1
        assert ctx._lib.mfs_selftest_fail_alloc(ctx._ctx, 0) == 0
        assert all(torch.equal(a, b) for a, b in zip(after(), want)), nth
    raise AssertionError("the call never completed")


@pytest.mark.parametrize("graphs", [0, 1])
def test_solve_with_more_right_hand_sides(graphs):
    wl = sphere_suspension(count=4, m=91, n=45, seed=2)
    ctx = _ctx(wl, autotune=0, max_rhs=4, graphs=graphs)
    F, T = np.random.default_rng(0).standard_normal((2, 4, 4, 3))

    def one():
        return ctx.solve_mobility(F[:1], T[:1])[:2]

    assert _refuse_in_turn(ctx, one, lambda: (), ()) >= 20  # a first solve: its basis, its kept solution, a plan
    want = one()
    assert _refuse_in_turn(ctx, lambda: ctx.solve_mobility(F, T), one, want) >= 17
    U, W, _ = ctx.solve_mobility(F, T)
    assert np.allclose(U[0], want[0][0], rtol=0, atol=1e-6) and np.allclose(W[0], want[1][0], rtol=0, atol=1e-6)
    ctx.close()


@pytest.mark.parametrize("farfield", [0, 1])
def test_gradient(farfield):
    wl = sphere_suspension(count=20, m=91, n=45, seed=2)
    ctx = _ctx(wl, autotune=0, max_rhs=1, farfield=farfield)
    g = np.random.default_rng(0).standard_normal((2, 1, 20, 3))
    want = ctx.solve_mobility(wl.F, wl.T)[:2]
    assert _refuse_in_turn(ctx, lambda: ctx.mobility_vjp(*g), lambda: ctx.solve_mobility(wl.F, wl.T)[:2], want) >= 10
    assert torch.isfinite(ctx.mobility_vjp(*g)[0]).all()
    ctx.close()


def test_moved_treecode():
    wl = sphere_suspension(count=60, m=91, n=45, seed=2)
    ctx = _ctx(wl, autotune=0, max_rhs=1, farfield=1)
    s = torch.tensor(np.random.default_rng(1).standard_normal((1, ctx.sum_N, 3)), device="cuda")
    want = ctx.pair_sum(s)

    def near():  # a refused rebuild leaves the direct sums: the same values to the treecode's accuracy
        got = ctx.pair_sum(s)
        return ((got - want).norm() < 1e-6 * want.norm(),)

    from paper_2409_04215_gb300.api import MFSError

    for nth in (1, 5, 20):
        assert ctx._lib.mfs_selftest_fail_alloc(ctx._ctx, nth) == 0
        with pytest.raises(MFSError):
            ctx.update_centers(wl.centres)
        assert ctx._lib.mfs_selftest_fail_alloc(ctx._ctx, 0) == 0
        assert all(near()), nth
        ctx.close()
        ctx = _ctx(wl, autotune=0, max_rhs=1, farfield=1)
    ctx.close()
