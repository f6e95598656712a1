"""Which Arnoldi step a batch of short lanes takes (gmres.cu, gmres_prepare), and that both give the
same solve: one launch per step for lanes that run at about one time, four launches for many lanes
(256 lanes of six spheres take 674 us an iteration in one launch, 422 us in four).

The step is read from the launches that two more iterations cost, against four lanes of the same
number of columns.  Solves are held to the same lanes solved one suspension at a time, in FP64 to the bar of
the other GMRES tests (1e-9 at tolerance 1e-12: in FP32 a lone suspension's columns run in another
one-body apply, whose results are 1e-6 away), and to themselves on a second call (the whole loop as
one graph) bit for bit.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from mfs_inputs.workloads import batched_suspensions  # noqa: E402

from test_gpu_parity import _ctx, _rel  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


def _launches_an_iteration(lanes, bodies):
    wl = batched_suspensions(num_suspensions=lanes, p_lo=bodies, p_hi=bodies, m=61, n=30, nrhs=1, seed=4)
    count = []
    for its in (2, 4):
        ctx = _ctx(wl, autotune=0, max_rhs=1, max_iter=its, restart=its, gmres_tol=1e-15)
        info = ctx.solve_mobility(wl.F, wl.T, allow_not_converged=True)[2]
        assert info.iters == its
        count.append(info.launches)
        ctx.close()
    return (count[1] - count[0]) / 2


@pytest.mark.parametrize("lanes,more", [(8, 0), (64, 3)])
def test_step_follows_the_number_of_lanes(lanes, more):
    few = _launches_an_iteration(4, 2 * lanes // 4)  # four short lanes of the same number of columns
    assert _launches_an_iteration(lanes, 2) == few + more


# lanes around the limit of the one-launch step, one block an SM and more, several blocks a lane
@pytest.mark.parametrize("lanes,bodies", [(5, 5), (11, 5), (13, 5), (17, 5), (40, 5), (75, 5), (77, 5), (90, 45)])
def test_lanes_agree_with_single_ones(lanes, bodies):
    wl = batched_suspensions(num_suspensions=lanes, p_lo=1, p_hi=bodies, m=61, n=30, nrhs=2, seed=lanes)
    ctx = _ctx(wl, autotune=0, max_rhs=2, precision=1, gmres_tol=1e-12)
    U, W, info = ctx.solve_mobility(wl.F, wl.T)
    U2, W2, info2 = ctx.solve_mobility(wl.F, wl.T)
    assert torch.equal(U, U2) and torch.equal(W, W2) and info2.iters == info.iters
    ctx.close()
    from paper_2409_04215_gb300 import MFS

    off = wl.body_offsets
    for s in sorted({0, lanes // 2, lanes - 1}):
        b = slice(off[s], off[s + 1])
        one = MFS("stokes", wl.centres[b], [(sh.proxy, sh.colloc) for sh in wl.shapes],
                  quats=None if wl.quats is None else wl.quats[b], shape_id=wl.shape_id[b], autotune=0, max_rhs=2,
                  mu=float(wl.mu), precision=1, gmres_tol=1e-12)
        u, w, _ = one.solve_mobility(wl.F[:, b], wl.T[:, b])
        assert _rel(torch.cat([U[:, b], W[:, b]]).numpy(), torch.cat([u, w]).numpy()) < 1e-9, s
        one.close()
