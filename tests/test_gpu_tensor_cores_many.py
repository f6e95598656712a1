"""The tensor-core apply and its transpose with at least nine columns of every shape.

Fewer Stokes columns take the few-column form (apply_few.cu), so these cases are the ones that hold the
tcgen05 apply itself: the forward and the transposed operator in both piece counts, a solve and a gradient.
Bars: those of test_gpu_tensor_cores.py, test_gpu_transposed.py and test_gpu_adjoint.py for the same calls.
That the tensor cores ran is read from the results: the few-column form does not look at the piece count,
so its two modes agree bit for bit, and those of the tensor cores do not.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import Problem  # noqa: E402

from test_gpu_parity import _ctx, _mixed, _rel, _seg  # noqa: E402
from test_gpu_tensor_cores import BACKWARD_TOL, MATVEC_TOL, _backward_err  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


def _many(P, nrhs, nsusp=1, m=150, n=75):
    wl = _mixed("stokes", P=P, m=m, n=n, seed=31, nsusp=nsusp)
    wl.shape_id = (np.arange(P) % 2).astype(np.int32)  # half of the bodies each
    assert P // 2 * nrhs >= 9
    return wl


@pytest.mark.parametrize("P,nrhs", [(18, 1), (7, 3), (6, 4)])
def test_apply_and_matvec(P, nrhs):
    wl = _many(P, nrhs)
    pr = Problem(wl)
    bodies = list(range(P))
    rng = np.random.default_rng(7)
    smooth = np.stack([np.concatenate(pr.pair_sum(bodies, [rng.standard_normal(pr.Y[k].shape[0] * 3) for k in bodies],
                                                  include_self=False)) for _ in range(nrhs)])
    gam = torch.tensor(smooth.reshape(nrhs, -1, 3), device="cuda")
    modes = {}
    for mode in (1, 2):
        ctx = _ctx(wl, tensor_cores=mode)
        lam, y = ctx.precond_apply(gam, project=False), ctx.matvec(gam)
        for h in range(nrhs):
            assert _backward_err(pr, bodies, lam[h].cpu().numpy().reshape(-1), smooth[h]) < BACKWARD_TOL[mode]
            assert _rel(y[h].cpu().numpy().reshape(-1), pr.matvec(bodies, smooth[h])) < MATVEC_TOL[mode]
        modes[mode] = lam
        ctx.close()
    assert not torch.equal(modes[1], modes[2])


@pytest.mark.parametrize("P,nrhs", [(18, 1), (10, 2)])
def test_transposed_matvec(P, nrhs):
    wl = _many(P, nrhs, nsusp=2)
    pr = Problem(wl)
    w = np.random.default_rng(21).standard_normal((nrhs, sum(len(pr.X[k]) for k in range(P)), 3))
    modes = {}
    for mode in (1, 2):
        ctx = _ctx(wl, tensor_cores=mode)
        modes[mode] = ctx.matvec_transposed(torch.tensor(w, device="cuda"))
        ctx.close()
        for h in range(nrhs):
            ref = np.concatenate([pr.matvec_T(list(pr.suspension_bodies(s)),
                                              w[h].reshape(-1)[_seg(pr, list(pr.suspension_bodies(s)), "colloc")])
                                  for s in range(wl.num_suspensions)])
            # 1e-6: the bar of both applies; two pieces are held to the 3e-6 of their forward matvec
            assert _rel(modes[mode][h].cpu().numpy().reshape(-1), ref) < MATVEC_TOL[mode]
    assert not torch.equal(modes[1], modes[2])


def test_solve_and_gradient():
    wl = _many(18, 1, nsusp=2, m=120, n=60)
    pr = Problem(wl)
    ctx = _ctx(wl, gmres_tol=1e-10, tensor_cores=1)
    F, T = torch.tensor(wl.F[:1], device="cuda"), torch.tensor(wl.T[:1], device="cuda")
    U, W, info = ctx.solve_mobility(F, T)
    Ur, Wr, _ = pr.solve_mobility(wl.F[0], wl.T[0], tol=1e-13)
    assert info.converged
    assert _rel(np.concatenate([U.cpu().numpy()[0], W.cpu().numpy()[0]], 1), np.concatenate([Ur, Wr], 1)) < 1e-5
    got = [g.cpu().numpy() for g in ctx.mobility_vjp(2.0 * U, 0.6 * W, want_force_grads=True)]
    want = pr.mobility_vjp(wl.F[0], wl.T[0], 2.0 * Ur, 0.6 * Wr)
    for a, b in zip((got[0], got[1][0], got[2][0]), want):
        assert np.abs(a - b).max() <= 1e-4 * np.abs(b).max()
    ctx.close()
