"""Where the one-body apply of few Stokes columns (apply_few.cu) and the packed stress policies change form.

* Applies of 1 to 9 columns of one shape (8 is the largest count taken by the few-column form, 9 the
  first of the tensor cores), on point counts that leave remainders in every loop: the apply itself by
  its backward error against the oracle's FP64 factors (1e-5, the bar of the tensor-core apply), the
  matvec and its transpose against the oracle (1e-6, the bar of both).
* Pressure and traction of 1 to 4 right-hand sides (one packed policy each), at point counts around
  the 256-point tiles, against the all-FP64 context: 1e-5, the bar of an FP32 solve, whose error and
  the sums' own rounding both enter.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from mfs_inputs import make_workload  # noqa: E402
from oracle import Problem  # noqa: E402

from test_gpu_parity import _ctx, _mixed, _rel  # noqa: E402
from test_gpu_tensor_cores import _backward_err  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("bodies,nrhs,m,n", [(1, 1, 61, 31), (2, 1, 150, 75), (3, 1, 97, 50), (7, 1, 129, 63),
                                             (2, 4, 150, 75), (4, 2, 101, 53), (3, 3, 150, 75)])
def test_apply_of_few_columns(bodies, nrhs, m, n):
    wl = _mixed("stokes", P=bodies, m=m, n=n, seed=31)
    wl.shape_id = np.zeros(bodies, np.int32)
    wl.shapes = wl.shapes[:1]
    pr, ctx = Problem(wl), _ctx(wl)
    ids = list(range(bodies))
    rng = np.random.default_rng(bodies * nrhs)
    gam = rng.standard_normal((nrhs, ctx.sum_M, 3))
    g = torch.tensor(gam, device="cuda")
    lam = ctx.precond_apply(g, project=False).cpu().numpy()
    y, yt = ctx.matvec(g).cpu().numpy(), ctx.matvec_transposed(g).cpu().numpy()
    for h in range(nrhs):
        assert _backward_err(pr, ids, lam[h].reshape(-1), gam[h].reshape(-1)) < 1e-5
        assert _rel(y[h].reshape(-1), pr.matvec(ids, gam[h].reshape(-1))) < 1e-6
        assert _rel(yt[h].reshape(-1), pr.matvec_T(ids, gam[h].reshape(-1))) < 1e-6
    ctx.close()


@pytest.mark.parametrize("nrhs", [1, 2, 3, 4])
@pytest.mark.parametrize("points", [33, 255, 257, 2001])
def test_packed_stress(nrhs, points):
    wl = make_workload("sphere100_mobility", count=6, m=240, n=120)
    a, b = _ctx(wl), _ctx(wl, precision=1, gmres_tol=1e-12)
    rng = np.random.default_rng(points)
    own = rng.integers(0, 6, points).astype(np.int32)
    nrm = rng.standard_normal((points, 3))
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    pts = wl.centres[own] + 1.02 * nrm  # just outside the unit spheres
    F, T = rng.standard_normal((nrhs, 6, 3)), rng.standard_normal((nrhs, 6, 3))
    for solve in ("solve_mobility", "solve_resistance"):
        out = []
        for c in (a, b):
            getattr(c, solve)(F, T)
            out.append(c.evaluate_stress(pts, nrm, own, nrhs=nrhs))
        for got, want in zip(*out):
            for h in range(nrhs):
                assert _rel(got[h], want[h]) < 1e-5, (solve, h)
    a.close()
    b.close()
