"""Evaluation points grouped on the device (eval_group.cu) at the sizes where its chunks and warps have
edges: 1, 31, 1023..1025 and several thousand points, unsorted owners, bodies without points, points
closest to each body found by the library.  Every call must equal the calls that evaluate a few points
at a time (one owner, one tile each) to FP32 summation order: 32 eps_32 of the largest value, the
bound on reordering sums of a few thousand terms that the pair kernel compensates per body; bad owners
and points are refused."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from mfs_inputs.workloads import batched_suspensions, sphere_suspension  # noqa: E402
from paper_2409_04215_gb300 import MFSError  # noqa: E402

from test_gpu_parity import _ctx  # noqa: E402

EPS = 32 * 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


def _solved(wl, **kw):
    ctx = _ctx(wl, autotune=0, **kw)
    ctx.solve_mobility(wl.F[:1], wl.T[:1])
    return ctx


@pytest.mark.parametrize("farfield", [0, 1])
@pytest.mark.parametrize("n", [1, 31, 257, 1023, 1025, 4099])
def test_grouping_matches_small_calls(n, farfield):
    wl = sphere_suspension(count=7, m=90, n=40, seed=3)
    ctx = _solved(wl, farfield=farfield)
    rng = np.random.default_rng(n)
    own = rng.choice([0, 2, 5, 6], n).astype(np.int32)  # bodies 1, 3 and 4 without points
    u = rng.standard_normal((n, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    x = wl.centres[own] + 1.02 * u
    out = ctx.evaluate(x, own)[0].numpy()
    p, t = (a[0].numpy() for a in ctx.evaluate_stress(x, u, own))
    nearest = ctx.evaluate(torch.tensor(x, device="cuda"))[0].cpu().numpy()  # the owner is the nearest body
    tol = EPS if not farfield else 2e-6  # other lists for other point sets: the treecode's accuracy
    assert np.abs(nearest - out).max() <= tol * np.abs(out).max()
    for i in sorted(set([0, n - 1, n // 2, min(n - 1, 31), min(n - 1, 1023)])):
        one = ctx.evaluate(x[i:i + 1], own[i:i + 1])[0, 0].numpy()
        pi, ti = ctx.evaluate_stress(x[i:i + 1], u[i:i + 1], own[i:i + 1])
        assert np.abs(one - out[i]).max() <= tol * np.abs(out).max()
        assert abs(pi[0, 0].item() - p[i]) <= (tol if not farfield else 1e-4) * np.abs(p).max()
        assert np.abs(ti[0, 0].numpy() - t[i]).max() <= (tol if not farfield else 1e-4) * np.abs(t).max()
    ctx.close()


def test_grouping_refusals_and_suspensions():
    wl = batched_suspensions(num_suspensions=2, p_lo=2, p_hi=4, m=60, n=30, nrhs=1, seed=4)
    ctx = _solved(wl)
    x = wl.centres + 2.0
    own = np.arange(wl.num_bodies, dtype=np.int32)
    good = ctx.evaluate(x, own)
    assert torch.isfinite(good).all()
    for bad in ((x, None), (x, own - 1), (x, own + 1), (np.where(own[:, None] == 1, np.inf, x), own)):
        with pytest.raises(MFSError):
            ctx.evaluate(*bad)
    assert torch.equal(ctx.evaluate(x, own), good)  # a refused call leaves the context usable
    ctx.close()
