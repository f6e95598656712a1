"""A solve that ends with a device error leaves no solution for evaluation and gradients.

The flag is set from the host (mfs_selftest_device_error): no kernel gives up.  Every solve entry then
reports MFS_ERR_DEVICE_TIMEOUT, evaluation and gradient refuse as before any solve, and the next
solve is what it was.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from mfs_inputs.workloads import sphere_suspension, two_sphere_elastance  # noqa: E402

from test_gpu_parity import _ctx  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("problem", ["mobility", "resistance", "elastance", "capacitance"])
def test_no_solution_after_a_device_error(problem):
    from paper_2409_04215_gb300.api import MFSError

    stokes = problem in ("mobility", "resistance")
    wl = sphere_suspension(count=3, m=91, n=45, seed=2) if stokes else two_sphere_elastance(m=91, n=45)
    ctx = _ctx(wl, autotune=0, max_rhs=1)
    rng = np.random.default_rng(0)
    args = rng.standard_normal((2, 1, 3, 3)) if stokes else rng.standard_normal((1, 1, wl.num_bodies))
    solve = getattr(ctx, "solve_" + problem)
    uses = [lambda: ctx.evaluate(10.0 + rng.standard_normal((4, 3)))]
    if problem == "mobility":
        uses.append(lambda: ctx.mobility_vjp(*args))
    want = solve(*args)[0]
    for use in uses:
        use()
    assert ctx._lib.mfs_selftest_device_error(ctx._ctx, None) == 0
    with pytest.raises(MFSError) as e:
        solve(*args)
    assert e.value.status == 7
    for use in uses:
        with pytest.raises(MFSError) as e:
            use()
        assert e.value.status == 1
    assert torch.equal(solve(*args)[0], want)
    for use in uses:
        use()
    ctx.close()
