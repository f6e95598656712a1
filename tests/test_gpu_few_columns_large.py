"""The few-column apply (apply_few.cu) on large factors: two warps a row beyond 1024 rows, one beyond 4096,
and on both sides of the line (2^24 columns times elements) at which three and more columns go to the
tensor cores.

Against the FP64 path (precision = 1, itself held to the oracle at 1e-11): the matvec on a smooth field at
the FP32 path's bar (1e-6, relative 2-norm), and the transpose through <A g, w> = <g, A^T w> at the bar of
that identity's other test (1e-6 |A g| |w|; A^T w by itself carries the rounding of its FP32 sums through
the transposed pseudo-inverse, 2e-5 to 3e-4 of it at these sizes whichever apply runs).  A wrong factor row
would show in either at 1e-4 or more.  The form that ran is read from the results of the two piece counts,
which the few-column form does not look at.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from mfs_inputs.workloads import sphere_suspension  # noqa: E402

from test_gpu_parity import _ctx  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


# factor rows 3 N and 3 M: 1056 and 2109 (two warps a row), 1209 and 4203 (two and one), then
# 3 x 3000 x 1800 = 0.97 x 2^24 and 3 x 3120 x 1800 = 1.004 x 2^24
@pytest.mark.parametrize("count,m,n,few", [(2, 703, 352, True), (2, 1401, 403, True), (3, 1000, 600, True),
                                           (3, 1040, 600, False)])
def test_large_factors(count, m, n, few):
    wl = sphere_suspension(count=count, m=m, n=n, volume_fraction=0.1, seed=5)
    exact = _ctx(wl, precision=1, autotune=0)
    rng = np.random.default_rng(count * m)
    g = exact.pair_sum(torch.tensor(rng.standard_normal((1, exact.sum_N, 3)), device="cuda"), include_self=True)
    w = torch.tensor(rng.standard_normal((1, exact.sum_M, 3)), device="cuda")
    want = exact.matvec(g)
    exact.close()
    got = []
    for mode in (1, 2):
        ctx = _ctx(wl, tensor_cores=mode, autotune=0)
        got.append((ctx.matvec(g), ctx.matvec_transposed(w), ctx.precond_apply(g, project=False)))
        ctx.close()
    assert float((got[0][0] - want).norm() / want.norm()) < 1e-6
    assert abs(float((want * w).sum() - (g * got[0][1]).sum())) <= 1e-6 * float(want.norm() * w.norm())
    assert torch.equal(got[0][2], got[1][2]) == few
    assert torch.equal(got[0][1], got[1][1]) == few
