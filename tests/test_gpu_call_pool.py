"""What calls keep between them does not grow with the number of contexts: 256 MB a device, all of it given
back with the last context."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from mfs_inputs.workloads import sphere_suspension  # noqa: E402

from test_gpu_parity import _ctx  # noqa: E402

MB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


def test_many_contexts_share_what_is_kept():
    wl = sphere_suspension(count=3, m=91, n=45, seed=2)
    rng = np.random.default_rng(0)
    F, T = rng.standard_normal((2, 4, 3, 3))
    points = 9.0 + rng.random((1000000, 3))  # about 230 MB of scratch: points, order, sums and outputs
    ctxs = [_ctx(wl, autotune=0) for _ in range(4)]
    for c in ctxs:
        c.solve_mobility(F, T)
        c.evaluate(points[:100], nrhs=4)  # the kernels are loaded
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    want = None
    for c in ctxs:
        got = c.evaluate(points, nrhs=4)
        want = got if want is None else want
        assert np.array_equal(got, want)
    torch.cuda.synchronize()
    # 32 MB: the granularity of the driver's own allocations
    assert free0 - torch.cuda.mem_get_info()[0] <= 256 * MB + 32 * MB
    for c in ctxs:
        c.close()
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] >= free0 - 32 * MB
