"""The treecode's sums of strengths whose far field is nearly constant over a body: of one direction, as in
sedimentation, and a long wave.

Against the FP64 sums (precision = 1), ellipsoids with enough targets for local expansions.  With one order
of equivalent sources and no local expansions these sums were 1.2e-8 to 2.0e-8 off for strengths of one
direction and 1.4e-8 to 3.1e-8 for the wave (400 to 1000 bodies): the bars are 2.5e-8 and 3.5e-8.  Carried by
the FP32 records of the local sources as a whole, the far field took them to 4.4e-8 to 6.1e-8.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from mfs_inputs.workloads import ellipsoid_cluster  # noqa: E402

from test_gpu_parity import _ctx  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("kind", ["stokes", "laplace"])
def test_nearly_constant_far_field(kind):
    wl = ellipsoid_cluster(count=400, n_v=22, seed=6)
    wl.kind = kind
    exact, tree = _ctx(wl, precision=1, autotune=0, max_rhs=2), _ctx(wl, farfield=1, max_rhs=2)
    one = np.array([0.3, -0.5, 1.0]) if kind == "stokes" else np.ones(1)
    body = np.repeat(wl.centres, [len(wl.shapes[i].proxy) for i in wl.shape_id], axis=0)
    wave = np.sin(body @ np.array([0.11, 0.07, -0.05]))
    s = torch.tensor(np.stack([np.tile(one, (len(body), 1)), np.repeat(wave[:, None], len(one), 1)]), device="cuda")
    want = exact.pair_sum(s)
    got = [tree.pair_sum(s), torch.cat([tree.pair_sum(s[h:h + 1].contiguous()) for h in (0, 1)])]
    for g in got:
        for h, bar in ((0, 2.5e-8), (1, 3.5e-8)):
            assert float((g[h] - want[h]).norm() / want[h].norm()) < bar
    exact.close()
    tree.close()
