"""Tile lengths of the treecode's sums (mfs_api.cu, build_plan_lists and ff_check_variant).

A cell of two bodies holds 2 M targets, cut into as few tiles as the forced pair-kernel entry allows,
of about equal length in whole target pairs; the sums at check points run in the packed entry of
256-target tiles.  For M at the edges (cells below one target pair a thread, exactly one tile, one
target more, a short remainder) and entries with tiles of 256 to 768 targets, and for the entries
that keep their own tile at the check points (scalar, several right-hand sides), the treecode's sums
are held to the direct sums: relative 2-norm 1e-6, the bar of the treecode's other tests.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from mfs_inputs import make_workload  # noqa: E402

from test_gpu_parity import _ctx, _rel  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("entry", ["PackedStokes<1,2,64>", "PackedStokes<1,4,64>", "PackedStokes<1,6,64>",
                                   "PackedStokesReg<1,1,128>", "Scalar<3,1,4,128>", "PackedStokes<4,1,64>"])
@pytest.mark.parametrize("m", [61, 128, 257, 385])
def test_tree_tiles(entry, m):
    from paper_2409_04215_gb300.api import pair_variants

    idx, _, _, nrhs, _ = [t for t in pair_variants() if t[1] == entry][0]
    wl = make_workload("batched256_mobility", num_suspensions=2, p_lo=30, p_hi=41, m=m, n=60, seed=17)
    direct, tree = _ctx(wl), _ctx(wl, farfield=1, pair_variant=idx)
    s = torch.tensor(np.random.default_rng(m).standard_normal((nrhs, direct.sum_N, 3)), device="cuda")
    for include_self in (False, True):
        a = direct.pair_sum(s, include_self=include_self).cpu().numpy()
        b = tree.pair_sum(s, include_self=include_self).cpu().numpy()
        assert _rel(b.reshape(-1), a.reshape(-1)) < 1e-6, include_self
    assert tree.pair_variant(nrhs) == entry
    direct.close()
    tree.close()
