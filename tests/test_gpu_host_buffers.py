"""Host inputs with device outputs: the caller may overwrite its (pinned) memory once the call returns.

The stream is busy with other work when the call comes, so a copy of the input that was still in flight
at the return would read the overwritten values.  The result has to be bit-identical to that of the
same input in device memory.
"""

import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from mfs_inputs import make_workload  # noqa: E402

from test_gpu_parity import _ctx  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("entry", ["precond_apply", "matvec"])
def test_pinned_input_may_be_overwritten(entry):
    wl = make_workload("sphere100_mobility", count=20, m=400, n=200)
    ctx = _ctx(wl)
    gamma = torch.tensor(np.random.default_rng(7).standard_normal((1, ctx.sum_M, 3)))
    pinned = gamma.clone().pin_memory()
    want = getattr(ctx, entry)(gamma.cuda())
    got = torch.empty_like(want)
    busy = torch.randn(4096, 4096, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    torch.cuda.synchronize()
    for _ in range(20):  # tens of milliseconds of work ahead of the call
        busy = busy @ busy.T / 4096.0
    args = [ctx._ctx, ctypes.c_void_p(pinned.data_ptr()), ctypes.c_void_p(got.data_ptr())]
    args += [1, 1] if entry == "precond_apply" else [1]
    rc = getattr(ctx._lib, "mfs_" + entry)(*args, ctypes.c_void_p(stream))
    pinned.zero_()
    torch.cuda.synchronize()
    assert rc == 0
    assert torch.equal(got, want)
    ctx.close()
