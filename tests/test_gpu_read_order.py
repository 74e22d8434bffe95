"""Host reads are ordered on the stream: work enqueued ahead of a read that still
uses the destination array sees its old contents."""
import ctypes
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HOST_FN = ctypes.CFUNCTYPE(None, ctypes.c_void_p)


def enqueue_snapshot(lib, stream, buf, seen):
    """A host function on the stream: waits, then copies buf into seen."""
    def work(_):
        time.sleep(0.3)
        seen[:] = buf
    fn = HOST_FN(work)
    lib.cudaLaunchHostFunc.argtypes = [ctypes.c_void_p, HOST_FN, ctypes.c_void_p]
    assert lib.cudaLaunchHostFunc(ctypes.c_void_p(stream), fn, None) == 0
    return fn  # to be kept until the stream has run it


@pytest.mark.parametrize("batch,pinned", [(False, False), (True, False), (True, True)])
def test_work_ahead_of_a_read_sees_the_old_contents(batch, pinned):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1701_07452_gb300 import binding as wb
    from paper_1701_07452_gb300.initial_conditions import random_box
    n = (33, 20, 17)
    nx, ny, nz = n
    st = random_box(n, seed=8)
    stream = torch.cuda.Stream()
    if batch:
        g = wb.Batch([{"n": n, "length": st["length"]}], stream=stream)
        g.load_state(0, st)
        want = g.read(0)
    else:
        g = wb.Grid(n, length=st["length"], stream=stream)
        g.load_state(st)
        want = g.read()
    sizes = [5 * nx * ny * nz, nz * ny * (nx + 1), nz * (ny + 1) * nx, (nz + 1) * ny * nx, 3 * nx * ny * nz]
    hold = torch.empty(sum(sizes), dtype=torch.float64, pin_memory=pinned)
    buf = hold.numpy()
    rng = np.random.default_rng(1)
    buf[:] = rng.standard_normal(buf.size)  # no zero byte where it would not show
    old = buf.copy()
    views = np.split(buf, np.cumsum(sizes)[:-1])
    ptrs = [ctypes.c_void_p(v.ctypes.data) for v in views]
    seen = np.empty_like(buf)
    keep = enqueue_snapshot(wb.lib(), stream.cuda_stream, buf, seen)
    if batch:
        g._check(wb.lib().wb_batch_read(g._h, 0, *ptrs, 0))
    else:
        g._check(wb.lib().wb_read_state(g._h, *ptrs, 0))
    stream.synchronize()
    del keep
    assert np.array_equal(seen, old)
    for v, w in zip(views, want):
        assert np.array_equal(v, w.ravel())
