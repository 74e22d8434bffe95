"""Host reads into arrays of any state: fresh pages, pages written before, a
buffer that starts and ends inside a page; whole arrays arrive and nothing
outside them is written."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(3, 2, 1), (20, 16, 12), (40, 33, 28)])
@pytest.mark.parametrize("batch", [False, True])
def test_reads_fill_their_arrays_and_no_more(n, batch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1701_07452_gb300 import binding as wb
    from paper_1701_07452_gb300.initial_conditions import random_box
    st = random_box(n, seed=5)
    nx, ny, nz = n
    shapes = [(5, nz, ny, nx), (nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx), (3, nz, ny, nx)]
    if batch:
        g = wb.Batch([{"n": n, "length": st["length"]}])
        g.load_state(0, st)
        want = g.read(0)
    else:
        g = wb.Grid(n, length=st["length"])
        g.load_state(st)
        want = g.read()
    # one buffer, each array between guard words, at odd multiples of 8 bytes
    sizes = [int(np.prod(s)) for s in shapes]
    guard = -7.25
    buf = np.full(sum(sizes) + 6, guard)
    at, views = 1, []
    for s, m in zip(shapes, sizes):
        views.append(buf[at:at + m])
        at += m + 1
    ptrs = [ctypes.c_void_p(v.ctypes.data) for v in views]
    if batch:
        g._check(wb.lib().wb_batch_read(g._h, 0, *ptrs, 0))
    else:
        g._check(wb.lib().wb_read_state(g._h, *ptrs, 0))
    for v, w in zip(views, want):
        assert np.array_equal(v, w.ravel())
    guards = [0] + [int(x) for x in np.cumsum([m + 1 for m in sizes])]
    assert np.all(buf[guards] == guard)
    for _ in range(2):  # fresh arrays again
        for a, b in zip(g.read(0) if batch else g.read(), want):
            assert np.array_equal(a, b)
