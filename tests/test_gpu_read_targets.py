"""Reads without the on_device flag into memory that is not the host's own: the
CUDA copy decides (whole arrays, or an error status); the host touches nothing."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("kind", ["device", "managed", "pinned"])
def test_other_targets(batch, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1701_07452_gb300 import binding as wb
    from paper_1701_07452_gb300.initial_conditions import random_box
    n = (20, 16, 12)
    nx, ny, nz = n
    st = random_box(n, seed=2)
    if batch:
        g = wb.Batch([{"n": n, "length": st["length"]}])
        g.load_state(0, st)
    else:
        g = wb.Grid(n, length=st["length"])
        g.load_state(st)
    want = np.concatenate([a.ravel() for a in (g.read(0) if batch else g.read())])
    sizes = [5 * nx * ny * nz, nz * ny * (nx + 1), nz * (ny + 1) * nx, (nz + 1) * ny * nx, 3 * nx * ny * nz]
    L, total, managed = wb.lib(), sum(sizes), ctypes.c_void_p()
    if kind == "managed":
        assert L.cudaMallocManaged(ctypes.byref(managed), ctypes.c_size_t(8 * total), 1) == 0
        base = managed.value
    else:
        hold = torch.zeros(total, dtype=torch.float64, pin_memory=kind == "pinned",
                           device="cuda" if kind == "device" else "cpu")
        base = hold.data_ptr()
    at = [base + 8 * int(x) for x in np.concatenate([[0], np.cumsum(sizes)[:-1]])]
    ptrs = [ctypes.c_void_p(a) for a in at]
    try:
        if batch:
            g._check(L.wb_batch_read(g._h, 0, *ptrs, 0))
        else:
            g._check(L.wb_read_state(g._h, *ptrs, 0))
    except wb.WombatError as e:
        assert kind == "device" and e.code != 0
        L.cudaGetLastError()
    else:
        torch.cuda.synchronize()
        if kind == "managed":
            got = np.ctypeslib.as_array(ctypes.cast(managed, ctypes.POINTER(ctypes.c_double)), (total,)).copy()
        else:
            got = hold.cpu().numpy()
        assert np.array_equal(got, want)
    if kind == "managed":
        L.cudaFree(managed)
    again = np.concatenate([a.ravel() for a in (g.read(0) if batch else g.read())])
    assert np.array_equal(again, want)
