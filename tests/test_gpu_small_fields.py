"""Fields that fall off through the end of the double range (Gaussian tails of
the transverse field and momentum, underflowing noise ahead of a front): an
interface gives the same bits whether its launch takes FP64 products (grids of at
most 152 tiles, blocks with fields beyond the integer products' range) or
integer ones (larger grids, patches, batches)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1701_07452_gb300 import binding
    binding.lib()
    return binding


def tail_box(n, low, seed):
    """Unit density and pressure, a uniform field along y and z that falls off
    along x from 1 to 2^low (a Gaussian tail) and to exactly 0 in the middle third,
    momenta likewise with other signs.  Face fields of axis x are 0.25 everywhere,
    so div B is 0."""
    nx, ny, nz = n
    rng = np.random.default_rng(seed)
    x = np.abs((np.arange(nx) + 0.5) / nx - 0.5) * 2.0       # 1 at the ends, 0 in the middle
    e = low * (1.0 - x) ** 2 * 2.2
    tail = np.where(e < low * 1.0001, 0.0, np.ldexp(1.0, 0) * np.exp2(np.maximum(e, -1080.0)))
    tail *= 1.0 + 0.3 * rng.random(nx)
    W = np.zeros((5, nz, ny, nx))
    W[0] = 1.0 + 0.1 * rng.random((nz, ny, nx))
    W[1] = 0.3 * tail
    W[2] = -0.2 * tail
    W[3] = 0.1 * tail[::-1]
    W[4] = 0.6
    bx = np.full((nz, ny, nx + 1), 0.25)
    by = np.broadcast_to(tail, (nz, ny + 1, nx)).copy()
    bz = np.broadcast_to(-tail[::-1], (nz + 1, ny, nx)).copy()
    return {"W": W, "bx": bx, "by": by, "bz": bz, "length": tuple(float(a) for a in n)}


def grid(wb, n, st, steps, **kw):
    g = wb.Grid(n, length=st["length"], **kw)
    g.load_state(st)
    g.advance(steps)
    return g.read()


@pytest.mark.parametrize("low", [-90, -150, -400, -1000, -1070])
@pytest.mark.parametrize("bc", [(0, 0, 0), (1, 0, 0)])
def test_small_grid_and_batch_agree(wb, low, bc):
    """A 64 x 6 x 4 grid (51 tiles: FP64 products) and a batch of the same box (integer)."""
    n = (64, 6, 4)
    st = tail_box(n, low, 3)
    want = grid(wb, n, st, 2, bc=bc)
    for form in ("staged", "persistent"):
        bt = wb.Batch([{"n": n, "length": st["length"], "bc": bc}])
        bt.set_form(form)
        bt.load_state(0, st)
        bt.set_steps(0, 2)
        bt.advance(2)
        for a, b in zip(bt.read(0), want):
            assert np.array_equal(a, b), (form, np.abs(a - b).max())


@pytest.mark.parametrize("low", [-150, -1000, -1070])
@pytest.mark.parametrize("kw", [{}, {"eps": (0.2, 0.1, 0.2, 0.05, 0.2, 0.1, 0.2)}])
def test_large_grid_its_patches_and_a_batch_agree(wb, low, kw):
    """Integer products on the whole grid, FP64 ones in passes of one patch."""
    n = (32, 32, 32)
    st = tail_box(n, low, 4)
    want = grid(wb, n, st, 2, **kw)
    for p, m in (((2, 4, 4), 1), ((2, 2, 2), 0)):
        for a, b in zip(grid(wb, n, st, 2, patches=p, batch_patches=m, **kw), want):
            assert np.array_equal(a, b), (p, np.abs(a - b).max())
    bt = wb.Batch([{"n": n, "length": st["length"]}], **kw)
    bt.load_state(0, st)
    bt.set_steps(0, 2)
    bt.advance(2)
    for a, b in zip(bt.read(0), want):
        assert np.array_equal(a, b), np.abs(a - b).max()
