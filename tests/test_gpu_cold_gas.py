"""Sound speeds down to the end of the normal range (a^2 from 2^-950 to 2^-1000,
floors off): the degenerate branches of the eigen-system (c_f = c_s, no transverse
field) are met there too."""
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


@pytest.mark.parametrize("n", [(8, 8, 8), (32, 32, 32)])
@pytest.mark.parametrize("p", [2.0 ** -950, 2.0 ** -970, 2.0 ** -990, 2.0 ** -1000])
def test_a_cold_box_at_rest_stays_at_rest(wb, n, p):
    """Uniform density and pressure without field: every flux is exactly the
    pressure's, so nothing changes."""
    nx, ny, nz = n
    W = np.zeros((5, nz, ny, nx))
    W[0], W[4] = 1.0, p
    st = {"W": W, "bx": np.zeros((nz, ny, nx + 1)), "by": np.zeros((nz, ny + 1, nx)),
          "bz": np.zeros((nz + 1, ny, nx)), "length": (1.0, 1.0, 1.0)}
    g = wb.Grid(n, length=st["length"], rho_floor=0.0, p_floor=0.0)
    g.load_state(st)
    before = g.read()
    g.advance(2)
    assert g.counters()["unphysical"] == 0
    for a, b in zip(g.read(), before):
        assert np.array_equal(a, b)


def shear_box(n, p):
    """A shear layer of a hundredth of the sound speed, drifting across itself at a
    tenth of it, in a gas of unit density and pressure p, without field."""
    nx, ny, nz = n
    a = np.sqrt(p)
    W = np.zeros((5, nz, ny, nx))
    W[0], W[4] = 1.0, p
    W[1] = 0.1 * a
    W[2] = 0.01 * a * np.sign(np.arange(nx) - nx / 2 + 0.5)
    W[3] = 0.005 * a * np.sign(np.arange(nx) - nx / 2 + 0.5)
    return {"W": W, "bx": np.zeros((nz, ny, nx + 1)), "by": np.zeros((nz, ny + 1, nx)),
            "bz": np.zeros((nz + 1, ny, nx)), "length": (1.0, 1.0, 1.0)}


@pytest.mark.parametrize("p", [2.0 ** -930, 2.0 ** -950, 2.0 ** -970])
def test_a_cold_shear_layer_moves_as_the_oracles(wb, oracle_mod, p):
    """The transverse velocity jump is carried without a transverse field to point
    along (the (1, 1)/sqrt 2 of a vanishing one)."""
    n = (32, 6, 4)
    st = shear_box(n, p)
    g = wb.Grid(n, length=st["length"], rho_floor=0.0, p_floor=0.0)
    o = oracle_mod.Grid(n, st["length"], rho_floor=0.0, p_floor=0.0)
    g.load_state(st)
    o.load_state(st)
    g.advance(2)
    o.advance(2)
    a, b = g.read()[0], o.read()[0]
    for c in range(5):
        scale = np.abs(b[c]).max()
        assert np.abs(a[c] - b[c]).max() <= 1e-9 * scale, c
