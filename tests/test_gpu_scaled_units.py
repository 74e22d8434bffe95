"""Units scaled by powers of two (rho by 2^kr, v by 2^kv, B by 2^(kr/2 + kv),
P by 2^(kr + 2 kv)) change no significand of the step, so the scaled run gives
the scaled bits -- also where the fields, or the sound speed, leave the range
of the integer products and the sweeps (whole blocks, or single interfaces)
take FP64 ones."""
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


def run(wb, n, st, kr, kv, **kw):
    """Two steps in scaled units, the result scaled back."""
    sr, sv = 2.0 ** kr, 2.0 ** kv
    sb = 2.0 ** (kr // 2) * sv
    W = st["W"] * np.array([sr, sv, sv, sv, sr * sv * sv])[:, None, None, None]
    g = wb.Grid(n, length=st["length"], rho_floor=0.0, p_floor=0.0, **kw)
    g.load(W, st["bx"] * sb, st["by"] * sb, st["bz"] * sb, primitive=True)
    t = g.advance(2)
    U, bx, by, bz, B = g.read()
    U = U / np.array([sr, sr * sv, sr * sv, sr * sv, sr * sv * sv])[:, None, None, None]
    return [U, bx / sb, by / sb, bz / sb, B / sb, np.array(t * sv)]


@pytest.mark.parametrize("n,kw", [((36, 33, 40), {}), ((64, 32, 32), {}), ((34, 30, 36), {"bc": (1, 0, 1)}),
                                  ((33, 30, 37), {"eps": (0.2, 0.1, 0.2, 0.05, 0.2, 0.1, 0.2), "sweby": 1.5}),
                                  ((32, 32, 32), {"prot_rho": 1e-300, "prot_p": 1e-300})])
@pytest.mark.parametrize("kr,kv", [(-60, 0), (60, 0), (0, 40), (0, -60), (-70, 30), (140, -130)])
def test_scaled_units_give_scaled_bits(wb, n, kw, kr, kv):
    from paper_1701_07452_gb300.initial_conditions import random_box
    st = random_box(n, seed=12)
    for a, b in zip(run(wb, n, st, 0, 0, **kw), run(wb, n, st, kr, kv, **kw)):
        assert np.array_equal(a, b)


def test_one_wild_zone_among_ordinary_ones(wb, oracle_mod):
    """A zone of density 2^-55 and one of energy 2^52 send their blocks to FP64
    products; every zone still matches the oracle."""
    from paper_1701_07452_gb300.initial_conditions import random_box
    from parity import state_err
    n = (40, 36, 34)
    st = random_box(n, seed=4)
    st["W"][0, 10, 11, 12] = 2.0 ** -55
    st["W"][4, 20, 21, 22] = 2.0 ** 52
    g, o = wb.Grid(n, length=st["length"]), oracle_mod.Grid(n, st["length"])
    g.load_state(st)
    o.load_state(st)
    g.advance(1)
    o.advance(1)
    assert state_err(g.read(), o.read()) < 1e-9
