"""The sweeps' thread layouts (wbu::sweep_tile) at the sizes where they change:
rings of periodic pencils of up to 128 zones (inside a warp, straddling two,
spanning a block), the open layout's block edges
(125 faces emitted from 128 zones, 3 zones between pencils), pencils shorter
than the stencil, and outflow boxes, whose pencils are never closed.  One step
against the oracle."""
import pytest

from parity import state_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1701_07452_gb300 import binding
    binding.lib()
    return binding


@pytest.mark.parametrize("n,bc", [
    ((16, 8, 4), (0, 0, 0)), ((32, 24, 5), (0, 0, 0)), ((30, 17, 33), (0, 0, 0)), ((122, 3, 2), (0, 0, 0)),
    ((125, 31, 1), (0, 0, 0)), ((2, 126, 6), (0, 0, 0)), ((1, 5, 40), (0, 0, 0)), ((20, 64, 42), (0, 0, 0)), ((128, 3, 21), (0, 0, 0)), ((127, 60, 3), (0, 0, 0)),
    ((16, 32, 8), (1, 1, 1)), ((59, 4, 61), (1, 0, 0)), ((119, 2, 3), (0, 0, 1)), ((1, 1, 7), (1, 1, 1)),
    ((40, 1, 3), (1, 1, 0)), ((3, 2, 1), (1, 1, 1)), ((20, 24, 1), (1, 0, 0)), ((4, 33, 18), (0, 1, 0)),
    # one-zone closed axes in launches of more than 152 tiles
    ((200, 120, 1), (0, 0, 0)), ((200, 120, 1), (1, 0, 0)), ((64, 1, 250), (0, 0, 0)), ((1, 150, 130), (0, 0, 0)),
    ((1, 64, 128), (0, 0, 0)),
])
def test_one_step_matches_the_oracle(wb, oracle_mod, n, bc):
    from paper_1701_07452_gb300.initial_conditions import random_box
    st = random_box(n, seed=sum(n))
    g = wb.Grid(n, length=st["length"], bc=bc)
    o = oracle_mod.Grid(n, st["length"], bc=bc)
    g.load_state(st)
    o.load_state(st)
    g.advance(1)
    o.advance(1)
    assert state_err(g.read(), o.read()) < 1e-11
