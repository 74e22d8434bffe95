"""Batches whose boxes agree or differ in the sweeps' thread layout (rings of
short closed pencils, open pencils), with more (box, axis) entries than one or
two rounds of the 32-wide entry search cover: the bits of the grid path."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

RINGS = [(16, 12, 32), (42, 31, 20), (64, 126, 18)]
OPEN = [(9, 12, 5), (33, 4, 7)]
MIXED = [(130, 5, 4), (20, 16, 32), (1, 1, 7), (12, 140, 1)]


@pytest.mark.parametrize("sizes,bc", [
    (RINGS, (0, 0, 0)), (OPEN, (1, 1, 1)), (OPEN, (0, 1, 0)), (MIXED, (0, 0, 0)),
    ([(5, 4, 3)] * 35 + MIXED, (0, 0, 0)), ([(2, 3, 4)] * 350 + RINGS, (0, 0, 0)),
])
@pytest.mark.parametrize("form", ["staged", "persistent"])
def test_same_bits_as_the_grid(sizes, bc, form):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1701_07452_gb300 import binding as wb
    from paper_1701_07452_gb300.initial_conditions import random_box
    states = [random_box(n, seed=300 + i) for i, n in enumerate(sizes)]
    bt = wb.Batch([{"n": n, "length": st["length"], "bc": bc} for n, st in zip(sizes, states)])
    bt.set_form(form)
    for i, st in enumerate(states):
        bt.load_state(i, st)
    bt.set_steps(-1, 2)
    bt.advance(2)
    for i in {0, len(sizes) // 2, *range(max(0, len(sizes) - 4), len(sizes))}:
        g = wb.Grid(sizes[i], length=states[i]["length"], bc=bc)
        g.load_state(states[i])
        g.advance(2)
        for a, b in zip(bt.read(i), g.read()):
            assert np.array_equal(a, b), i
