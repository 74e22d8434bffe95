"""Patched grids whose pipeline passes hold whole rows or layers of patches (the
intermediates' ghosts along those axes are images of the pass's own patches), in
part or not at all, with periodic, outflow and one-patch axes, down to patches
thinner than the images are deep: the bits of the single grid."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,patches,batch,bc", [
    # layers, rows, everything in one pass; a last pass that is not full
    ((64, 32, 24), (4, 2, 2), 8, (0, 0, 0)), ((64, 32, 72), (4, 2, 6), 16, (0, 0, 0)),
    ((160, 48, 40), (2, 2, 2), 2, (0, 0, 0)), ((20, 18, 10), (2, 3, 2), 0, (0, 0, 0)),
    # too small a pass, or no whole row in it
    ((32, 16, 12), (4, 2, 2), 4, (0, 0, 0)), ((15, 8, 7), (3, 1, 1), 2, (0, 0, 0)),
    # with outflow and one-patch axes
    ((50, 54, 20), (2, 3, 2), 6, (0, 0, 1)), ((50, 54, 60), (2, 3, 2), 2, (0, 1, 0)),
    ((50, 54, 20), (2, 3, 2), 6, (1, 0, 0)), ((50, 54, 20), (2, 3, 2), 0, (0, 1, 0)),
    ((130, 33, 34), (2, 1, 2), 2, (0, 0, 0)), ((40, 39, 28), (1, 3, 2), 3, (0, 0, 0)),
    ((40, 39, 28), (1, 3, 2), 3, (1, 0, 0)), ((128, 6, 4), (1, 2, 1), 1, (0, 0, 0)),
    # patches thinner than the images are deep
    ((16, 64, 96), (16, 2, 3), 32, (0, 0, 0)), ((16, 64, 96), (8, 2, 3), 16, (0, 0, 1)),
    ((4, 4, 6), (4, 2, 3), 0, (0, 0, 0)),
    # one plane
    ((128, 96, 1), (4, 2, 1), 4, (0, 0, 0)), ((128, 96, 1), (4, 2, 1), 0, (0, 0, 0)),
    ((128, 96, 1), (4, 2, 1), 0, (1, 0, 0)),
])
def test_same_bits_as_one_patch(n, patches, batch, bc):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1701_07452_gb300 import binding as wb
    from paper_1701_07452_gb300.initial_conditions import random_box
    st = random_box(n, seed=11)
    out = []
    for kw in ({}, {"patches": patches, "batch_patches": batch}):
        g = wb.Grid(n, length=st["length"], bc=bc, **kw)
        g.load_state(st)
        g.advance(3)
        out.append(g.read())
    for a, b in zip(*out):
        assert np.array_equal(a, b)
