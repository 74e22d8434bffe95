"""The dt that a step's update prepares for the next step (its last block)
against one dt launch a step: the same states, clock and counters, with and
without a time limit, around the 64-step clock reads, and after a run that has
become unphysical."""
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


def make(wb, kw):
    from paper_1701_07452_gb300.initial_conditions import random_box
    n = (12, 8, 10)
    st = random_box(n, seed=3)
    g = wb.Grid(n, length=st["length"], **kw)
    g.load_state(st)
    return g


@pytest.mark.parametrize("kw", [{}, {"bc": (1, 0, 1)}, {"patches": (2, 2, 1)}, {"patches": (3, 2, 2), "batch_patches": 5},
                                {"dt_lag": True}])
@pytest.mark.parametrize("steps,frac", [(3, None), (70, None), (130, 63.5), (130, 64.5), (70, 64.0)])
def test_one_call_equals_single_steps(wb, kw, steps, frac):
    one, many = make(wb, kw), make(wb, kw)
    t_end = 0.0 if frac is None else frac * make(wb, kw).dt()
    t1 = one.advance(steps, t_end=t_end)
    for _ in range(steps):
        t2 = many.advance(1, t_end=t_end)
    assert t1 == t2 and one.counters() == many.counters()
    for a, b in zip(one.read(), many.read()):
        assert np.array_equal(a, b)


def test_an_unphysical_run_counts_the_steps_it_could_not_take(wb):
    grids = []
    for calls in ((4,), (1, 1, 1, 1)):
        g = make(wb, {})
        U, bx, by, bz, _ = g.read()
        U[4, 2, 3, 4] = np.nan
        g.load(U, bx, by, bz)
        for c in calls:
            with pytest.raises(wb.WombatError):
                g.advance(c)
        grids.append(g.counters())
    a, b = grids
    # the step that meets the state counts its zones, each later one itself
    assert a == b and a["steps"] == 1 and a["unphysical"] > 3
