"""What the autotuner spends and decides on: one trial of real steps for each
configuration that differs in what runs, none that has no steps left to time."""
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


def batch(wb, sizes, steps):
    from paper_1701_07452_gb300.initial_conditions import random_box
    states = [random_box(n, seed=40 + i) for i, n in enumerate(sizes)]
    bt = wb.Batch([{"n": n, "length": st["length"]} for n, st in zip(sizes, states)])
    for i, st in enumerate(states):
        bt.load_state(i, st)
    bt.set_steps(-1, steps)
    return bt


@pytest.mark.parametrize("trial", [1, 3])
def test_one_trial_a_configuration(wb, trial):
    """The persistent form once for each number of blocks per SM, the staged form,
    which has no such number, once."""
    bt = batch(wb, [(13, 9, 8), (10, 11, 6 + trial)], 1000)  # sizes of its own: tuned ones start as tuned
    blocks = bt.get_config()["blocks_per_sm"]  # the most that fit
    bt.config(blocks_per_sm=1)
    assert bt.autotune(trial_steps=trial) > 0.0
    assert [bt.counters(i)["steps"] for i in range(2)] == [trial * (blocks + 1)] * 2


def test_trials_without_steps_decide_nothing(wb):
    """With steps for one trial only, the first configuration is the only one that
    was timed and is kept; a batch of the same sizes later starts from the default,
    not from a comparison that did not take place."""
    sizes = [(14, 9, 8), (10, 12, 7)]
    bt = batch(wb, sizes, 2)
    default = bt.get_config()
    ms = bt.autotune(trial_steps=2)
    assert [bt.counters(i)["steps"] for i in range(2)] == [2, 2]
    assert bt.get_config() == default
    # 2 steps of some 20 stages of one persistent launch, not an empty launch
    assert ms > 0.0
    other = batch(wb, sizes, 2)
    assert other.get_config() == default


def test_no_steps_at_all(wb):
    bt = batch(wb, [(15, 9, 8)], 0)
    default = bt.get_config()
    bt.autotune(trial_steps=1)
    assert bt.counters(0)["steps"] == 0
    assert bt.get_config() == default
