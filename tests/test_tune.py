"""The launch-shape tuner times what a shape decides: steps one a call. The bulk-copy pipeline,
which shares no launches, is kept only where it takes many steps a call faster too."""
import pytest

from paper_1008_2865_gb300 import tune


def test_pick():
    single = {(64, 16, 0): 3.0, (128, 32, 0): 2.0, (128, 32, 1): 1.5}
    # pipeline 0 takes many steps a call two at a time
    assert tune._pick(single, lambda s: {0: 1.2, 1: 1.5}[s[2]]) == (128, 32, 0)
    assert tune._pick(single, lambda s: {0: 2.0, 1: 1.5}[s[2]]) == (128, 32, 1)
    only = {(64, 16, 0): 3.0, (96, 8, 0): 2.5}
    assert tune._pick(only, None) == (96, 8, 0)


@pytest.mark.gpu
def test_shapes_are_timed_one_step_a_call(monkeypatch):
    import paper_1008_2865_gb300 as lb
    calls = []

    class Recorded(lb.Lattice):
        def step(self, n):
            calls.append((self.launch[2], n))
            super().step(n)

    class RecordedBatch(lb.Batch):
        def step(self, n):
            calls.append((0, n))
            super().step(n)

    monkeypatch.setattr(lb, "Lattice", Recorded)
    monkeypatch.setattr(lb, "Batch", RecordedBatch)
    best, table = tune.tune(512, 96, steps=10, save=False)
    assert best in table and {s[2] for s in table} == {0, 1}
    assert sum(n == 1 for _, n in calls) >= 13 * len(table)
    # calls of many steps: one to align and one timed for each pipeline's best
    assert sorted(p for p, n in calls if n > 1) == [0, 0, 1, 1]
    calls.clear()
    from paper_1008_2865_gb300 import inputs
    rhos = [inputs.noisy_density(n, n, n, mean=0.7, amp=0.01, mode="rel") for n in (48, 64)]
    best, table = tune.tune_batch(rhos, [0.1, 0.2], steps=4, save=False)
    assert best in table and all(n == 1 for _, n in calls)
