"""The autotuner's choice over several batches, with a fake solve: a slow solve of
one batch counts as much as it would if that batch were tuned alone."""
import pytest

torch = pytest.importorskip("torch")


def run(monkeypatch, plan, reps):
    """plan[split_min] = per batch its solves' seconds in turn."""
    from paper_2601_21552_gb300 import api, autotune
    clock = {"t": 0.0}
    calls = {}

    def fake_solve(batch, want_model=False, stats=False, time_budget_ms=0, split_min=0):
        k = calls[(split_min, batch)] = calls.get((split_min, batch), -1) + 1
        clock["t"] += plan[split_min][batch][k]

    monkeypatch.setattr(api, "solve", fake_solve)
    monkeypatch.setattr(api, "status", lambda *a: 0)
    monkeypatch.setattr(autotune.time, "perf_counter", lambda: clock["t"])
    monkeypatch.setattr(torch.cuda, "synchronize", lambda *a: None)
    return autotune.sweep(0, reps=reps, space={"split_min": list(plan)}, more=(1, 2))


def test_a_tail_of_one_batch_is_not_steady(monkeypatch):
    # 64: one solve of four of the large batch takes 2.2x, 1.30x over the three
    # batches; 128: 1 % slower in the mean, steady
    plan = {64: [[0.75, 0.75, 0.75, 1.65], [0.005] * 4, [0.012] * 4],
            128: [[0.985] * 4, [0.00505] * 4, [0.012] * 4]}
    best, trials = run(monkeypatch, plan, 4)
    assert trials[0]["mean_s"] < trials[1]["mean_s"] < 1.05 * trials[0]["mean_s"]
    assert best["options"] == {"split_min": 128}


def test_the_mean_is_each_batch_s_own(monkeypatch):
    # 64: median 0.70, but one solve of four takes 5x (mean 1.40); 128: always 1.1
    plan = {64: [[0.70, 0.70, 0.70, 3.5], [0.005] * 4, [0.012] * 4],
            128: [[1.1] * 4, [0.005] * 4, [0.012] * 4]}
    best, trials = run(monkeypatch, plan, 4)
    assert best["options"] == {"split_min": 128}
    assert trials[0]["mean_s"] == pytest.approx((1.40 * 0.005 * 0.012) ** (1 / 3))
    assert trials[1]["median_s"] == pytest.approx((1.1 * 0.005 * 0.012) ** (1 / 3))
    assert [len(t) for t in trials[0]["times"]] == [4, 4, 4]


def test_the_file_that_every_tuned_call_reads_stays_small(monkeypatch):
    import json
    import os

    from paper_2601_21552_gb300 import autotune
    plan = {s: [[0.8] * 63 + [2.5], [0.005] * 64, [0.012] * 64] for s in range(16)}
    _, trials = run(monkeypatch, plan, 64)
    kept = [autotune.summary(t) for t in trials]
    assert len(json.dumps(kept)) < 16 * 400
    # (63 * 0.8 + 2.5) / 64 = 0.8265625, kept to six decimals
    assert kept[3]["batches"][0] == {"mean_s": pytest.approx(0.8265625, abs=5.1e-7, rel=0),
                                     "median_s": 0.8, "max_s": 2.5}
    assert kept[3]["options"] == {"split_min": 3} and "times" not in kept[3]
    assert os.path.getsize(autotune.DEFAULT_OUT) < 8000
