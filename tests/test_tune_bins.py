"""The autotuner's choice of the point bins, on the CPU with a clock and operators of the test's own."""
from paper_2411_01955_gb300 import tune


def test_bins_are_chosen_for_both_operators(monkeypatch):
    """Bins of 16 are best for the adjoint alone, bins of 8 for the two operators together."""
    cost = {"forward": {8: 1.0, 16: 4.0, 32: 3.0}, "adjoint": {8: 2.0, 16: 1.5, 32: 2.5}}
    state = {"tile": None, "t": 0.0}

    def ran(what):
        state["t"] += cost[what][state["tile"]]

    def clock(fn, reps):
        t0 = state["t"]
        for _ in range(reps):
            fn()
        return (state["t"] - t0) / reps

    monkeypatch.setattr(tune.L, "plan_set_tuning", lambda plan, key, value: state.update(tile=value))
    monkeypatch.setattr(tune.L, "forward", lambda plan, x, y: ran("forward"))
    monkeypatch.setattr(tune.L, "adjoint", lambda plan, y, out: ran("adjoint"))
    monkeypatch.setattr(tune, "_time", clock)
    t = tune.time_bins(None, tune.valid_tiles(640, 6), None, None, None, 3)
    assert t == {8: 3.0, 16: 5.5, 32: 5.5} and tune.pick(t) == 8
