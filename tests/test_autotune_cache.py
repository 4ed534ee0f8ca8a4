"""Which cached schedules the autotuner uses (no GPU): none tuned for the other potential scheme,
none timed on another library's kernels, none timed at the other kind of count."""
import json

import pytest

from paper_2407_01654_gb300 import autotune
from paper_2407_01654_gb300 import workloads as wl


@pytest.fixture
def tuner(tmp_path, monkeypatch):
    path = tmp_path / "tune.json"
    monkeypatch.setenv("EHD_AUTOTUNE_CACHE", str(path))
    calls = []

    def timer(params, fields, ov, steps, fixed_iter):
        calls.append(ov)
        fast = 2 if params["potential_scheme"] else 4  # loop 4 has no conventional form
        return 1.0 if ov["poisson_loop"] == fast else 2.0

    return path, calls, timer


def test_a_schedule_is_not_served_to_the_other_scheme(tuner):
    path, calls, timer = tuner
    p = wl.make_params(nx=512, ny=1024)
    assert autotune.tune(p, timer=timer, device_name="dev")["poisson_loop"] == 4
    conv = dict(p, potential_scheme=1, chi=2.0)
    assert autotune.tune(conv, timer=timer, device_name="dev")["poisson_loop"] == 2
    calls.clear()
    for q, loop in ((p, 4), (conv, 2)):
        assert autotune.tune(q, timer=timer, device_name="dev")["poisson_loop"] == loop
    assert calls == []


@pytest.mark.parametrize("edit", ["other", "none"])
def test_a_schedule_of_another_library_is_tuned_again(tuner, edit):
    path, calls, timer = tuner
    p = wl.make_params(nx=64, ny=64)
    reqs = [(p, {})]
    rate = lambda requests, schedule, steps, budget: calls.append(schedule) or 1.0
    autotune.tune(p, timer=timer, device_name="dev")
    autotune.tune_batch(reqs, timer=rate, device_name="dev")
    d = json.loads(path.read_text())
    for e in d.values():
        if edit == "other":
            e["library"] = "0" * 16
        else:
            del e["library"]  # as entries written before libraries were told apart
        e["overrides"] = {"poisson_loop": 1, "tile_rows": 64}
    path.write_text(json.dumps(d))
    calls.clear()
    assert autotune.tune(p, timer=timer, device_name="dev")["poisson_loop"] == 4
    assert calls == autotune.candidates(p)
    calls.clear()
    assert autotune.tune_batch(reqs, timer=rate, device_name="dev") in autotune.batch_candidates()
    assert calls == autotune.batch_candidates()
    calls.clear()
    autotune.tune(p, timer=timer, device_name="dev")
    autotune.tune_batch(reqs, timer=rate, device_name="dev")
    assert calls == []  # and kept from then on


class FakeSim:
    """Records the parameters a candidate is timed with."""
    seen = []

    def __init__(self, params):
        FakeSim.seen.append(params)
        self.params = params

    def loop_kind(self):
        return self.params["poisson_loop"]

    def set_fields(self, *fields):
        pass

    def step(self, n, stats=True):
        pass

    def read_stats(self):
        pass

    def close(self):
        pass


@pytest.mark.parametrize("count", [0, 5])
def test_candidates_run_the_kernels_that_the_parameters_run(monkeypatch, tuner, count):
    """Under the rule the candidates are timed under the rule (its smallest and largest count
    set), at a fixed count at a fixed one; the two have cached schedules of their own."""
    from paper_2407_01654_gb300 import ehd
    path, calls, timer = tuner
    monkeypatch.setattr(ehd, "Sim", FakeSim)
    FakeSim.seen = []
    p = wl.make_params(nx=64, ny=64, poisson_fixed_iter=count)
    ov = {"poisson_loop": 2, "tile_rows": 32}
    assert autotune.time_candidate(p, autotune._default_fields(p), ov, 4, 32) >= 0.0
    q, = FakeSim.seen
    assert q["poisson_loop"] == 2 and q["tile_rows"] == 32
    if count:
        assert q["poisson_fixed_iter"] == 32
    else:
        assert q["poisson_fixed_iter"] == 0
        assert q["poisson_min_iter"] == q["poisson_max_iter"] == 32 and 0 < q["poisson_tol"] < 1e-9
    autotune.tune(p, timer=timer, device_name="dev")
    calls.clear()
    autotune.tune(dict(p, poisson_fixed_iter=0 if count else 5), timer=timer, device_name="dev")
    assert calls == autotune.candidates(p)
