"""The scheme comparison of bench.py against fakes of the solver and of torch (no GPU): only
MUSCL-FV2's run may be shortened, what failed is reported, and ratios compare equal windows."""
import importlib.util
import os
import types

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
COST = {"dg2_nl": 2.0, "dg2_ll": 3.0, "fv2": 1.0, "fv1": 0.5, "dg2_nl_4m": 0.25}  # ms per second


@pytest.fixture(scope="module")
def bench():
    spec = importlib.util.spec_from_file_location("bench_host2", os.path.join(ROOT, "bench.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    return m


def fakes(limits, early=1.0):
    """A binding whose runs of a scheme longer than its limit (s) go non-finite, and a clock
    of COST ms per simulated second, `early` times that in the first 70 s."""
    class Dg2Error(RuntimeError):
        def __init__(self, code, msg):
            super().__init__(msg)
            self.code = code

    clock = {"ms": 0.0}
    open_solvers = []

    class Solver:
        stream = None

        def __init__(self, cs, kw):
            self.name = {0: "dg2_nl", 1: "dg2_ll"}.get(kw.get("variant"), kw.get("scheme"))
            self.name += "_4m" if cs.dx == 4.0 else ""
            self.t = 0.0
            open_solvers.append(self)

        def set_state(self, planes, t):
            if self.name.startswith("fv"):
                assert not planes[[1, 2, 4, 5, 7, 8]].any()
            self.t = t

        def step(self, dt):
            self.t += 0.1

        def time(self):
            return self.t, 0.1

        def steps(self):
            return int(10 * self.t)

        def launches(self):
            return 0

        def run_to(self, t):
            span = t - self.t
            if span > limits.get(self.name, 1e9):
                raise Dg2Error(-4, f"non-finite state or step near t={self.t}")
            clock["ms"] += COST[self.name] * (early * min(span, 70.0) + max(span - 70.0, 0.0))
            self.t = t

        def close(self):
            open_solvers.remove(self)

    class Event:
        def __init__(self, enable_timing):
            pass

        def record(self, stream):
            self.ms = clock["ms"]

        def elapsed_time(self, other):
            return other.ms - self.ms

    B = types.SimpleNamespace(Dg2Error=Dg2Error, DG2_E_NONFINITE=-4, DG2_NL=0, DG2_LL=1,
                              DG2_SCHEME_FV2="fv2", DG2_SCHEME_FV1="fv1",
                              solver_from_case=lambda cs, **kw: Solver(cs, kw))
    cuda = types.SimpleNamespace(Event=Event, synchronize=lambda: None, empty_cache=lambda: None)
    return B, types.SimpleNamespace(cuda=cuda), open_solvers


def compare(bench, limits, **kw):
    B, torch, left = fakes(limits, **kw)
    fine, coarse = (types.SimpleNamespace(nx=8, ny=4, dx=dx, cfl=0.33) for dx in (2.0, 4.0))
    start = (np.ones((9, 4, 8)), 3600.0)
    try:
        out = bench.scheme_cost_variant(B, torch, fine, start, coarse, start, window=120.0)
    finally:
        assert not left and (start[0] == 1.0).all()   # closed whatever happened; not written to
    return out


def test_all_windows_in_full(bench):
    out = compare(bench, {})
    assert out["failed"] == [] and {r["window_s"] for r in out["runs"].values()} == {120.0}
    assert set(out["runs"]) == set(COST) and "fv2" not in out["workload"]
    assert out["time_ratios"]["fv2/dg2_nl"] == pytest.approx(0.5)


def test_a_shortened_fv2_run_is_reported_and_divided_by_the_same_window(bench):
    out = compare(bench, {"fv2": 50.0}, early=3.0)
    runs, ratios = out["runs"], out["time_ratios"]
    assert [f["window_s"] for f in out["failed"]] == [120.0, 60.0]
    assert all(f["run"] == "fv2" and "non-finite" in f["error"] for f in out["failed"])
    assert runs["fv2"]["window_s"] == runs["dg2_nl_30s"]["window_s"] == 30.0
    assert runs["dg2_nl_4m_30s"]["window_s"] == 30.0 and runs["dg2_nl"]["window_s"] == 120.0
    assert "fv2 and its ratios: 30 s" in out["workload"]
    assert ratios["fv2/dg2_nl"] == pytest.approx(0.5)
    assert ratios["fv2_2m/dg2_nl_4m"] == pytest.approx(4.0)
    assert ratios["dg2_ll/dg2_nl"] == pytest.approx(1.5)
    assert ratios["fv1/dg2_nl"] == pytest.approx(0.25)


@pytest.mark.parametrize("name", ["dg2_nl", "dg2_ll", "fv1", "dg2_nl_4m"])
def test_another_scheme_that_goes_non_finite_fails_the_bench(bench, name):
    with pytest.raises(RuntimeError, match="non-finite"):
        compare(bench, {name: 100.0})


def test_fv2_failing_over_every_window_fails_the_bench(bench):
    with pytest.raises(RuntimeError, match="non-finite"):
        compare(bench, {"fv2": 1.0})
