"""The autotuner sweeps shapes only where the shower has a launch shape, and for
the trial scheme that it is asked for."""
import pytest


@pytest.fixture(scope="module")
def A():
    from paper_2511_19633_gb300 import build
    build.build()
    from paper_2511_19633_gb300 import autotune
    return autotune


def _run(A, monkeypatch, **kw):
    calls = []

    def timed(process, sqrt_s, pdf, shape, n_events, precision, **k):
        cfg = A.G.make_config(process, sqrt_s, precision=precision, schedule=k["schedule"],
                              trial_mode=k.get("trial_mode"), **shape)
        calls.append(cfg.trial_mode)
        return {**shape, "ms": 100.0 - len(calls), "events_per_s": 1.0, "lane_efficiency": 1.0}

    monkeypatch.setattr(A, "time_shape", timed)
    return A.autotune(0, 91.2, None, n_events=1, **kw), calls


@pytest.mark.parametrize("schedule", ["PERSISTENT", "WAVE"])
def test_one_launch_shape_is_timed_once(A, monkeypatch, schedule):
    out, calls = _run(A, monkeypatch, schedule=getattr(A.G, "GAPS_SCHED_" + schedule))
    assert calls == [A.G.GAPS_TRIALS_KEEP] and len(out["table"]) == 1
    assert set(out["best"]) <= set(out["table"][0])


def test_fp64_is_timed_once(A, monkeypatch):
    assert len(_run(A, monkeypatch, precision=A.G.GAPS_FP64)[1]) == 1


@pytest.mark.parametrize("schedule,name", [("PERSISTENT", "REDRAW"), ("PERSISTENT", "SELECT"),
                                           ("PERSISTENT", "VETOMAX"), ("WAVE", "SELECT")])
def test_other_schemes_are_swept(A, monkeypatch, schedule, name):
    mode = getattr(A.G, "GAPS_TRIALS_" + name)
    out, calls = _run(A, monkeypatch, schedule=getattr(A.G, "GAPS_SCHED_" + schedule), trial_mode=mode)
    assert len(calls) > 10 and set(calls) == {mode}
    assert out["best"] == {k: out["table"][-1][k] for k in out["best"]}
