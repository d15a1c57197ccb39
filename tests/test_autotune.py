"""What the launch-shape tuner tries, keeps and remembers (its timings made up, so
without a GPU)."""
import json
import types

import pytest

from paper_2609_24294_gb300 import autotune, zfpx as z


@pytest.fixture
def tuner(monkeypatch, tmp_path):
    """tune_codec over given times: {(direction, units per warp): ms}."""
    state = {"set": {}, "calls": 0, "library": "a" * 16}
    plan = types.SimpleNamespace(n=(8, 8, 8), src_strides=(1, 8, 64), dst_strides=(1, 8, 64), pr=1, pc=1,
                                 transposition=0, dims=3)
    monkeypatch.setattr(autotune, "CACHE", str(tmp_path / "tune.json"))
    monkeypatch.setattr(autotune.torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(autotune.torch.cuda, "get_device_properties",
                        lambda i: types.SimpleNamespace(name="gpu", multi_processor_count=152))
    stamp = tmp_path / "stamp"
    monkeypatch.setattr(autotune._build, "STAMP", str(stamp))
    monkeypatch.setattr(z, "zfpx_set_units_per_warp",
                        lambda encode, rate, u: state["set"].__setitem__("encode" if encode else "decode", u))
    monkeypatch.setattr(z, "zfpx_pack_compress", lambda *a, **k: "encode")
    monkeypatch.setattr(z, "zfpx_decompress_unpack", lambda *a, **k: "decode")

    def run(ms, **kw):
        def time_call(fn, reps):
            state["calls"] += 1
            d = fn()
            return ms(d, state["set"][d])

        monkeypatch.setattr(autotune, "time_call", time_call)
        stamp.write_text(state["library"])
        return autotune.tune_codec(plan, 8, None, None, None, **kw)[0]

    run.state = state
    return run


def test_the_librarys_choice_is_kept_within_the_margin(tuner):
    assert tuner(lambda d, u: 10.0 if u else 9.0, use_cache=False) == {"encode": 0, "decode": 0}
    assert tuner.state["set"] == {"encode": 0, "decode": 0}
    assert tuner(lambda d, u: 10.1 if u == 0 else 10.0 + u, use_cache=False) == {"encode": 0, "decode": 0}
    # 1 beats it by a tenth in one direction
    times = lambda d, u: 10.0 if u == 0 else (9.0 if d == "decode" and u == 1 else 11.0)
    assert tuner(times, use_cache=False) == {"encode": 0, "decode": 1}
    assert tuner.state["set"] == {"encode": 0, "decode": 1}


def test_given_candidates_are_the_only_ones(tuner):
    assert tuner(lambda d, u: float(u), candidates=(5, 3), use_cache=False) == {"encode": 3, "decode": 3}


def test_choices_of_another_library_are_not_taken(tuner):
    ms = lambda d, u: 10.0 if u != 4 else 5.0
    assert tuner(ms) == {"encode": 4, "decode": 4}
    n = tuner.state["calls"]
    assert n == 2 * len(autotune.UPW_CANDIDATES)
    assert tuner(lambda d, u: 1.0) == {"encode": 4, "decode": 4} and tuner.state["calls"] == n
    tuner.state["library"] = "b" * 16
    assert tuner(lambda d, u: 1.0) == {"encode": 0, "decode": 0} and tuner.state["calls"] == 2 * n
    with open(autotune.CACHE) as f:
        assert len(json.load(f)) == 2
