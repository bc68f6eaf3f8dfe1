"""One Batch fixed several times while the file of tuned FFT plans changes or cannot be written: the plan of the
first fix stays, and with it the captured graph and the weight table that it reads."""
import json

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

DIMS = [(16, 16, 16, 16), (8, 8, 8, 8), (16, 16, 16, 16)]  # the fixed-length and the general passes both take them


def fix(b, precision):
    Us = [synth.config(d, 121 + k, 0.4) for k, d in enumerate(DIMS)]
    res = b.fix(Us, 0.08, 1e-15, precision)
    assert all(r["theta"] < 1e-15 for r in res)
    return Us, b.describe()


def same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("first", ["generic", "fixed"])
def test_cache_rewritten_between_fixes(first, precision, tmp_path, monkeypatch):
    import paper_1210_8018_gb300 as lgf
    path = tmp_path / "tune.json"
    monkeypatch.setenv("LGF_TUNE_CACHE", str(path))
    with lgf.Batch(DIMS) as b:  # fills the file, so that its keys are known
        fix(b, precision)
    keys = list(json.loads(path.read_text()))

    def write(plan):
        path.write_text(json.dumps({k: {"plan": plan, "C": 0 if plan == "generic" else 16, "ms": 1.0} for k in keys}))

    write(first)
    with lgf.Batch(DIMS) as b:
        runs = [fix(b, precision)]
        write("fixed" if first == "generic" else "generic")
        runs.append(fix(b, precision))
        path.unlink()
        runs.append(fix(b, precision))
    plans = runs[0][1]["fft_f64"] + runs[0][1]["fft_f32"]
    assert plans.count("=" + first + "/") == plans.count("=") > 0
    for Us, info in runs[1:]:
        assert same(Us, runs[0][0])
        assert (info["fft_f64"], info["fft_f32"]) == (runs[0][1]["fft_f64"], runs[0][1]["fft_f32"])


def test_cache_not_writable(tmp_path, monkeypatch):
    import paper_1210_8018_gb300 as lgf
    (tmp_path / "file").write_text("")
    monkeypatch.setenv("LGF_TUNE_CACHE", str(tmp_path / "file" / "tune.json"))
    with lgf.Batch(DIMS) as b:
        runs = [fix(b, p) for p in ("mixed", "mixed", "fp64", "mixed")]
    assert same(runs[0][0], runs[1][0]) and same(runs[0][0], runs[3][0])
    assert runs[0][1]["fft_f32"] == runs[1][1]["fft_f32"] == runs[3][1]["fft_f32"]


def test_entries_of_other_keys(tmp_path, monkeypatch):
    """Times taken in other arithmetic, for another number of configurations or by an earlier version do not count,
    nor do widths that no kernel has; forms of the same passes share an entry."""
    import paper_1210_8018_gb300 as lgf
    path = tmp_path / "tune.json"
    monkeypatch.setenv("LGF_TUNE_CACHE", str(path))

    def keys(dims):
        before = set(json.loads(path.read_text())) if path.exists() else set()
        Us = [synth.config(d, 124 + k, 0.4) for k, d in enumerate(dims)]
        with lgf.Batch(dims) as b:
            b.fix(Us, 0.08, 1e-15, "fp64")
            info = b.describe()
        return set(json.loads(path.read_text())) - before, info

    two = [(16, 16, 16, 16)] * 2
    path.write_text(json.dumps({"16x16x16x16:f64": {"plan": "generic", "C": 0, "ms": 1e-6}}))
    first, _ = keys(two)
    assert len(first) == 1
    assert len(keys(two)[0]) == 0
    assert len(keys(two + two[:1])[0]) == 1
    with monkeypatch.context() as m:
        m.setenv("LGF_FFT_ZT", "0")
        assert len(keys(two)[0]) == 0
    with monkeypatch.context() as m:
        m.setenv("LGF_FFT_NATIVE_F64", "1")
        assert len(keys(two)[0]) == 1
    path.write_text(json.dumps({k: {"plan": "fixed", "C": 8, "ms": 1e-6} for k in first}))
    assert "/8 " not in keys(two)[1]["fft_f64"]


def test_pass_over_z_and_t_in_a_batch(monkeypatch):
    """Without the tuner the plan is the fixed-length one, and its pass over z and t gives the bits of the three."""
    import paper_1210_8018_gb300 as lgf
    monkeypatch.setenv("LGF_AUTOTUNE", "0")
    runs = []
    for flag in ("1", "0"):
        monkeypatch.setenv("LGF_FFT_ZT", flag)
        with lgf.Batch(DIMS) as b:
            runs.append(fix(b, "mixed"))
    assert same(runs[0][0], runs[1][0])
    assert runs[0][1]["launches_per_replay"] < runs[1][1]["launches_per_replay"]
