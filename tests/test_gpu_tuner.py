"""The tuner at a size that CPRA_ENGINE_WARP does not name: the warp kernels are
timed there as AUTO, and its answer is an engine that cpra_plan takes."""
import json

import numpy as np
import pytest

from test_gpu_parity import cp  # noqa: F401

pytestmark = pytest.mark.gpu


def test_unlisted_size(cp, tmp_path, monkeypatch):  # noqa: F811
    path = str(tmp_path / "t.json")
    eng, ms = cp.cpra_autotune(160, cp.FP32, path)
    line = [l for l in open(path) if '"N=160,' in l]
    assert len(line) == 1 and "ms_engine_0" in line[0] and "ms_engine_1" in line[0] and "ms_engine_3" not in line[0]
    e = json.loads(line[0].rstrip().rstrip(","))
    assert eng in (cp.ENGINE_AUTO, cp.ENGINE_TWO_PASS) and ms == pytest.approx(min(e["ms_engine_0"], e["ms_engine_1"]))
    assert eng == cp.ENGINE_AUTO  # 0.19 us an angle against 0.40: not a close call
    assert cp.cpra_autotune(160, cp.FP32, path)[0] == eng  # from the cache
    # TUNED and the answer itself run what AUTO runs
    monkeypatch.setenv("CPRA_TUNE_CACHE", path)
    rng = np.random.default_rng(1)
    I = rng.random((4, 160, 160)).astype(np.float32)
    out = []
    for engine in (cp.ENGINE_AUTO, cp.ENGINE_TUNED, eng):
        p = cp.Plan(cp.make_config(160, 4, engine=engine))
        p.load_intensities(I, 0, np.arange(4) * np.pi / 4)
        p.iterate(2)
        out.append(p.result(cp.RESULT_STATE))
        p.close()
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])


def test_an_entry_from_before_is_timed_anew(cp, tmp_path):  # noqa: F811
    """A cache written when TWO_PASS was the only engine there: replaced, and
    the other entries stay."""
    path = str(tmp_path / "t.json")
    cp.cpra_autotune(160, cp.FP32, path)
    key = json.loads([l for l in open(path) if '"N=160,' in l][0].rstrip().rstrip(","))["key"]
    other = '{"key": "N=96,prec=0,sms=1,dev=other", "engine": 1, "ms": 0.5, "ms_engine_1": 0.5}'
    with open(path, "w") as f:
        f.write('{"cpra_tune_cache": 1, "entries": [\n%s,\n{"key": "%s", "engine": 1, "ms": 9.0, "ms_engine_1": 9.0}\n]}\n' % (other, key))
    eng, ms = cp.cpra_autotune(160, cp.FP32, path)
    assert eng == cp.ENGINE_AUTO and ms < 9.0
    entries = json.load(open(path))["entries"]
    assert [e["key"] for e in entries].count(key) == 1 and json.loads(other) in entries
