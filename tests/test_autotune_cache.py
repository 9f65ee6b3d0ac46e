"""CPU test of the autotuner's saved picks: a pick is applied to the build of
the library it was measured with and to no other.  The library's tuner is
replaced by a counter, so nothing is launched."""
import json
import types

import pytest

torch = pytest.importorskip("torch")


class _Tuner:
    """Stands in for the loaded library: counts the calls of the tuner."""

    def __init__(self):
        self.calls = 0

    def rbsm_batch_autotune(self, desc, workspace, nbytes, stream, repeats, tuning):
        self.calls += 1
        t = tuning._obj
        t.tile_threads, t.ctas_per_sm, t.chunk_tiles, t.ms, t.candidates = 128, 0, 2, 1.0, 28
        return 0


@pytest.fixture
def tuned(monkeypatch):
    """(tune(build), tuner): autotunes one batch with the library of `build`."""
    from paper_1711_07793_gb300 import _native as N
    from paper_1711_07793_gb300 import api
    tuner = _Tuner()
    monkeypatch.setattr(N, "lib", lambda: tuner)
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda dev: "a GPU")
    plane = torch.zeros(1000)
    job = types.SimpleNamespace(map_index=0, mode=3, x=plane, codes=None)
    stream = types.SimpleNamespace(cuda_stream=0)

    def tune(build, cache):
        monkeypatch.setattr(N, "_fingerprint", build, raising=False)
        batch = types.SimpleNamespace(maps=[torch.zeros(64, 64)], jobs=[job], desc=N.rbsm_batch(),
                                      workspace=plane, workspace_bytes=4096, shape=None)
        batch.set_launch = lambda *a: setattr(batch, "shape", a)
        return api.rbsm_batch_autotune(batch, stream=stream, cache=cache), batch

    return tune, tuner


def test_a_pick_is_kept_for_its_own_build_only(tuned, tmp_path):
    tune, tuner = tuned
    cache = str(tmp_path / "tune.json")
    first, _ = tune("build a", cache)
    again, batch = tune("build a", cache)
    assert not first["cached"] and again["cached"] and tuner.calls == 1
    assert batch.shape == (128, 0, 2, 0)
    other, _ = tune("build b", cache)                  # the kernels were rebuilt: measured again
    assert not other["cached"] and tuner.calls == 2
    assert tune("build a", cache)[0]["cached"] and tune("build b", cache)[0]["cached"] and tuner.calls == 2


def test_picks_saved_without_a_build_are_not_applied(tuned, tmp_path):
    """Files of picks whose keys do not say which build they were measured with."""
    tune, tuner = tuned
    cache = tmp_path / "tune.json"
    old = json.dumps(["v2", "a GPU", [[64, 64]], [[0, 3, 1000, False]]])
    cache.write_text(json.dumps({old: {"tile_threads": 512, "ctas_per_sm": 1, "chunk_tiles": 4, "flags": 0}}))
    res, batch = tune("build a", str(cache))
    assert not res["cached"] and tuner.calls == 1 and batch.shape == (128, 0, 2, 0)


def test_the_fingerprint_is_the_loaded_file_s():
    import hashlib

    from paper_1711_07793_gb300 import _native as N
    from paper_1711_07793_gb300 import build as B
    B.build()
    N.lib()
    with open(N.LIB_PATH, "rb") as f:
        assert N.library_fingerprint() == hashlib.sha256(f.read()).hexdigest()[:16]
