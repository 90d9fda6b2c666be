"""The autotuner's JSON cache (hgm.autotune): what it keeps, and for which library. Host logic only, with a stand-in
for the library."""
import json

import numpy as np
import pytest

from paper_1505_00581_gb300 import hgm


class _Lib:
    def __init__(self, times):
        self.times, self.tuned, self.set = times, 0, []

    def hgm_autotune(self, mh, nm, sh, ns, params, stream, sample, best, ms):
        self.tuned += 1
        np.ctypeslib.as_array(ms, (hgm.N_VARIANTS,))[:] = self.times
        best._obj.value = int(np.argmin(self.times))
        return 0

    def hgm_set_recurse_variant(self, v):
        self.set.append(v)
        return 0


@pytest.fixture
def tune(tmp_path, monkeypatch):
    monkeypatch.setenv("HGM_TUNE_CACHE", str(tmp_path / "tune.json"))
    monkeypatch.setattr(hgm, "LIB_PATH", str(tmp_path / "lib.so"))
    monkeypatch.setattr(hgm, "_stream", lambda s: None)
    (tmp_path / "lib.so").write_bytes(b"first build")

    def call(lib, K=64):
        monkeypatch.setattr(hgm, "load", lambda: lib)
        p = hgm.Params()
        p.K = K
        return hgm.autotune([], [], p)

    return call, tmp_path


def test_a_choice_is_cached_for_the_library_that_made_it(tune):
    call, tmp = tune
    lib = _Lib([3.0, 1.0, 2.0])
    assert call(lib) == (1, {0: 3.0, 1: 1.0, 2: 2.0}) and lib.tuned == 1
    assert call(lib) == (1, None) and lib.tuned == 1 and lib.set == [1]
    (tmp / "lib.so").write_bytes(b"kernels changed")
    assert call(lib)[0] == 1 and lib.tuned == 2      # timed again


def test_no_choice_is_not_cached(tune):
    call, tmp = tune
    lib = _Lib([2.0, 2.0, 2.0])       # one measurement: no launch of this call takes a variant
    call(lib, K=16)
    call(lib, K=16)
    assert lib.tuned == 2 and lib.set == []
    assert not (tmp / "tune.json").exists() or json.load(open(tmp / "tune.json")) == {}
