"""The autotuner tunes what has a tile: workloads of the scalar chain (no GPU)."""
import numpy as np
import pytest

from paper_2104_04582_gb300 import _build
from paper_2104_04582_gb300 import fewsum as F
from paper_2104_04582_gb300 import tune
from paper_2104_04582_gb300 import workloads as W

FULL, FEW, PAST = W.mode_grid(10, 30), np.array([[2, 2, 0]], dtype=np.int32), W.mode_grid(11, 4)


@pytest.fixture(scope="module", autouse=True)
def lib():
    _build.build()
    return F.load()


def _request(modes, n, prec=F.FEW_MIXED):
    return (W.knot_times(10.0 * n, 50), modes, 0.0, 10.0, n, prec)


def test_only_the_scalar_chain_has_a_tile(tmp_path, monkeypatch):
    assert not tune.has_tile([_request(FULL, 100000), _request(FEW, 100000)])
    assert tune.has_tile([_request(FULL, 100000), _request(PAST, 100000)])
    monkeypatch.setattr(F, "few_get_tiles", lambda h, prec: (8, 256, 1024))
    monkeypatch.setattr(tune, "install", lambda *a: pytest.fail("installed a tile that makes no difference"))
    monkeypatch.setattr(tune, "tune", lambda *a, **k: pytest.fail("timed a workload without a tile"))
    path = str(tmp_path / "t.json")
    tune._save(path, {tune.bucket(F.FEW_MIXED, 1281, 100000): {"R": 2, "threads": 128, "stage_slots": 256}})
    assert tune.ensure(0, None, F.FEW_MIXED, 1281, 100000, path, requests=[_request(FULL, 100000)]) == ((8, 256, 1024), False)


def test_a_scalar_workload_is_still_tuned(tmp_path, monkeypatch):
    monkeypatch.setattr(tune, "tune", lambda *a, **k: ((2, 128, 256), {}))
    assert tune.ensure(0, None, F.FEW_MIXED, 99, 100000, str(tmp_path / "t.json"),
                       requests=[_request(PAST, 100000)]) == ((2, 128, 256), True)
