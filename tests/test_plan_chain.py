"""Which of the two summations a request takes (few_plan_chain): the limits of the tensor cores, and the line
between them for sets of a few frequencies, on both sides of what was measured."""
import numpy as np
import pytest

from paper_2104_04582_gb300 import _build
from paper_2104_04582_gb300 import fewsum as F
from paper_2104_04582_gb300 import workloads as W

MIXED, FP64 = F.FEW_MIXED, F.FEW_FP64


@pytest.fixture(scope="module", autouse=True)
def lib():
    _build.build()
    return F.load()


def _chain(modes, K, n, prec, dt=10.0):
    T = max(n, K) * dt
    return F.few_plan_chain(W.knot_times(T, K), np.asarray(modes, dtype=np.int32), 0.0, dt, n, prec)


PAIR = [(2, 2, 0)]
M10 = [(10, 10, n) for n in (-1, 0, 1)]
ROW = [(2, 2, n) for n in range(-5, 6)]


@pytest.mark.parametrize("modes,K,n,prec,tc", [
    # measured us, tensor cores against scalar, at 100 knots and dt = 2 s or 10 s
    (PAIR, 100, 40000000, MIXED, False),     # 884, 740
    (PAIR, 100, 3155760, MIXED, True),       # 82, 90
    (PAIR, 4096, 1000000, MIXED, True),      # 136, 204
    (PAIR, 100, 20000, MIXED, True),         # 12, 32
    (ROW, 100, 40000000, MIXED, True),       # 884, 966
    (W.mode_grid(4, 5), 100, 40000000, MIXED, True),
    (PAIR, 100, 20000, FP64, True),          # 38, 61
    (PAIR, 100, 3155760, FP64, True),        # 557, 1048
    (PAIR, 1000, 1000, FP64, False),         # 110, 77
    (PAIR, 4096, 20000, FP64, False),        # 371, 229
    (M10, 4096, 100000, FP64, False),        # 747, 326
    (M10, 100, 100000, FP64, True),          # 113, 133
    (M10, 4, 1000000, FP64, True),           # 489, 604
    ([(10, 10, 0), (10, 10, 30)], 300, 20000, FP64, False),  # 135, 110
    (W.mode_grid(4, 5), 1000, 1000, FP64, True),     # 138, 211
    (W.mode_grid(4, 5), 4096, 20000, FP64, True),    # 534, 784
    (W.mode_grid(10, 30), 4096, 1000, FP64, True),
    # past the limits, whatever the size
    ([(11, 11, 0)], 100, 20000, MIXED, False),
    ([(2, 2, 0), (2, 2, 32)], 100, 20000, FP64, False),
    (W.mode_grid(10, 32), 100, 3155760, MIXED, False),
])
def test_line_between_the_chains(modes, K, n, prec, tc):
    on, scalar_bytes, tc_bytes = _chain(modes, K, n, prec)
    assert on == tc
    past = max(m for _, m, _ in np.asarray(modes).tolist()) > 10 or np.abs(np.asarray(modes)[:, 2]).max() > 31
    assert scalar_bytes > 0 and (tc_bytes == 0) == past


def test_sizes_grow_as_the_layouts_do():
    # FP64, full grid: 7 digit slices of 11 row pairs and 64 basis values against 64 bytes a slot
    on, s, t = _chain(W.mode_grid(10, 30), 101, 1000000, FP64)
    assert on and abs(s - 100 * 1281 * 64) < 65536 and abs(t - 100 * 512 * 7 * 11 * 4 - 1000000) < 65536
    # mixed, a sample: 3 bytes of anchors against one of tile records
    _, s1, t1 = _chain(W.mode_grid(4, 5), 101, 1000000, MIXED)
    _, s2, t2 = _chain(W.mode_grid(4, 5), 101, 2000000, MIXED)
    assert abs((s2 - s1) - 3000000) < 30000 and abs((t2 - t1) - 1000000) < 30000


@pytest.mark.parametrize("modes,K,n,dt,status", [
    ([(2, 3, 0)], 10, 100, 10.0, F.FEW_ERR_MODES), (PAIR, 3, 100, 10.0, F.FEW_ERR_KNOTS),
    (PAIR, 10, 100, -1.0, F.FEW_ERR_RANGE), (PAIR, 10, 2 ** 31, 10.0, F.FEW_ERR_RANGE)])
def test_refusals(modes, K, n, dt, status):
    with pytest.raises(F.FewError) as e:
        F.few_plan_chain(W.knot_times(1e12, K), np.asarray(modes, dtype=np.int32), 0.0, dt, n, MIXED)
    assert e.value.status == status
    with pytest.raises(F.FewError) as e:
        F.few_plan_chain(W.knot_times(1e3, 10), np.asarray(PAIR, dtype=np.int32), 0.0, 1.0, 10, 7)
    assert e.value.status == F.FEW_ERR_INVALID_ARG


@pytest.mark.parametrize("modes,K,n,tc", [
    # FP64, measured us of 48 waveforms in one graph (6 for 2000 knots), tensor cores against scalar
    ([(10, 10, 0), (10, 10, 1)], 50, 300, False),   # 402, 176
    ([(10, 10, 0), (10, 10, 30)], 50, 2000, False), # 952, 492
    ([(10, 10, 0), (10, 10, 30)], 300, 60000, True),  # 6945, 7976 (one: 171, 292)
    (PAIR, 300, 3000, False),                       # 1179, 685
    (PAIR, 300, 60000, True),                       # 1685, 1897
    (PAIR, 10, 2000, True),                         # 81, 103
    (PAIR, 10, 200, False),                         # 68, 49
    ([(2, 2, -30), (2, 2, 30), (2, 1, 3)], 50, 300, True),  # 382, 567
    ([(2, 2, -30), (2, 2, 30), (2, 1, 3)], 2000, 2000, True),  # 1415, 2107
])
def test_line_between_the_chains_in_batches(modes, K, n, tc):
    assert _chain(modes, K, n, FP64)[0] == tc
