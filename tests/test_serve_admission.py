"""What the serving engine counts for a request: the plan of the summation that it takes (no GPU)."""
import types

import numpy as np
import pytest

from paper_2104_04582_gb300 import _build
from paper_2104_04582_gb300 import fewsum as F
from paper_2104_04582_gb300 import workloads as W
from paper_2104_04582_gb300.serve import AdmissionError, GpuEngine, Request, Server

FULL, PAST = W.mode_grid(10, 30), W.mode_grid(11, 4)


@pytest.fixture(scope="module", autouse=True)
def lib():
    _build.build()
    return F.load()


def _engine(modes, K, T):
    """The engine's host side with one resident trajectory."""
    e = GpuEngine.__new__(GpuEngine)
    slots = F.few_mode_slots(modes)[0]
    e.trajs = {"t": types.SimpleNamespace(t_knots=W.knot_times(T, K), modes=modes, info=(K, len(modes), slots))}
    e._announced = {}
    return e


def test_admission_counts_the_plan_that_runs():
    n = 100000
    for prec, seg in ((F.FEW_MIXED, 1024 * 11 * 4), (F.FEW_FP64, 3584 * 11 * 4)):
        need = _engine(FULL, 101, 10.0 * n).scratch_bytes(Request("t", n, 10.0, prec=prec))
        assert abs(need - (100 * seg + n)) <= 200 * 1024  # tables, a byte a sample of tile records
    # two modes 60 apart: tables of 64 basis values against 122 slots
    far = np.array([[10, 10, -30], [10, 10, 30]], dtype=np.int32)
    need = _engine(far, 101, 1e8).scratch_bytes(Request("t", 1000000, 10.0, prec=F.FEW_FP64))
    assert need >= 100 * 3584 * 11 * 4
    # past the limits: the scalar chain's slots and anchors
    slots = F.few_mode_slots(PAST)[0]
    need = _engine(PAST, 101, 10.0 * n).scratch_bytes(Request("t", n, 10.0, prec=F.FEW_MIXED))
    assert abs(need - (100 * slots * 32 + 3 * n)) <= 200 * 1024


def test_unknown_trajectory_and_knot_data():
    e = _engine(FULL, 20, 1e6)
    with pytest.raises(KeyError):
        e.scratch_bytes(Request("new", 100, 10.0))
    w = W.make_inputs(1e6, 20, 10.0, FULL, 1)
    assert e.scratch_bytes(Request("new", 1000, 10.0, traj_inputs=w)) > 0


def test_a_request_whose_smaller_plan_fits_is_still_admitted():
    """FP64 on the full grid: tables of 157 KB a segment, slots of 82 KB."""
    class Engine:
        sizes = _engine(FULL, 1001, 1e6)
        scratch_bytes = staticmethod(sizes.scratch_bytes)
        least_scratch_bytes = staticmethod(sizes.least_scratch_bytes)

        def alloc_out(self, req):
            return None

        def launch(self, reqs, outs):
            return None

        def wait(self, handle):
            pass

        def release(self, handle):
            pass

    req = Request("t", 1000, 10.0, prec=F.FEW_FP64)
    big, least = (f(req) + req.out_bytes() for f in (Engine.scratch_bytes, Engine.least_scratch_bytes))
    assert least < 0.6 * big
    for budget, runs in ((big, True), (least, True), (least - 1, False)):
        srv = Server(Engine(), hbm_budget_bytes=budget)
        f = srv.submit(req)
        if runs:
            f.result(timeout=5)
            assert srv.stats()["max_bytes_in_use"] <= budget
        else:
            with pytest.raises(AdmissionError):
                f.result(timeout=5)
        srv.close()
