"""Edges of the tensor-core summations (tcsum.cu, tcsum64.cu): tile and segment remainders, row and
basis limits on both sides of their dispatch, batches and budgets that mix them with the scalar chain.

FP64 tolerance: the operands' digits and the products left out (2^-50 of the table's largest entry,
which is at most a few times a sample's size in these sets) and the phases (FP64 rounding of ~1e3 rad,
1e-13, times |m| + |n| <= 70) add up to at most 1e-11.

Mixed tolerance: the basis and table splits (2^-24 and 2^-23 of a term), the reduced phases (2^-28 turn,
a chain of at most four products), up to 12 accumulation steps (2^-23 each if truncated) and the
11-step chain in z_phi^2 add up to at most 4e-6 of the terms of a sample.
"""
import numpy as np
import pytest

import oracle
from paper_2104_04582_gb300 import fewsum as F
from paper_2104_04582_gb300 import runtime as RT
from paper_2104_04582_gb300 import workloads as W
from tests.gpu_common import MIXED_MISMATCH, oracle_threads, rel_l2, to_host

pytestmark = pytest.mark.gpu
REL = {F.FEW_MIXED: 4e-6, F.FEW_FP64: 1e-11}
PRECS = [F.FEW_MIXED, F.FEW_FP64]


def _modes(ms, ns, l=None):
    return np.asarray([(l or max(2, m), m, n) for m in ms for n in ns], dtype=np.int32)


SETS = {
    "one_m0_mode": _modes([0], [3]),
    "one_m2_mode": _modes([2], [-1]),
    "n_range_15": _modes([0, 2], range(-7, 8)),            # one K step full
    "n_range_17": _modes([0, 2], range(-8, 9)),            # one value into the second
    "n_range_63": _modes([0, 1], range(-31, 32)),          # the whole basis
    "n_range_64": _modes([0], range(-32, 32)),             # an even range: half-width 32, scalar
    "n_shifted": _modes([0], range(40, 90)),               # m = 0 only: a centre far from zero
    "m0_wider_one_way": np.concatenate([_modes([0], range(-23, 23)), _modes([2], range(-5, 7))]),
    "m0_one_sided": np.concatenate([_modes([0], range(-31, -9)), _modes([1, 4], range(-3, 4))]),
    "rows_21": _modes(range(11), [-2, 0, 5], l=10),
    "rows_22_empty": _modes([0, 10], [-30, 30], l=10),     # empty rows in between
    "rows_23": _modes(range(12), [0, 1], l=11),            # too many rows: scalar
}


# just past the limits: these stay on the scalar chain, whose contract is the mixed path's gate
PAST = ("n_range_64", "rows_23")


@pytest.mark.parametrize("name", PAST)
def test_mode_sets_past_the_limits(gpu_ctx, name):
    import torch
    w = W.make_inputs(4.0e5, 9, 100.0, SETS[name], 5, 4.0, 60.0)
    tr = RT.from_inputs(gpu_ctx, w)
    h = RT.waveform_inputs(gpu_ctx, tr, w, F.FEW_MIXED)
    torch.cuda.synchronize()
    assert gpu_ctx.sync_status() == F.FEW_OK
    o = oracle.waveform_inputs(w, nthreads=oracle_threads())
    assert oracle.mismatch(to_host(h), o) <= MIXED_MISMATCH
    tr.release()


@pytest.mark.parametrize("name", [s for s in SETS if s not in PAST])
@pytest.mark.parametrize("n_samples", [1, 128, 4001])
@pytest.mark.parametrize("prec", PRECS)
def test_mode_set_edges(gpu_ctx, prec, name, n_samples):
    import torch
    w = W.make_inputs(4.0e5, 9, 4.0e5 / max(n_samples, 200), SETS[name], 5, 4.0, 60.0,
                      n_samples=n_samples)
    tr = RT.from_inputs(gpu_ctx, w)
    h = RT.waveform_inputs(gpu_ctx, tr, w, prec)
    torch.cuda.synchronize()
    assert gpu_ctx.sync_status() == F.FEW_OK
    assert rel_l2(to_host(h), oracle.waveform_inputs(w, nthreads=oracle_threads())) <= REL[prec]
    tr.release()


@pytest.mark.parametrize("K,n_samples,i0,count", [
    (4, 127, 0, 127), (4, 129, 0, 129), (5, 1000, 1, 998), (300, 400, 0, 400),
    (300, 5000, 77, 4097), (40, 152 * 128 + 1, 0, 152 * 128 + 1)])
@pytest.mark.parametrize("prec", PRECS)
def test_sample_and_segment_edges(gpu_ctx, prec, K, n_samples, i0, count):
    """Segments shorter than a tile, empty segments, windows that start inside one, a run of tiles
    that leaves CTAs with one tile and with two."""
    import torch
    w = W.make_inputs(3.0e5, K, 3.0e5 / n_samples, W.mode_grid(4, 9), 11, 3.0, 20.0,
                      n_samples=n_samples)
    tr = RT.from_inputs(gpu_ctx, w)
    out = torch.full((count + 2,), complex(7.0, 7.0), device="cuda",
                     dtype=torch.complex64 if prec == F.FEW_MIXED else torch.complex128)
    h = RT.waveform_inputs(gpu_ctx, tr, w, prec, i_begin=i0, count=count, out=out[1:-1])
    torch.cuda.synchronize()
    assert gpu_ctx.sync_status() == F.FEW_OK
    g = to_host(out)
    assert g[0] == g[-1] == complex(7.0, 7.0)
    o = oracle.waveform_inputs(w, i0, count, nthreads=oracle_threads())
    assert rel_l2(g[1:-1], o) <= REL[prec]
    tr.release()


def test_long_request_equals_its_windows(gpu_ctx):
    """More tiles than one a thread of the blocks that fill their records: the same samples as short
    requests (whose records are formed one by one), to the bit where the first sample's time is the
    same number (t0 + i_begin dt is rounded)."""
    import torch
    n = 128 * (152 * 4 * 128 + 1000) + 5
    w = W.make_inputs(3.0e7, 300, 3.0e7 / n, SETS["n_range_15"], 5, 4.0, 60.0, n_samples=n)
    tr = RT.from_inputs(gpu_ctx, w)
    h = RT.waveform_inputs(gpu_ctx, tr, w, F.FEW_MIXED)
    torch.cuda.synchronize()
    for i0 in (0, n // 3, n // 2 + 77, n - 5000):
        g = to_host(RT.waveform_inputs(gpu_ctx, tr, w, F.FEW_MIXED, i_begin=i0, count=5000))
        if i0 == 0:
            np.testing.assert_array_equal(to_host(h[:5000]), g)
        assert rel_l2(to_host(h[i0:i0 + 5000]), g) <= 4e-6
        assert rel_l2(g, oracle.waveform_inputs(w, i0, 5000, nthreads=oracle_threads())) <= 4e-6
    tr.release()


@pytest.mark.parametrize("prec,scale", [(F.FEW_MIXED, 1e-30), (F.FEW_MIXED, 1e-22), (F.FEW_MIXED, 1e25),
                                        (F.FEW_FP64, 1e-290), (F.FEW_FP64, 1e-22), (F.FEW_FP64, 1e290)])
def test_amplitude_range(gpu_ctx, prec, scale):
    """The table's power-of-two scaling: amplitudes far from one keep their relative accuracy."""
    import torch
    w = W.make_inputs(3.0e5, 12, 100.0, W.mode_grid(4, 9), 3, 3.0, 20.0)
    tr = RT.from_inputs(gpu_ctx, w)
    h = RT.waveform(gpu_ctx, tr, w.n_samples, w.t0, w.dt, w.theta, w.phi, prec, False, scale)
    torch.cuda.synchronize()
    o = oracle.waveform_inputs(w, nthreads=oracle_threads(), scale=scale)
    assert rel_l2(to_host(h) / scale, o / scale) <= REL[prec]
    tr.release()


@pytest.mark.parametrize("prec", PRECS)
def test_batch_of_both_variants(gpu_ctx, prec):
    """A batch whose mode sets need both summation variants: each waveform as computed alone."""
    import torch
    sets = ["n_range_63", "rows_23", "n_range_15", "n_range_64"]
    ws = [W.make_inputs(2.0e5, 7, 50.0, SETS[s], k, 4.0, 60.0) for k, s in enumerate(sets)]
    trs = [RT.from_inputs(gpu_ctx, w) for w in ws]
    outs = [RT.alloc_out(w.n_samples, prec == F.FEW_MIXED) for w in ws]
    reqs = [RT.request(tr, o, w.n_samples, w.t0, w.dt, w.theta, w.phi, prec, w.scale)
            for tr, o, w in zip(trs, outs, ws)]
    for flags in (0, F.FEW_BATCH_NO_GRAPH):
        b = F.few_batch_plan(gpu_ctx.handle, reqs, flags)
        F.few_batch_run(gpu_ctx.handle, b, RT.current_stream())
        torch.cuda.synchronize()
        assert gpu_ctx.sync_status() == F.FEW_OK
        for w, tr, o in zip(ws, trs, outs):
            np.testing.assert_array_equal(to_host(o), to_host(RT.waveform_inputs(gpu_ctx, tr, w, prec)))
            o.zero_()
        F.few_batch_release(gpu_ctx.handle, b)
    for tr in trs:
        tr.release()


def test_budget_that_only_the_scalar_plan_fits():
    """Two modes on 4096 knots: the operand tables (rows x basis) are far larger than the scalar
    plan's two slots a segment; under a budget between the two the request still runs."""
    import torch
    w = W.make_inputs(3.0e6, 4096, 300.0, _modes([2], [-31, 31]), 3)
    with RT.Context(0) as free:
        tr = RT.from_inputs(free, w)
        ref = to_host(RT.waveform_inputs(free, tr, w, F.FEW_MIXED))
        held = free.memory()[0]
        tr.release()
    for extra, runs in ((16 << 20, True), (200 << 20, True), (1 << 10, False)):
        with RT.Context(0, held + extra) as ctx:
            tr = RT.from_inputs(ctx, w)
            if not runs:
                with pytest.raises(F.FewError) as e:
                    RT.waveform_inputs(ctx, tr, w, F.FEW_MIXED)
                assert e.value.status == F.FEW_ERR_BUDGET
            else:
                h = RT.waveform_inputs(ctx, tr, w, F.FEW_MIXED)
                torch.cuda.synchronize()
                assert ctx.sync_status() == F.FEW_OK
                # under the small budget the scalar chain ran: the mixed path's gate
                assert oracle.mismatch(to_host(h), ref) <= MIXED_MISMATCH
            tr.release()


@pytest.mark.parametrize("how", ["pageable", "rebuild"])
def test_budget_with_buffers_beside_the_plan(how):
    """The same two modes with a buffer next to the plan: staging of a pageable output, or the build jobs
    of a batch.  A budget that holds the tensor-core plan alone, but not that buffer beside it, still
    runs the request (by the scalar plan)."""
    import torch
    w = W.make_inputs(3.0e6, 4096, 300.0, _modes([2], [-31, 31]), 3)
    out = np.empty(w.n_samples, dtype=np.complex64)

    def run(ctx, tr):
        if how == "pageable":
            out[:] = 0
            F.few_waveform(ctx.handle, RT.request(tr, out, w.n_samples, w.t0, w.dt, w.theta, w.phi, F.FEW_MIXED,
                                                  out_where=F.FEW_MEM_HOST), RT.current_stream())
            return out.astype(np.complex128)
        dev = RT.alloc_out(w.n_samples, True)
        req = RT.request(tr, dev, w.n_samples, w.t0, w.dt, w.theta, w.phi, F.FEW_MIXED)
        b = F.few_batch_plan(ctx.handle, [req], F.FEW_BATCH_REBUILD_SPLINES)
        F.few_batch_run(ctx.handle, b, RT.current_stream())
        torch.cuda.synchronize()
        F.few_batch_release(ctx.handle, b)
        return to_host(dev)

    with RT.Context(0) as free:
        tr = RT.from_inputs(free, w)
        held = free.memory()[0]
        ref = to_host(RT.waveform_inputs(free, tr, w, F.FEW_MIXED))
        b = F.few_batch_plan(free.handle, [RT.request(tr, RT.alloc_out(w.n_samples, True), w.n_samples, w.t0, w.dt,
                                                      w.theta, w.phi, F.FEW_MIXED)], 0)
        plan = free.memory()[0] - held  # the tensor-core plan
        F.few_batch_release(free.handle, b)
        tr.release()
    with RT.Context(0, held + plan) as ctx:
        tr = RT.from_inputs(ctx, w)
        assert oracle.mismatch(run(ctx, tr), ref) <= MIXED_MISMATCH
        assert ctx.sync_status() == F.FEW_OK
        tr.release()


@pytest.mark.parametrize("prec", PRECS)
def test_budget_moves_only_the_waves_that_do_not_fit(prec):
    """A batch of one full and three sparse mode sets (two modes on 1500 knots): under a budget that does
    not hold the sparse sets' tables beside the full one's, the full set keeps its plan, to the bit."""
    import torch
    ws = [W.make_inputs(2.0e5, 1500, 200.0, _modes([2], [-31, 31]), 3 + k) for k in range(3)]
    ws.insert(1, W.make_inputs(2.0e5, 20, 50.0, W.mode_grid(10, 30), 9, 4.0, 60.0))

    def setup(ctx):
        trs = [RT.from_inputs(ctx, w) for w in ws]
        outs = [RT.alloc_out(w.n_samples, prec == F.FEW_MIXED) for w in ws]
        return trs, outs, [RT.request(tr, o, w.n_samples, w.t0, w.dt, w.theta, w.phi, prec)
                           for tr, o, w in zip(trs, outs, ws)]

    def plan_bytes(ctx, reqs):
        held = ctx.memory()[0]
        b = F.few_batch_plan(ctx.handle, reqs, 0)
        held = ctx.memory()[0] - held
        F.few_batch_release(ctx.handle, b)
        return held

    with RT.Context(0) as free:
        trs, outs, reqs = setup(free)
        held, both, full = free.memory()[0], plan_bytes(free, reqs), plan_bytes(free, reqs[1:2])
        refs = [to_host(RT.waveform(free, tr, w.n_samples, w.t0, w.dt, w.theta, w.phi, prec)) for tr, w in zip(trs, ws)]
        for tr in trs:
            tr.release()
    budget = held + full + (both - full) // 2  # the sparse sets by the scalar chain: a third at most
    with RT.Context(0, budget) as ctx:
        trs, outs, reqs = setup(ctx)
        b = F.few_batch_plan(ctx.handle, reqs, 0)
        F.few_batch_run(ctx.handle, b, RT.current_stream())
        torch.cuda.synchronize()
        assert ctx.sync_status() == F.FEW_OK
        for k, (o, ref) in enumerate(zip(outs, refs)):
            if k == 1:
                np.testing.assert_array_equal(to_host(o), ref)
            elif prec == F.FEW_FP64:
                assert rel_l2(to_host(o), ref) <= REL[prec]
            else:
                assert oracle.mismatch(to_host(o), ref) <= MIXED_MISMATCH
        F.few_batch_release(ctx.handle, b)
        for tr in trs:
            tr.release()


def test_fp64_records_of_many_short_segments(gpu_ctx):
    """About one sample a segment (many of them empty): blocks that fill tile records meet more segments than
    they cache at once.  The call stays near its latency (140 us; 400 us while a block took 128 tiles
    whatever their segments)."""
    import torch
    w = W.make_inputs(1.0e4, 1000, 10.0, W.mode_grid(4, 5), 7, 2.0, 8.0)
    tr = RT.from_inputs(gpu_ctx, w)
    out = RT.alloc_out(w.n_samples, False)
    best = float("inf")
    for _ in range(20):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        RT.waveform_inputs(gpu_ctx, tr, w, F.FEW_FP64, out=out)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3)
    assert gpu_ctx.sync_status() == F.FEW_OK
    assert rel_l2(to_host(out), oracle.waveform_inputs(w, nthreads=oracle_threads())) <= REL[F.FEW_FP64]
    assert best <= 270.0
    tr.release()


@pytest.mark.parametrize("modes,K,n,prec", [
    (_modes([2], [0]), 1000, 1000, F.FEW_FP64), (_modes([2], [0]), 100, 20000, F.FEW_FP64),
    (_modes([2], [0]), 20, 24000000, F.FEW_MIXED), (_modes([2], [0]), 20, 300000, F.FEW_MIXED),
    (W.mode_grid(4, 5), 60, 50000, F.FEW_MIXED), (_modes([11], [0, 1], l=11), 40, 20000, F.FEW_FP64)])
def test_requests_take_the_chain_that_few_plan_chain_names(gpu_ctx, modes, K, n, prec):
    """The memory that a planned batch holds is that of the chain it names, and so are the two entry points'
    results."""
    import torch
    w = W.make_inputs(max(n, K) * 10.0, K, 10.0, modes, 5, 2.0, 8.0, n_samples=n)
    on, scalar_bytes, tc_bytes = F.few_plan_chain(w.t_knots, w.modes, w.t0, w.dt, n, prec)
    tr = RT.from_inputs(gpu_ctx, w)
    out = RT.alloc_out(n, prec == F.FEW_MIXED)
    req = RT.request(tr, out, n, w.t0, w.dt, w.theta, w.phi, prec)
    held = gpu_ctx.memory()[0]
    b = F.few_batch_plan(gpu_ctx.handle, [req], 0)
    held = gpu_ctx.memory()[0] - held
    F.few_batch_release(gpu_ctx.handle, b)
    assert abs(held - (tc_bytes if on else scalar_bytes)) <= 16384 + 1024
    F.few_waveform(gpu_ctx.handle, req, RT.current_stream())
    if min(scalar_bytes, tc_bytes or scalar_bytes) < (8 << 20):  # of the 16 MiB that the other entry point has
        other = torch.empty_like(out)
        F.few_waveform_noalloc(gpu_ctx.handle, RT.request(tr, other, n, w.t0, w.dt, w.theta, w.phi, prec),
                               RT.current_stream())
        np.testing.assert_array_equal(to_host(other), to_host(out))
    torch.cuda.synchronize()
    assert gpu_ctx.sync_status() == F.FEW_OK
    i0, count = n // 3, min(n, 4000)
    g, o = to_host(out[i0:i0 + count]), oracle.waveform_inputs(w, i0, min(count, n - i0), nthreads=oracle_threads())
    assert rel_l2(g, o) <= REL[prec] if prec == F.FEW_FP64 else oracle.mismatch(g, o) <= MIXED_MISMATCH
    tr.release()


@pytest.mark.parametrize("span", [1e-4, 2e-2, 1.0])
def test_fp64_phase_of_one_frequency(gpu_ctx, span):
    """One frequency (n = 31, m = 0) over a small phase `span` (rad, quadratic in time: the splines reproduce
    it): the sample's phase against extended precision.  The expansion's coefficients c0 and c1 are rounded
    to 2^-65 turn, the latter times 127 samples and n: 31 x 127 x 2^-65 x 2 pi = 7e-16; sine and cosine,
    digits and sums 2^-50; the phases themselves and the oracle of this test 31 x 2^-53 x span: 4e-15 +
    4e-15 span in all.  (c2 rounded likewise: 31 x 127^2 x 2^-65 x 2 pi = 8.5e-14.)"""
    import torch
    K, n, dt = 60, 20000, 10.0
    w = W.make_inputs(n * dt, K, dt, _modes([0], [31]), 3, n_samples=n)
    LD = np.longdouble

    def phase(t):
        x = np.asarray(t, dtype=LD) / LD(n * dt)
        return LD(span) * (LD(0.3) + LD(0.5) * x + LD(0.2) * x * x)

    w.phi_r = phase(w.t_knots).astype(np.float64)
    w.phi_phi = np.zeros(K)
    w.amp_re, w.amp_im = np.ones((K, 1)), np.zeros((K, 1))
    assert F.few_plan_chain(w.t_knots, w.modes, w.t0, dt, n, F.FEW_FP64)[0]
    tr = RT.from_inputs(gpu_ctx, w)
    h = to_host(RT.waveform_inputs(gpu_ctx, tr, w, F.FEW_FP64))
    torch.cuda.synchronize()
    assert gpu_ctx.sync_status() == F.FEW_OK
    tr.release()
    a = -31 * (phase(np.arange(n) * dt) - phase(0.0))
    c, s = np.cos(a), np.sin(a)
    re, im = LD(h[0].real), LD(h[0].imag)
    err = np.hypot(h.real - (re * c - im * s), h.imag - (re * s + im * c)) / np.hypot(re, im)
    assert float(err.max()) <= 4e-15 + 4e-15 * span
