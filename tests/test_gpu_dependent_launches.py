"""Calls that follow one another on a stream without a wait, their kernels overlapping and their scratch
at the same addresses: every result equals, to the bit, that of the call by itself."""
import numpy as np
import pytest

from paper_2104_04582_gb300 import fewsum as F
from paper_2104_04582_gb300 import runtime as RT
from paper_2104_04582_gb300 import workloads as W
from tests.gpu_common import to_host

pytestmark = pytest.mark.gpu
REPEATS = 24


def _same(alone, chained):
    np.testing.assert_array_equal(to_host(chained), to_host(alone))


@pytest.mark.parametrize("prec", [F.FEW_MIXED, F.FEW_FP64])
@pytest.mark.parametrize("K,n_samples", [(20, 3000), (60, 90001), (200, 20000)])
def test_resident_waveforms_back_to_back(gpu_ctx, prec, K, n_samples):
    """Angles, offsets and trajectories of equal shape alternate (K = 200: a plan too long for the kernel
    parameters)."""
    import torch
    ws = [W.make_inputs(4.0e5, K, 4.0e5 / n_samples, W.mode_grid(6, 12), 40 + k, 3.0, 20.0, n_samples=n_samples)
          for k in range(2)]
    trs = [RT.from_inputs(gpu_ctx, w) for w in ws]

    def call(k, out=None):
        w = ws[k & 1]
        return RT.waveform(gpu_ctx, trs[k & 1], n_samples, w.t0, w.dt, 0.3 + 0.1 * k, 0.2 * k, prec,
                           dphi_phi0=0.05 * k, dphi_r0=-0.03 * k, out=out)

    alone = []
    for k in range(REPEATS):
        alone.append(call(k))
        torch.cuda.synchronize()
    outs = [torch.zeros_like(h) for h in alone]
    torch.cuda.synchronize()
    for k in range(REPEATS):
        call(k, outs[k])
    torch.cuda.synchronize()
    assert gpu_ctx.sync_status() == F.FEW_OK
    for a, b in zip(alone, outs):
        _same(a, b)
    for tr in trs:
        tr.release()


@pytest.mark.parametrize("prec", [F.FEW_MIXED, F.FEW_FP64])
def test_new_data_then_waveform_back_to_back(gpu_ctx, prec):
    """One trajectory whose knot data change before every waveform."""
    import torch
    ws = [W.make_inputs(2.0e5, 40, 50.0, W.mode_grid(4, 9), 60 + k, 3.0, 20.0) for k in range(3)]
    tr = RT.Trajectory(gpu_ctx, ws[0].t_knots, ws[0].modes)
    data = [tuple(torch.as_tensor(np.ascontiguousarray(a)).cuda() for a in (w.phi_phi, w.phi_r, w.amp_re, w.amp_im))
            for w in ws]

    def call(k, out=None):
        w = ws[0]
        tr.set_data_device(data[k % 3])
        return RT.waveform(gpu_ctx, tr, w.n_samples, w.t0, w.dt, 0.4 + 0.1 * k, 0.1, prec, out=out)

    alone = []
    for k in range(REPEATS):
        alone.append(call(k))
        torch.cuda.synchronize()
    outs = [torch.zeros_like(h) for h in alone]
    torch.cuda.synchronize()
    for k in range(REPEATS):
        call(k, outs[k])
    torch.cuda.synchronize()
    for a, b in zip(alone, outs):
        _same(a, b)
    tr.release()


@pytest.mark.parametrize("prec", [F.FEW_MIXED, F.FEW_FP64])
def test_direct_sums_back_to_back(gpu_ctx, prec):
    """Viewing angles, and with them the tables that the first kernel of a call writes, alternate."""
    import torch
    modes = W.mode_grid(6, 9)
    g = torch.Generator(device="cuda").manual_seed(3)
    n = 1500
    pp, pr = (torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * 1e4 for _ in range(2))
    re, im = (torch.randn(n, len(modes), generator=g, device="cuda", dtype=torch.float64) for _ in range(2))

    def call(k, out):
        F.few_direct_sum(gpu_ctx.handle, pp, pr, re, im, modes, 0.3 + 0.1 * k, 0.2 * k, out, prec=prec,
                         stream=RT.current_stream())
        return out

    dtype = torch.complex64 if prec == F.FEW_MIXED else torch.complex128
    alone = []
    for k in range(REPEATS):
        alone.append(call(k, torch.empty(n, device="cuda", dtype=dtype)))
        torch.cuda.synchronize()
    outs = [torch.zeros_like(h) for h in alone]
    torch.cuda.synchronize()
    for k in range(REPEATS):
        call(k, outs[k])
    torch.cuda.synchronize()
    for a, b in zip(alone, outs):
        _same(a, b)
