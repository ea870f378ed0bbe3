"""Mode amplitudes from reduced-basis coefficients (Sec. 3.E) on the GPU against the oracle:
the FP64 GEMM and the tensor-core (split bf16, FP32 accumulation) product, with and without
the per-knot renormalisation, at the paper's size (99 coefficients, 3843 modes) and at ragged
sizes that leave partial tiles in every dimension; then the amplitudes feed a trajectory and
its waveform is compared with the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2104_04582_gb300 import fewsum as F
from paper_2104_04582_gb300 import runtime as RT
from paper_2104_04582_gb300 import workloads as W
from tests.gpu_common import MIXED_MISMATCH, oracle_threads, to_host

pytestmark = pytest.mark.gpu

# Per-row bounds in the form of the dot-product error bound |fl(x.y) - x.y| <= g |x|.|y|:
# FP64, a 2 Nb-term complex dot product per output; mixed, FP32 accumulation of six partial
# products of bf16 parts (the three-way split keeps ~24 bits of each operand) over 12 Nb terms,
# so g = 2e-6 (about 32 FP32 ulps, the typical sqrt(12 Nb) growth with margin).
FP64_GAMMA = 1e-14
MIXED_GAMMA = 2e-6


def _dev(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _gpu_rb(ctx, alpha, basis, norms, prec, basis_on_device=False):
    import torch
    M, N = alpha.shape[0], basis.shape[1]
    if basis_on_device:
        h = F.few_basis_create(ctx.handle, _dev(basis.real), _dev(basis.imag), RT.current_stream())
    else:
        h = F.few_basis_create(ctx.handle, basis.real, basis.imag, RT.current_stream())
    try:
        ore = torch.full((M, N), np.nan, dtype=torch.float64, device="cuda")
        oim = torch.full((M, N), np.nan, dtype=torch.float64, device="cuda")
        F.few_rb_amplitudes(ctx.handle, h, _dev(alpha.real), _dev(alpha.imag), ore, oim,
                            None if norms is None else _dev(norms), prec, RT.current_stream())
        torch.cuda.synchronize()
        assert ctx.sync_status() == F.FEW_OK
        return to_host(ore) + 1j * to_host(oim)
    finally:
        F.few_basis_release(ctx.handle, h)


def _check_rows(g, o, alpha, basis, norms, prec):
    """||g_k - o_k|| <= gamma || |s_k alpha_k| |B| || for every knot k."""
    raw = np.abs(alpha) @ np.abs(basis)
    if norms is not None:
        plain = np.linalg.norm(oracle.rb_amplitudes(alpha, basis), axis=1)
        s = np.where(plain > 0, norms / np.where(plain > 0, plain, 1.0), 0.0)
        raw = raw * s[:, None]
    gamma = FP64_GAMMA if prec == F.FEW_FP64 else MIXED_GAMMA
    err = np.linalg.norm(g - o, axis=1)
    bound = gamma * np.linalg.norm(raw, axis=1)
    assert np.all(err <= bound), np.max(err / np.where(bound > 0, bound, 1e-300))


@pytest.mark.parametrize("prec", [F.FEW_FP64, F.FEW_MIXED])
@pytest.mark.parametrize("renorm", [False, True])
def test_rb_paper_size_matches_oracle(gpu_ctx, prec, renorm):
    alpha, basis, nu = W.rb_inputs(100)
    g = _gpu_rb(gpu_ctx, alpha, basis, nu if renorm else None, prec)
    o = oracle.rb_amplitudes(alpha, basis, nu if renorm else None, oracle_threads())
    assert np.all(np.isfinite(g))
    _check_rows(g, o, alpha, basis, nu if renorm else None, prec)


@pytest.mark.parametrize("M,Nb,N", [(1, 1, 1), (129, 7, 130), (300, 99, 257), (5, 256, 64),
                                    (257, 33, 1)])
@pytest.mark.parametrize("prec", [F.FEW_FP64, F.FEW_MIXED])
def test_rb_ragged_sizes(gpu_ctx, M, Nb, N, prec):
    rng = np.random.default_rng(M * 1000 + Nb * 10 + N)
    alpha = rng.standard_normal((M, Nb)) + 1j * rng.standard_normal((M, Nb))
    basis = rng.standard_normal((Nb, N)) + 1j * rng.standard_normal((Nb, N))
    nu = rng.uniform(0.5, 2.0, M)
    g = _gpu_rb(gpu_ctx, alpha, basis, nu, prec, basis_on_device=(M % 2 == 1))
    o = oracle.rb_amplitudes(alpha, basis, nu)
    _check_rows(g, o, alpha, basis, nu, prec)


@pytest.mark.parametrize("prec", [F.FEW_FP64, F.FEW_MIXED])
def test_rb_norms_and_zero_rows(gpu_ctx, prec):
    alpha, basis, nu = W.rb_inputs(40, Nb=20, N=500)
    alpha[[3, 17]] = 0.0
    g = _gpu_rb(gpu_ctx, alpha, basis, nu, prec)
    norms = np.linalg.norm(g, axis=1)
    live = np.ones(40, bool)
    live[[3, 17]] = False
    tol = 1e-13 if prec == F.FEW_FP64 else 3e-6
    assert np.all(np.abs(norms[live] - nu[live]) <= tol * nu[live])
    assert np.all(g[~live] == 0)


def test_rb_bad_norm_latches_invalid(gpu_ctx):
    import torch
    alpha, basis, nu = W.rb_inputs(8, Nb=4, N=16)
    nu[5] = np.nan
    nu[6] = -1.0
    h = F.few_basis_create(gpu_ctx.handle, basis.real, basis.imag, RT.current_stream())
    try:
        ore = torch.empty((8, 16), dtype=torch.float64, device="cuda")
        oim = torch.empty_like(ore)
        F.few_rb_amplitudes(gpu_ctx.handle, h, _dev(alpha.real), _dev(alpha.imag), ore, oim,
                            _dev(nu), F.FEW_MIXED, RT.current_stream())
        torch.cuda.synchronize()
        assert gpu_ctx.sync_status() == F.FEW_ERR_INVALID_ARG
        assert gpu_ctx.sync_status() == F.FEW_OK  # the latch is cleared once read
    finally:
        F.few_basis_release(gpu_ctx.handle, h)


def test_rb_zero_knots_is_noop(gpu_ctx):
    import torch
    alpha, basis, _ = W.rb_inputs(4, Nb=3, N=8)
    h = F.few_basis_create(gpu_ctx.handle, basis.real, basis.imag, RT.current_stream())
    try:
        e = torch.empty((0, 3), dtype=torch.float64, device="cuda")
        o = torch.empty((0, 8), dtype=torch.float64, device="cuda")
        F.few_rb_amplitudes(gpu_ctx.handle, h, e, e, o, o, None, F.FEW_MIXED, RT.current_stream())
        torch.cuda.synchronize()
        assert gpu_ctx.sync_status() == F.FEW_OK
    finally:
        F.few_basis_release(gpu_ctx.handle, h)


def test_rb_amplitudes_feed_a_waveform(gpu_ctx):
    """Amplitudes produced on the device straight into the arrays a trajectory reads, then the
    interpolated summation, against the oracle waveform built from the oracle's amplitudes."""
    import torch
    w = W.config1()  # one week, 40 knots, 132 modes
    K, N = len(w.t_knots), len(w.modes)
    alpha, basis, nu = W.rb_inputs(K, Nb=12, N=N)
    h = F.few_basis_create(gpu_ctx.handle, basis.real, basis.imag, RT.current_stream())
    tr = RT.Trajectory(gpu_ctx, w.t_knots, w.modes)
    try:
        ore = torch.empty((K, N), dtype=torch.float64, device="cuda")
        oim = torch.empty_like(ore)
        F.few_rb_amplitudes(gpu_ctx.handle, h, _dev(alpha.real), _dev(alpha.imag), ore, oim,
                            _dev(nu), F.FEW_MIXED, RT.current_stream())
        tr.set_data_device((_dev(w.phi_phi), _dev(w.phi_r), ore, oim))
        out = RT.waveform(gpu_ctx, tr, w.n_samples, w.t0, w.dt, w.theta, w.phi, F.FEW_MIXED,
                          scale=w.scale)
        torch.cuda.synchronize()
        assert gpu_ctx.sync_status() == F.FEW_OK
        A = oracle.rb_amplitudes(alpha, basis, nu)
        ref = oracle.waveform(w.t_knots, w.phi_phi, w.phi_r, w.modes, A.real, A.imag, w.theta,
                              w.phi, w.scale, w.t0, w.dt, 0, w.n_samples, oracle_threads())
        assert oracle.mismatch(to_host(out), ref) <= MIXED_MISMATCH
    finally:
        tr.release()
        F.few_basis_release(gpu_ctx.handle, h)


def test_rb_basis_limit(gpu_ctx):
    b = np.zeros((257, 4))  # one more basis vector than FEW_MAX_BASIS
    with pytest.raises(F.FewError) as e:
        F.few_basis_create(gpu_ctx.handle, b, b)
    assert e.value.status == F.FEW_ERR_LIMIT


@pytest.mark.parametrize("M", [1, 2, 7, 8, 9, 15, 17])
def test_rb_fp64_knot_groups(gpu_ctx, M):
    """Every size of a knot group of the FP64 product, with a last mode warp that is partly past N."""
    rng = np.random.default_rng(M)
    alpha = rng.standard_normal((M, 33)) + 1j * rng.standard_normal((M, 33))
    basis = rng.standard_normal((33, 161)) + 1j * rng.standard_normal((33, 161))
    nu = rng.uniform(0.5, 2.0, M)
    g = _gpu_rb(gpu_ctx, alpha, basis, nu, F.FEW_FP64)
    assert np.all(np.isfinite(g))
    _check_rows(g, oracle.rb_amplitudes(alpha, basis, nu), alpha, basis, nu, F.FEW_FP64)


@pytest.mark.parametrize("M,N,shift", [(1, 28, 0), (16, 32, 1), (17, 33, 0), (33, 60, 1), (255, 61, 3), (257, 63, 2),
                                       (300, 3843, 1), (520, 3841, 0)])
@pytest.mark.parametrize("Nb", [3, 99, 128])
def test_rb_mixed_store_edges(gpu_ctx, M, N, Nb, shift):
    """Every way the output rows can start in a sector, groups of modes that just fit, parts of tiles; the
    output is written whole and nothing around it."""
    import torch
    rng = np.random.default_rng(M + 7 * N + Nb)
    alpha = rng.standard_normal((M, Nb)) + 1j * rng.standard_normal((M, Nb))
    basis = rng.standard_normal((Nb, N)) + 1j * rng.standard_normal((Nb, N))
    nu = rng.uniform(0.5, 2.0, M)
    h = F.few_basis_create(gpu_ctx.handle, basis.real, basis.imag, RT.current_stream())
    try:
        out = [torch.full((M * N + 8,), 7.0, dtype=torch.float64, device="cuda") for _ in range(2)]
        re, im = (o[2 + shift:2 + shift + M * N].view(M, N) for o in out)
        F.few_rb_amplitudes(gpu_ctx.handle, h, _dev(alpha.real), _dev(alpha.imag), re, im, _dev(nu),
                            F.FEW_MIXED, RT.current_stream())
        torch.cuda.synchronize()
        assert gpu_ctx.sync_status() == F.FEW_OK
        plain = alpha @ basis
        s = (nu / np.linalg.norm(plain, axis=1))[:, None]
        err = np.linalg.norm(to_host(re) + 1j * to_host(im) - s * plain, axis=1)
        assert np.all(err <= MIXED_GAMMA * np.linalg.norm(s * (np.abs(alpha) @ np.abs(basis)), axis=1))
        for o in out:
            assert torch.all(o[:2 + shift] == 7.0) and torch.all(o[2 + shift + M * N:] == 7.0)
    finally:
        F.few_basis_release(gpu_ctx.handle, h)


@pytest.mark.parametrize("M,Nb,N,kind", [
    (1, 102, 43200, "plain"), (64, 102, 640, "plain"), (65, 103, 641, "plain"), (130, 192, 321, "plain"),
    (200, 256, 130, "plain"), (300, 9, 1600, "plain"), (70, 60, 1025, "ranges"), (70, 60, 1025, "special"),
    (1, 1, 1, "plain"), (127, 13, 64, "plain")])
def test_rb_fp64_digit_slices(gpu_ctx, M, Nb, N, kind):
    """Tiles and parts of the digit-slice product, element by element; rows and columns whose entries span
    30 decades or are not finite or far from one go to the plain chain.  Bound: both operands to 2^-62 of
    their largest entry with sums of magnitudes above 2^-7 of the two, or FP64's own (2 Nb roundings):
    below 1e-13 of the sum of magnitudes."""
    import torch
    rng = np.random.default_rng(M + Nb + N)
    alpha = rng.standard_normal((M, Nb)) + 1j * rng.standard_normal((M, Nb))
    basis = rng.standard_normal((Nb, N)) + 1j * rng.standard_normal((Nb, N))
    if kind == "ranges":
        alpha *= 10.0 ** rng.uniform(-30, 0, (M, Nb))
        basis *= 10.0 ** rng.uniform(-30, 0, (Nb, N))
        alpha[3], basis[:, 5] = 0.0, 0.0
        alpha[4] *= 1e130
        basis[:, 7] *= 1e-130
    if kind == "special":
        alpha[2, 1], alpha[9, 0], basis[4, 3], basis[0, 70] = np.nan, np.inf, np.inf, np.nan
    h = F.few_basis_create(gpu_ctx.handle, basis.real, basis.imag, RT.current_stream())
    try:
        out = [torch.full((M * N + 2,), 7.0, dtype=torch.float64, device="cuda") for _ in range(2)]
        re, im = (o[1:-1].view(M, N) for o in out)
        F.few_rb_amplitudes(gpu_ctx.handle, h, _dev(alpha.real), _dev(alpha.imag), re, im, None, F.FEW_FP64,
                            RT.current_stream())
        torch.cuda.synchronize()
        assert gpu_ctx.sync_status() == F.FEW_OK
        g = to_host(re) + 1j * to_host(im)
        assert all(float(o[0]) == float(o[-1]) == 7.0 for o in out)
    finally:
        F.few_basis_release(gpu_ctx.handle, h)
    with np.errstate(all="ignore"):
        ref = alpha.real @ basis.real - alpha.imag @ basis.imag + 1j * (alpha.real @ basis.imag + alpha.imag @ basis.real)
        bound = 1e-13 * (np.abs(alpha) @ np.abs(basis))
    bad = ~np.isfinite(alpha).all(axis=1)[:, None] | ~np.isfinite(basis).all(axis=0)[None, :]
    assert np.all(np.abs(g - ref)[~bad] <= bound[~bad])
    assert not np.isfinite(g[bad]).any()


@pytest.mark.parametrize("kind", ["unit", "blocks"])
def test_rb_fp64_localised_basis(gpu_ctx, kind):
    """A localised basis (each mode in one vector, or in a few neighbouring ones) and decaying coefficients:
    most outputs are below the digit product's guard and take the plain chain.  Bound of
    test_rb_fp64_digit_slices; and the call stays below the 1.7 ms that the plain chain of every output
    takes (it took 2.6 ms with one output at a time in flight a thread)."""
    import torch
    M, Nb, N = 400, 99, 3843
    rng = np.random.default_rng(5)
    alpha = (rng.standard_normal((M, Nb)) + 1j * rng.standard_normal((M, Nb))) * np.exp(-np.arange(Nb) / 5.0)
    basis = rng.standard_normal((Nb, N)) + 1j * rng.standard_normal((Nb, N))
    place = np.abs(np.arange(N)[None, :] * Nb // N - np.arange(Nb)[:, None])
    basis *= (place == 0) if kind == "unit" else np.exp(-place)
    nu = rng.uniform(0.5, 2.0, M)
    h = F.few_basis_create(gpu_ctx.handle, basis.real, basis.imag, RT.current_stream())
    try:
        dev = [_dev(alpha.real), _dev(alpha.imag), _dev(nu)]
        re, im = (torch.empty(M, N, dtype=torch.float64, device="cuda") for _ in range(2))
        best = float("inf")
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            F.few_rb_amplitudes(gpu_ctx.handle, h, dev[0], dev[1], re, im, dev[2], F.FEW_FP64, RT.current_stream())
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) * 1e3)
        assert gpu_ctx.sync_status() == F.FEW_OK
        plain = alpha @ basis
        s = (nu / np.linalg.norm(plain, axis=1))[:, None]
        g = to_host(re) + 1j * to_host(im)
        assert np.all(np.abs(g - s * plain) <= 1e-13 * s * (np.abs(alpha) @ np.abs(basis)) + 1e-300)
        assert best <= 1700.0
    finally:
        F.few_basis_release(gpu_ctx.handle, h)


def _slices_case(rng, M=40, Nb=99, N=3843):
    alpha = rng.standard_normal((M, Nb)) + 1j * rng.standard_normal((M, Nb))
    basis = rng.standard_normal((Nb, N)) + 1j * rng.standard_normal((Nb, N))
    return alpha, basis, rng.uniform(0.5, 2.0, M)


def _room_for_basis_alone(basis, modes, knots):
    """Bytes that a context holds for a basis (with its digit slices) and for a trajectory."""
    with RT.Context(0) as free:
        h = F.few_basis_create(free.handle, basis.real, basis.imag, RT.current_stream())
        held = free.memory()[0]
        tr = RT.Trajectory(free, knots, modes)
        traj = free.memory()[0] - held
        tr.release()
        F.few_basis_release(free.handle, h)
    return held, traj


@pytest.mark.parametrize("prec", [F.FEW_FP64, F.FEW_MIXED])
def test_rb_slices_give_way_to_other_allocations(prec):
    """A budget that holds a basis with its FP64 digit slices, or the basis and a trajectory: the trajectory
    is not refused, and the basis' amplitudes stay what they were (FP64 by the plain chain)."""
    import torch
    alpha, basis, nu = _slices_case(np.random.default_rng(8))
    modes, knots = W.mode_grid(10, 10), W.knot_times(1e6, 200)
    held, traj = _room_for_basis_alone(basis, modes, knots)
    with RT.Context(0, held + traj // 4) as ctx:
        h = F.few_basis_create(ctx.handle, basis.real, basis.imag, RT.current_stream())
        assert ctx.memory()[0] == held
        tr = RT.Trajectory(ctx, knots, modes)
        assert ctx.memory()[0] < held + traj
        re, im = (torch.empty(len(nu), basis.shape[1], dtype=torch.float64, device="cuda") for _ in range(2))
        F.few_rb_amplitudes(ctx.handle, h, _dev(alpha.real), _dev(alpha.imag), re, im, _dev(nu), prec,
                            RT.current_stream())
        torch.cuda.synchronize()
        assert ctx.sync_status() == F.FEW_OK
        _check_rows(to_host(re) + 1j * to_host(im), oracle.rb_amplitudes(alpha, basis, nu), alpha, basis, nu, prec)
        tr.release()
        F.few_basis_release(ctx.handle, h)


def test_rb_slices_of_a_captured_call_stay():
    """A captured graph reads the slices: they are kept, the trajectory is refused, and the replay is right."""
    import torch
    alpha, basis, nu = _slices_case(np.random.default_rng(9))
    modes, knots = W.mode_grid(10, 10), W.knot_times(1e6, 200)
    held, traj = _room_for_basis_alone(basis, modes, knots)
    with RT.Context(0, held + traj // 4) as ctx:
        h = F.few_basis_create(ctx.handle, basis.real, basis.imag, RT.current_stream())
        dev = [_dev(alpha.real), _dev(alpha.imag), _dev(nu)]
        re, im = (torch.zeros(len(nu), basis.shape[1], dtype=torch.float64, device="cuda") for _ in range(2))

        def call():
            F.few_rb_amplitudes(ctx.handle, h, dev[0], dev[1], re, im, dev[2], F.FEW_FP64, RT.current_stream())

        call()
        torch.cuda.synchronize()
        ref = to_host(re) + 1j * to_host(im)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            call()
        with pytest.raises(F.FewError) as e:
            RT.Trajectory(ctx, knots, modes)
        assert e.value.status == F.FEW_ERR_BUDGET
        re.zero_()
        im.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert ctx.sync_status() == F.FEW_OK
        np.testing.assert_array_equal(to_host(re) + 1j * to_host(im), ref)
        del g
        F.few_basis_release(ctx.handle, h)


@pytest.mark.parametrize("prec", [F.FEW_MIXED, F.FEW_FP64])
def test_rb_more_outputs_than_2_to_the_31(gpu_ctx, prec):
    """559,200 knots of 3841 modes (2 x 17 GB): the rows' places in memory past 2^31 elements, around that
    boundary and at both ends."""
    import torch
    M, N, Nb = 559200, 3841, 2
    assert M * N > 2 ** 31
    if torch.cuda.mem_get_info()[0] < 48 << 30:
        pytest.skip("needs 48 GB")
    rng = np.random.default_rng(2)
    basis = rng.standard_normal((Nb, N)) + 1j * rng.standard_normal((Nb, N))
    are, aim = (_dev(rng.standard_normal((M, Nb))) for _ in range(2))
    bre, bim = _dev(basis.real), _dev(basis.imag)
    re, im = (torch.full((M, N), 7.0, dtype=torch.float64, device="cuda") for _ in range(2))
    h = F.few_basis_create(gpu_ctx.handle, basis.real, basis.imag, RT.current_stream())
    try:
        F.few_rb_amplitudes(gpu_ctx.handle, h, are, aim, re, im, None, prec, RT.current_stream())
        torch.cuda.synchronize()
        assert gpu_ctx.sync_status() == F.FEW_OK
        edge = 2 ** 31 // N
        for k0 in (0, edge - 1000, M - 3000):
            s = slice(k0, k0 + 3000)
            bound = (FP64_GAMMA if prec == F.FEW_FP64 else MIXED_GAMMA) * torch.linalg.vector_norm(
                (are[s].abs() + aim[s].abs()) @ (bre.abs() + bim.abs()), dim=1)
            for g, o in ((re, are[s] @ bre - aim[s] @ bim), (im, are[s] @ bim + aim[s] @ bre)):
                assert torch.all(torch.linalg.vector_norm(g[s] - o, dim=1) <= bound)
        assert not torch.any(re[::997] == 7.0) and not torch.any(im[::997] == 7.0)
    finally:
        F.few_basis_release(gpu_ctx.handle, h)
        del re, im
        torch.cuda.empty_cache()


@pytest.mark.parametrize("kind,Nb", [("dense", 20), ("dense", 99), ("dense", 200), ("edge", 99)])
def test_rb_fp64_against_extended_precision(gpu_ctx, kind, Nb):
    """The digit product's error, of each output's sum of magnitudes S: its rounding, at most 2^-53 (rms 2^-54 or
    less), and the products left out, ~2^-58 sqrt(Nb / 99) of the two scales, which S exceeds 2^-5 times at the
    least ("edge": the large entries of rows and columns do not meet): below 2^-53 in the root mean square.
    (An FP64 chain of 2 Nb steps: 2e-16 to 6e-16.)"""
    if np.finfo(np.longdouble).nmant < 60:
        pytest.skip("needs extended precision")
    M, N = 64, 256
    rng = np.random.default_rng(Nb)
    alpha = rng.standard_normal((M, Nb)) + 1j * rng.standard_normal((M, Nb))
    basis = rng.standard_normal((Nb, N)) + 1j * rng.standard_normal((Nb, N))
    if kind == "edge":
        alpha[:, 1:] *= 2.0 ** -5
        alpha[:, 0] = 1.9 + 1.9j
        basis[1, :] = 1.9 - 1.9j
        basis[[0] + list(range(2, Nb)), :] *= 2.0 ** -5
    g = _gpu_rb(gpu_ctx, alpha, basis, None, F.FEW_FP64)
    ar, ai, br, bi = (np.asarray(x, dtype=np.longdouble) for x in (alpha.real, alpha.imag, basis.real, basis.imag))
    re, im = ar @ br - ai @ bi, ar @ bi + ai @ br
    S = np.abs(ar) @ np.abs(br) + np.abs(ai) @ np.abs(bi), np.abs(ar) @ np.abs(bi) + np.abs(ai) @ np.abs(br)
    for x, ref, s in ((g.real, re, S[0]), (g.imag, im, S[1])):
        e = np.asarray((x - ref) / s, dtype=np.float64)
        assert np.sqrt(np.mean(e * e)) < 2.0 ** -53
