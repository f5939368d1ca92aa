"""Launch shapes of the fused smoother: sizes at the edges of the lanes per block,
of the steps per lane and of the grid level, every compiled form, against the
oracle; and the shape that a run chooses against a fixed one.

Tolerances: FP64 differs by rounding order (1e-9); one FP32 iteration on a stable
linear model, or from a nominal near the truth, is the exact smoother up to FP32
rounding through some tens of operator applications (1e-4); the refined iteration
is held to 1e-5 as elsewhere."""
import numpy as np
import pytest
import torch

import oracle
from paper_2102_00514_gb300 import pes, synth
from tests.gpu_common import (ORACLE_METHOD, TOL_FP32, TOL_FP64, gpu_run, oracle_run, prior_only,
                              random_linear_workload, rel_err, to_dev, workload_to_dev)
from tests.test_gpu_refined import TOL_REFINED, final_iteration_errors, float_inputs

pytestmark = pytest.mark.gpu

# 1 to 2 blocks of 32 lanes, a block's tree at odd counts, the first sizes of 64,
# 96 and 128 lanes, several steps per lane, odd grid levels
EDGES = [1, 2, 30, 31, 32, 33, 62, 63, 64, 65, 127, 128, 2049, 4863, 4865, 9729, 20011]


@pytest.fixture(scope="module")
def sm():
    s = pes.Smoother(1 << 18, 64)
    yield s
    s.close()


def linear_case(T, seed=3):
    """A stable linear-Gaussian model and its data, rounded to float on both sides."""
    rng = np.random.default_rng(seed)
    r32 = lambda a: np.asarray(a, dtype=np.float32).astype(np.float64)
    F = r32(0.95 * np.eye(5) + 0.01 * rng.standard_normal((5, 5)))
    A = rng.standard_normal((5, 5))
    Q, R = r32(1e-2 * (A @ A.T + np.eye(5))), r32(0.05 * np.eye(2))
    H, c, d = r32(rng.standard_normal((2, 5))), r32(0.01 * rng.standard_normal(5)), r32(0.1 * rng.standard_normal(2))
    off = synth.offsets_from_lengths(np.array([T]))
    y = r32(rng.standard_normal((2, T + 1)))
    P0 = oracle.sym_packed(np.eye(5))[None]
    return dict(om=oracle.Model.linear(F, c, Q, H, d, R),
                gm=pes.Model.linear(F, c, oracle.sym_packed(Q), H, d, oracle.sym_packed(R)), off=off, y=y,
                m0=np.zeros((1, 5)), P0=P0)


def linear_run(sm, w, method, prec, iters=1):
    dt = torch.float64 if prec == pes.FP64 else torch.float32
    x, P, _, _ = sm.ieks_run(w["gm"], method, prec, to_dev(w["y"], dt), to_dev(w["off"], torch.int64),
                             to_dev(w["m0"], dt), to_dev(w["P0"], dt), iters=iters, want_iters=True)
    return x.double().cpu().numpy(), P.double().cpu().numpy()


@pytest.mark.parametrize("prec,tol", [(pes.FP64, TOL_FP64), (pes.FP32, TOL_FP32)])
@pytest.mark.parametrize("method", [pes.IEKS, pes.CUBATURE, pes.GAUSS_HERMITE])
def test_linear_model_at_edge_sizes(sm, method, prec, tol):
    for T in EDGES:
        w = linear_case(T)
        ref = oracle.iterated_smoother(w["om"], ORACLE_METHOD[method], w["off"], w["y"], w["m0"], w["P0"], iters=1)
        x, P = linear_run(sm, w, method, prec)
        assert rel_err(x, ref["x"], w["off"]) < tol, T
        assert rel_err(P, ref["P"], w["off"]) < tol, T


@pytest.mark.parametrize("method", [pes.IEKS, pes.CUBATURE])
def test_coordinated_turn_at_edge_sizes(sm, method):
    for T in EDGES:
        wl = synth.ct_bearings([T], seed=T, sensor_jitter=0.2, omega0_halfwidth=1.0)
        ref = oracle_run(wl, method, iters=2)
        x, P, _, _ = gpu_run(sm, wl, method, pes.FP64, iters=2)
        assert rel_err(x, ref["x"], wl["offsets"]) < TOL_FP64, T
        assert rel_err(P, ref["P"], wl["offsets"]) < TOL_FP64, T


@pytest.mark.parametrize("method", [pes.IEKS, pes.CUBATURE, pes.GAUSS_HERMITE])
def test_chosen_shape_matches_oracle_with_damping_tolerance_and_prior_only_trajectories(sm, method):
    wl = synth.ct_bearings([1, 31, 1, 64, 500], seed=8, sensor_jitter=0.2, omega0_halfwidth=1.0)
    wl = prior_only(wl, (0, 2))
    ref = oracle_run(wl, method, iters=4, lm=0.5)
    x, P, _, _ = gpu_run(sm, wl, method, pes.FP64, iters=4, lm=0.5)
    assert rel_err(x, ref["x"], wl["offsets"]) < TOL_FP64
    assert rel_err(P, ref["P"], wl["offsets"]) < TOL_FP64
    w = linear_case(500)
    ref = oracle.iterated_smoother(w["om"], ORACLE_METHOD[method], w["off"], w["y"], w["m0"], w["P0"], iters=9, tol=1e-6)
    x, P, used, _ = sm.ieks_run(w["gm"], method, pes.FP64, to_dev(w["y"]), to_dev(w["off"], torch.int64),
                                to_dev(w["m0"]), to_dev(w["P0"]), iters=9, tol=1e-6, want_iters=True)
    assert used == ref["iters_used"]
    assert rel_err(x.cpu().numpy(), ref["x"], w["off"]) < TOL_FP64


@pytest.mark.parametrize("prec,threads,tol", [(pes.FP64, 128, TOL_FP64), (pes.FP32, 256, TOL_FP32),
                                              (pes.FP32, 128, TOL_FP32)])
def test_fixed_shapes_match_the_chosen_one(prec, threads, tol):
    """A chosen shape against all lanes with nine steps each (at 100,004 states a
    grid level of more blocks than one pass takes, with 128 threads)."""
    s = pes.Smoother(1 << 17, 4)
    try:
        for T in (60, 700, 12863, 100003):
            w = linear_case(T)
            x, P = linear_run(s, w, pes.IEKS, prec)
            chosen = s.launch_shape(pes.IEKS, prec, T + 1)
            s.set_launch_shape(pes.IEKS, prec, threads, 9)
            nb, nt, L = s.launch_shape(pes.IEKS, prec, T + 1)
            assert nt == threads and L <= 9 and (T < 100000 or L == 9) and (nb, nt, L) != chosen
            xf, Pf = linear_run(s, w, pes.IEKS, prec)
            s.set_launch_shape(pes.IEKS, prec, 0, 0)
            assert rel_err(x, xf, w["off"]) < tol, T
            assert rel_err(P, Pf, w["off"]) < tol, T
    finally:
        s.close()


def test_workspace_of_exactly_as_many_states():
    """The lane padding of a chosen shape fits a workspace made for just that size."""
    for N in (2, 33, 4865, 9728, 20000):
        w = linear_case(N - 1)
        s = pes.Smoother(N, 1)
        for prec, tol in ((pes.FP64, TOL_FP64), (pes.FP32, TOL_FP32)):
            ref = oracle.iterated_smoother(w["om"], oracle.CUBATURE, w["off"], w["y"], w["m0"], w["P0"], iters=1)
            x, P = linear_run(s, w, pes.CUBATURE, prec)
            assert rel_err(x, ref["x"], w["off"]) < tol, N
        s.close()


@pytest.mark.parametrize("prec,threads,tol", [(pes.FP64, 128, TOL_FP64), (pes.FP32, 256, TOL_FP32),
                                              (pes.FP32, 128, TOL_FP32)])
def test_a_minimum_of_steps_is_followed(prec, threads, tol):
    """Any minimum but the defaults' own (8) gives full blocks of lanes with at least so
    many steps, few as they may be; 8 with the default threads is the default."""
    s = pes.Smoother(1 << 15, 4)
    try:
        for T in (60, 700, 20011):
            N = T + 1
            w = linear_case(T)
            ref = oracle.iterated_smoother(w["om"], oracle.IEKS, w["off"], w["y"], w["m0"], w["P0"], iters=1)
            default = s.launch_shape(pes.IEKS, prec, N)
            for steps in (1, 2, 4, 7, 9, 32):
                s.set_launch_shape(pes.IEKS, prec, threads, steps)
                nb, nt, L = s.launch_shape(pes.IEKS, prec, N)
                want = -(-N // (threads * steps))
                assert nt == threads and nb <= want and L == -(-N // (nb * nt))
                assert nb == want or nb >= 152, (steps, nb, want)
                x, P = linear_run(s, w, pes.IEKS, prec)
                assert rel_err(x, ref["x"], w["off"]) < tol, (T, steps)
                assert rel_err(P, ref["P"], w["off"]) < tol, (T, steps)
            s.set_launch_shape(pes.IEKS, prec, 128 if prec == pes.FP64 else 256, 8)
            assert s.launch_shape(pes.IEKS, prec, N) == default
            s.set_launch_shape(pes.IEKS, prec, 0, 0)
    finally:
        s.close()


def near_truth(T, seed, q_form=0):
    """Coordinated turns of T + 1 states in all, with float inputs, a nominal at the
    true states and covariances of the size of the smoothed ones. Up to 5,000 states
    one trajectory, else 16: a longer one leaves the sensors behind, and the
    sequential FP32 smoother alone is then off by up to 3e-4."""
    N = T + 1
    lens = [T] if N <= 5000 else [N // 16 - 1 + (i < N % 16) for i in range(16)]
    wl = float_inputs(synth.ct_bearings(lens, seed=seed, q_form=q_form, sensor_jitter=0.2, omega0_halfwidth=1.0))
    x = wl["x_true"].astype(np.float32).astype(np.float64)
    P = np.repeat(oracle.sym_packed(np.diag([0.01, 0.01, 0.1, 0.1, 0.1]))[:, None], T + 1, 1)
    return wl, x, P.astype(np.float32).astype(np.float64)


def one_iteration(sm, wl, method, prec, x, P):
    dt = torch.float64 if prec == pes.FP64 else torch.float32
    d = workload_to_dev(wl, prec)
    got = sm.ieks_run(d["model"], method, prec, d["y"], d["offsets"], d["m0"], d["P0"], x_init=to_dev(x, dt),
                      P_init=to_dev(P, dt) if method != pes.IEKS else None, iters=1)
    torch.cuda.synchronize()
    return got[0].double().cpu().numpy(), got[1].double().cpu().numpy()


@pytest.mark.parametrize("threads", [256, 128])
@pytest.mark.parametrize("method", [pes.IEKS, pes.CUBATURE])
def test_coordinated_turn_fp32_at_edge_sizes(sm, method, threads):
    sm.set_launch_shape(method, pes.FP32, threads, 8)
    try:
        for T in EDGES:
            wl, x0, P0 = near_truth(T, T)
            ref = oracle_run(wl, method, iters=1, x_init=x0, P_init=P0)
            x, P = one_iteration(sm, wl, method, pes.FP32, x0, P0)
            assert rel_err(x, ref["x"], wl["offsets"]) < TOL_FP32, T
            assert rel_err(P, ref["P"], wl["offsets"]) < TOL_FP32, T
    finally:
        sm.set_launch_shape(method, pes.FP32, 0, 0)


@pytest.mark.parametrize("threads", [256, 128])
@pytest.mark.parametrize("method", [pes.IEKS, pes.CUBATURE])
def test_refined_iteration_at_edge_sizes(sm, method, threads):
    """The residual kernels read the smoother kernel's handoff over the edges of
    lanes, warps and blocks, and its scans run with fewer lanes than threads."""
    sm.set_launch_shape(method, pes.FP32, threads, 8)
    try:
        for T in EDGES:
            wl = synth.ct_bearings([T], seed=T, sensor_jitter=0.2, omega0_halfwidth=1.0)
            ex, eP, _, _ = final_iteration_errors(sm, wl, method, pes.REFINED, iters=2)
            assert ex < TOL_REFINED and eP < TOL_REFINED, (T, ex, eP)
    finally:
        sm.set_launch_shape(method, pes.FP32, 0, 0)


@pytest.mark.parametrize("prec,tol", [(pes.FP64, TOL_FP64), (pes.FP32, TOL_FP32)])
def test_scans_over_given_arrays_at_edge_sizes(sm, prec, tol):
    """One to three steps per lane, blocks that fill and that overflow by one."""
    dt = torch.float64 if prec == pes.FP64 else torch.float32
    for T in (1, 30, 31, 32, 62, 63, 64, 126, 127, 128, 254, 255, 256, 511, 1023, 1024, 2047, 2048, 4095, 4096):
        lin, y, m0, P0, off = random_linear_workload([T], T)
        ref = oracle.kf_rts(off, lin, y, m0, P0)
        dlin = {k: to_dev(v, dt) for k, v in lin.items()}
        xf, Pf = sm.filter_scan(prec, dlin, to_dev(y, dt), to_dev(m0, dt), to_dev(P0, dt), to_dev(off, torch.int64))
        xs, Ps = sm.smooth_scan(prec, dlin, xf, Pf, to_dev(off, torch.int64))
        sm.sync()
        for k, v in (("xf", xf), ("Pf", Pf), ("xs", xs), ("Ps", Ps)):
            assert rel_err(v.double().cpu().numpy(), ref[k], off) < tol, (T, k)


@pytest.mark.parametrize("q_form", [0, 1])
@pytest.mark.parametrize("prec,wmax,sd,tol", [(pes.FP64, 300.0, (1e-2, 100.0), TOL_FP64),
                                              (pes.FP64, 20.0, (0.1, 10.0), TOL_FP64),
                                              (pes.FP32, 20.0, (0.1, 10.0), TOL_FP32)])
def test_cubature_regression_over_wide_turn_rates(sm, prec, wmax, sd, tol, q_form):
    """The coordinated turn's own regression: turn angles of a step from 0 to wmax / 100
    and sigma-point offsets of them from 2e-4 to 0.2 (FP64: 2), both sides of its
    series. (Relative changes of 1e-12 of the inputs change the result by 3e-9 at most
    in the widest case, 1e-12 in the others: rounding stays within the tolerance.)"""
    T = 300
    wl = synth.ct_bearings([T], seed=9, q_form=q_form, sensor_jitter=0.2, omega0_halfwidth=1.0)
    rng = np.random.default_rng(9)
    x = wl["x_true"].copy()
    x[4] = rng.permutation(np.linspace(-wmax, wmax, T + 1))
    s = np.exp(rng.uniform(np.log(sd[0]), np.log(sd[1]), T + 1))
    Lc = 0.3 * np.tril(0.2 * rng.standard_normal((T + 1, 5, 5)), -1) + np.diag([0.1, 0.1, 0.3, 0.3, 1.0])
    Lc[:, 4] *= s[:, None]
    P = oracle.sym_packed(Lc @ np.swapaxes(Lc, 1, 2)).T.copy()
    if prec == pes.FP32:
        wl, x, P = float_inputs(wl), x.astype(np.float32).astype(np.float64), P.astype(np.float32).astype(np.float64)
    ref = oracle_run(wl, pes.CUBATURE, iters=1, x_init=x, P_init=P)
    gx, gP = one_iteration(sm, wl, pes.CUBATURE, prec, x, P)
    assert rel_err(gx, ref["x"], wl["offsets"]) < tol
    assert rel_err(gP, ref["P"], wl["offsets"]) < tol


@pytest.mark.parametrize("method", [pes.CUBATURE, pes.UNSCENTED])
def test_full_process_noise_through_the_stored_regression(sm, method):
    """q_form 1 (a full 5 x 5 Q): what the compact stored form leaves out is the model's."""
    for T in (40, 3000):
        wl, x0, P0 = near_truth(T, T, q_form=1)
        for prec, tol in ((pes.FP64, TOL_FP64), (pes.FP32, TOL_FP32)):
            ref = oracle_run(wl, method, iters=1, x_init=x0, P_init=P0)
            x, P = one_iteration(sm, wl, method, prec, x0, P0)
            assert rel_err(x, ref["x"], wl["offsets"]) < tol, (T, prec)
            assert rel_err(P, ref["P"], wl["offsets"]) < tol, (T, prec)


def test_a_tuning_at_a_large_size_keeps_the_choice_for_small_ones():
    """At sizes at which every lane has steps enough, small minima give one launch: the
    tuning then records the library's own choice, which other sizes go by."""
    T = (1 << 18) + 300000
    s = pes.Smoother(T + 1, 1)
    try:
        w = linear_case(T)
        small = s.launch_shape(pes.IEKS, pes.FP64, 501)
        d = [to_dev(w["y"]), to_dev(w["off"], torch.int64), to_dev(w["m0"]), to_dev(w["P0"])]
        assert s.autotune(w["gm"], pes.IEKS, pes.FP64, *d, iters=1)[1] == 8
        assert s.launch_shape(pes.IEKS, pes.FP64, 501) == small
    finally:
        s.close()


@pytest.mark.parametrize("prec,threads,tol", [(pes.FP64, 128, TOL_FP64), (pes.FP32, 256, TOL_FP32)])
def test_layout_copies_at_whole_chunks_and_pieces(prec, threads, tol):
    """Steps per lane around the widths at which the copies' tiles change (banks' words,
    the widest whole chunk of 63 steps), in a block whose last lane lacks a state."""
    s = pes.Smoother(1 << 15, 1)
    try:
        for L in (1, 2, 3, 5, 8, 15, 16, 17, 31, 32, 33, 62, 63, 64, 65, 126, 127):
            N = L * threads - (1 if L > 1 else 0)
            w = linear_case(N - 1, seed=L)
            s.set_launch_shape(pes.IEKS, prec, threads, L if L != 8 else 9)   # 8 leaves the steps to the library
            assert L == 8 or s.launch_shape(pes.IEKS, prec, N) == (1, threads, L)
            ref = oracle.iterated_smoother(w["om"], oracle.IEKS, w["off"], w["y"], w["m0"], w["P0"], iters=1)
            x, P = linear_run(s, w, pes.IEKS, prec)
            assert rel_err(x, ref["x"], w["off"]) < tol, L
            assert rel_err(P, ref["P"], w["off"]) < tol, L
    finally:
        s.close()
