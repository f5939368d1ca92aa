"""Launch shapes of the fused smoother: sizes at the edges of the lanes per block,
of the steps per lane and of the grid level, every compiled form, against the
oracle; and the shape that a run chooses against a fixed one.

Tolerances: FP64 differs by rounding order (1e-9); one FP32 iteration on a stable
linear model is the exact smoother up to FP32 rounding through some tens of
operator applications (1e-4)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2102_00514_gb300 import pes, synth
from tests.gpu_common import ORACLE_METHOD, TOL_FP32, TOL_FP64, gpu_run, oracle_run, prior_only, rel_err, to_dev

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
