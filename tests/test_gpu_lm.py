"""GPU parity of the Levenberg-Marquardt iteration with adaptive
per-trajectory damping (pes_ieks_run_lm) against the oracle
(orc_iterated_smoother_lm), on models with a positive definite Q."""
import numpy as np
import pytest
import torch

import oracle
from paper_2102_00514_gb300 import pes, synth
from tests.gpu_common import TOL_FP32, TOL_FP64, rel_err, to_dev, workload_to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sm():
    s = pes.Smoother(1 << 16, 64)
    yield s
    s.close()


def starts(wl, seed):
    """Starts off the truth (positions shifted by up to 1.5 units, turn rate by
    up to 3 rad/s), where lightly damped steps overshoot and are rejected."""
    rng = np.random.default_rng(seed)
    off = wl["offsets"]
    x = wl["x_true"].copy()
    for b in range(len(off) - 1):
        sl = slice(int(off[b]), int(off[b + 1]))
        x[:, sl] += np.array([rng.uniform(-1.5, 1.5), rng.uniform(-1.5, 1.5), 0.0, 0.0, rng.uniform(-3, 3)])[:, None]
    return x


@pytest.mark.parametrize("lam0", [1e-4, 1.0])
def test_lm_fp64_matches_oracle(sm, lam0):
    wl = synth.ct_bearings([15, 40, 200, 1000], seed=31, q_form=1, sensor_jitter=0.2)
    x0 = starts(wl, 31)
    model = oracle.Model.from_workload(wl)
    d = workload_to_dev(wl, pes.FP64)
    for iters in (3, 8):
        ref = oracle.iterated_smoother_lm(model, wl["offsets"], wl["y"], wl["m0"], wl["P0"], x_init=x0, iters=iters,
                                          lambda0=lam0, nu=10.0)
        x, P, used, info = sm.ieks_run_lm(d["model"], pes.FP64, d["y"], d["offsets"], d["m0"], d["P0"],
                                          x_init=to_dev(x0), iters=iters, lambda0=lam0, nu=10.0)
        print(f"lam0 {lam0} iters {iters}: kept {info['accepted']} (oracle {ref['accepted']}), "
              f"lambda {info['lam']}")
        assert used == iters
        np.testing.assert_array_equal(info["accepted"], ref["accepted"])
        np.testing.assert_allclose(info["lam"], ref["lam"], rtol=1e-12)
        assert rel_err(x.cpu().numpy(), ref["x"], wl["offsets"]) < TOL_FP64
        assert rel_err(P.cpu().numpy(), ref["P"], wl["offsets"]) < TOL_FP64
    # the case exercises both decisions
    assert (ref["accepted"] < iters).any() and (ref["accepted"] > 0).all()


def test_lm_tolerance_mode_matches_oracle(sm):
    wl = synth.ct_bearings([60, 300], seed=32, q_form=1, sensor_jitter=0.2)
    x0 = starts(wl, 32)
    model = oracle.Model.from_workload(wl)
    d = workload_to_dev(wl, pes.FP64)
    ref = oracle.iterated_smoother_lm(model, wl["offsets"], wl["y"], wl["m0"], wl["P0"], x_init=x0, iters=60,
                                      tol=1e-8, lambda0=1e-2, nu=10.0)
    assert ref["status"] == oracle.OK
    x, P, used, info = sm.ieks_run_lm(d["model"], pes.FP64, d["y"], d["offsets"], d["m0"], d["P0"], x_init=to_dev(x0),
                                      iters=60, tol=1e-8, lambda0=1e-2, nu=10.0)
    # a step whose relative size is within rounding of tol may count on either
    # side of it: the converged iteration agrees to within one
    assert abs(used - ref["iters_used"]) <= 1
    assert np.abs(info["conv_iter"] - ref["conv_iter"]).max() <= 1
    assert rel_err(x.cpu().numpy(), ref["x"], wl["offsets"]) < TOL_FP64
    # at convergence the result is the IEKS fixed point: plain iterations leave it in place
    one = oracle.iterated_smoother(model, oracle.IEKS, wl["offsets"], wl["y"], wl["m0"], wl["P0"], x_init=ref["x"],
                                   iters=1)
    assert rel_err(one["x"], ref["x"], wl["offsets"]) < 1e-7


def test_lm_fp32_matches_oracle(sm):
    """FP32 steps, FP64 objective: the decisions of the first iterations (steps
    far larger than FP32 rounding) agree with the oracle's; near convergence
    the objective of a float trajectory no longer separates a step from the
    nominal, so a longer FP32 run may keep or reject differently there."""
    wl = synth.ct_bearings([40, 200], seed=33, q_form=1, sensor_jitter=0.2)
    x0 = starts(wl, 33)
    model = oracle.Model.from_workload(wl)
    d = workload_to_dev(wl, pes.FP32)
    ref = oracle.iterated_smoother_lm(model, wl["offsets"], wl["y"], wl["m0"], wl["P0"], x_init=x0, iters=3,
                                      lambda0=1.0, nu=10.0)
    x, P, used, info = sm.ieks_run_lm(d["model"], pes.FP32, d["y"], d["offsets"], d["m0"], d["P0"],
                                      x_init=to_dev(x0, torch.float32), iters=3, lambda0=1.0, nu=10.0)
    np.testing.assert_array_equal(info["accepted"], ref["accepted"])
    assert rel_err(x.double().cpu().numpy(), ref["x"], wl["offsets"]) < TOL_FP32
    assert rel_err(P.double().cpu().numpy(), ref["P"], wl["offsets"]) < TOL_FP32


def test_lm_rejects_singular_q_and_bad_arguments(sm):
    wl = synth.ct_bearings([20], seed=34, q_form=0)
    d = workload_to_dev(wl, pes.FP64)
    with pytest.raises(pes.PesError) as ei:
        sm.ieks_run_lm(d["model"], pes.FP64, d["y"], d["offsets"], d["m0"], d["P0"], iters=2)
    assert ei.value.status == pes.UNSUPPORTED
    wl = synth.ct_bearings([20], seed=34, q_form=1)
    d = workload_to_dev(wl, pes.FP64)
    for kw in (dict(lambda0=0.0), dict(nu=1.0), dict(iters=0)):
        with pytest.raises(pes.PesError) as ei:
            sm.ieks_run_lm(d["model"], pes.FP64, d["y"], d["offsets"], d["m0"], d["P0"], **kw)
        assert ei.value.status == pes.INVALID_ARG


L = np.longdouble


def inverse(a):
    """Inverse in long doubles: Newton steps on the double one."""
    a = np.asarray(a, dtype=L)
    v = np.linalg.inv(a.astype(np.float64)).astype(L)
    for _ in range(4):
        v = v + v @ (np.eye(len(a), dtype=L) - a @ v)
    return v


def objective(e, r, e0, model, P0):
    """Half the squared norms of process residuals, innovations and prior residual."""
    Q, R = np.asarray(model.Q()).reshape(5, 5), np.asarray(model.R()).reshape(2, 2)
    return ((e * (inverse(Q) @ e)).sum() + (r * (inverse(R) @ r)).sum() + e0 @ inverse(P0) @ e0) / 2


def turn_objective(wl, model, x):
    """The MAP objective of a single coordinated-turn trajectory."""
    x, dt = np.asarray(x, dtype=L), L(wl["dt"])
    px, py, vx, vy, w = x[:, :-1]
    a = w * dt
    safe = np.where(w == 0, L(1), w)
    A1 = np.where(w == 0, dt, np.sin(a) / safe)
    A2 = np.where(w == 0, L(0), 2 * np.sin(a / 2) ** 2 / safe)
    f = np.stack([px + A1 * vx - A2 * vy, py + A2 * vx + A1 * vy, np.cos(a) * vx - np.sin(a) * vy,
                  np.sin(a) * vx + np.cos(a) * vy, w])
    s = np.asarray(wl["sensors"], dtype=L).reshape(-1)
    r = np.stack([wl["y"][i, 1:] - np.arctan2(x[1, 1:] - s[2 * i + 1], x[0, 1:] - s[2 * i]) for i in range(2)])
    pi = np.arccos(L(-1))
    r = r - 2 * pi * np.round(r / (2 * pi))
    return objective(x[:, 1:] - f, r, x[:, 0] - np.asarray(wl["m0"][0], dtype=L), model,
                     oracle.sym_full(wl["P0"][0], 5))


def rounding_steps(sm, gm, y, off, m0, P0, opt, value, tol):
    """FP32 steps about an optimum are rounding noise, up or down: each decision
    against `value`, the objective in long doubles."""
    x0 = opt.float()
    J0 = value(x0.double().cpu().numpy())
    kept = []
    f32 = lambda a: to_dev(a, torch.float32)
    for lam0 in (1e-6, 1e-5, 1e-4, 1e-3, 1e-2, 1e-1, 1.0, 10.0):
        x1, _, _, info = sm.ieks_run_lm(gm, pes.FP32, f32(y), to_dev(off, torch.int64), f32(m0), f32(P0), x_init=x0,
                                        iters=1, tol=tol, lambda0=lam0, allow_not_converged=True)
        dJ = float(value(x1.double().cpu().numpy()) - J0)
        kept.append(int(info["accepted"][0]))
        print(f"lambda0 {lam0:g}: kept {kept[-1]}, change {dJ:.3e} of {float(J0):.3e}")
        if kept[-1]:
            assert dJ < 0.0
            np.testing.assert_allclose(info["lam"], lam0 / 10.0, rtol=1e-6)
        else:
            assert torch.equal(x1, x0)
            np.testing.assert_allclose(info["lam"], lam0 * 10.0, rtol=1e-6)
    return kept


@pytest.mark.parametrize("tol", [0.0, 1e-3])
@pytest.mark.parametrize("offset", [0.0, 1e5])
def test_lm_keeps_a_step_only_if_it_lowers_the_objective(sm, offset, tol):
    """Linear model; an innovation that no state explains (a zero row of H) makes the
    objective up to 1e12, of which the steps' changes are 1e-18."""
    rng = np.random.default_rng(41)
    r32 = lambda a: np.asarray(a, dtype=np.float32).astype(np.float64)
    T = 200
    F = r32(0.95 * np.eye(5) + 0.01 * rng.standard_normal((5, 5)))
    A = rng.standard_normal((5, 5))
    Q, R = r32(1e-4 * (A @ A.T + np.eye(5))), np.eye(2)
    H = r32(np.stack([rng.standard_normal(5), np.zeros(5)]))
    c, d, m0, P0 = r32(0.1 * rng.standard_normal(5)), np.zeros(2), np.zeros((1, 5)), np.eye(5)
    y = r32(np.stack([rng.standard_normal(T + 1), np.full(T + 1, offset)]))
    off = np.array([0, T + 1])
    model = oracle.Model.linear(F, c, Q, H, d, R)
    gm = pes.Model.linear(F, c, oracle.sym_packed(Q), H, d, oracle.sym_packed(R))
    opt = oracle.iterated_smoother(model, oracle.IEKS, off, y, m0, oracle.sym_packed(P0)[None], iters=2)["x"]

    def value(x):
        x = np.asarray(x, dtype=L)
        return objective(x[:, 1:] - (F.astype(L) @ x[:, :-1] + c[:, None]), y[:, 1:] - H.astype(L) @ x[:, 1:], x[:, 0],
                         model, P0)

    kept = rounding_steps(sm, gm, y, off, m0, oracle.sym_packed(P0)[None], to_dev(opt), value, tol)
    assert 0 in kept


@pytest.mark.parametrize("tol", [0.0, 1e-3])
@pytest.mark.parametrize("turn", [0.0, 20.0])
def test_lm_keeps_a_step_of_the_turn_only_if_it_lowers_the_objective(sm, turn, tol):
    """Small turn angles (series) and larger ones (differences of sine and cosine)."""
    wl = synth.ct_bearings([200], seed=41, q_form=1, omega0_halfwidth=turn)
    r32 = lambda a: np.asarray(a, dtype=np.float32).astype(np.float64)
    for k in ("y", "m0", "P0"):
        wl[k] = r32(wl[k])
    model = oracle.Model.from_workload(wl)
    d64 = workload_to_dev(wl, pes.FP64)
    opt, _, _, _ = sm.ieks_run_lm(d64["model"], pes.FP64, d64["y"], d64["offsets"], d64["m0"], d64["P0"],
                                  x_init=to_dev(wl["x_true"]), iters=40, lambda0=1e-2)
    kept = rounding_steps(sm, d64["model"], wl["y"], wl["offsets"], wl["m0"], wl["P0"], opt,
                          lambda x: turn_objective(wl, model, x), tol)
    assert 0 in kept


def test_lm_change_of_the_objective_for_each_branch_of_the_turn(sm):
    """Decisions at zero, small and large turn rates and turn-rate steps, FP64: the
    oracle keeps and rejects the same steps while they are far from rounding."""
    for shift in (0.0, 1e-3, 0.5, 3.0, 40.0):
        wl = synth.ct_bearings([80], seed=43, q_form=1, sensor_jitter=0.2)
        x0 = wl["x_true"].copy()
        x0[4] = shift
        model = oracle.Model.from_workload(wl)
        d = workload_to_dev(wl, pes.FP64)
        ref = oracle.iterated_smoother_lm(model, wl["offsets"], wl["y"], wl["m0"], wl["P0"], x_init=x0, iters=5,
                                          lambda0=1e-3, nu=10.0)
        x, _, _, info = sm.ieks_run_lm(d["model"], pes.FP64, d["y"], d["offsets"], d["m0"], d["P0"], x_init=to_dev(x0),
                                       iters=5, lambda0=1e-3, nu=10.0)
        np.testing.assert_array_equal(info["accepted"], ref["accepted"])
        assert rel_err(x.cpu().numpy(), ref["x"], wl["offsets"]) < TOL_FP64, shift
