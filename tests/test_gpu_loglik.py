"""Log-likelihood terms of the filter scan at their limits. With H = 0 the innovation
covariance is the given R' and the innovation the given y, to the bit, so the sum of
log N(y_k; 0, R'_k) is known from the inputs alone (numpy long doubles here).

Tolerance: a term in FP64 forms det = R00 R11 - R01^2 and the quadratic form from
three products each; both lose at most a few eps / (1 - rho^2) of themselves, so the
sum is within 16 eps / (1 - rho^2) of the sum of the terms' magnitudes."""
import numpy as np
import pytest
import torch

from paper_2102_00514_gb300 import pes
from tests.gpu_common import to_dev

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


def run(T_list, R, y, prec):
    """Filter with H = 0: R [3][N], y [2][N] (first state of a trajectory not used)."""
    off = np.concatenate([[0], np.cumsum(np.array(T_list) + 1)])
    N, B = int(off[-1]), len(T_list)
    dt = torch.float64 if prec == pes.FP64 else torch.float32
    eye = np.eye(5)
    packed = np.array([eye[i, j] for i in range(5) for j in range(i, 5)])
    lin = dict(F=np.repeat(0.9 * eye.reshape(25, 1), N, 1), c=np.zeros((5, N)), Qp=np.repeat(packed[:, None], N, 1),
               H=np.zeros((10, N)), d=np.zeros((2, N)), Rp=R)
    sm = pes.Smoother(N, B)
    _, _, ll = sm.filter_loglik(prec, {k: to_dev(v, dt) for k, v in lin.items()}, to_dev(y, dt),
                                to_dev(np.zeros((B, 5)), dt), to_dev(np.repeat(packed[None], B, 0), dt),
                                to_dev(off, torch.int64))
    return sm, off, ll


def terms(R, y):
    a, b, c, u, v = (np.asarray(t, dtype=np.longdouble) for t in (R[0], R[1], R[2], y[0], y[1]))
    det = a * c - b * b
    q = (c * u * u - 2 * b * u * v + a * v * v) / det
    log_2pi = np.log(np.longdouble(2) * np.arccos(np.longdouble(-1)))
    return -(q + np.log(det)) / 2 - log_2pi, q + np.abs(np.log(det)) + 2 * log_2pi


@pytest.mark.parametrize("prec", [pes.FP64, pes.FP32])
@pytest.mark.parametrize("scale", [1.0, 1e-15, 1e14])
@pytest.mark.parametrize("one_less_rho2", [1.0, 0.02, 2e-3])
def test_terms_have_fp64_accuracy(prec, scale, one_less_rho2):
    rng = np.random.default_rng(5)
    T_list = [3] * 200 + [1, 700]
    N = sum(T_list) + len(T_list)
    f = np.float32 if prec == pes.FP32 else np.float64
    s0, s1 = scale * np.exp(rng.uniform(-1, 1, (2, N)))
    rho = np.sqrt(1 - one_less_rho2)
    R = np.stack([s0, rho * np.sqrt(s0 * s1), s1]).astype(f).astype(np.float64)
    y = (np.sqrt(scale) * rng.standard_normal((2, N))).astype(f).astype(np.float64)
    sm, off, ll = run(T_list, R, y, prec)
    sm.sync()
    ll = ll.cpu().numpy()
    t, mag = terms(R, y)
    for b in range(len(T_list)):
        k = slice(off[b] + 1, off[b + 1])
        assert abs(ll[b] - t[k].sum()) <= 16 * EPS / one_less_rho2 * mag[k].sum(), b
    sm.close()


def test_products_of_determinants_stay_in_range():
    """Determinants of 1e-200 and 1e200, a thousand of one kind in a row."""
    T = 3000
    s = np.where(np.arange(T + 1) < T // 2, 1e-100, 1e100)
    R, y = np.stack([s, np.zeros(T + 1), s]), np.sqrt(s) * np.ones((2, 1))
    sm, off, ll = run([T], R, y, pes.FP64)
    sm.sync()
    t, mag = terms(R[:, 1:], y[:, 1:])
    assert abs(ll.item() - t.sum()) <= 16 * EPS * mag.sum()
    sm.close()


@pytest.mark.parametrize("prec", [pes.FP64, pes.FP32])
@pytest.mark.parametrize("bad", [[3], [3, 4], [2, 3, 5, 6]])
def test_indefinite_innovation_covariances_give_nan(prec, bad):
    """Also an even number of them in one lane's chunk, whose determinants' product
    is positive; the other trajectories keep their values."""
    T_list = [7] * 256   # 2,048 states: eight steps per lane, a trajectory each
    N = sum(T_list) + len(T_list)
    R = np.stack([np.ones(N), np.zeros(N), np.ones(N)])
    R[2, [8 + k for k in bad]] = -1.0
    y = np.ones((2, N))
    sm, off, ll = run(T_list, R, y, prec)
    with pytest.raises(pes.PesError) as ei:
        sm.sync()
    assert ei.value.status == pes.NOT_PD
    ll = ll.cpu().numpy()
    assert np.isnan(ll[1])
    others = np.delete(ll, 1)
    want = 7 * (-1.0 - np.log(2 * np.pi))
    assert np.abs(others - want).max() < 16 * EPS * 7 * (2.0 + 2 * np.log(2 * np.pi))
    sm.close()
