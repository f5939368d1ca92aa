"""The work that programs have this library do, as cases that can be timed.

The model is the one of the repository's workloads: a coordinated turn with
bearings from two sensors (dt 0.01, q_c 0.1, q_w 0.01, r_std 0.05). Two
geometries: the "experiment" has its two sensors 2.5 units apart near the start
of the track, which long tracks leave far behind; "stations" stand around the
track, at a distance of its own extent, as a tracker's would. In the experiment's
geometry the iterations amplify rounding by orders of magnitude, so that two
correct runs in single precision differ: there the runs are short ones in FP64,
from the prior. Longer ones, those in single precision and those at the oracle's
tolerance have stations, and start from a nominal near the truth (a previous
window's solution, or the learned initialiser's start) with the few iterations
that such a start needs; one, the final iteration, for a single long trajectory.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2102_00514_gb300 import learned_init, pes

METHODS = {"ieks": pes.IEKS, "cubature": pes.CUBATURE}
PRECISIONS = {"fp64": pes.FP64, "fp32": pes.FP32, "refined": pes.REFINED}
DT, Q_C, Q_W, R_STD = 0.01, 0.1, 0.01, 0.05
SENSORS = (-1.5, 0.5, 1.0, 1.0)
M0 = (0.1, 0.2, 1.0, 0.0, 0.0)
IU = np.triu_indices(5)


def _run(name, method, prec, B, lo, hi, iters, warm, geometry):
    return dict(name=name, kind="run", method=method, prec=prec, B=B, lo=lo, hi=hi, iters=iters, warm=warm, geometry=geometry)


def listed():
    return [
        # the smallest call: a short window re-smoothed as measurements arrive; latency is all there is
        _run("window_T61_ieks_fp32", "ieks", "fp32", 1, 61, 61, 2, True, "stations"),
        # the plain experiment: one trajectory of 500 steps, ten iterations from the prior in double precision
        _run("T500_ieks_fp64", "ieks", "fp64", 1, 500, 500, 10, False, "experiment"),
        # the sigma-point length: one trajectory of 10,000 steps in double precision, from a nominal near the truth
        _run("T10000_cubature_fp64", "cubature", "fp64", 1, 10000, 10000, 5, True, "stations"),
        # a few dozen ragged tracks of at most 400 steps (a tracker's batch)
        _run("tracks64_T1_400_cubature_fp32", "cubature", "fp32", 64, 1, 400, 3, True, "stations"),
        # an offline batch of ragged trajectories, both linearisations
        _run("batch1024_T100_2000_ieks_fp32", "ieks", "fp32", 1024, 100, 2000, 3, True, "stations"),
        _run("batch1024_T100_2000_cubature_fp32", "cubature", "fp32", 1024, 100, 2000, 3, True, "stations"),
        # the batch of long ragged trajectories, at the oracle's tolerance; the largest case
        _run("batch2048_T100_5000_ieks_refined", "ieks", "refined", 2048, 100, 5000, 3, True, "stations"),
        # one long trajectory (the length sweep), the final iteration at the oracle's tolerance, both linearisations
        _run("T1048576_ieks_refined", "ieks", "refined", 1, 1 << 20, 1 << 20, 1, True, "stations"),
        _run("T262147_cubature_refined", "cubature", "refined", 1, 262147, 262147, 1, True, "stations"),
        # one iteration through the layer entry points: linearise, filter (with log-likelihoods), smooth
        dict(name="layers128_T1000_ieks_fp32", kind="layers", method="ieks", prec="fp32", B=128, lo=1000, hi=1000, geometry="stations"),
        # the learned initialiser: the start of a batch, and a training minibatch's gradient
        dict(name="init_forward_B256_T1000_10000", kind="forward", B=256, lo=1000, hi=10000),
        dict(name="init_gradient_B128_T1000", kind="gradient", B=128, lo=1000, hi=1000),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    pick = rng.random()
    if pick < 0.10:
        B = log_int(8, 256)
        lo = log_int(100, 2000)
        return dict(kind=rng.choice(["forward", "gradient"]), B=B, lo=lo, hi=lo + log_int(1, 500))
    method = rng.choice(["ieks", "cubature"])
    if pick < 0.20:
        B, lo = log_int(1, 256), log_int(50, 1000)
        return dict(kind="layers", method=method, prec=rng.choice(["fp32", "fp64"]), B=B, lo=lo, hi=lo + log_int(1, 300), geometry="stations")
    if pick < 0.35:   # double precision: short tracks from the prior, long ones from near the truth
        T = log_int(20, 12000)
        return dict(kind="run", method=method, prec="fp64", B=1, lo=T, hi=T, iters=rng.randint(2, 10), warm=T > 1500,
                    geometry="stations" if T > 1500 else "experiment")
    if pick < 0.55:   # long trajectories at the oracle's tolerance
        T = log_int(20000, 1000000)
        return dict(kind="run", method=method, prec="refined", B=1, lo=T, hi=T, iters=1, warm=True, geometry="stations")
    # batches of ragged trajectories, from single windows to a million states
    B, hi = log_int(1, 1200), log_int(40, 2000)
    return dict(kind="run", method=method, prec=rng.choice(["fp32", "fp32", "refined"]), B=B, lo=max(1, hi // rng.randint(1, 20)),
                hi=hi, iters=rng.randint(1, 3), warm=True, geometry="stations")


def _lengths(case):
    """Measurements per trajectory: fixed by the case, so that every seed has the same sizes."""
    if case["lo"] == case["hi"]:
        return np.full(case["B"], case["lo"], dtype=np.int64)
    return np.random.default_rng(case["B"] * 1000003 + case["hi"]).integers(case["lo"], case["hi"] + 1, case["B"])


def _offsets(case):
    T = _lengths(case)
    off = np.zeros(len(T) + 1, dtype=np.int64)
    off[1:] = np.cumsum(T + 1)
    return off


def _cumsum(v):
    """Running sums of a vector, added in the same order on every run: rows of 1024, then the rows' totals."""
    n, width = v.shape[0], 1024
    if n <= width:
        return torch.cumsum(torch.stack([v, v]), 1)[0]
    rows = torch.nn.functional.pad(torch.view_as_real(v) if v.is_complex() else v[:, None], (0, 0, 0, -n % width))
    rows = torch.cumsum(rows.T.reshape(rows.shape[1], -1, width), 2)
    total = torch.stack([_cumsum(t) for t in rows[:, :, -1]])
    rows[:, 1:] += total[:, :-1, None]
    out = rows.reshape(rows.shape[0], -1)[:, :n]
    return torch.complex(out[0], out[1]) if v.is_complex() else out[0]


def _simulate(case, seed):
    """A ragged batch in float64 on the GPU: truth x [5][N], measurements y [2][N] (0 at a first state), sensors [B][4].

    The model's recursion in closed form: turn rates and turn angles are running sums, the velocity (a complex number)
    is the first one plus the noises turned back to the start, all turned by the angle.
    """
    off = _offsets(case)
    B, N = len(off) - 1, int(off[-1])
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    normal = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.float64)
    offd = torch.as_tensor(off, device="cuda")
    traj = torch.repeat_interleave(torch.arange(B, device="cuda"), offd[1:] - offd[:-1])
    k = torch.arange(N, device="cuda") - offd[traj]
    first = k == 0

    def running(v):
        """Sums within each trajectory, up to and with the entry itself."""
        s = _cumsum(v)
        return s - (s - v)[offd[:-1]][traj]

    x0 = torch.tensor(M0, dtype=torch.float64, device="cuda") + normal(B, 5)
    if B > 1:
        x0[:, 4] = torch.rand(B, generator=g, device="cuda", dtype=torch.float64) * 2 - 1
    zero = torch.zeros((), dtype=torch.float64, device="cuda")
    w = running(torch.where(first, x0[traj, 4], math.sqrt(Q_W * DT) * normal(N)))
    wprev = torch.where(first, zero, w.roll(1))
    theta = running(wprev * DT)
    turn = torch.polar(torch.ones_like(theta), theta)
    noise = torch.complex(normal(N), normal(N)) * math.sqrt(Q_C * DT)
    v0 = torch.complex(x0[:, 2], x0[:, 3])
    v = turn * running(torch.where(first, v0[traj], turn.conj() * noise))
    half = 0.5 * wprev * DT
    inc = v.roll(1) * torch.polar(DT * torch.sinc(half / math.pi), half)
    p = running(torch.where(first, torch.complex(x0[:, 0], x0[:, 1])[traj], inc))
    x = torch.stack([p.real, p.imag, v.real, v.imag, w])
    sensors = torch.tensor(SENSORS, dtype=torch.float64, device="cuda").repeat(B, 1)
    if case.get("geometry") == "stations":
        centre = (running(p)[offd[1:] - 1]) / (offd[1:] - offd[:-1])
        extent = torch.zeros(B, dtype=torch.float64, device="cuda").scatter_reduce_(0, traj, (p - centre[traj]).abs(), "amax")
        side = torch.rand(2, B, generator=g, device="cuda", dtype=torch.float64)
        for i, angle in enumerate((6.3 * side[0], 6.3 * side[0] + 1.2 + side[1])):
            at = torch.view_as_real(centre + torch.polar(10.0 + 1.5 * extent, angle))
            sensors[:, 2 * i], sensors[:, 2 * i + 1] = at[:, 0], at[:, 1]
    elif B > 1:
        sensors = sensors + 0.4 * (torch.rand(B, 4, generator=g, device="cuda", dtype=torch.float64) - 0.5)
    y = _bearings(x, sensors[traj]) + R_STD * normal(2, N)
    y[:, first] = 0.0
    return dict(off=offd, traj=traj, k=k, x=x, y=y, sensors=sensors, normal=normal)


def _bearings(x, s):
    return torch.stack([torch.atan2(x[1] - s[:, 1], x[0] - s[:, 0]), torch.atan2(x[1] - s[:, 3], x[0] - s[:, 2])])


def _nominal(w):
    """A nominal near the truth: its error varies slowly along a trajectory, as a smoother's does; and its covariance."""
    B = w["sensors"].shape[0]
    a = w["normal"](2, 5, B)[:, :, w["traj"]] * torch.tensor([[0.05], [0.05], [0.05], [0.05], [0.02]], dtype=torch.float64, device="cuda")
    ph = w["k"] * DT
    x = w["x"] + a[0] * torch.cos(0.7 * ph) + a[1] * torch.sin(0.3 * ph)
    root = torch.diag(torch.tensor([0.12, 0.12, 0.15, 0.15, 0.08], dtype=torch.float64, device="cuda"))
    root = root @ (torch.eye(5, dtype=torch.float64, device="cuda") + 0.3 * torch.tril(w["normal"](5, 5), -1))
    P = root @ root.T
    size = 1.0 + 0.3 * torch.sin(0.5 * ph)
    return x, P[IU[0], IU[1]][:, None] * size


def _inputs(case, seed):
    """The arrays of a call, in the precision it takes them."""
    w = _simulate(case, seed)
    dt = torch.float64 if case.get("prec") == "fp64" else torch.float32
    B = case["B"]
    d = dict(off=w["off"], y=w["y"].to(dt).contiguous(), sensors=w["sensors"],
             m0=torch.tensor(M0, dtype=dt, device="cuda").repeat(B, 1), P0=torch.eye(5, dtype=dt, device="cuda")[IU[0], IU[1]].repeat(B, 1),
             x=None, P=None, truth=w["x"].to(dt).contiguous())
    if case.get("warm") or case["kind"] == "layers":
        x, P = _nominal(w)
        d["x"], d["P"] = x.to(dt).contiguous(), P.to(dt).contiguous()
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    N = d["y"].shape[1]
    if case["kind"] in ("forward", "gradient"):
        net = pes.InitNet(N, case["B"])
        net.set_params(learned_init.initial_params(int(seed)), np.array(M0), np.array([2.0, 2.0, 1.0, 1.0, 0.5]))
        return dict(case=case, net=net, **d)
    model = pes.Model(dt=DT, q_c=Q_C, q_w=Q_W, r_std=R_STD, sensors=d["sensors"])
    return dict(case=case, sm=pes.Smoother(N, case["B"]), model=model, **d)


def run(s):
    case = s["case"]
    if case["kind"] == "forward":
        return s["net"].forward(pes.FP32, s["y"], s["off"])
    if case["kind"] == "gradient":
        loss, grad = s["net"].loss_grad(pes.FP32, s["y"], s["off"], s["truth"])
        return [loss, grad]
    method, prec = METHODS[case["method"]], PRECISIONS[case["prec"]]
    if case["kind"] == "layers":
        lin = s["sm"].linearize(s["model"], method, prec, s["x"], s["P"], s["y"], s["off"])
        xf, Pf, ll = s["sm"].filter_loglik(prec, lin, lin["y_used"], s["m0"], s["P0"], s["off"])
        xs, Ps = s["sm"].smooth_scan(prec, lin, xf, Pf, s["off"])
        return [lin, xf, Pf, ll, xs, Ps]
    x, P, _, _ = s["sm"].ieks_run(s["model"], method, prec, s["y"], s["off"], s["m0"], s["P0"], x_init=s["x"],
                                  P_init=s["P"] if case["method"] == "cubature" else None, iters=case["iters"])
    return [x, P]


# Multiply-adds of one state and iteration: linearisation, filter (predict, update), smoother (gain, element, step).
LINEARISE = {"ieks": 100, "cubature": 700}
SMOOTH = 110 + 95 + 260 + 225
NET_MACS = 5 * 6 * 64 + 3 * 5 * 64 * 64 + 64 * 64 + 64 * 5   # four convolutions of five taps and the head, per state


def work(case):
    off = _offsets(case)
    B, N = len(off) - 1, int(off[-1])
    if case["kind"] == "forward":
        return {"bytes": 4 * 7 * N + 8 * (B + 1), "flops": 2 * NET_MACS * N}
    if case["kind"] == "gradient":
        return {"bytes": 4 * 7 * N + 8 * (B + 1) + 2 * 4 * pes.INIT_NPARAMS, "flops": 6 * NET_MACS * N}
    size = 8 if case["prec"] == "fp64" else 4
    flops = 2 * (LINEARISE[case["method"]] + SMOOTH) * N
    fixed = size * 20 * B + 8 * (B + 1) + 32 * B
    if case["kind"] == "layers":
        # nominal and measurements in; the linearisation (62 values), filtered and smoothed moments out
        return {"bytes": size * N * (22 + 62 + 20 + 20) + fixed + 8 * B, "flops": flops}
    nominal = (20 if case["method"] == "cubature" else 5) if case["warm"] else 0
    return {"bytes": size * N * (2 + nominal + 20) + fixed, "flops": flops * case["iters"]}


# ---- the same results in 64 bits, with torch alone --------------------------------------


def _sym(p):
    """Packed [15][N] (or [3][N]) to full [N][n][n]."""
    n = 5 if p.shape[0] == 15 else 2
    M = torch.zeros(p.shape[1], n, n, dtype=torch.float64, device=p.device)
    i, j = np.triu_indices(n)
    M[:, i, j] = p.T
    M[:, j, i] = p.T
    return M


def _pack(M):
    i, j = np.triu_indices(M.shape[-1])
    return M[:, i, j].T.contiguous()


def _turn(x):
    """The transition f of [..., 5] states."""
    a = x[..., 4] * DT
    half = 0.5 * a
    A = torch.polar(DT * torch.sinc(half / math.pi), half)
    v = torch.complex(x[..., 2], x[..., 3])
    p = torch.complex(x[..., 0], x[..., 1]) + A * v
    v = torch.polar(torch.ones_like(a), a) * v
    return torch.stack([p.real, p.imag, v.real, v.imag, x[..., 4]], -1)


def _turn_jacobian(x):
    a, w = x[:, 4] * DT, x[:, 4]
    half = 0.5 * a
    A = torch.polar(DT * torch.sinc(half / math.pi), half)
    rot = torch.polar(torch.ones_like(a), a)
    # d/dw of (exp(i w dt) - 1) / (i w), its series in a where that cancels
    near = a.abs() < 0.02
    ws = torch.where(near, torch.ones_like(w), w)
    far_d = (rot * DT - A) / ws
    series = torch.zeros_like(A)
    term = torch.full_like(A, 1.0)
    for n in range(2, 12):   # sum over n of i^{n-1} (n-1) a^{n-2} / n!  dt^2
        series = series + (1j ** (n - 1)) * (n - 1) / math.factorial(n) * term
        term = term * a
    dA = torch.where(near, series * DT * DT, far_d)
    v = torch.complex(x[:, 2], x[:, 3])
    F = torch.zeros(x.shape[0], 5, 5, dtype=torch.float64, device=x.device)
    F[:, 0, 0] = F[:, 1, 1] = F[:, 4, 4] = 1.0
    for r, c in ((0, A), (2, rot)):
        F[:, r, 2], F[:, r, 3], F[:, r + 1, 2], F[:, r + 1, 3] = c.real, -c.imag, c.imag, c.real
    F[:, 0, 4], F[:, 1, 4] = (dA * v).real, (dA * v).imag
    dv = 1j * DT * rot * v
    F[:, 2, 4], F[:, 3, 4] = dv.real, dv.imag
    return F


def _nearest(angle, reference):
    return angle - 2 * math.pi * torch.round((angle - reference) / (2 * math.pi))


def _linearise(method, x, P, y, s):
    """F, c, Q', H, d, R' and the unwrapped measurement of every state (x [N][5], P [N][5][5], y [2][N], s [N][4])."""
    N = x.shape[0]
    Q = torch.diag(torch.tensor([0, 0, Q_C * DT, Q_C * DT, Q_W * DT], dtype=torch.float64, device=x.device))
    R = R_STD ** 2 * torch.eye(2, dtype=torch.float64, device=x.device)
    hx = _bearings(x.T, s).T
    yu = _nearest(y.T, hx)
    if method == "ieks":
        F = _turn_jacobian(x)
        fx = _turn(x)
        H = torch.zeros(N, 2, 5, dtype=torch.float64, device=x.device)
        for r in range(2):
            dx, dy = x[:, 0] - s[:, 2 * r], x[:, 1] - s[:, 2 * r + 1]
            H[:, r, 0], H[:, r, 1] = -dy / (dx * dx + dy * dy), dx / (dx * dx + dy * dy)
        Qp, Rp, zy = Q.expand(N, 5, 5), R.expand(N, 2, 2), hx
    else:
        L = torch.linalg.cholesky(P) * math.sqrt(5.0)
        pts = torch.cat([x[:, None, :] + L.transpose(1, 2), x[:, None, :] - L.transpose(1, 2)], 1)
        zf = _turn(pts)
        flat = pts.reshape(-1, 5)
        zh = _nearest(_bearings(flat.T, s.repeat_interleave(10, 0)).T, hx.repeat_interleave(10, 0)).reshape(N, 10, 2)
        dev = pts - x[:, None, :]

        def regress(z):
            mean = z.mean(1)
            dz = z - mean[:, None, :]
            slope = torch.linalg.solve(P, dev.transpose(1, 2) @ dz / 10).transpose(1, 2)
            rest = dz - dev @ slope.transpose(1, 2)
            return mean, slope, rest.transpose(1, 2) @ rest / 10

        fx, F, lam = regress(zf)
        zy, H, om = regress(zh)
        Qp, Rp = Q + lam, R + om
    c = fx - (F @ x[:, :, None])[:, :, 0]
    d = zy - (H @ x[:, :, None])[:, :, 0]
    return F, c, Qp, H, d, Rp, yu


def _scan(op, e):
    """Inclusive scan of the elements (tuples of [n][...] tensors) under op(earlier, later)."""
    n = e[0].shape[0]
    if n == 1:
        return e
    m = n // 2
    pair = op(tuple(t[0:2 * m:2] for t in e), tuple(t[1:2 * m:2] for t in e))
    odd = _scan(op, pair)
    rest = (n - 1) // 2
    even = op(tuple(t[:rest] for t in odd), tuple(t[2:2 * rest + 1:2] for t in e)) if rest else None
    out = []
    for i, t in enumerate(e):
        o = torch.empty_like(t)
        o[1::2] = odd[i]
        o[0] = t[0]
        if rest:
            o[2:2 * rest + 1:2] = even[i]
        out.append(o)
    return tuple(out)


def _mv(A, x):
    return (A @ x[..., None])[..., 0]


def _T(A):
    return A.transpose(-1, -2)


def _filter_op(a, b):
    A1, b1, C1, e1, J1 = a
    A2, b2, C2, e2, J2 = b
    eye = torch.eye(5, dtype=torch.float64, device=A1.device)
    M = _T(torch.linalg.solve(_T(eye + C1 @ J2), _T(A2)))          # A2 (I + C1 J2)^-1
    W = _T(torch.linalg.solve(_T(eye + J2 @ C1), A1))               # A1' (I + J2 C1)^-1
    C = M @ C1 @ _T(A2) + C2
    J = W @ J2 @ A1 + J1
    return (M @ A1, _mv(M, b1 + _mv(C1, e2)) + b2, 0.5 * (C + _T(C)), _mv(W, e2 - _mv(J2, b1)) + e1, 0.5 * (J + _T(J)))


def _smooth_op(later, earlier):
    E2, g2, L2 = later
    E1, g1, L1 = earlier
    L = E1 @ L2 @ _T(E1) + L1
    return E1 @ E2, _mv(E1, g2) + g1, 0.5 * (L + _T(L))


def _filter(lin, y, off, traj, m0, P0):
    """Filtered moments and per-trajectory log-likelihoods."""
    F, c, Q, H, d, R = lin
    first = torch.zeros(y.shape[0], dtype=torch.bool, device=y.device)
    first[off[:-1]] = True
    eye = torch.eye(5, dtype=torch.float64, device=y.device)
    Fp, cp, Qp = F.roll(1, 0), c.roll(1, 0), Q.roll(1, 0)
    S = H @ Qp @ _T(H) + R
    S = torch.where(first[:, None, None], torch.eye(2, dtype=torch.float64, device=y.device), S)
    K = _T(torch.linalg.solve(S, H @ Qp))
    v = y - _mv(H, cp) - d
    A = (eye - K @ H) @ Fp
    HF = H @ Fp
    SiHF = torch.linalg.solve(S, HF)
    b, C = cp + _mv(K, v), (eye - K @ H) @ Qp
    eta, J = _mv(_T(SiHF), v), _T(HF) @ SiHF
    A[first], b[first], C[first], eta[first], J[first] = 0.0, m0, P0, 0.0, 0.0
    C, J = 0.5 * (C + _T(C)), 0.5 * (J + _T(J))
    _, m, P, _, _ = _scan(_filter_op, (A, b, C, eta, J))
    P = 0.5 * (P + _T(P))
    mp, Pp = _mv(Fp, m.roll(1, 0)) + cp, Fp @ P.roll(1, 0) @ _T(Fp) + Qp
    S = H @ Pp @ _T(H) + R
    S = torch.where(first[:, None, None], torch.eye(2, dtype=torch.float64, device=y.device), S)
    v = y - _mv(H, mp) - d
    term = -0.5 * ((v * torch.linalg.solve(S, v)).sum(1) + torch.logdet(S)) - math.log(2 * math.pi)
    term[first] = 0.0
    ll = torch.zeros(len(off) - 1, dtype=torch.float64, device=y.device).index_add_(0, traj, term)
    return m, P, ll


def _smooth(lin, m, P, off):
    F, c, Q = lin[:3]
    last = off[1:] - 1
    Fs, Qs = F.clone(), Q.clone()
    Fs[last] = 0.0
    Qs[last] = torch.eye(5, dtype=torch.float64, device=F.device)
    FP = Fs @ P
    Pp = FP @ _T(Fs) + Qs
    E = _T(torch.linalg.solve(0.5 * (Pp + _T(Pp)), FP))
    g = m - _mv(E, _mv(Fs, m) + c)
    L = P - E @ Pp @ _T(E)
    L = 0.5 * (L + _T(L))
    flip = lambda t: t.flip(0)
    _, g, L = _scan(_smooth_op, (flip(E), flip(g), flip(L)))
    return flip(g), flip(L)


def exact(case, seed):
    if case["kind"] in ("forward", "gradient"):
        return None   # bfloat16 activations by design: the rounding between the layers is part of the result
    d = _inputs(case, seed)
    off, B = d["off"], case["B"]
    traj = torch.repeat_interleave(torch.arange(B, device="cuda"), off[1:] - off[:-1])
    y = d["y"].double()
    s = d["sensors"][traj]
    m0, P0 = d["m0"].double(), _sym(d["P0"].double().T)
    x = d["x"].double().T if d["x"] is not None else m0[traj]
    P = _sym(d["P"].double()) if d["P"] is not None else P0[traj]
    for _ in range(case.get("iters", 1)):
        F, c, Q, H, dd, R, yu = _linearise(case["method"], x, P, y, s)
        lin = (F, c, Q, H, dd, R)
        m, Pf, ll = _filter(lin, yu, off, traj, m0, P0)
        x, P = _smooth(lin, m, Pf, off)
    if case["kind"] == "run":
        return [x.T.contiguous(), _pack(P)]
    first, last = off[:-1], off[1:] - 1
    out = {"F": F.reshape(-1, 25).T, "c": c.T, "Qp": _pack(Q), "H": H.reshape(-1, 10).T, "d": dd.T, "Rp": _pack(R), "y_used": yu.T}
    out = {k: v.contiguous().clone() for k, v in out.items()}
    for k in ("F", "c", "Qp"):
        out[k][:, last] = 0.0
    for k in ("H", "d", "Rp", "y_used"):
        out[k][:, first] = 0.0
    return [out, m.T.contiguous(), _pack(Pf), ll, x.T.contiguous(), _pack(P)]
