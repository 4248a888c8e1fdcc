"""The 3D edge kernel's sensor (edge3d.cu: eig32, to_char32, weno3_32), emulated on the CPU: Roe state,
eigenvectors, projections and WENO test in FP32 from end states rounded to FP32 and differences formed in
FP64 and rounded once.  An edge is taken as smooth where the test clears a 4e-3 band around both thresholds; all
other components are decided again in FP64, so the one error to look for is a clear decision that FP64 does
not share."""
import numpy as np
import pytest

from oracle import hfd3d as O
from synth import three_d as T

F = np.float32
GUARD = F(4e-3)


def _eig32(wi, wj, n, t1, t2, g1):
    """Rows of L in FP32 (5 x 5 x E), as eig32 and to_char32 form them."""
    def sq(w):
        return w[1] * w[1] + w[2] * w[2] + w[3] * w[3]
    sl, sr = F(1) / np.sqrt(wi[0]), F(1) / np.sqrt(wj[0])
    pl = g1 * (wi[4] - F(0.5) * (sq(wi) * (sl * sl)))
    pr = g1 * (wj[4] - F(0.5) * (sq(wj) * (sr * sr)))
    s = F(1) / (wi[0] * sl + wj[0] * sr)
    u = (wi[1:4] * sl + wj[1:4] * sr) * s
    H = ((wi[4] + pl) * sl + (wj[4] + pr) * sr) * s
    K = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
    ic = F(1) / np.sqrt(g1 * (H - F(0.5) * K))
    dot = lambda a: u[0] * a[0] + u[1] * a[1] + u[2] * a[2]
    qn, q1, q2 = dot(n), dot(t1), dot(t2)
    b1 = g1 * ic * ic
    b2 = F(0.5) * b1 * K

    def to_char(a):
        um = dot(a[1:4])
        nm = (n[0] * a[1] + n[1] * a[2] + n[2] * a[3]) * ic
        qc = qn * ic
        return [F(0.5) * ((b2 + qc) * a[0] - b1 * um - nm + b1 * a[4]),
                (F(1) - b2) * a[0] + b1 * um - b1 * a[4],
                t1[0] * a[1] + t1[1] * a[2] + t1[2] * a[3] - q1 * a[0],
                t2[0] * a[1] + t2[1] * a[2] + t2[2] * a[3] - q2 * a[0],
                F(0.5) * ((b2 - qc) * a[0] - b1 * um + nm + b1 * a[4])]
    return to_char


def _weno_t(u, eps):
    u0, u1, u2, u3, u4 = u
    e1, f1 = u0 - F(2) * u1 + u2, u0 - F(4) * u1 + F(3) * u2
    e2, f2 = u1 - F(2) * u2 + u3, u1 - u3
    e3, f3 = u2 - F(2) * u3 + u4, F(3) * u2 - F(4) * u3 + u4
    s1 = (F(eps) + (F(13.0 / 12.0) * (e1 * e1) + F(0.25) * (f1 * f1))) ** 2
    s2 = (F(eps) + (F(13.0 / 12.0) * (e2 * e2) + F(0.25) * (f2 * f2))) ** 2
    s3 = (F(eps) + (F(13.0 / 12.0) * (e3 * e3) + F(0.25) * (f3 * f3))) ** 2
    t0 = F(0.0625) * (s2 * s3)
    return t0, t0 + F(0.625) * (s1 * s3) + F(0.3125) * (s1 * s2)


@pytest.fixture(scope="module")
def box8():
    m = T.periodic_tet_box(8, 8, 8, 10.0, 10.0, 10.0, seed=3)
    return m, O.prepare(m)


def _state(name, m, P):
    if name == "vortex":
        return T.vortex_tube(m)
    if name == "wave":
        return T.density_wave(m, amp=0.1)
    if name.startswith("mach"):          # smooth waves of all families on a fast stream, in part with jumps
        mach, x, y, z = float(name[4:]), m["x"], m["y"], m["z"]
        rng = np.random.default_rng(int(mach))
        k = 2 * np.pi / 10.0
        wave = lambda: sum(0.1 * np.sin(k * (rng.integers(1, 3) * c) + rng.uniform(0, 6)) for c in (x, y, z))
        rho, p = 1.0 + wave(), 1.0 + wave()
        u = [mach * 1.2 * d + wave() for d in (0.6, -0.5, 0.62)]
        rho, p = np.where(x > 7, 2.0 * rho, rho), np.where(y > 6, 1.5 * p, p)
        U = np.zeros((20, len(x)))
        U[:5] = rho, rho * u[0], rho * u[1], rho * u[2], p / 0.4 + 0.5 * rho * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        return U
    U = T.planar_sod3(m)
    if name == "sod_after_2_steps":
        dt = 0.5 * O.cfl_dt(m, P, U)
        U = O.step(m, P, O.step(m, P, U, dt), dt)
    return U


@pytest.mark.parametrize("state", ["vortex", "wave", "sod", "sod_after_2_steps", "mach1", "mach10", "mach100"])
def test_clear_fp32_decisions_are_those_of_fp64(box8, state):
    m, P = box8
    opts = P.opts
    W = _state(state, m, P)[:, P.stencil]
    wi, wj = W[0:5, :, 2], W[0:5, :, 3]
    vel, H, c = O.roe_average(wi, wj, opts.gamma)
    L, _ = O.eigenvectors(vel, H, c, P.normal, P.t1, P.t2, opts.gamma)
    C64 = np.einsum("eij,jek->eik", L, W[0:5])
    frame = [np.asarray(a).astype(F).T for a in (P.normal, P.t1, P.t2)]
    to_char = _eig32(wi.astype(F), wj.astype(F), *frame, F(opts.gamma - 1.0))
    C32 = np.stack([to_char((W[0:5, :, k] - wi).astype(F)) for k in range(6)], 2)        # 5 x E x 6
    wrong = taken = 0
    for order in ([0, 1, 2, 3, 4], [5, 4, 3, 2, 1]):
        o1, _, _ = O.weno_weights(*[C64[:, :, k] for k in order], opts.weno_eps)
        smooth64 = ((o1 > opts.sens_lo) & (o1 < opts.sens_hi)).T
        with np.errstate(over="ignore", invalid="ignore"):
            t0, S = _weno_t([C32[:, :, k] for k in order], opts.weno_eps)
            clear = np.isfinite(S) & (t0 - F(opts.sens_lo) * S > GUARD * S) & (F(opts.sens_hi) * S - t0 > GUARD * S)
        wrong += int(np.sum(clear & ~smooth64))
        taken += int(np.sum(clear))
    assert wrong == 0 and taken > 0
