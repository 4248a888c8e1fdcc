"""GPU tests of the FP64 divergence in fixed point (div_fixed.cu) against the plain FP64 divergence,
which the persistent stage kernel runs: one RK3 step of the same state on the same mesh."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

VISC = dict(viscous=True, mu=0.01, prandtl=0.72, R_gas=1.0 / (1.4 * 0.01))


def _pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2109_01286_gb300 as pkg
    return pkg


def _irregular(n, seed):
    """A periodic Delaunay mesh of strongly jittered points: rows of more than 127 products."""
    from scipy.spatial import Delaunay
    rng = np.random.default_rng(seed)
    gx, gy = np.meshgrid(np.arange(n) / n, np.arange(n) / n)
    x = (gx.ravel() + rng.uniform(-0.6, 0.6, n * n) / n) % 1
    y = (gy.ravel() + rng.uniform(-0.6, 0.6, n * n) / n) % 1
    P = np.concatenate([np.stack([x + i, y + j], 1) for i in (-1, 0, 1) for j in (-1, 0, 1)])
    t = Delaunay(P).simplices
    c = P[t].mean(1)
    t = t[(c >= 0).all(1) & (c < 1).all(1)]
    d1, d2 = P[t[:, 1]] - P[t[:, 0]], P[t[:, 2]] - P[t[:, 0]]
    neg = d1[:, 0] * d2[:, 1] - d1[:, 1] * d2[:, 0] < 0
    t[neg] = t[neg][:, [0, 2, 1]]
    return {"x": 10 * x, "y": 10 * y, "tri": (t % (n * n)).astype(np.int32), "Lx": 10.0, "Ly": 10.0,
            "periodic_x": True, "periodic_y": True}


def _case(name):
    if name == "irregular":
        m = _irregular(20, 2)
        return m, synth.isentropic_vortex(m, beta=2.0), {}
    if name == "quad":
        m = synth.jittered_box_with_ghosts(37, 29, (0.0, 1.0), (0.0, 1.0), 5, seed=2)
        return m, synth.four_quadrant(m), {}
    if name == "tgv":
        m = synth.jittered_grid(19, 23, 2 * np.pi, 2 * np.pi, seed=3)
        return m, synth.taylor_green(m), VISC
    nx, ny = {"torus3": (3, 3), "row_edge": (17, 16), "tiles16": (150, 137)}[name]
    m = synth.jittered_grid(nx, ny, 10.0, 10.0, seed=1)
    return m, synth.isentropic_vortex(m), {}


@pytest.mark.parametrize("name", ["torus3", "row_edge", "tiles16", "quad", "tgv", "irregular"])
def test_fixed_point_step_equals_plain_fp64(name):
    """Partial tiles (rows not a multiple of 8 or 16), both tile sizes, viscous rows, zeros beside
    nonzero fluxes, rows of more than 127 products (28-bit limbs).  A row's FP64 sum of up to 150
    products rounds by at most 150 x 2^-53 of its largest partial sum, and the rows' terms cancel by up
    to 1e3 (1e4 at Mach 0.1): the increments agree to 1.7e-14 x 1e3 (1e4)."""
    pkg = _pkg()
    m, U, kw = _case(name)
    mesh = pkg.Mesh(m, **kw)
    U0 = mesh.import_state(torch.from_numpy(U).cuda())
    dt, out = 1e-3, {}
    for persistent in (False, True):
        mesh.set_launch(persistent, 0)
        out[persistent] = mesh.step(U0.clone(), dt)
    mesh.check()
    a, b = out[False] - U0, out[True] - U0
    tol = 2e-10 if name == "tgv" else 2e-11
    for rows in (slice(0, 4), slice(4, 8), slice(8, 12)):
        assert torch.linalg.norm(a[rows] - b[rows]) <= tol * torch.linalg.norm(b[rows])
    R = {}
    mesh.set_launch(False, 0)
    for lanes in (4, 8):                    # the sums are exact: lane counts agree bit for bit
        mesh.set_lanes(lanes)
        R[lanes] = mesh.residual(U0.clone())
    assert torch.equal(R[4], R[8])


def test_fixed_point_divergence_follows_the_scale_of_the_state():
    """The Euler fluxes are homogeneous of degree one and even powers of two are exact (the Roe
    average takes square roots of the density): with the branch fixed, R(2^k U) = 2^k R(U) bit for bit
    (exponents up to those where energies squared still fit)."""
    pkg = _pkg()
    m = synth.jittered_grid(17, 16, 10.0, 10.0, seed=1)
    mesh = pkg.Mesh(m, force_branch="hermite")
    U = mesh.import_state(torch.from_numpy(synth.isentropic_vortex(m)).cuda())
    R = mesh.residual(U.clone())
    for k in (-400, -40, 4, 40, 400):
        assert torch.equal(mesh.residual(U * 2.0 ** k), R * 2.0 ** k), k


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_nonfinite_fluxes_reach_the_same_rows(value):
    """A non-finite state: the rows that read it are evaluated in FP64, and the step has NaN and
    infinities where the plain divergence has them."""
    pkg = _pkg()
    m = synth.jittered_grid(17, 16, 10.0, 10.0, seed=1)
    mesh = pkg.Mesh(m)
    U0 = mesh.import_state(torch.from_numpy(synth.isentropic_vortex(m)).cuda())
    U0[3, 40] = value
    out = {}
    for persistent in (False, True):
        mesh.set_launch(persistent, 0)
        out[persistent] = mesh.step(U0.clone(), 1e-4)
    a, b = out[False], out[True]
    assert torch.equal(torch.isnan(a), torch.isnan(b))
    assert torch.equal(torch.isposinf(a), torch.isposinf(b)) and torch.equal(torch.isneginf(a), torch.isneginf(b))
    assert not torch.isfinite(b).all() and torch.isfinite(b).any()
    with pytest.raises(pkg.HfdError):
        mesh.check()


def test_edge_kernels_of_small_and_large_meshes_give_the_same_bits():
    """A mesh of few edges gives every edge 8 lanes; a batch of copies has one thread an edge and lists
    the edges with a 3-node component.  Sums are exact and the rest is the same code: equal bits."""
    pkg = _pkg()
    m = synth.jittered_grid(40, 33, 4.0, 3.3, seed=1)          # 3,960 edges; shocked part of the box
    U = synth.isentropic_vortex(m, center=(2.0, 1.6))
    U[:4, np.hypot(m["x"] - 1.0, m["y"] - 1.0) < 0.6] *= 2.0
    prep = pkg.Prep(m)
    one, many = prep.upload(), pkg.Prep.concat([prep] * 4).upload()
    a = one.import_state(torch.from_numpy(U).cuda())
    b = many.import_state(torch.from_numpy(np.concatenate([U] * 4, 1)).cuda())
    assert one.edge_branches(a.clone()).any() and not one.edge_branches(a.clone()).all()
    Ra = one.export_state(one.residual(a))
    Rb = many.export_state(many.residual(b))
    for k in range(4):
        assert torch.equal(Rb[:, k * len(m["x"]):(k + 1) * len(m["x"])], Ra)
