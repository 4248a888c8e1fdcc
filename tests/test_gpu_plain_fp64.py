"""FP64 meshes whose rows have no fixed-point form: the plain FP64 kernels, chosen by the mesh and not by the
caller."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

VISC = dict(viscous=True, mu=0.01, prandtl=0.72, R_gas=1.0 / (1.4 * 0.01))
K = 600                                            # the exponent field of the fixed-point rows ends at 500


def _pair(nx, kind):
    """A mesh and the same with its divergence coefficients times 2^K (exact), and a state."""
    import paper_2109_01286_gb300 as pkg
    if kind == "tgv":
        m = synth.jittered_grid(nx, nx, 2 * np.pi, 2 * np.pi, seed=3)
        kw, U = VISC, synth.taylor_green(m)
    else:
        m = synth.jittered_grid(nx, nx, 10.0, 10.0, seed=1)
        kw, U = {}, synth.isentropic_vortex(m)
        U[:4, np.hypot(m["x"] - 3.0, m["y"] - 3.0) < 1.5] *= 1.5
    a, b = pkg.Prep(m, **kw), pkg.Prep(m, **kw)
    for name in ("div_coef", "visc_coef") if kw else ("div_coef",):
        b.set(name, a.get(name) * 2.0 ** K)
    return m, kw, U, a.upload(), b.upload()


def _l2(a, b):
    return max((torch.linalg.norm(a[g] - b[g]) / torch.linalg.norm(b[g])).item()
               for g in (slice(0, 4), slice(4, 8), slice(8, 12)))


@pytest.mark.parametrize("kind", ["vortex", "tgv"])
@pytest.mark.parametrize("nx", [24, 60])           # 1,728 edges: 8 lanes an edge; 10,800: one thread
def test_rows_without_a_fixed_point_form_take_fp64_sums(nx, kind):
    """Powers of two scale FP64 sums exactly: lanes 1 and 2 give the bits of the unscaled mesh with those
    lanes, 4 and 8 sums in orders of their own (110 products, sqrt(110) x 2^-53 of terms that cancel by up
    to 1e3, 1e4 at Mach 0.1, as between lane counts 1 and 2)."""
    m, kw, U, a, b = _pair(nx, kind)
    Ui = a.import_state(torch.from_numpy(U).cuda())
    ref = {}
    for lanes in (1, 2, 4):
        a.set_lanes(lanes)
        ref[lanes] = a.residual(Ui.clone())
    scale = 2.0 ** -K
    assert torch.equal(b.residual(Ui.clone()) * scale, ref[1])          # the default of such a mesh: 1 lane
    R = {}
    for lanes in (1, 2, 4, 8):
        b.set_lanes(lanes)
        R[lanes] = b.residual(Ui.clone()) * scale
        S = torch.empty_like(Ui)
        b.residual_static(Ui.clone(), S)
        assert torch.equal(S * scale, R[lanes])
    b.check()
    assert torch.equal(R[1], ref[1]) and torch.equal(R[2], ref[2])
    assert not torch.equal(R[4], R[8]) and not torch.equal(R[4], ref[4])
    for lanes in (4, 8):
        assert _l2(R[lanes], ref[1]) < (1.3e-11 if kw else 1.3e-12)
    P = oracle.prepare(m, oracle.Options(**kw) if kw else None)
    want = torch.from_numpy(oracle.residual(m, P, U.copy())[:, a.perm]).cuda()
    assert (torch.linalg.norm(R[8] - want) / torch.linalg.norm(want)).item() < 1e-7


@pytest.mark.parametrize("kind", ["vortex", "tgv"])
def test_steps_and_adjoint_of_such_meshes(kind):
    """A step and its adjoint with dt times 2^-K: the bits of the unscaled mesh with 1 lane."""
    m, kw, U, a, b = _pair(24, kind)
    a.set_lanes(1)
    Ui = a.import_state(torch.from_numpy(U).cuda())
    dt = 1e-3
    assert torch.equal(a.step(Ui.clone(), dt), b.step(Ui.clone(), dt * 2.0 ** -K))
    lam = torch.randn(Ui.shape, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    assert torch.equal(a.adjoint(Ui, lam, dt=dt), b.adjoint(Ui, lam, dt=dt * 2.0 ** -K))
