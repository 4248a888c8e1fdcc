"""The 3D divergence in fixed point (the default) against the FP64 gather (chosen lanes)."""
import numpy as np
import pytest
import torch

from synth import three_d as T

pytestmark = pytest.mark.gpu


def _mesh(shape):
    from paper_2109_01286_gb300 import hfd3d
    nx, ny, nz = shape
    m = T.periodic_tet_box(nx, ny, nz, 10.0, 10.0 * ny / nx, 10.0 * nz / nx, seed=3)
    return m, hfd3d.Mesh3(m)


def _bound(M, U):
    """Rows' bounds on the difference of the two sums: each is off by at most K units of 2^-53 of
    sum |c| |f| (K <= 512 products; the fixed-point factors' roundings, 2^-56 of their scales, are below
    that), with |f| at most 8 times the largest vertex flux of its kind (an edge's states are
    combinations of its stencil's with weights of sum 10/3 at most, its flux their fluxes' mean and
    a dissipation of (|u| + c) / 2 times their difference)."""
    w = U[:5]
    u = w[1:4] / w[0]
    p = 0.4 * (w[4] - 0.5 * (w[1:4] * u).sum(0))
    top = [np.abs(w[1:4]).max(), (np.abs(w[1:4]).max(0) * np.abs(u).max(0) + np.abs(p)).max(),
           ((np.abs(w[4]) + np.abs(p)) * np.abs(u).max(0)).max()]
    top = 8.0 * np.array([top[0], top[1], top[1], top[1], top[2]])
    vp, ep = M.prep_get("vptr"), M.prep_get("eptr")
    cv, ce = np.abs(M.prep_get("cv")).reshape(-1, 4, 3).sum(2), np.abs(M.prep_get("ce")).reshape(-1, 4)
    S = np.add.reduceat(cv, vp[:-1]) + np.add.reduceat(ce, ep[:-1])          # V x 4
    assert (3 * np.diff(vp) + np.diff(ep)).max() <= 512
    return (2 * 512 * 2.0 ** -53) * (S.T[:, None, :] * top[None, :, None]).reshape(20, -1)


@pytest.mark.parametrize("shape,case", [((7, 7, 7), "smooth"), ((7, 9, 8), "smooth"), ((12, 7, 10), "smooth"),
                                        ((7, 9, 8), "spread")])
def test_fixed_point_rows_match_fp64(shape, case):
    m, M = _mesh(shape)
    U = T.vortex_tube(m) if case == "smooth" else T.uniform_state3(m)
    if case == "spread":                 # neighbours' fluxes 2^-40 apart: shifts of more than 32 bits
        U[:, ::3] *= 2.0 ** -40
    Ud = torch.from_numpy(U).cuda()
    R = M.residual(Ud)
    again = M.residual(Ud)
    M.set_lanes(4)
    P = M.residual(Ud)
    torch.cuda.synchronize()
    assert torch.equal(R, again)
    d = (R - P).abs().cpu().numpy()
    assert (d <= _bound(M, U)).all()


def test_coefficients_scaled_by_a_power_of_two_scale_the_residual():
    m, M = _mesh((7, 9, 8))
    Ud = torch.from_numpy(T.vortex_tube(m)).cuda()
    R = M.residual(Ud)
    for k in (-30, 90):
        for name in ("cv", "ce"):
            M.prep_set(name, M.prep_get(name) * 2.0 ** k)
        assert torch.equal(M.residual(Ud), R * 2.0 ** k)
        for name in ("cv", "ce"):
            M.prep_set(name, M.prep_get(name) * 2.0 ** -k)


def test_rows_with_non_finite_fluxes_match_fp64():
    from paper_2109_01286_gb300 import hfd3d
    m, M = _mesh((7, 9, 8))
    U = T.vortex_tube(m)
    U[4, 100] = np.inf
    U[0, 300] = np.nan
    Ud = torch.from_numpy(U).cuda()
    R = M.residual(Ud).cpu()
    with pytest.raises(hfd3d.HfdError):
        M.check()
    M.set_lanes(4)
    P = M.residual(Ud).cpu()
    with pytest.raises(hfd3d.HfdError):
        M.check()
    assert torch.equal(torch.isfinite(R), torch.isfinite(P))
    assert not torch.isfinite(R[:, 100]).all() and torch.isfinite(R).any()
    ok = torch.isfinite(P).numpy()
    U[4, 100] = U[4, 101]
    U[0, 300] = U[0, 301]
    assert (np.abs(R.numpy() - P.numpy())[ok] <= _bound(M, U)[ok]).all()


@pytest.mark.parametrize("shape", [(7, 7, 7), (12, 7, 10)])
@pytest.mark.parametrize("force", [0, 1, 2])
def test_edge_sums_in_fixed_point_match_fp64(shape, force):
    """A weight that is not finite turns the edges' fixed-point sums off for the whole mesh; rows that do
    not read that edge agree.  A sum of 20 products is off by 20 units of 2^-53 of sum |w| |v| < 4 |v| either
    way, a flux by at most 10 times its states: within 2 * 800 units of the row's sum |c| |f|."""
    from paper_2109_01286_gb300 import hfd3d
    nx, ny, nz = shape
    m = T.periodic_tet_box(nx, ny, nz, 10.0, 10.0 * ny / nx, 10.0 * nz / nx, seed=3)
    M = hfd3d.Mesh3(m, force_branch=force)
    U = T.vortex_tube(m)
    Ud = torch.from_numpy(U).cuda()
    R = M.residual(Ud).cpu().numpy()
    M.check()
    w5 = M.prep_get("w5").copy()
    w5.reshape(-1, 40)[5, 7] = np.nan
    M.prep_set("w5", w5)
    P = M.residual(Ud).cpu().numpy()
    torch.cuda.synchronize()
    ep, ei = M.prep_get("eptr"), M.prep_get("eidx")
    far = np.array([5 not in ei[ep[v]:ep[v + 1]] for v in range(U.shape[1])])
    assert far.any() and np.isfinite(P[:, far]).all()
    assert (np.abs(R - P)[:, far] <= 2 * _bound(M, U)[:, far]).all()
