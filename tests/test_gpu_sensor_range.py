"""The FP32 sensor of the FP64 edge kernels on states in units that FP32 does not hold."""
import numpy as np
import pytest

import synth
from synth import three_d as T

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _scaled(U, n, k):
    """The state in units of velocity 2^-k: exact in FP64, and the decisions of the acoustic and entropy
    components, whose characteristic values are densities, stay the same."""
    V = U.copy()
    for d in range(U.shape[0] // n):
        V[n * d + 1:n * d + n - 1] *= 2.0 ** k
        V[n * d + n - 1] *= 4.0 ** k
    return V


def _jumps(x, y, moving):
    """Jumps of density, velocity and pressure in boxes: 3-node branches for waves of every family."""
    rho = np.where(np.abs(x - 4.0) < 1.5, 1.0, 0.7)
    u = np.where(np.abs(y - 5.0) < 2.0, 0.6, 0.0) * moving
    p = np.where(np.abs(x + y - 10.0) < 2.5, 1.0, 0.8)
    return rho, u, p


@pytest.mark.parametrize("moving,k", [(1, -40), (1, -50), (1, -56), (0, 62), (0, 66), (0, 100)])
@pytest.mark.parametrize("nx", [40, 60])          # 4,800 and 10,800 edges: both edge kernels
def test_branches_do_not_depend_on_the_unit_of_velocity(nx, moving, k):
    import paper_2109_01286_gb300 as pkg
    m = synth.jittered_grid(nx, nx, 10.0, 10.0, seed=1)
    rho, u, p = _jumps(m["x"], m["y"], moving)
    U = np.zeros((12, len(rho)))
    U[0], U[1], U[2], U[3] = rho, rho * u, -0.5 * rho * u, p / 0.4 + 0.625 * rho * u * u
    mesh = pkg.Mesh(m)
    got = [mesh.edge_branches(mesh.import_state(torch.from_numpy(V).cuda())) & 0xbb for V in (U, _scaled(U, 4, k))]
    assert (got[0] != 0).sum() > 100
    assert np.array_equal(*got)


@pytest.mark.parametrize("moving,k", [(1, -40), (1, -50), (1, -56), (0, 62), (0, 66), (0, 100)])
def test_3d_fluxes_follow_the_unit_of_velocity(moving, k):
    """A weight that is not finite on one edge sends the mesh's sums and the sensor's inputs to FP64: rows
    that do not read that edge take the same branches and agree to the sums' rounding, 1e-11 of the rows
    of their kind (20 products, cancellation up to 1e4)."""
    from paper_2109_01286_gb300 import hfd3d
    m = T.periodic_tet_box(9, 8, 7, 10.0, 10.0, 10.0, seed=3)
    rho, u, p = _jumps(m["x"], m["y"], moving)
    U = np.zeros((20, len(rho)))
    U[0], U[1], U[2], U[4] = rho, rho * u, -0.5 * rho * u, p / 0.4 + 0.625 * rho * u * u
    M = hfd3d.Mesh3(m)
    Ud = torch.from_numpy(_scaled(U, 5, k)).cuda()
    R = M.residual(Ud).cpu().numpy()
    w5 = M.prep_get("w5").copy()
    w5.reshape(-1, 40)[5, 7] = np.nan
    M.prep_set("w5", w5)
    P = M.residual(Ud).cpu().numpy()
    torch.cuda.synchronize()
    ep, ei = M.prep_get("eptr"), M.prep_get("eidx")
    far = np.array([5 not in ei[ep[v]:ep[v + 1]] for v in range(U.shape[1])])
    assert far.any() and np.isfinite(P[:, far]).all()
    for r in range(20):
        top = np.abs(P[r - r % 5 + (1 if r % 5 in (1, 2, 3) else r % 5):, far][:3 if r % 5 in (1, 2, 3) else 1]).max()
        assert (np.abs(R[r] - P[r])[far] <= 1e-11 * top).all(), r
