"""5-node sums of the FP64 edges whose two sides lie orders of magnitude apart."""
import numpy as np
import pytest

import synth
from synth import three_d as T

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rows(vptr, vidx, eptr, eidx, stencil, K):
    """Rows that read no flux at vertex K and no edge with K among the four nodes of both sides, but an edge
    with K as the far node of one side."""
    out = []
    for r in range(len(vptr) - 1):
        if K in vidx[vptr[r]:vptr[r + 1]]:
            continue
        s = stencil[eidx[eptr[r]:eptr[r + 1]]]
        if not (s[:, 1:5] == K).any() and (s[:, [0, 5]] == K).any():
            out.append(r)
    return np.array(out)


# One vertex 2^30 above the others (the same velocity and temperature): an edge with it as far node takes 3-node
# values without it on that side, whose weights at the vertex are below 1e-30, and 5-node sums of five
# ordinary nodes on the other.  Rows that read only such edges are sums of up to 110 (2D) or 512 (3D) products
# of ordinary values, off by that many units of 2^-53 of terms that cancel by up to 1e2 here; their norms see
# the root of the number: 23 x 1.1e-16 x 1e2 < 1e-12 over all groups.  A side held at the far node's scale
# has an error of 2^-57 x 2^30 = 7e-9.
TOL = 1e-12


@pytest.mark.parametrize("nx", [40, 60])          # 4,800 edges: 8 lanes an edge; 10,800: one thread
@pytest.mark.parametrize("ratio", [2.0 ** 10, 2.0 ** 30])
def test_a_side_does_not_lose_bits_to_the_other_sides_far_node(nx, ratio):
    import paper_2109_01286_gb300 as pkg
    m = synth.jittered_grid(nx, nx, 10.0, 10.0, seed=1)
    U = synth.isentropic_vortex(m)
    prep = pkg.Prep(m)
    pos = np.full(len(prep.get("edges")) // 2, -1)
    pos[prep.get("flux_edges")] = np.arange(len(prep.get("flux_edges")))
    K = int(np.argmin(np.hypot(m["x"] - 4.0, m["y"] - 4.5)))
    rows = _rows(prep.get("div_vptr"), prep.get("div_vidx"), prep.get("div_eptr"), pos[prep.get("div_eidx")],
                 prep.get("stencil").reshape(-1, 6), K)
    rows = prep.get("active")[rows]
    assert len(rows) >= 4
    U[:, K] *= ratio
    mesh = pkg.Mesh(prep=prep)
    Ui = mesh.import_state(torch.from_numpy(U).cuda())
    R = {}
    for lanes in (8, 1):                           # the default's fixed-point sums and FP64 sums
        mesh.set_lanes(lanes)
        R[lanes] = mesh.export_state(mesh.residual(Ui.clone()))[:, rows]
    mesh.check()
    for g in (slice(0, 4), slice(4, 8), slice(8, 12)):
        assert torch.linalg.norm(R[8][g] - R[1][g]) <= TOL * torch.linalg.norm(R[1][g])


@pytest.mark.parametrize("ratio", [2.0 ** 10, 2.0 ** 30])
def test_3d_side_does_not_lose_bits_to_the_other_sides_far_node(ratio):
    from paper_2109_01286_gb300 import hfd3d
    m = T.periodic_tet_box(11, 10, 12, 10.0, 10.0, 10.0, seed=3)
    M = hfd3d.Mesh3(m)
    U = T.vortex_tube(m)
    K = int(np.argmin(np.abs(m["x"] - 4.0) + np.abs(m["y"] - 4.5) + np.abs(m["z"] - 5.0)))
    rows = _rows(M.prep_get("vptr"), M.prep_get("vidx"), M.prep_get("eptr"), M.prep_get("eidx"),
                 M.prep_get("sten").reshape(-1, 6), K)
    assert len(rows) >= 4
    U[:, K] *= ratio
    Ud = torch.from_numpy(U).cuda()
    R = M.residual(Ud)[:, rows]
    w5 = M.prep_get("w5").copy()                   # a weight that is not finite on an edge that these rows do
    ep, ei = M.prep_get("eptr"), M.prep_get("eidx")         # not read: FP64 sums for all edges
    e = np.setdiff1d(np.arange(len(w5) // 40), np.concatenate([ei[ep[r]:ep[r + 1]] for r in rows]))[0]
    w5.reshape(-1, 40)[e, 7] = np.nan
    M.prep_set("w5", w5)
    P = M.residual(Ud)[:, rows]
    assert torch.isfinite(P).all()
    for g in range(4):
        d = slice(5 * g, 5 * g + 5)
        assert torch.linalg.norm(R[d] - P[d]) <= TOL * torch.linalg.norm(P[d])


@pytest.mark.parametrize("nx", [40, 60])
def test_adjoint_of_edges_in_fp64_sums(nx):
    """One vertex 8 times the others: some edges lie outside the fixed-point range of the sums.  lambda_n is lambda
    and dt (1e-3) times sums whose terms are off by up to 110 units of 2^-53 and cancel by up to 1e2: the
    norms agree to 1e-3 x 110 x 1.1e-16 x 1e2 and lambda's own rounding, below 1e-13."""
    import paper_2109_01286_gb300 as pkg
    m = synth.jittered_grid(nx, nx, 10.0, 10.0, seed=1)
    U = synth.isentropic_vortex(m)
    U[:, int(np.argmin(np.hypot(m["x"] - 4.0, m["y"] - 4.5)))] *= 8.0
    mesh = pkg.Mesh(m)
    Ui = mesh.import_state(torch.from_numpy(U).cuda())
    lam = torch.randn(Ui.shape, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    out = {}
    for lanes in (8, 1):
        mesh.set_lanes(lanes)
        out[lanes] = mesh.adjoint(Ui, lam, dt=1e-3)
    mesh.check()
    assert not torch.equal(out[8], out[1])
    assert torch.linalg.norm(out[8] - out[1]) <= 1e-13 * torch.linalg.norm(out[1])
