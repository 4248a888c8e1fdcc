"""The FP64 divergence in fixed point on rows of many products, and beside such rows."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _hub(n, spokes, seed):
    """A periodic Delaunay mesh of jittered points around a wheel of `spokes` neighbours: rows of up to 282
    products (40 spokes) and 582 (100 spokes; there the coefficients of one row add up to more than 127 times
    their scale)."""
    from scipy.spatial import Delaunay
    rng = np.random.default_rng(seed)
    gx, gy = np.meshgrid((np.arange(n) + 0.5) / n, (np.arange(n) + 0.5) / n)
    x = (gx.ravel() + rng.uniform(-0.25, 0.25, n * n) / n) % 1
    y = (gy.ravel() + rng.uniform(-0.25, 0.25, n * n) / n) % 1
    radius = 2.2 / n
    keep = np.hypot(x - 0.5, y - 0.5) > 1.25 * radius
    a = 2 * np.pi * (np.arange(spokes) + rng.uniform(-0.2, 0.2, spokes)) / spokes
    x = np.concatenate([x[keep], 0.5 + radius * np.cos(a), [0.5]])
    y = np.concatenate([y[keep], 0.5 + radius * np.sin(a), [0.5]])
    P = np.concatenate([np.stack([x + i, y + j], 1) for i in (-1, 0, 1) for j in (-1, 0, 1)])
    t = Delaunay(P).simplices
    c = P[t].mean(1)
    t = t[(c >= 0).all(1) & (c < 1).all(1)]
    d1, d2 = P[t[:, 1]] - P[t[:, 0]], P[t[:, 2]] - P[t[:, 0]]
    neg = d1[:, 0] * d2[:, 1] - d1[:, 1] * d2[:, 0] < 0
    t[neg] = t[neg][:, [0, 2, 1]]
    return {"x": 10 * x, "y": 10 * y, "tri": (t % len(x)).astype(np.int32), "Lx": 10.0, "Ly": 10.0,
            "periodic_x": True, "periodic_y": True}


VISC = dict(viscous=True, mu=0.01, prandtl=0.72, R_gas=1.0 / (1.4 * 0.01))


def _prep(spokes, kw):
    import paper_2109_01286_gb300 as pkg
    m = _hub(14, spokes, 1)
    return pkg.Prep(m, **kw), synth.isentropic_vortex(m, beta=2.0)


@pytest.mark.parametrize("spokes", [40, 100])
@pytest.mark.parametrize("kw", [{}, VISC], ids=["euler", "viscous"])
def test_rows_of_many_products_match_fp64(spokes, kw):
    """Both lane counts of the fixed-point kernel give the same bits, other than FP64 sums and within their
    rounding: K <= 582 products, sqrt(K) x 2^-53 of terms that cancel by up to 1e4: 24 x 1.1e-16 x 1e4."""
    prep, U = _prep(spokes, kw)
    mesh = prep.upload()
    Ui = mesh.import_state(torch.from_numpy(U).cuda())
    R = {}
    for lanes in (8, 4, 1):
        mesh.set_lanes(lanes)
        R[lanes] = mesh.residual(Ui.clone())
    mesh.check()
    assert torch.equal(R[8], R[4]) and not torch.equal(R[8], R[1])
    for g in (slice(0, 4), slice(4, 8), slice(8, 12)):
        assert torch.linalg.norm(R[8][g] - R[1][g]) <= 2.7e-11 * torch.linalg.norm(R[1][g])


@pytest.mark.parametrize("spokes", [40, 100])
@pytest.mark.parametrize("nx", [24, 60])
def test_members_of_a_batch_do_not_depend_on_a_neighbour_with_long_rows(spokes, nx):
    import paper_2109_01286_gb300 as pkg
    m = synth.jittered_grid(nx, nx, 10.0, 10.0, seed=1)
    preps = [(pkg.Prep(m), synth.isentropic_vortex(m)), _prep(spokes, {})]
    alone = []
    for prep, U in preps:
        mesh = prep.upload()
        alone.append(mesh.export_state(mesh.residual(mesh.import_state(torch.from_numpy(U).cuda()))))
    both = pkg.Prep.concat([p for p, _ in preps]).upload()
    R = both.export_state(both.residual(both.import_state(torch.from_numpy(
        np.concatenate([U for _, U in preps], 1)).cuda())))
    both.check()
    assert torch.equal(R, torch.cat(alone, 1))
