"""force_branch = "weno" on small meshes (8 lanes an edge) and large ones (one thread an edge)."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flux", ["roe", "rusanov"])
def test_forced_three_node_edges_of_small_and_large_meshes_give_the_same_bits(flux):
    """3,960 edges alone and in a batch of five copies (19,800): the same operations in the same order."""
    import paper_2109_01286_gb300 as pkg
    m = synth.jittered_grid(40, 33, 4.0, 3.3, seed=1)
    U = synth.isentropic_vortex(m, center=(2.0, 1.6))
    U[:4, np.hypot(m["x"] - 1.0, m["y"] - 1.0) < 0.6] *= 2.0
    prep = pkg.Prep(m, force_branch="weno", flux=flux)
    one, many = prep.upload(), pkg.Prep.concat([prep] * 5).upload()
    a = one.import_state(torch.from_numpy(U).cuda())
    b = many.import_state(torch.from_numpy(np.concatenate([U] * 5, 1)).cuda())
    assert (one.edge_branches(a.clone()) == 0xff).all() and (many.edge_branches(b.clone()) == 0xff).all()
    for lanes in (8, 1):                           # fixed-point and FP64 sums
        one.set_lanes(lanes)
        many.set_lanes(lanes)
        Ra = one.export_state(one.residual(a.clone()))
        Rb = many.export_state(many.residual(b.clone()))
        for k in range(5):
            assert torch.equal(Rb[:, k * len(m["x"]):(k + 1) * len(m["x"])], Ra)


def test_long_lists_of_three_node_edges_give_the_same_bits():
    """3,960 edges alone (8 lanes each) and in a batch of 60 copies, whose list is above the length from which
    it takes one thread an edge (20,000)."""
    import paper_2109_01286_gb300 as pkg
    m = synth.jittered_grid(40, 33, 4.0, 3.3, seed=1)
    U = synth.isentropic_vortex(m, center=(2.0, 1.6))
    U *= 1.0 + 0.3 * np.random.default_rng(0).random(U.shape[1])
    U[:, 700] *= 2.0 ** 30                         # sides far below their scale, in FP64 sums
    prep = pkg.Prep(m)
    one, many = prep.upload(), pkg.Prep.concat([prep] * 60).upload()
    a = one.import_state(torch.from_numpy(U).cuda())
    b = many.import_state(torch.from_numpy(np.concatenate([U] * 60, 1)).cuda())
    taken = one.edge_branches(a.clone())
    assert 60 * (taken != 0).sum() > 20000 and not taken.all()
    assert np.array_equal(many.edge_branches(b.clone()), np.tile(taken, 60))
    for lanes in (8, 1):
        one.set_lanes(lanes)
        many.set_lanes(lanes)
        Ra = one.export_state(one.residual(a.clone()))
        Rb = many.export_state(many.residual(b.clone()))
        assert torch.equal(Rb, Ra.repeat(1, 60))
