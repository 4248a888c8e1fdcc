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
