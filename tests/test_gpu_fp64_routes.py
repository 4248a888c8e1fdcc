"""The FP64 sums beside the fixed-point ones: the routes that call them, and what they compute."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2109_01286_gb300 as pkg
    return pkg


def _l2(a, b):
    return max((torch.linalg.norm(a[g] - b[g]) / torch.linalg.norm(b[g])).item()
               for g in (slice(0, 4), slice(4, 8), slice(8, 12)))


@pytest.mark.parametrize("nx", [24, 60])          # 1,728 edges: 8 lanes an edge; 10,800: one thread
def test_one_and_two_lanes_take_fp64_sums(nx):
    """Lane counts 1 and 2 sum in FP64, in orders of their own: other bits than the fixed-point sums, whose
    lane counts agree bit for bit, and the same residual.  A row's FP64 sum of up to 110 products is off by
    110 units of 2^-53 of its largest partial sum and the terms cancel by up to 1e3; the norms see the
    root of that number: 11 x 1.1e-16 x 1e3 = 1.3e-12.  The oracle's coefficients come from other
    arithmetic, 1e-7 apart (the full path's parity tests)."""
    pkg = _pkg()
    m = synth.jittered_grid(nx, nx, 10.0, 10.0, seed=1)
    U = synth.isentropic_vortex(m)
    mesh = pkg.Mesh(m)
    Ui = mesh.import_state(torch.from_numpy(U).cuda())
    R = {}
    for lanes in (4, 8, 1, 2):
        mesh.set_lanes(lanes)
        R[lanes] = mesh.residual(Ui.clone())
        S = torch.empty_like(Ui)
        mesh.residual_static(Ui.clone(), S)
        assert torch.equal(S, R[lanes])
    mesh.check()
    assert torch.equal(R[4], R[8])
    assert not torch.equal(R[1], R[4]) and not torch.equal(R[1], R[2])
    for lanes in (1, 2):
        assert _l2(R[lanes], R[4]) < 1.3e-12
    P = oracle.prepare(m)
    ref = torch.from_numpy(oracle.residual(m, P, U.copy())[:, mesh.perm]).cuda()
    assert (torch.linalg.norm(R[1] - ref) / torch.linalg.norm(ref)).item() < 1e-7
    a = Ui.clone()
    mesh.set_lanes(1)
    mesh.steps(a, 0.0, 2)                          # captured with the FP64 sums
    b = Ui.clone()
    mesh.set_lanes(8)
    mesh.steps(b, 0.0, 2)
    mesh.check()
    assert not torch.equal(a, b) and (torch.linalg.norm(a - b) / torch.linalg.norm(b)).item() < 1e-12
