"""hfd3_mesh_set_lanes: 4 lanes are the default's fixed-point divergence, 1 and 2 the FP64 gather."""
import numpy as np
import pytest
import torch

from synth import three_d as T
from test_gpu_3d_fixed import _bound, _mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,case", [((7, 9, 8), "smooth"), ((12, 7, 10), "smooth"), ((7, 9, 8), "spread")])
def test_four_lanes_are_the_default_and_one_and_two_the_fp64_gather(shape, case):
    m, M = _mesh(shape)
    U = T.vortex_tube(m) if case == "smooth" else T.uniform_state3(m)
    if case == "spread":
        U[:, ::3] *= 2.0 ** -40
    Ud = torch.from_numpy(U).cuda()
    R = M.residual(Ud)
    bound = _bound(M, U)
    for lanes in (1, 2, 4):
        M.set_lanes(lanes)
        P = M.residual(Ud)
        assert torch.equal(P, R) == (lanes == 4)
        assert ((R - P).abs().cpu().numpy() <= bound).all()


def test_rows_with_non_finite_fluxes_match_the_fp64_gather():
    from paper_2109_01286_gb300 import hfd3d
    m, M = _mesh((7, 9, 8))
    U = T.vortex_tube(m)
    U[4, 100] = np.inf
    U[0, 300] = np.nan
    Ud = torch.from_numpy(U).cuda()
    out = []
    for lanes in (4, 1):
        M.set_lanes(lanes)
        out.append(M.residual(Ud).cpu())
        with pytest.raises(hfd3d.HfdError):
            M.check()
    R, P = out
    assert torch.equal(torch.isfinite(R), torch.isfinite(P))
    assert not torch.isfinite(R[:, 100]).all() and torch.isfinite(R).any()
    ok = torch.isfinite(P).numpy()
    U[4, 100] = U[4, 101]
    U[0, 300] = U[0, 301]
    assert (np.abs(R.numpy() - P.numpy())[ok] <= _bound(M, U)[ok]).all()
