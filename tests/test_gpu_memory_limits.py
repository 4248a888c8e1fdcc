"""Meshes that fit the memory only without the second, fixed-point form of their rows and weights."""
import numpy as np
import pytest

import synth
from synth import three_d as T

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class _Left:
    """Leaves `nbytes` of the device's memory free."""

    def __init__(self, nbytes):
        self.nbytes = int(nbytes)

    def __enter__(self):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.hog = torch.empty(torch.cuda.mem_get_info()[0] - self.nbytes, dtype=torch.uint8, device="cuda")

    def __exit__(self, *exc):
        del self.hog
        torch.cuda.empty_cache()


class _Limit:
    """Lets PyTorch's allocator take `nbytes` more."""

    def __init__(self, nbytes):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.share = (torch.cuda.memory_reserved() + nbytes) / torch.cuda.mem_get_info()[1]

    def __enter__(self):
        torch.cuda.set_per_process_memory_fraction(self.share)

    def __exit__(self, *exc):
        torch.cuda.empty_cache()
        torch.cuda.set_per_process_memory_fraction(1.0)


@pytest.mark.parametrize("allocator", ["cuda", "torch"])
def test_2d_mesh_falls_back_to_fp64_sums(allocator):
    """85% of what the mesh takes with both forms (1.5 times what it takes with one)."""
    import paper_2109_01286_gb300 as pkg
    m = synth.jittered_grid(300, 300, 10.0, 10.0, seed=1)
    prep = pkg.Prep(m, allocator=None if allocator == "cuda" else "torch")
    U = torch.from_numpy(synth.isentropic_vortex(m)).cuda()
    mesh = prep.upload()
    both = mesh.stats.device_bytes
    Ui = mesh.import_state(U)
    fixed = mesh.residual(Ui.clone())
    mesh.set_lanes(1)
    fp64 = mesh.residual(Ui.clone())
    mesh.close()
    R = torch.empty_like(Ui)
    with (_Left if allocator == "cuda" else _Limit)(0.85 * both):
        mesh = prep.upload()
        mesh.residual(Ui, R)
        mesh.check()
        assert mesh.stats.device_bytes < 0.75 * both
        mesh.close()
    assert torch.equal(R, fp64) and not torch.equal(R, fixed)


def test_3d_mesh_falls_back_to_fp64_sums():
    """80% of what the mesh takes with both forms (1.9 times what it takes with one)."""
    from paper_2109_01286_gb300 import hfd3d
    m = T.periodic_tet_box(18, 17, 18, 10.0, 10.0, 10.0, seed=3)
    U = torch.from_numpy(T.vortex_tube(m)).cuda()
    before = torch.cuda.mem_get_info()[0]
    M = hfd3d.Mesh3(m)
    both = before - torch.cuda.mem_get_info()[0]
    fixed = M.residual(U)
    del M
    R = torch.empty_like(U)
    with _Left(0.8 * both):
        M = hfd3d.Mesh3(m)
        M.residual(U, R)
        M.check()
        assert M.prep_get("cv").size > 0
        M.prep_set("cv", M.prep_get("cv"))         # packs again where there is a second form
        M.prep_set("w5", M.prep_get("w5"))
        again = M.residual(U, torch.empty_like(U))
        del M
    assert torch.equal(R, again) and not torch.equal(R, fixed)
    assert (torch.linalg.norm(R - fixed) / torch.linalg.norm(fixed)).item() < 1e-11
