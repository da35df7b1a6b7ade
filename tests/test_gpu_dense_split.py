"""Dense coarsest solves with the contraction split between four groups of a block, at and around the size where it begins."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_07172_gb300 import FP64, MIXED, Plan, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [FP64, MIXED], ids=["fp64", "mixed"])
@pytest.mark.parametrize("dims", [(34, 4, 22), (38, 8, 20), (34, 16, 46), (50, 4, 30), (62, 8, 66)])
def test_stretched_mesh_matches_oracle(dims, precision):
    """Coarsest levels of 374 to 1023 cells, no multiples of the tile."""
    p = W.annulus(*dims)
    w = 1.01 ** np.arange(p.nz)
    p = p.with_z_faces(p.z0 + (p.z1 - p.z0) * np.r_[0.0, np.cumsum(w)] / w.sum())
    rho = W.rho_plasma(p, 9)
    g = oracle.grid_from_problem(p)
    ref, _ = oracle.solve3d(g, rho, tol=1e-15)
    with Plan(p, precision=precision) as plan:
        phi, info = plan.solve(torch.from_numpy(rho).cuda(), tol=1e-12)
    assert info["status"] == 0
    assert np.linalg.norm(phi.cpu().numpy() - ref) <= 1e-9 * np.linalg.norm(ref)
    # the coarsest solve is exact up to binary32: as few cycles as the other dense sizes of the repository
    assert info["cycles"] <= 40
