"""Dense coarsest solves of 195 and 204 cells, on either side of the size from which the contraction is split."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_07172_gb300 import FP64, MIXED, Plan, workloads as W
from paper_2609_07172_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [FP64, MIXED], ids=["fp64", "mixed"])
@pytest.mark.parametrize("dims,cells", [((26, 4, 30), 195), ((34, 4, 12), 204)])
def test_stretched_mesh_matches_oracle(dims, cells, precision):
    p = W.annulus(*dims)
    w = 1.01 ** np.arange(p.nz)
    p = p.with_z_faces(p.z0 + (p.z1 - p.z0) * np.r_[0.0, np.cumsum(w)] / w.sum())
    q = B.query(p)
    assert q["nr"][-1] * q["nz"][-1] == cells
    rho = W.rho_plasma(p, 9)
    ref, _ = oracle.solve3d(oracle.grid_from_problem(p), rho, tol=1e-15)
    with Plan(p, precision=precision) as plan:
        phi, info = plan.solve(torch.from_numpy(rho).cuda(), tol=1e-12)
    assert info["status"] == 0 and info["cycles"] <= 40
    assert np.linalg.norm(phi.cpu().numpy() - ref) <= 1e-9 * np.linalg.norm(ref)
