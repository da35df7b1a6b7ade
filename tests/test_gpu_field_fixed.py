"""Face fields with the products by integer multiplies, over the whole range of binary64."""
import numpy as np
import pytest
import torch

from paper_2609_07172_gb300 import Plan, workloads as W

pytestmark = pytest.mark.gpu


def _fields(plan, phi):
    return [e.cpu().numpy() for e in plan.face_field(torch.from_numpy(phi).cuda())]


@pytest.mark.parametrize("dims", [(1, 2, 1), (33, 4, 17), (64, 8, 40), (136, 64, 128), (256, 128, 288)])
@pytest.mark.parametrize("spread", [1.0, 280.0])
def test_products_are_those_of_binary64(dims, spread):
    """Faces between cells, bit for bit; the inverse distances are read off a field of alternating 0 and 1."""
    nr, nt, nz = dims
    p = W.annulus(nr, nt, nz)
    rng = np.random.default_rng(nr)
    phi = rng.standard_normal((nz, nt, nr)) * 10.0 ** rng.uniform(-spread, spread, (nz, nt, nr))
    phi.flat[rng.integers(0, phi.size, phi.size // 16 + 1)] = 0.0
    phi.flat[rng.integers(0, phi.size, phi.size // 64 + 1)] = 5e-324
    board = (np.indices(phi.shape).sum(0) % 2).astype(np.float64)
    with Plan(p) as plan:
        (ir, ia, iz), (er, ea, ez) = _fields(plan, board), _fields(plan, phi)
    assert np.array_equal(er[..., 1:-1], (phi[..., :-1] - phi[..., 1:]) * np.abs(ir[..., 1:-1]))
    assert np.array_equal(ea, (phi - np.roll(phi, -1, axis=1)) * np.abs(ia))
    assert np.array_equal(ez[1:-1], (phi[:-1] - phi[1:]) * np.abs(iz[1:-1]))


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan, 1.7e308])
def test_values_beyond_the_normal_range(bad):
    p = W.annulus(16, 4, 12)
    phi = np.ones((12, 4, 16))
    phi[5, 2, 7] = bad
    with Plan(p) as plan:
        er, ea, ez = [e.cpu().numpy() for e in plan.face_field(torch.from_numpy(phi).cuda())]
    for v in (er[5, 2, 7], er[5, 2, 8], ea[5, 2, 7], ea[5, 1, 7], ez[5, 2, 7], ez[6, 2, 7]):
        assert np.isnan(v) if np.isnan(bad) else np.isinf(v)
    assert np.all(np.isfinite(np.delete(er.ravel(), [(5 * 4 + 2) * 17 + 7, (5 * 4 + 2) * 17 + 8])))
