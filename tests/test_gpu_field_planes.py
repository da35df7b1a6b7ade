"""Face field of a domain with more than 2^20 planes (more pieces along z than a grid's second dimension holds)."""
import pytest
import torch

from paper_2609_07172_gb300 import Plan, workloads as W

pytestmark = pytest.mark.gpu


def test_more_than_a_million_planes():
    p = W.annulus(2, 2, 33 << 15, z0=0.0, z1=0.001, phi_z0=3.0)
    g = torch.Generator().manual_seed(1)
    phi = torch.randn(p.shape, generator=g, dtype=torch.float64).cuda()
    with Plan(p) as plan:
        er, ea, ez = plan.face_field(phi)
    dz = (p.z1 - p.z0) / p.nz
    want = (phi[:-1] - phi[1:]) / dz
    assert (ez[1:-1] - want).abs().max() <= 4 * 2.0 ** -53 * want.abs().max()
    assert (ez[0] - (3.0 - phi[0]) / (0.5 * dz)).abs().max() <= 8 * 2.0 ** -53 * ez[0].abs().max()
    assert (ez[-1] - phi[-1] / (0.5 * dz)).abs().max() <= 8 * 2.0 ** -53 * ez[-1].abs().max()
    dr = (p.r_out - p.r_in) / p.nr
    assert (er[:, :, 1] - (phi[:, :, 0] - phi[:, :, 1]) / dr).abs().max() <= 8 * 2.0 ** -53 * er[:, :, 1].abs().max()
    rc = torch.tensor([p.r_in + 0.5 * dr, p.r_in + 1.5 * dr], dtype=torch.float64, device="cuda")
    want = (phi - phi.roll(-1, 1)) / (rc * (p.theta_span / 2))
    assert (ea - want).abs().max() <= 16 * 2.0 ** -53 * want.abs().max()
