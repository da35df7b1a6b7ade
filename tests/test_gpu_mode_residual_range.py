"""The mode residual takes binary64's whole range, and shows what is not finite where it enters."""
import pytest
import torch

from paper_2609_07172_gb300 import Plan, workloads as W

pytestmark = pytest.mark.gpu

MESHES = {
    "annulus": lambda: W.annulus(16, 8, 12),
    "plume": lambda: W.channel_plume(32, 8, 24),
    "one_level": lambda: W.annulus(5, 8, 6),
}


@pytest.mark.parametrize("power", [-960, -900, -800, 800, 940, 980])
@pytest.mark.parametrize("name", list(MESHES))
def test_mode_residual_scales_exactly(name, power):
    p = MESHES[name]()
    g = torch.Generator().manual_seed(3)
    with Plan(p) as plan:
        u, b = [torch.randn(plan.mode_shape, generator=g, dtype=torch.float64).cuda() for _ in range(2)]
        r = plan.mode_residual(u, b)[0]
        f = 2.0 ** power
        rs = plan.mode_residual(f * u, f * b)[0]
    assert torch.isfinite(rs).all() and torch.equal(rs, f * r)


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
def test_mode_residual_shows_what_is_not_finite(value):
    p = W.annulus(16, 8, 12)
    with Plan(p) as plan:
        u = torch.ones(plan.mode_shape, dtype=torch.float64, device="cuda")
        b = torch.ones_like(u)
        for part in (0, 1):
            x = u.clone()
            x[5, 7, 2, part] = value
            r = plan.mode_residual(x, b)[0]
            bad = ~torch.isfinite(r)
            want = torch.zeros_like(bad)
            for k, i in ((5, 7), (4, 7), (6, 7), (5, 6), (5, 8)):
                want[k, i, 2, part] = True
            assert torch.equal(bad, want)
