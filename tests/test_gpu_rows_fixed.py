"""Stencils of a composite domain with the imaginary part in fixed point: residuals against extended precision,
strips of the smoother bitwise equal, scaled problems."""
import numpy as np
import pytest
import torch

from paper_2609_07172_gb300 import Plan, cell_coeffs, workloads as W

pytestmark = pytest.mark.gpu
L = np.longdouble


@pytest.mark.parametrize("dims", [(32, 8, 32), (64, 16, 48), (96, 2, 64)])
@pytest.mark.parametrize("spread", [0.0, 6.0, 30.0])
def test_mode_residual_matches_extended_precision(dims, spread):
    nr, nt, nz = dims
    p = W.channel_plume(nr, nt, nz)
    act = np.zeros((nz, nr), bool)
    for i0, i1, k0, k1 in p.patches:
        act[k0:k1, i0:i1] = True
    g = np.array([[cell_coeffs(p, i, k) if act[k, i] else [0.0] * 12 for i in range(nr)] for k in range(nz)], dtype=object)
    g = np.array([[list(map(float, c))[:11] for c in row] for row in g])
    cond = [g[..., f] * (1 - g[..., 4 + f]) for f in range(4)]
    rng = np.random.default_rng(nr)

    def field():
        v = rng.standard_normal((nz, nr, p.n_modes, 2)) * 10.0 ** rng.uniform(-spread, spread, (nz, nr, p.n_modes, 2))
        v[..., 0, 1] = 0.0
        return v * act[..., None, None]
    u, b = field(), field()
    with Plan(p) as plan:
        r = plan.mode_residual(torch.from_numpy(u).cuda(), torch.from_numpy(b).cuda())[0].cpu().numpy()
    m = np.arange(p.n_modes)
    lam = 4.0 / (p.theta_span / p.ntheta) ** 2 * np.sin(np.pi * m / p.ntheta) ** 2
    d = (g[..., 10, None] + lam * g[..., 8, None])[..., None]
    pad = np.pad(u.astype(L), ((1, 1), (1, 1), (0, 0), (0, 0)))
    near = [pad[1:-1, :-2], pad[1:-1, 2:], pad[:-2, 1:-1], pad[2:, 1:-1]]
    terms = [c[..., None, None] * x for c, x in zip(cond, near)] + [-d * u.astype(L), b.astype(L)]
    # binary64: six operations and coefficients rounded once, each within 2^-53 of the sum of magnitudes
    err = np.abs(r - sum(terms)) * act[..., None, None]
    assert np.all(err <= 8 * 2.0 ** -53 * sum(np.abs(t) for t in terms))
    assert np.all(r[~act] == 0.0)


@pytest.mark.parametrize("kw", [dict(), dict(pre_sweeps=1, post_sweeps=2, fmg=1)])
def test_strips_are_bitwise_and_solutions_scale_exactly(kw):
    p = W.channel_plume(64, 16, 48, phi_z0=0.0)   # linear in the charge
    rho = torch.from_numpy(W.rho_plasma(p, 3)).cuda()
    out = []
    for strip, e in ((0, 0), (2, 0), (0, 300)):
        with Plan(p, smooth_strip=strip, **kw) as plan:
            phi, info = plan.solve(torch.ldexp(rho, torch.tensor(e, device="cuda")), tol=1e-10)
        assert info["status"] == 0
        out.append(np.ldexp(phi.cpu().numpy(), -e))
    assert all(np.array_equal(out[0], x) for x in out[1:])
