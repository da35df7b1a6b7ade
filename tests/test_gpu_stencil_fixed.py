"""The stencils' imaginary parts in fixed point: residuals against extended precision where
operands lie far apart, at walls and on odd sizes; scaled problems; infinities and NaN."""
import math

import numpy as np
import pytest
import torch

from paper_2609_07172_gb300 import Plan, PicPoissonError, cell_coeffs, workloads as W

pytestmark = pytest.mark.gpu
L = np.longdouble


def _operator(p):
    """Face conductances (nz, nr) of the W, E, S, N neighbours (0 at walls), D0 and mu."""
    g = np.array([[cell_coeffs(p, i, k) for i in range(p.nr)] for k in range(p.nz)])
    return [g[..., f] * (1 - g[..., 4 + f]) for f in range(4)], g[..., 10], g[..., 8]


def _residual(p, u, b):
    (gw, ge, gs, gn), d0, mu = _operator(p)
    m = np.arange(p.n_modes)
    lam = 4.0 / (p.theta_span / p.ntheta) ** 2 * np.sin(np.pi * m / p.ntheta) ** 2
    d = (d0[..., None] + lam * mu[..., None])[..., None]
    u, b = u.astype(L), b.astype(L)
    pad = np.pad(u, ((1, 1), (1, 1), (0, 0), (0, 0)))
    terms = [gw[..., None, None] * pad[1:-1, :-2], ge[..., None, None] * pad[1:-1, 2:],
             gs[..., None, None] * pad[:-2, 1:-1], gn[..., None, None] * pad[2:, 1:-1], -d * u, b]
    return sum(terms), sum(np.abs(t) for t in terms)


@pytest.mark.parametrize("nr,nt,nz", [(2, 2, 1), (9, 4, 7), (16, 8, 2), (33, 16, 20), (24, 64, 15)])
@pytest.mark.parametrize("spread", [0.0, 6.0, 30.0])
def test_mode_residual_matches_extended_precision(nr, nt, nz, spread):
    p = W.annulus(nr, nt, nz)
    rng = np.random.default_rng(nr + nt)

    def field():   # neighbours up to `spread` decades apart
        v = rng.standard_normal((nz, nr, p.n_modes, 2)) * 10.0 ** rng.uniform(-spread, spread, (nz, nr, p.n_modes, 2))
        v[..., 0, 1] = 0.0
        return v
    u, b = field(), field()
    with Plan(p) as plan:
        r, _ = plan.mode_residual(torch.from_numpy(u).cuda(), torch.from_numpy(b).cuda())
    want, size = _residual(p, u, b)
    err = np.abs(r.cpu().numpy() - want)
    # binary64: five operations and coefficients rounded once, each within 2^-53 of the sum of magnitudes
    assert np.all(err <= 8 * 2.0 ** -53 * size)
    assert np.all(err[..., 0, 1] == 0.0)


@pytest.mark.parametrize("dims", [(48, 16, 40), (50, 8, 27)])
@pytest.mark.parametrize("e", [-400, 400])
def test_solution_scales_exactly_with_the_charge(dims, e):
    p = W.annulus(*dims, phi_z0=0.0)
    rho = W.rho_plasma(p, 5)
    with Plan(p, fmg=1) as plan:
        a, ia = plan.solve(torch.from_numpy(rho).cuda())
        b, ib = plan.solve(torch.from_numpy(np.ldexp(rho, e)).cuda())
    assert ia["status"] == ib["status"] == 0 and ia["cycles"] == ib["cycles"]
    assert np.array_equal(b.cpu().numpy(), np.ldexp(a.cpu().numpy(), e))


@pytest.mark.parametrize("bad", [math.inf, math.nan])
def test_non_finite_guess_is_reported(bad):
    p = W.annulus(32, 8, 24)
    rho = torch.from_numpy(W.rho_plasma(p, 1)).cuda()
    with Plan(p) as plan:
        plan.solve(rho)
        u = plan.get_modes()
        u[3, 4, 2, 1] = bad      # one imaginary part
        with pytest.raises(PicPoissonError):
            plan.solve_modes(rho, u)
        phi, info = plan.solve(rho)
    assert info["status"] == 0 and bool(torch.isfinite(phi).all())
