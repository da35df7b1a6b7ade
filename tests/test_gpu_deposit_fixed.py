"""The fixed-point deposit where it can go wrong: cell boundaries, walls, thin and shifted domains,
runs that cross threads, warps and blocks, unaligned arrays."""
import numpy as np
import pytest
import torch

import oracle
from oracle import deposit as D
from paper_2609_07172_gb300 import Plan, workloads as W

pytestmark = pytest.mark.gpu

W0 = 1e8


def _check(p, r, a, z, shift=0):
    dev = []
    for x in (r, a, z):      # `shift` values past the allocation's start
        t = torch.empty(x.size + 2, dtype=torch.float64, device="cuda")
        t[shift:shift + x.size] = torch.from_numpy(x)
        dev.append(t[shift:shift + x.size])
    with Plan(p) as plan:
        got = plan.deposit(*dev, W0).cpu().numpy()
    # (the oracle takes finite positions only; what lies outside deposits nothing)
    ok = (r >= p.r_in) & (r < p.r_out) & (a >= 0.0) & (a < p.theta_span) & (z >= p.z0) & (z < p.z1)
    want = D.deposit(oracle.grid_from_problem(p), r[ok], a[ok], z[ok], W0)
    # binary64 positions round to 2^-53 of a coordinate, at most 2^-53 max(nr, nt, nz) cells from the
    # oracle's (thin domains: of the coordinate over the width), the rest far below
    span = max(p.nr * p.r_out / (p.r_out - p.r_in), p.ntheta, p.nz * max(abs(p.z0), abs(p.z1)) / (p.z1 - p.z0))
    assert np.abs(got - want).max() <= (1e-12 + 16 * span * 2.0 ** -53) * np.abs(want).max()
    return got


def _inside(p, n, seed):
    rng = np.random.default_rng(seed)
    return (rng.uniform(p.r_in, p.r_out, n), rng.uniform(0.0, p.theta_span, n), rng.uniform(p.z0, p.z1, n))


GRIDS = {
    "annulus": lambda: W.annulus(38, 4, 19),
    "one_cell": lambda: W.annulus(1, 2, 1),
    "thin_and_far": lambda: W.annulus(32, 8, 16, r_in=100.0, r_out=100.03125, z0=-40.0, z1=-39.875),
    "across_zero": lambda: W.annulus(20, 4, 24, z0=-0.01, z1=0.02),
    "large_counts": lambda: W.annulus(1030, 2, 4),
}


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("name", list(GRIDS))
def test_random_particles(name, shift):
    p = GRIDS[name]()
    _check(p, *_inside(p, 5003, 3), shift=shift)


@pytest.mark.parametrize("name", ["annulus", "across_zero", "thin_and_far"])
def test_particles_on_and_beside_faces_and_walls(name):
    p = GRIDS[name]()
    rf = p.r_in + (p.r_out - p.r_in) / p.nr * np.arange(p.nr + 1)
    zf = p.z0 + (p.z1 - p.z0) / p.nz * np.arange(p.nz + 1)
    af = p.theta_span / p.ntheta * np.arange(p.ntheta + 1)
    r, a, z = [np.concatenate([f, np.nextafter(f, -np.inf), np.nextafter(f, np.inf)]) for f in (rf, af, zf)]
    n = 600
    rng = np.random.default_rng(4)
    bad = np.array([np.nan, np.inf, -np.inf, 0.0, -1.0, 1e300, 5e-324])
    r = np.concatenate([rng.choice(r, n), bad, np.full(14, 0.5 * (p.r_in + p.r_out))])
    a = np.concatenate([rng.choice(a, n), np.full(7, 0.1), bad, np.full(7, 0.1)])
    z = np.concatenate([rng.choice(z, n), np.full(14, 0.5 * (p.z0 + p.z1)), bad])
    # a particle on a face belongs to the cell on either side (its weight toward the far node is then
    # 0), but one on an upper wall is inside or outside by the last bit: those are left out
    dr, dz, da = p.r_out - p.r_in, p.z1 - p.z0, p.theta_span
    wall = (np.abs(r - p.r_out) < 1e-9 * dr) | (np.abs(r - p.r_in) < 1e-9 * dr) | (np.abs(a - da) < 1e-9 * da)
    wall |= (np.abs(z - p.z1) < 1e-9 * dz) | (np.abs(z - p.z0) < 1e-9 * dz)
    _check(p, r[~wall], a[~wall], z[~wall])


@pytest.mark.parametrize("ppc", [1, 3, 4, 27, 130, 1500])
def test_sorted_runs(ppc):
    """Cell-sorted particles: runs inside a thread, over lanes, warps and blocks, row ends included."""
    p = W.annulus(37, 4, 6)
    rng = np.random.default_rng(ppc)
    cells = np.arange(37 * 4 * (6 if ppc < 200 else 1))
    cell = np.repeat(cells, ppc)
    u = rng.uniform(0.001, 0.999, (3, cell.size))
    r = p.r_in + (p.r_out - p.r_in) / p.nr * (cell % p.nr + u[0])
    a = p.theta_span / p.ntheta * (cell // p.nr % p.ntheta + u[1])
    z = p.z0 + (p.z1 - p.z0) / p.nz * (cell // (p.nr * p.ntheta) + u[2])
    _check(p, r, a, z)


@pytest.mark.parametrize("nr", [1, 30, 31, 32, 62, 63])
@pytest.mark.parametrize("nz", [1, 8, 9])
def test_projection_blocks(nr, nz):
    p = W.annulus(nr, 4, nz)
    rng = np.random.default_rng(nr + nz)
    nodes = rng.uniform(1.0, 2.0, (nz + 1, 4, nr + 1))
    g = oracle.grid_from_problem(p)
    with Plan(p) as plan:
        rho = plan.project(torch.from_numpy(nodes).cuda(), 2.0)
        plan.project(torch.from_numpy(nodes).cuda(), 0.5, rho, accumulate=True)
        got = rho.cpu().numpy()
    want = D.project(g, nodes, 2.0) + D.project(g, nodes, 0.5)
    assert np.abs(got - want).max() <= 1e-14 * np.abs(want).max()
