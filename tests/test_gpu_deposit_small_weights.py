"""Deposit weights of isolated particles close to cell corners, node by node: a weight's error is that of
the offsets in binary64 arithmetic, however small the weight."""
import numpy as np
import pytest
import torch

import oracle
from oracle import deposit as D
from paper_2609_07172_gb300 import Plan, workloads as W

pytestmark = pytest.mark.gpu

GRIDS = {
    "annulus": lambda: W.annulus(64, 16, 48),
    "near_axis": lambda: W.annulus(64, 16, 48, r_in=1e-5, r_out=1.0, z0=1e-7, z1=1.0),
    "across_zero": lambda: W.annulus(64, 16, 48, z0=-0.01, z1=0.02),
    "thin_and_far": lambda: W.annulus(64, 16, 48, r_in=100.0, r_out=100.0625, z0=-40.0, z1=-39.625),
    "one_cell": lambda: W.annulus(1, 2, 1),
    "patches": lambda: W.channel_plume(64, 16, 48),
}


def _faces(lo, hi, n):
    lo, hi = np.longdouble(lo), np.longdouble(hi)
    return lo + (hi - lo) * np.arange(n + 1) / np.longdouble(n)


@pytest.mark.parametrize("seed", [0, 1])
@pytest.mark.parametrize("name", list(GRIDS))
def test_every_corner_weight(name, seed):
    p = GRIDS[name]()
    g = oracle.grid_from_problem(p)
    rng = np.random.default_rng(seed)
    # one particle in every other cell along each axis: no two share a node
    shift = [int(rng.integers(0, 2)) if n > 2 else 0 for n in (p.nr, p.ntheta, p.nz)]
    i, j, k = [x.ravel() for x in np.meshgrid(np.arange(shift[0], p.nr, 2), np.arange(shift[1], p.ntheta - 1 + shift[1] // 2, 2),
                                              np.arange(shift[2], p.nz, 2), indexing="ij")]
    L = np.longdouble
    ends = [(p.r_in, p.r_out, p.nr, i), (0.0, p.theta_span, p.ntheta, j), (p.z0, p.z1, p.nz, k)]
    pos, t, width = [], [], []
    for lo, hi, n, c in ends:
        s = 10.0 ** -rng.choice([0.4, 1, 2, 3, 4, 5, 6, 7, 8, 10, 12], c.size) * rng.uniform(0.5, 1.0, c.size)
        s = np.where(rng.integers(0, 2, c.size) == 1, 1.0 - s, s)
        x = np.asarray(L(lo) + (L(hi) - L(lo)) * (c + s.astype(L)) / L(n), dtype=np.float64)
        x = np.clip(x, lo, np.nextafter(hi, -np.inf))
        at = (x.astype(L) - L(lo)) * L(n) / (L(hi) - L(lo))
        # (a particle that rounding moved onto a face or over it stays out)
        keep = np.floor(at) == c
        pos.append(x)
        t.append((at, keep))
    ok = t[0][1] & t[1][1] & t[2][1]
    if g.active is not None:
        ok &= g.active.astype(bool)[k, i]
    pos = [x[ok] for x in pos]
    i, j, k = i[ok], j[ok], k[ok]
    at = [x[ok] for x, _ in t]
    assert i.size >= 1
    off = [x - np.floor(x) for x in at]
    # the offset in binary64: a subtraction, the spacing (two roundings), its inverse and a product, each
    # within 2^-53 of the position, and half as much again
    err = [8 * 2.0 ** -53 * x for x in at]
    vol = D.node_volumes(g)
    order = rng.permutation(i.size)
    dev = [torch.from_numpy(np.ascontiguousarray(x[order])).cuda() for x in pos]
    with Plan(p) as plan:
        got = plan.deposit(*dev, 1.0).cpu().numpy()
    seen = np.zeros(got.shape, bool)
    for corner in range(8):
        bits = corner & 1, (corner >> 1) & 1, corner >> 2
        w = [o if b else 1 - o for o, b in zip(off, bits)]
        node = (k + bits[2], (j + bits[1]) % p.ntheta, i + bits[0])
        want = (w[0] * w[1] * w[2]) / vol[node[0], node[2]]
        # 2^-44: four products of 2^-47 and the volume's own rounding
        rel = sum(e / np.maximum(x, np.finfo(float).tiny) for e, x in zip(err, w)) + 2.0 ** -44
        bad = np.abs(got[node] - want) > rel * want
        if p.ntheta == 2:       # (both azimuthal nodes of every cell are the same two)
            continue
        assert not bad.any(), (corner, int(bad.sum()), [x[bad][:3] for x in w], got[node][bad][:3], want[bad][:3])
        seen[node] = True
    if p.ntheta > 2:
        assert not got[~seen].any()


@pytest.mark.parametrize("power", [-1000, -960, -300, 300, 960])
def test_the_weight_scales_exactly(power):
    """One particle, so that no order of additions enters: a power of two times the weight is exact."""
    p = W.annulus(16, 8, 12)
    pos = [torch.tensor([x], dtype=torch.float64, device="cuda")
           for x in (p.r_in + 0.37 * (p.r_out - p.r_in), 0.61, p.z0 + 0.23 * (p.z1 - p.z0))]
    with Plan(p) as plan:
        one, scaled = plan.deposit(*pos, 1.7), plan.deposit(*pos, 1.7 * 2.0 ** power)
    if one.max().item() * 2.0 ** power < 1e308:
        assert torch.equal(one * 2.0 ** power, scaled)


@pytest.mark.parametrize("s", [1e-2, 1e-4, 1e-6])
@pytest.mark.parametrize("count", [2, 3, 7, 40, 200, 1500])
def test_many_particles_near_one_corner(count, s):
    """Sorted runs inside a thread, over lanes, warps and blocks whose sums toward the far corners are small, beside a
    run of the radial neighbour with ordinary offsets."""
    p = W.annulus(8, 4, 6)
    g = oracle.grid_from_problem(p)
    rng = np.random.default_rng(count)
    L = np.longdouble
    cell = [np.repeat([3, 4], count), np.full(2 * count, 2), np.full(2 * count, 4)]
    far = np.arange(2 * count) < count
    off = [np.where(far, s * rng.uniform(0.5, 1.0, 2 * count), rng.uniform(0.2, 0.8, 2 * count)) for _ in range(3)]
    pos, at = [], []
    for (lo, hi, n), c, o in zip(((p.r_in, p.r_out, p.nr), (0.0, p.theta_span, p.ntheta), (p.z0, p.z1, p.nz)), cell, off):
        x = np.asarray(L(lo) + (L(hi) - L(lo)) * (c + o.astype(L)) / L(n), dtype=np.float64)
        pos.append(x)
        at.append((x.astype(L) - L(lo)) * L(n) / (L(hi) - L(lo)))
    frac = [t - c for t, c in zip(at, cell)]
    vol = D.node_volumes(g)
    want, tol = np.zeros((p.nz + 1, p.ntheta, p.nr + 1), L), np.zeros((p.nz + 1, p.ntheta, p.nr + 1), L)
    for corner in range(8):
        bits = corner & 1, (corner >> 1) & 1, corner >> 2
        w = [f if b else 1 - f for f, b in zip(frac, bits)]
        node = (cell[2] + bits[2], (cell[1] + bits[1]) % p.ntheta, cell[0] + bits[0])
        val = w[0] * w[1] * w[2] / vol[node[0], node[2]]
        np.add.at(want, node, val)
        # the offsets as above, 2^-44 of a weight, and the additions in any order
        np.add.at(tol, node, val * (sum(8 * 2.0 ** -53 * t / x for t, x in zip(at, w)) + 2.0 ** -44 + 2 * count * 2.0 ** -53))
    with Plan(p) as plan:
        got = plan.deposit(*[torch.from_numpy(x).cuda() for x in pos], 1.0).cpu().numpy()
    assert np.all(np.abs(got - want) <= tol)
