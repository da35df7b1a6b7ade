"""V-cycles in shared memory (one cluster per mode) against the level kernels: bitwise equal."""
import threading

import pytest
import torch

from paper_2609_07172_gb300 import FP64, MIXED, BatchPlan, Plan, workloads as W

pytestmark = pytest.mark.gpu

# one smoothed level, semi-coarsening either way, odd coarsest rows and columns, few rows (one block a mode),
# two modes, many modes, and levels too large for a cluster above ones that fit
SIZES = [(32, 16, 32), (16, 8, 12), (26, 8, 70), (64, 2, 24), (90, 32, 70), (152, 32, 90), (16, 8, 400), (256, 8, 16),
         (512, 8, 12), (48, 256, 33), (128, 64, 96), (320, 16, 288), (512, 128, 64)]


def _solve(p, rho, guess=None, **kw):
    with Plan(p, **kw) as plan:
        phi, info = plan.solve(rho, tol=1e-10) if guess is None else plan.solve(rho, guess.clone(), tol=1e-10)
    assert info["status"] == 0
    return phi, info["cycles"]


def _level_kernels(p, rho, guess=None, **kw):
    """By separate launches.  A full-multigrid start with the mode-local bottom smooths the two coarsest levels
    together, without it one by one: there the reference is a batch, whose problems take the mode-local bottom."""
    if not kw.get("fmg"):
        return _solve(p, rho, guess, local_bottom=-1, **kw)
    with BatchPlan([p, p], **kw) as plan:
        phis, infos = plan.solve([rho, rho], None if guess is None else [guess.clone(), guess.clone()], tol=1e-10)
    assert infos[0]["status"] == 0 and torch.equal(phis[0], phis[1])
    return phis[0], infos[0]["cycles"]


@pytest.mark.parametrize("dims", SIZES, ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("kw", [dict(precision=FP64), dict(precision=FP64, pre_sweeps=2, post_sweeps=1, fmg=1),
                                dict(precision=MIXED, pre_sweeps=2, post_sweeps=2, inner_cycles=3, smooth_fused=1),
                                dict(precision=MIXED, pre_sweeps=1, post_sweeps=1, inner_cycles=1, inner_first=2)],
                         ids=["fp64", "fp64fmg", "mixedfused", "mixed"])
def test_bitwise_the_level_kernels(dims, kw):
    p = W.annulus(*dims, phi_z0=300.0)
    rho = torch.from_numpy(W.rho_plasma(p, 7)).cuda()
    a, ca = _level_kernels(p, rho, **kw)
    b, cb = _solve(p, rho, graph=True, **kw)
    assert ca == cb and torch.equal(a, b)


@pytest.mark.parametrize("fmg", [0, 1])
@pytest.mark.parametrize("dims", [(32, 16, 32), (90, 32, 70), (320, 16, 288)])
def test_from_a_given_iterate(dims, fmg):
    p = W.annulus(*dims)
    rho = torch.from_numpy(W.rho_plasma(p, 8)).cuda()
    g = 0.9 * _solve(p, rho)[0]
    a, ca = _level_kernels(p, rho, g, fmg=fmg, initial_guess=True)
    b, cb = _solve(p, rho, g, fmg=fmg, initial_guess=True)
    assert ca == cb and torch.equal(a, b)


def test_two_threads_on_their_own_streams():
    """Two solves of one launch each that fill most of the chip, at the same time: neither waits on the other's blocks."""
    p = W.annulus(64, 64, 64)
    rho = torch.from_numpy(W.rho_plasma(p, 9)).cuda()
    want, _ = _solve(p, rho)
    torch.cuda.synchronize()
    errors = []

    def work():
        try:
            st = torch.cuda.Stream()
            with torch.cuda.stream(st), Plan(p, graph=True) as plan:
                for _ in range(40):
                    phi, info = plan.solve(rho, tol=1e-10)
                    assert info["status"] == 0 and torch.equal(phi, want)
        except BaseException as e:      # noqa: B036 (reported by the test's thread)
            errors.append(e)
    threads = [threading.Thread(target=work) for _ in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
