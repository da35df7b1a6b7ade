"""Plans whose kernels need different amounts of shared memory, used by host threads at a time: no thread's
launch depends on the size that another one last asked for."""
import contextlib
import threading

import pytest
import torch

from paper_2609_07172_gb300 import FP64, MIXED, BatchPlan, Plan, workloads as W
from paper_2609_07172_gb300.unet import P, _ok, _st, nn_lib

pytestmark = pytest.mark.gpu


def _transforms(dims):
    p = W.annulus(*dims)
    rho = torch.from_numpy(W.rho_plasma(p, 2)).cuda()
    plan = Plan(p)
    modes = plan.analyze(rho)

    def call():
        plan.analyze(rho, modes)
        plan.inverse(modes, rho)
    return plan, call


def _solves(dims, batch, precision):
    p = W.annulus(*dims)
    rho = torch.from_numpy(W.rho_plasma(p, 2)).cuda()
    phi = torch.empty_like(rho)
    kw = dict(precision=precision, max_cycles=1)      # (only the launches matter)
    if batch:
        plan = BatchPlan([p, p], **kw)
        phi2 = torch.empty_like(rho)
        return plan, lambda: plan.solve([rho, rho], [phi, phi2], tol=1e-30)
    plan = Plan(p, local_bottom=-1, **kw)
    return plan, lambda: plan.solve(rho, phi, tol=1e-30)


def _conv(w, cin, cout):
    lib = nn_lib()
    x, y = torch.randn(1, 8, w, cin, device="cuda").bfloat16(), torch.empty(1, 8, w, cout, device="cuda", dtype=torch.bfloat16)
    k, b = torch.randn(9, cout, cin, device="cuda").bfloat16(), torch.zeros(cout, device="cuda")
    call = lambda: _ok(lib.pic_nn_conv3x3(P(x), cin, P(k), P(b), P(y), None, cout, 1, 8, w, 1, _st()))  # noqa: E731
    call()
    return contextlib.nullcontext(), call


# per kernel a plan that needs much and one that needs little: the transforms, the exact coarsest solve by
# itself (45 x 35 and 8 x 4) and below a smoothed level (64 x 31 and 8 x 4)
PAIRS = {
    "transforms": (3000, lambda: _transforms((32, 256, 4)), lambda: _transforms((32, 8, 4))),
    "coarse_fp64": (1000, lambda: _solves((90, 2, 70), False, FP64), lambda: _solves((16, 2, 8), False, FP64)),
    "coarse_mixed": (1000, lambda: _solves((90, 2, 70), False, MIXED), lambda: _solves((16, 2, 8), False, MIXED)),
    "bottom_fp64": (1000, lambda: _solves((64, 2, 62), True, FP64), lambda: _solves((32, 2, 16), True, FP64)),
    "conv": (10000, lambda: _conv(64, 64, 128), lambda: _conv(64, 16, 16)),
    "conv_resident": (10000, lambda: _conv(128, 160, 16), lambda: _conv(128, 32, 16)),
    "bottom_mixed": (1000, lambda: _solves((64, 2, 62), True, MIXED), lambda: _solves((32, 2, 16), True, MIXED)),
}


@pytest.mark.parametrize("name", list(PAIRS))
def test_threads_with_different_sizes(name):
    times, much, little = PAIRS[name]
    errors, done = [], threading.Event()

    def work(make, leader):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                plan, call = make()
                with plan:
                    n = 0
                    while n < times if leader else not done.is_set():
                        call()
                        n += 1
                        if errors:
                            break
                    torch.cuda.current_stream().synchronize()
        except BaseException as e:      # noqa: B036 (reported by the test's thread)
            errors.append(e)
        finally:
            if leader:
                done.set()
    threads = [threading.Thread(target=work, args=a) for a in ((much, True), (little, False), (little, False))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
