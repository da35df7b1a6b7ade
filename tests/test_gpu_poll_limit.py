"""The one-launch solve's bounded wait: when it runs out the call fails, and the plan stays usable."""
import ctypes
import math

import pytest
import torch

from paper_2609_07172_gb300 import Plan, workloads as W
from paper_2609_07172_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("dims", [(32, 16, 32), (90, 32, 70)], ids=lambda d: "x".join(map(str, d)))
def test_a_wait_that_runs_out_is_an_error(dims, graph):
    p = W.annulus(*dims)
    rho = torch.from_numpy(W.rho_plasma(p, 5)).cuda()
    with Plan(p, graph=graph) as plan:
        want, first = plan.solve(rho, tol=1e-10)
        plan.set_poll_limit(0)          # no block looks for the others even once
        with pytest.raises(B.PicPoissonError, match="ran out") as e:
            plan.solve(rho, tol=1e-10)
        assert e.value.status == B.ECUDA
        info = B.Info()
        phi = torch.empty_like(want)
        assert B.load().pic_poisson_solve(plan._plan, ctypes.c_void_p(rho.data_ptr()), ctypes.c_void_p(phi.data_ptr()),
                                          1e-10, ctypes.byref(info)) == B.ECUDA
        assert info.status == B.ECUDA and math.isnan(info.rel_res) and math.isnan(info.rel_res0)
        plan.set_poll_limit(1 << 22)
        again, last = plan.solve(rho, tol=1e-10)
        assert torch.equal(again, want) and (last["cycles"], last["rel_res"]) == (first["cycles"], first["rel_res"])
        with pytest.raises(B.PicPoissonError):
            plan.set_poll_limit(-1)
