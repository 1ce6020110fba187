"""The fault switch of the bounded waits (cip_set_test_fault) on priors whose row pass waits for nothing (T = I:
the l1 prior and the dictionary codes): there is no wait to give up, so nothing is reported or changed."""
import numpy as np
import pytest

from test_gpu_timeout import _plan
from paper_2006_08303_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prior", ["l1", "convdict"])
@pytest.mark.parametrize("N", [64, 256])
def test_the_switch_changes_nothing_without_a_staged_copy(prior, N):
    from paper_2006_08303_gb300 import api
    import torch
    P = inputs.tiny_tv(N=N, M=2, iters=3, dtype="f32")
    out = []
    for fault in (0, 1):
        if prior == "l1":
            P.prior = "l1"
            p = _plan(api, torch, P)
        else:
            f = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32).cuda()
            p = api.Plan(P.N, P.K, P.M, "f32")
            p.set_prior("convdict", P.lam, P.rho, P.beta)
            p.set_dictionary(f(np.eye(9).reshape(9, 3, 3)[:4]))
            p.set_psfs(f(P.h))
            p.set_measurements(f(P.y))
        p.set_test_fault(fault)
        p.iterate(3)
        p.residuals()
        out.append((p.get_x().cpu().numpy(), p.get_u().cpu().numpy()))
        p.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
