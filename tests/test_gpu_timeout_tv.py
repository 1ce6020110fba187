"""The bounded wait of the TV prior passes that stage u in shared memory (complex64, N <= 512): a wait that
gives up (cip_set_test_fault: nothing in flight, 64 polls) is reported and leaves the iterate what it is,
as for the DCT prior.  Forms without a staged copy do not wait, and the switch changes nothing there."""
import numpy as np
import pytest

from test_gpu_timeout import CIP_ERR_TIMEOUT, _plan
from paper_2006_08303_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prior", ["tv", "tv_iso"])
@pytest.mark.parametrize("N,width,waits", [(64, 0, True), (128, 0, True), (256, 8, True), (256, 16, True), (512, 8, True),
                                           (512, 16, True), (1024, 0, False)])
def test_timeout_is_reported_and_the_iterate_is_the_same(prior, N, width, waits):
    from paper_2006_08303_gb300 import api
    import torch
    P = inputs.tiny_tv(N=N, M=2, iters=3, dtype="f32")
    P.prior = prior
    out = []
    for fault in (0, 1):
        p = _plan(api, torch, P, prior_fft=width)
        p.set_test_fault(fault)
        p.iterate(3)
        if fault and waits:
            with pytest.raises(api.CipError) as ei:
                p.residuals()
            assert ei.value.status == CIP_ERR_TIMEOUT
        else:
            p.residuals()
        out.append((p.get_x().cpu().numpy(), p.get_u().cpu().numpy()))
        if fault:  # switched off and reset, the same plan runs cleanly
            p.set_test_fault(0)
            p.reset_state()
            p.iterate(3)
            p.residuals()
            assert np.array_equal(p.get_x().cpu().numpy(), out[0][0])
        p.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
