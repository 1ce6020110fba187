"""Dictionary column pass on both sides of the rule that chooses between one kernel and three: the form that runs
(kernels per iteration: row pass and one or three), and one step against the FP64 oracle with the same
bounds as the fused pass's own test.  GPU only."""
import pytest

from test_gpu_convdict_fused import test_dictionary_step as check_step

pytestmark = pytest.mark.gpu

CASES = [(1024, 1, 7, "f32", 3), (1024, 1, 8, "f32", 1), (512, 1, 1, "f32", 1), (1024, 11, 1, "f32", 3),
         (1024, 12, 1, "f32", 1), (128, 5, 1, "f64", 1), (256, 1, 4, "f64", 1),
         (256, 2, 3, "f64", 1), (256, 2, 4, "f64", 3), (256, 3, 1, "f64", 3), (512, 1, 3, "f64", 1), (512, 1, 4, "f64", 3)]


@pytest.mark.parametrize("N,M,L,dtype,kernels", CASES)
def test_form_and_step(N, M, L, dtype, kernels):
    import torch
    from paper_2006_08303_gb300 import api
    real = torch.float32 if dtype == "f32" else torch.float64
    g = torch.Generator(device="cuda").manual_seed(N + L)
    p = api.Plan(N, M, M, dtype)
    p.set_prior("convdict", 1e-2, 1.0)
    p.set_dictionary(torch.rand(L, 3, 3, device="cuda", generator=g, dtype=real))
    p.set_psfs(torch.rand(M, M, N, N, device="cuda", generator=g, dtype=real) / (N * N))
    p.set_measurements(torch.rand(M, N, N, device="cuda", generator=g, dtype=real))
    p.iterate(2)
    n0 = p.launches()
    p.iterate(5)
    n1 = p.launches()
    p.iterate(10)
    assert (p.launches() - n1) - (n1 - n0) == 5 * (1 + kernels)
    p.close()
    if M <= 8:  # the oracle's setup at 1024^2 with 12 channels takes minutes
        check_step(N, M, L, dtype, 0.0)
