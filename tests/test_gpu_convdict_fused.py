"""One dictionary step from a random state on both sides of the fused column pass's limits (a channel's
L column spectra in shared memory, FFT teams inside a warp), against the FP64 oracle.  GPU only.
Tolerances: the per-step bounds, 1e-5 (complex64) and 1e-10 (complex128), relative L2 on x and z."""
import numpy as np
import pytest

from oracle import fast
from paper_2006_08303_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,M,L,dtype", [(64, 1, 1, "f32"), (64, 3, 32, "f32"), (128, 2, 17, "f32"), (256, 2, 32, "f32"),
                                         (512, 2, 31, "f32"), (1024, 1, 25, "f32"), (1024, 1, 27, "f32"),
                                         (2048, 1, 2, "f32"), (64, 2, 5, "f64"), (512, 1, 26, "f64"), (512, 1, 27, "f64"),
                                         (1024, 1, 2, "f64")])
@pytest.mark.parametrize("mu", [0.0, 0.3])
def test_dictionary_step(N, M, L, dtype, mu):
    import torch
    from paper_2006_08303_gb300 import api
    if mu and N > 512:
        pytest.skip("the gradient penalty does not depend on the column pass's form")
    lam, rho, beta, P = 0.15, 8.0, 4.0, 7
    rng = np.random.default_rng(N + L)
    real = np.float32 if dtype == "f32" else np.float64
    r = lambda *s: rng.standard_normal(s).astype(real).astype(np.float64)  # noqa: E731
    h = inputs.gaussian_psf_bank(N, M, M).astype(real).astype(np.float64)
    d = inputs.gabor_filters(rng, L, P).astype(real).astype(np.float64)
    y, z, t, u = r(M, N, N), r(L, M, N, N), r(L, M, N, N), 0.1 * r(L, M, N, N)
    C = fast.convdict_setup(h, y, d, lam, rho, beta, mu)
    x1, z1, _, _ = fast.convdict_step(C, z, t, u)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a).astype(real)).cuda()  # noqa: E731
    plan = api.Plan(N, M, M, dtype)
    plan.set_prior("convdict", lam, rho, beta)
    plan.set_dictionary(dev(d))
    plan.set_code_gradient_weight(mu)
    plan.set_psfs(dev(h))
    plan.set_measurements(dev(y))
    plan.state_import_coefficients(*(dev(a.transpose(1, 0, 2, 3)) for a in (z, t, u)))
    plan.iterate(1)
    tol = 1e-5 if dtype == "f32" else 1e-10
    gx = plan.get_x().double().cpu().numpy()
    gz = plan.get_coefficients().double().cpu().numpy().transpose(1, 0, 2, 3)
    assert np.linalg.norm(gx - x1) <= tol * np.linalg.norm(x1)
    assert np.linalg.norm(gz - z1) <= tol * np.linalg.norm(z1)
