"""One 3D dictionary step from a random state for odd, even, one and sixteen channels, few and many
filters (complex128 with 16 channels and 32 filters takes the smaller bin tile), against the FP64 oracle.
GPU only.  Tolerances: the per-step bounds, 1e-5 (complex64) and 1e-10 (complex128), relative L2."""
import numpy as np
import pytest

from oracle import fast
from paper_2006_08303_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,L,Q,dtype", [(1, 3, 1, "f32"), (2, 1, 2, "f32"), (3, 9, 2, "f32"), (5, 7, 5, "f32"), (7, 2, 3, "f32"),
                                         (10, 8, 3, "f32"), (13, 5, 4, "f32"), (16, 32, 3, "f32"), (15, 4, 3, "f64"),
                                         (16, 32, 2, "f64"), (4, 6, 3, "f64")])
def test_step(M, L, Q, dtype):
    import torch
    from paper_2006_08303_gb300 import api
    N, P, lam, rho, beta = 64, 5, 0.15, 8.0, 4.0
    rng = np.random.default_rng(100 * M + L)
    real = np.float32 if dtype == "f32" else np.float64
    r = lambda *s: rng.standard_normal(s).astype(real).astype(np.float64)  # noqa: E731
    h = inputs.gaussian_psf_bank(N, M, M).astype(real).astype(np.float64)
    d = 0.1 * r(L, Q, P, P)
    d = d.astype(real).astype(np.float64)
    y, z, t, u = r(M, N, N), r(L, M, N, N), r(L, M, N, N), r(L, M, N, N)
    C = fast.convdict3d_setup(h, y, d, lam, rho, beta)
    x1, z1, _, _ = fast.convdict3d_step(C, z, t, u)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a).astype(real)).cuda()  # noqa: E731
    plan = api.Plan(N, M, M, dtype)
    plan.set_prior("convdict", lam, rho, beta)
    plan.set_dictionary_3d(dev(d))
    plan.set_psfs(dev(h))
    plan.set_measurements(dev(y))
    plan.state_import_coefficients(*(dev(a.transpose(1, 0, 2, 3)) for a in (z, t, u)))
    plan.iterate(1)
    tol = 1e-5 if dtype == "f32" else 1e-10
    gx = plan.get_x().double().cpu().numpy()
    gz = plan.get_coefficients().double().cpu().numpy().transpose(1, 0, 2, 3)
    assert np.linalg.norm(gx - x1) <= tol * np.linalg.norm(x1)
    assert np.linalg.norm(gz - z1) <= tol * np.linalg.norm(z1)
