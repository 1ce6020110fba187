"""One step of the wavelet x channel-DCT prior from a random state with 16- and 32-wide subband tiles
(the wide ones run from two CTAs per SM on) and every band size, against the FP64 oracle.  GPU only.
Tolerances: the per-step bounds, 1e-5 (complex64) and 1e-10 (complex128)."""
import numpy as np
import pytest

from oracle import fast
from paper_2006_08303_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,M,dtype", [(64, 1, "f32"), (128, 3, "f32"), (256, 16, "f32"), (512, 4, "f32"), (512, 5, "f32"),
                                       (1024, 2, "f32"), (2048, 1, "f32"), (512, 5, "f64"), (128, 2, "f64")])
def test_wavelet_step(N, M, dtype):
    import torch
    from paper_2006_08303_gb300 import api
    lam, rho = 5e-2, 0.5
    rng = np.random.default_rng(N + M)
    real = np.float32 if dtype == "f32" else np.float64
    r = lambda *s: rng.standard_normal(s).astype(real).astype(np.float64)  # noqa: E731
    h = inputs.disk_gaussian_psf_bank(N, M, M).astype(real).astype(np.float64)
    y, t, u = r(M, N, N), 0.2 * r(M, 1, N, N), 0.1 * r(M, 1, N, N)
    t, u = (a.astype(real).astype(np.float64) for a in (t, u))
    S = fast.analysis_setup(h, y, "wdct", lam, rho, 1.0)
    x1, t1, u1, w1 = fast.analysis_step(S, t, u)
    dev = lambda a: torch.as_tensor(a.astype(real)).cuda()  # noqa: E731
    P = api.Plan(N, M, M, dtype)
    P.set_prior("wdct", lam, rho, 1.0)
    P.set_psfs(dev(h))
    P.set_measurements(dev(y))
    P.state_import(dev(t), dev(u))
    P.iterate(1)
    tol = 1e-5 if dtype == "f32" else 1e-10
    gx, gu = P.get_x().double().cpu().numpy(), P.get_u().double().cpu().numpy()
    assert np.linalg.norm(gx - x1) <= tol * np.linalg.norm(x1)
    assert np.linalg.norm(gu - u1) <= tol * max(np.linalg.norm(u1), np.linalg.norm(w1))
    r0, s0 = P.residuals()
    r1 = np.linalg.norm(w1 - t1) / max(np.linalg.norm(w1), np.linalg.norm(t1))
    s1 = np.linalg.norm(t1 - t) / np.linalg.norm(u1)
    assert abs(r0 - r1) <= 10 * tol * r1 and abs(s0 - s1) <= 10 * tol * s1
