"""One step of the complex128 priors that run the row pass (T = I, and the row transforms of the wavelet chain) from a
random state at the sizes where its tile or FFT width changes, against the FP64 oracle.  GPU only.
Tolerances: the per-step bound of complex128, 1e-10, on x and, at the scale of u and T x, on u; the relative
residuals, ratios of norms of the same quantities, to ten times that."""
import numpy as np
import pytest

from oracle import fast
from paper_2006_08303_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prior,N,M", [("l1", 64, 1), ("l1", 64, 3), ("l1", 128, 2), ("l1", 256, 1), ("l1", 256, 3),
                                       ("l1", 512, 2), ("wdct", 64, 2), ("wdct", 128, 1), ("wdct", 256, 2)])
def test_step(prior, N, M):
    import torch
    from paper_2006_08303_gb300 import api
    lam, rho, tol = 2e-2, 1.0, 1e-10
    rng = np.random.default_rng(N + M)
    h = inputs.gaussian_psf_bank(N, M, M)
    y, _ = inputs.measure(rng, inputs.rectangles_image(rng, N, M, n_rect=4), h, 30.0)
    t, u = 0.1 * rng.standard_normal((M, 1, N, N)), 0.02 * rng.standard_normal((M, 1, N, N))
    S = fast.analysis_setup(h, y, prior, lam, rho, 1.0)
    x1, t1, u1, w1 = fast.analysis_step(S, t, u)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()  # noqa: E731
    P = api.Plan(N, M, M, "f64")
    P.set_prior(prior, lam, rho, 1.0)
    P.set_psfs(dev(h))
    P.set_measurements(dev(y))
    P.state_import(dev(t), dev(u))
    P.iterate(1)
    gx, gu = P.get_x().cpu().numpy(), P.get_u().cpu().numpy()
    assert np.linalg.norm(gx - x1) <= tol * np.linalg.norm(x1)
    assert np.linalg.norm(gu - u1) <= tol * max(np.linalg.norm(u1), np.linalg.norm(w1))
    r, s = P.residuals()
    r1 = np.linalg.norm(w1 - t1) / max(np.linalg.norm(w1), np.linalg.norm(t1))
    s1 = np.linalg.norm(t1 - t) / np.linalg.norm(u1)
    assert abs(r - r1) <= 10 * tol * r1 and abs(s - s1) <= 10 * tol * s1
