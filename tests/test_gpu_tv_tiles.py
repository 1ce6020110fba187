"""One TV step from a random state at every image size (each has its own row-group, walk or staging
form of the prior pass) and both FFT widths, against the FP64 oracle: the state makes the first and
last rows and columns, the borders of the 8-row tiles and of a warp's 64 columns all matter.  GPU only.

Tolerances are the repository's per-step bounds: 1e-5 (complex64), 1e-10 (complex128) on x and, at the
scale of u and T x, on u; the relative residuals, ratios of norms of the same quantities, to ten times
that."""
import numpy as np
import pytest

from oracle import admm, fast
from paper_2006_08303_gb300 import inputs

pytestmark = pytest.mark.gpu

CASES = [(N, "f32", 0) for N in (64, 128, 2048)] + [(N, "f32", e) for N in (256, 512, 1024) for e in (8, 16)] + [
    (N, "f64", 0) for N in (64, 256, 1024)]


@pytest.mark.parametrize("prior", ["tv", "tv_iso"])
@pytest.mark.parametrize("N,dtype,width", CASES)
def test_tv_step(N, dtype, width, prior):
    import torch
    from paper_2006_08303_gb300 import api
    K, M, lam, rho = 2, 2, 2e-2, 1.0
    rng = np.random.default_rng(N + width)
    x = inputs.rectangles_image(rng, N, M, n_rect=4)
    h = inputs.gaussian_psf_bank(N, K, M)
    y, _ = inputs.measure(rng, x, h, 30.0)
    t = 0.1 * rng.standard_normal((M, 2, N, N))
    u = 0.02 * rng.standard_normal((M, 2, N, N))
    real = np.float32 if dtype == "f32" else np.float64
    h, y, t, u = (a.astype(real).astype(np.float64) for a in (h, y, t, u))
    S = fast.analysis_setup(h, y, prior, lam, rho, 1.0)
    x1, t1, u1, w1 = fast.analysis_step(S, t, u)
    dev = lambda a: torch.as_tensor(a.astype(real)).cuda()  # noqa: E731
    P = api.Plan(N, K, M, dtype, prior_fft=width)
    P.set_prior(prior, lam, rho, 1.0)
    P.set_psfs(dev(h))
    P.set_measurements(dev(y))
    P.state_import(dev(t), dev(u))
    P.iterate(1)
    tol = 1e-5 if dtype == "f32" else 1e-10
    gx, gu = P.get_x().double().cpu().numpy(), P.get_u().double().cpu().numpy()
    assert np.linalg.norm(gx - x1) <= tol * np.linalg.norm(x1)
    assert np.linalg.norm(gu - u1) <= tol * max(np.linalg.norm(u1), np.linalg.norm(w1))
    assert np.max(np.abs(gu - u1)) <= 100 * tol * np.max(np.abs(w1))
    r, s = P.residuals()
    r1 = np.linalg.norm(w1 - t1) / max(np.linalg.norm(w1), np.linalg.norm(t1))
    s1 = np.linalg.norm(t1 - t) / np.linalg.norm(u1)
    assert abs(r - r1) <= 10 * tol * r1 and abs(s - s1) <= 10 * tol * s1
