"""Min-norm inverse of the DC bin of TV (g = 0) against numpy's pseudo-inverse, in FP64: odd and even M,
one channel, the largest M, full and deficient rank.  GPU only.

The first iterate from the zero state is Psi^+ beta Lambda^H F y, so its channel means are the DC bin.
Tolerance 1e-10, the FP64 per-step bound: the eigenvalues kept span at most ~1e6 here, times 2^-53."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,M", [(1, 1), (3, 2), (2, 3), (5, 5), (3, 8), (7, 15), (16, 16), (5, 16)])
@pytest.mark.parametrize("unit_sum", [False, True])
def test_dc_bin_is_the_min_norm_solution(K, M, unit_sum):
    import torch
    from paper_2006_08303_gb300 import api, inputs
    N, beta = 64, 1.5
    rng = np.random.default_rng(100 * K + M)
    h = inputs.gaussian_psf_bank(N, K, M)
    if not unit_sum:
        h = h * rng.uniform(0.2, 2.0, size=(K, M, 1, 1)) * rng.choice([-1.0, 1.0], size=(K, M, 1, 1))
    y = rng.standard_normal((K, N, N)) + 1.0
    P = api.Plan(N, K, M, "f64")
    P.set_prior("tv", 1e-2, 1.0, beta)
    P.set_psfs(torch.as_tensor(h).cuda())
    P.set_measurements(torch.as_tensor(y).cuda())
    P.iterate(1)
    got = P.get_x().mean((1, 2)).cpu().numpy()
    L = h.sum((2, 3))
    want = np.linalg.pinv(beta * L.T @ L, rcond=1e-10, hermitian=True) @ (beta * L.T @ y.mean((1, 2)))
    assert np.linalg.norm(got - want) <= 1e-10 * np.linalg.norm(want)
