"""The filter update divides a bin's filters and sums between two groups of threads, four filters at a
time: filter counts below, at and beside multiples of four and eight, both support classes (<= 16, <= 32), the smallest and largest channel counts,
and the residuals of a check, against the oracle."""
import numpy as np
import pytest

from test_gpu_dictlearn import BETA, LAM, RHO, fast, learning_plan, problem, rel, torch  # noqa: F401

pytestmark = pytest.mark.gpu

# float32: the bounds of the parity tests beside this file (rounding of 3 steps)
CASES = [(64, 1, L, P) for L, P in ((1, 3), (2, 3), (3, 17), (4, 5))] + \
        [(64, 8, 5, 17), (128, 4, 31, 11), (64, 6, 32, 16)]


@pytest.mark.parametrize("dtype,tol", [("f32", 1e-4), ("f64", 1e-9)])
@pytest.mark.parametrize("N,M,L,P", CASES)
def test_filter_groups(torch, N, M, L, P, dtype, tol):  # noqa: F811
    h, y, d0 = problem(seed=17, N=N, K=2, M=M, L=L, Pf=P)
    sigma, iters = 5.0, 3
    x_or, _, _, _, f_or = fast.run_convdict_learn(h, y, d0, LAM, RHO, BETA, sigma, iters)
    got = []
    for every in (0, 1):  # with the check's residual sums and without
        plan, _ = learning_plan(torch, h, y, d0, LAM, RHO, BETA, sigma, dtype, check_every=every)
        plan.iterate(iters)
        got.append((plan.get_x().double().cpu().numpy(), plan.get_dictionary().double().cpu().numpy()))
        plan.close()
    x, f = got[0]
    assert rel(f, f_or) <= tol, rel(f, f_or)
    assert rel(x, x_or) <= tol, rel(x, x_or)
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])


def test_learning_in_a_batch_equals_alone(torch):  # noqa: F811
    """The three launches recorded into a batch's graph: bit for bit the plan alone."""
    from paper_2006_08303_gb300 import api

    def plans():
        out = []
        for N, M, L, P in ((64, 3, 5, 7), (128, 5, 9, 11)):
            h, y, d0 = problem(seed=23, N=N, K=2, M=M, L=L, Pf=P)
            out.append(learning_plan(torch, h, y, d0, LAM, RHO, BETA, 5.0)[0])
        return out

    alone, together = plans(), plans()
    for p in alone:
        p.iterate(8)
    batch = api.Batch(together)
    batch.iterate(8)
    for a, b in zip(alone, together):
        assert torch.equal(a.get_x(), b.get_x()) and torch.equal(a.get_dictionary(), b.get_dictionary())
    batch.close()
    for p in alone + together:
        p.close()
