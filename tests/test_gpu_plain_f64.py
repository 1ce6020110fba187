"""complex128 iterations on both sides of the rule that launches their kernels plainly or programmatically: many
iterations alone, split into calls, and recorded in a batch give the same bits (a kernel that started before its
input was complete would not).  GPU only."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prior,N,M", [("l1", 256, 1), ("l1", 256, 2), ("tv", 256, 5), ("tv", 256, 6), ("dct8", 512, 4),
                                       ("dct8", 512, 5), ("wdct", 64, 3), ("wdct", 128, 8)])
def test_repeated_iterations_have_the_same_bits(prior, N, M):
    import torch
    from paper_2006_08303_gb300 import api

    def plan():
        g = torch.Generator(device="cuda").manual_seed(N + M)
        p = api.Plan(N, M, M, "f64", column_pass=2)
        p.set_prior(prior, 1e-2, 1.0)
        p.set_psfs(torch.rand(M, M, N, N, device="cuda", generator=g, dtype=torch.float64) / (N * N))
        p.set_measurements(torch.rand(M, N, N, device="cuda", generator=g, dtype=torch.float64))
        return p

    a, b, c = plan(), plan(), plan()
    a.iterate(24)
    for _ in range(24):
        b.iterate(1)
        torch.cuda.synchronize()
    batch = api.Batch([c])
    batch.iterate(24)
    for q in (b, c):
        assert torch.equal(a.get_x(), q.get_x()) and torch.equal(a.get_u(), q.get_u())
    batch.close()
