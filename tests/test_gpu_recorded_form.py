"""Column-pass form of iterations recorded for a batch: where a plan alone runs the fused form without the
ring, the autotuner keeps the faster of the other two for them.  GPU only; the decisions go through the
tuning file, in processes of their own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import torch
from paper_2006_08303_gb300 import api
def plan(N, M, prior):
    g = torch.Generator(device="cuda").manual_seed(N + M)
    p = api.Plan(N, M, M, "f32")
    p.set_prior(prior, 1e-3, 1e-2)
    p.set_psfs(torch.rand(M, M, N, N, device="cuda", generator=g) / (N * N))
    p.set_measurements(torch.rand(M, N, N, device="cuda", generator=g))
    return p
"""


def run(code, cache):
    subprocess.run([sys.executable, "-c", CODE + code], cwd=ROOT, check=True, timeout=300,
                   env=dict(os.environ, CIP_TUNE_CACHE=str(cache), PYTHONPATH=ROOT))


def test_the_recorded_form_of_a_decision_is_the_one_that_runs(tmp_path):
    f = tmp_path / "tune.txt"
    # N M dtype prior form tile variant [recorded form]; forms: 1 ring (one kernel), 2 split (three), 3 no ring
    f.write_text("128 2 0 0 3 1 0 2\n128 3 0 0 3 1 0 1\n64 2 0 2 3 1 0\n256 2 0 0 2 0 0 2\n")
    run("""
for N, M, prior, kernels in ((128, 2, "tv", 4), (128, 3, "tv", 2), (64, 2, "l1", 2), (256, 2, "tv", 4)):
    a, b = plan(N, M, prior), plan(N, M, prior)
    a.iterate(6)
    batch = api.Batch([b])
    n0 = b.launches()
    batch.iterate(6)
    assert b.launches() - n0 == 6 * kernels + 1, (N, M, b.launches() - n0)  # the last one is the residual sum
    assert torch.equal(a.get_x(), b.get_x()) and torch.equal(a.get_u(), b.get_u())
    batch.close()
""", f)


def test_the_autotuner_keeps_a_recorded_form(tmp_path):
    f = tmp_path / "tune.txt"
    run("""
for N, M in ((1024, 1), (1024, 3), (64, 3)):
    a, b = plan(N, M, "tv"), plan(N, M, "tv")
    a.iterate(4)
    batch = api.Batch([b])
    batch.iterate(4)
    assert torch.equal(a.get_x(), b.get_x())
    batch.close()
""", f)
    lines = [list(map(int, s.split())) for s in f.read_text().splitlines()]
    assert len(lines) == 3
    for n in lines:
        assert n[7] in (1, 2) and (n[4] == 3 or n[7] == n[4]), n
