"""The fused column pass without the ring gives the ring kernel's bits: every size, one channel to the
most it takes, more bins than solving threads and the reverse, several iterations.  The autotuner's
decision file selects it, in a process of its own.  GPU only."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

SIZES = [(64, 1), (64, 3), (64, 8), (128, 2), (128, 5), (256, 1), (256, 4), (256, 8), (512, 3), (512, 8), (1024, 1), (1024, 5),
         (1024, 7)]

CODE = """
import sys, torch
from paper_2006_08303_gb300 import api
for N, M in %r:
    g = torch.Generator(device="cuda").manual_seed(N + M)
    h = torch.rand(M, M, N, N, device="cuda", generator=g) / (N * N)
    y = torch.rand(M, N, N, device="cuda", generator=g)
    out = []
    for kw in ({}, {"column_pass": 1}):
        P = api.Plan(N, M, M, "f32", **kw)
        P.set_prior("l1", 1e-3, 1e-2)
        P.set_psfs(h)
        n0 = P.launches()
        P.set_measurements(y)
        assert kw or P.launches() - n0 == 3, "the decision of the file was not taken"
        P.iterate(3)
        out.append((P.get_x(), P.get_u()))
    assert all(torch.equal(a, b) for a, b in zip(*out)), (N, M)
"""


def test_same_bits_as_the_ring(tmp_path):
    f = tmp_path / "tune.txt"
    f.write_text("".join(f"{N} {M} 0 2 3 1 0\n" for N, M in SIZES))  # N M dtype prior form tile variant
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    subprocess.run([sys.executable, "-c", CODE % (SIZES,)], cwd=root, check=True, timeout=300,
                   env=dict(os.environ, CIP_TUNE_CACHE=str(f), PYTHONPATH=root))
