"""Autotuner decisions of dictionary plans are kept per number of maps M L and for 2D and 3D apart: the row pass of one filter and of 32
fill the device differently, so a plan's width must not depend on which plan came first.  GPU only; the
decisions go through the tuning file, in processes of their own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import torch
from paper_2006_08303_gb300 import api
def plan(L, Q=0):
    g = torch.Generator(device="cuda").manual_seed(L)
    p = api.Plan(256, 2, 2, "f32")
    p.set_prior("convdict", 1e-3, 1e-2)
    if Q: p.set_dictionary_3d(torch.rand(L, Q, 3, 3, device="cuda", generator=g))
    else: p.set_dictionary(torch.rand(L, 3, 3, device="cuda", generator=g))
    p.set_psfs(torch.rand(2, 2, 256, 256, device="cuda", generator=g) / 65536)
    p.set_measurements(torch.rand(2, 256, 256, device="cuda", generator=g))
    return p
width = lambda p: p.config()["prior_fft_elems"]
"""


def run(code, cache):
    subprocess.run([sys.executable, "-c", CODE + code], cwd=ROOT, check=True, timeout=300,
                   env=dict(os.environ, CIP_TUNE_CACHE=str(cache), PYTHONPATH=ROOT))


def test_each_number_of_maps_has_its_own_decision(tmp_path):
    f = tmp_path / "tune.txt"
    # N M dtype prior form tile variant recorded [maps]; widths of the variants 0, 1, 2: 8, 16, 32
    f.write_text("256 2 0 3 1 1 0 1 4\n256 2 0 3 1 1 1 1 10\n256 2 0 3 1 1 0 1 -10\n256 2 0 3 1 1 2 1\n")
    run("""
assert [width(plan(L)) for L in (2, 5, 3)] == [8, 16, 32]  # the last one: a line for any dictionary
assert width(plan(5, Q=2)) == 8 and width(plan(3, Q=2)) == 32  # -10: the 3D dictionary of 10 maps
""", f)
    assert len(f.read_text().splitlines()) == 4


def test_the_autotuner_keeps_a_decision_per_number_of_maps(tmp_path):
    f = tmp_path / "tune.txt"
    run("""
a, b, c, d = plan(1), plan(32), plan(1), plan(32, Q=2)
assert width(a) == width(c)
""", f)
    lines = [list(map(int, s.split())) for s in f.read_text().splitlines()]
    assert sorted(n[8] for n in lines) == [-64, 2, 64], lines
