"""The TV step test at the complex128 sizes whose register budget differs (two CTAs per SM from N = 128 on).  GPU only."""
import pytest

from test_gpu_tv_tiles import test_tv_step as check_step

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prior", ["tv", "tv_iso"])
@pytest.mark.parametrize("N", [128, 512])
def test_step(N, prior):
    check_step(N, "f64", 0, prior)
