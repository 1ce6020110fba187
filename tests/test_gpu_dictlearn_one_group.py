"""The filter update at the sizes where one group of threads per bin runs instead of two, beside the sizes of its
other test: same problems, same bounds.  GPU only."""
import pytest

from test_gpu_dictlearn import torch  # noqa: F401
from test_gpu_dictlearn_groups import test_filter_groups as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,M,L,P,dtype", [(256, 8, 5, 11, "f32"), (256, 7, 3, 17, "f32"), (512, 1, 9, 17, "f32"), (512, 6, 2, 5, "f32"),
                                           (512, 5, 2, 5, "f32"), (256, 1, 9, 17, "f64"), (256, 7, 3, 5, "f64"), (256, 8, 2, 5, "f64"),
                                           (512, 2, 5, 11, "f64")])
def test_groups_and_step(torch, N, M, L, P, dtype):  # noqa: F811
    check(torch, N, M, L, P, dtype, 1e-4 if dtype == "f32" else 1e-9)
