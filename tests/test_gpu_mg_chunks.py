"""The coarse operator's form with 5 to 8 chunks per thread (11 to 14 test vectors),
as the others in test_gpu_mg_kernels.py."""
import pytest

from test_gpu_mg_kernels import SMALL, WIDE
from test_gpu_mg_kernels import test_restriction_and_coarse_operator as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,n", [(SMALL, 11), (SMALL, 14), (WIDE, 12)])
def test_coarse_operator_with_eight_chunks(shape, n):
    check(shape, n)
