"""FP64 cores of more than 128 columns: the cluster form with 6 and 8 rows a lane, and the first size
beyond it."""
import pytest

from tests import test_gpu_core_sizes as base
from tests.test_gpu_core_sizes import ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("l", [129, 192, 193, 256, 257])
@pytest.mark.parametrize("kind", ["spread", "repeated"])
def test_core_fp64_sizes(ctx, l, kind):   # noqa: F811
    base.test_core_sizes(ctx, l, 0, kind)
