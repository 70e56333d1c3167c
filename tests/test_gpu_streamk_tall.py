"""Stream-K sketches of more tiles than SMs, few of which are cut: one, two and more column blocks, and
reductions of a few stages (cuts that fall on tile boundaries)."""
import pytest

from tests import test_gpu_streamk_pieces as base

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,l", [(19457, 200, 17), (20033, 90, 130), (25601, 33, 200), (38913, 64, 40)])
@pytest.mark.parametrize("mode,dt", [("TF32X3", "f32"), ("TF32", "f32"), ("TF32_RN", "f32"), ("BF16", "bf16")])
@pytest.mark.parametrize("op", ["N", "H"])
def test_many_tiles(m, n, l, mode, dt, op):
    base.test_pieces(m, n, l, mode, dt, op)
