"""Allocation-free sketches whose staged operand would leave little or none of the scratch array: pure and full
quaternion A, the widest blocks of the fused staging, long reductions."""
import pytest
import torch

from tests.test_gpu_tall_products import _gauss

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("planes,m,n,l,op", [(3, 10000, 20000, 60, "N"), (3, 20000, 10000, 60, "H"), (4, 4000, 30000, 30, "N"),
                                             (3, 3000, 20000, 100, "N"), (3, 1000, 60000, 60, "N")])
@pytest.mark.parametrize("compute", ["TF32X3", "TF32"])
def test_noalloc_long_reduction(planes, m, n, l, op, compute):
    from paper_2507_13731_gb300 import build, qlr
    build.build()
    comp, o = getattr(qlr, "COMPUTE_" + compute), getattr(qlr, "OP_" + op)
    A = _gauss(1, planes, m, n)
    k, r = (n, m) if op == "N" else (m, n)
    X = qlr.to_thin(_gauss(2, 4, k, l))
    Y, W = qlr.empty_thin(r, l), qlr.empty_thin(r, l)
    qlr.qsketch_noalloc(o, A, X, Y, comp)
    c = qlr.Context(0)
    qlr.qsketch(c, o, A, X, W, comp)
    assert c.sync() == 0
    torch.cuda.synchronize()
    # sums of 4 k products of unit size in other pieces: each of at most a few hundred roundings of the running
    # sum differs, and a TF32 accumulator truncates at every one of its 4 k / 8 additions
    tol = (64 if compute == "TF32X3" else 4 * k / 8) * 2.0 ** -23 * (4 * k) ** 0.5
    assert float((Y - W).abs().max()) <= tol * 6
    c.close()
