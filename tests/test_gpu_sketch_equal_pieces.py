"""FP32-accurate sketches of few tiles whose reduction is cut into equal pieces (down to one stage) against the
FP64 product, element by element; with and without a pure A, and the same bits from a poisoned output."""
import numpy as np
import pytest
import torch

import synth
from oracle import quaternion as Q
from tests._qutil import dev_thin, host

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24


# rows x reduction x columns: one stage in all; fewer stages than SMs; a remainder stage; 76 and 77 row
# tiles (two pieces each, and none); column-block groups; the last length below 24 stages a piece
@pytest.mark.parametrize("m,n,l", [(5, 7, 3), (100, 100, 15), (517, 389, 23), (9728, 65, 9), (9729, 65, 9),
                                   (390, 517, 140), (1500, 600, 100), (128, 24 * 152 * 8 - 8, 16)])
@pytest.mark.parametrize("mode", ["TF32X3", "TF32_RN"])
@pytest.mark.parametrize("op", ["N", "H"])
@pytest.mark.parametrize("pure", [True, False])
def test_equal_pieces(m, n, l, mode, op, pure):
    from paper_2507_13731_gb300 import build, qlr
    build.build()
    ctx = qlr.Context(0)
    rows, cols = (m, n) if op == "N" else (n, m)      # the reduction is n long either way
    planes = 3 if pure else 4
    A = qlr.empty_rowmajor(rows, cols, planes, torch.float32)
    A.copy_(torch.from_numpy(synth.gaussian_qmat(5 + m, rows, cols)[4 - planes:]))
    X = dev_thin(synth.gaussian_qmat(6 + l, n, l), "f32")
    Y = qlr.empty_thin(m, l)
    outs = []
    for _ in range(2):
        Y.fill_(float("nan"))
        qlr.qsketch(ctx, qlr.OP_N if op == "N" else qlr.OP_H, A, X, Y, getattr(qlr, "COMPUTE_" + mode))
        assert ctx.sync() == 0
        outs.append(host(Y))
    assert np.array_equal(outs[0], outs[1])
    Ah, Xh = host(A), host(X)
    Aop = Ah if op == "N" else Q.qH(Ah)
    # operands: 2^-19 for the hi / lo split, 2^-10 for rounded TF32; sums: half an ulp for each of up to
    # n accumulations, as in the other sketch tests
    tol = {"TF32X3": 2.0 ** -19, "TF32_RN": 2.0 ** -10}[mode] + 4.0 * n * U32
    bound = 2 * tol * (Q.qnorm(Aop) @ Q.qnorm(Xh)) + 1e-30
    assert np.all(Q.qnorm(outs[0] - Q.qmatmul(Aop, Xh)) <= bound)
    ctx.close()
