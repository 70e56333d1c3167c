"""Stream-K sketches whose tiles are reduced in many pieces (few tiles, a long reduction), in few, and in
column-block groups: the pieces' sum against the FP64 product, element by element, and the same bits on a
second call into a poisoned output."""
import numpy as np
import pytest
import torch

import synth
from oracle import quaternion as Q
from tests._qutil import dev_rowmajor, dev_thin, host

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24


# rows x reduction x columns: one tile of up to 152 pieces; 3 tiles; a ragged last tile and column
# block; several column blocks; nearly one tile per SM
@pytest.mark.parametrize("m,n,l", [(100, 9000, 15), (129, 5000, 33), (300, 2600, 70), (257, 3000, 130), (700, 1100, 200),
                                   (9601, 640, 17)])
@pytest.mark.parametrize("mode,dt", [("TF32X3", "f32"), ("TF32", "f32"), ("TF32_RN", "f32"), ("BF16", "bf16")])
@pytest.mark.parametrize("op", ["N", "H"])
def test_pieces(m, n, l, mode, dt, op):
    from paper_2507_13731_gb300 import build, qlr
    build.build()
    ctx = qlr.Context(0)
    rows, cols = (m, n) if op == "N" else (n, m)      # the reduction is n long either way
    A = qlr.empty_rowmajor(rows, cols, 3, {"f32": torch.float32, "bf16": torch.bfloat16}[dt])
    A.copy_(torch.from_numpy(synth.gaussian_qmat(5 + m, rows, cols)[1:]))
    X = dev_thin(synth.gaussian_qmat(6 + l, n, l), "f32")
    Y = qlr.empty_thin(m, l)
    outs = []
    for _ in range(2):
        Y.fill_(float("nan"))
        qlr.qsketch(ctx, qlr.OP_N if op == "N" else qlr.OP_H, A, X, Y, getattr(qlr, "COMPUTE_" + mode))
        assert ctx.sync() == 0
        outs.append(host(Y))
    assert np.array_equal(outs[0], outs[1])
    Ah, Xh = host(A), host(X.to(torch.bfloat16)) if mode == "BF16" else host(X)
    Aop = Ah if op == "N" else Q.qH(Ah)
    # operands: 2^-9 for truncated, 2^-10 for rounded TF32, 2^-19 for its hi / lo split; sums: half an
    # ulp for each of up to n accumulations, as in the other sketch tests
    tol = {"TF32X3": 2.0 ** -19, "TF32": 2.0 ** -9, "TF32_RN": 2.0 ** -10, "BF16": 0.0}[mode] + 4.0 * n * U32
    bound = 2 * tol * (Q.qnorm(Aop) @ Q.qnorm(Xh)) + 1e-30
    assert np.all(Q.qnorm(outs[0] - Q.qmatmul(Aop, Xh)) <= bound)
    ctx.close()
