"""The truncation error of 3xTF32 sketches whose reduction is cut into equal pieces: that of chunks of at most
12 stages, however long the pieces are."""
import numpy as np
import pytest
import torch

import synth
from oracle import quaternion as Q
from tests._qutil import dev_thin, host

pytestmark = pytest.mark.gpu


# 51 row tiles take two pieces each of 24 stages (8 steps of the reduction); TMEM sums and sums in memory
@pytest.mark.parametrize("l", [40, 110])
@pytest.mark.parametrize("op", ["N", "H"])
@pytest.mark.parametrize("pure", [True, False])
def test_long_equal_pieces(l, op, pure):
    from paper_2507_13731_gb300 import build, qlr
    build.build()
    ctx = qlr.Context(0)
    m, n, planes = 6500, 376, 3 if pure else 4
    rows, cols = (m, n) if op == "N" else (n, m)
    A = qlr.empty_rowmajor(rows, cols, planes, torch.float32)
    A.copy_(torch.from_numpy(synth.gaussian_qmat(31, rows, cols)[4 - planes:]))
    X = dev_thin(synth.gaussian_qmat(32, n, l), "f32")
    Y = qlr.empty_thin(m, l)
    qlr.qsketch(ctx, qlr.OP_N if op == "N" else qlr.OP_H, A, X, Y, qlr.COMPUTE_TF32X3)
    assert ctx.sync() == 0
    Ah, Xh, Yh = host(A), host(X), host(Y)
    want = Q.qmatmul(Ah if op == "N" else Q.qH(Ah), Xh)
    # Each of the 3 products per stage and plane truncates the sum so far by half an ulp, 0.36 * 2^-23 of it on
    # average over mantissas; the sum of random terms after i of s steps is sqrt(i / s) of the last, 2 / 3 on average.
    # A quarter on top for the lo x lo product left out and the spread of the data.
    steps = 12 * 3 * planes
    tol = 1.25 * (2 / 3) * steps * 0.36 * 2.0 ** -23
    assert np.linalg.norm(Yh - want) <= tol * np.linalg.norm(want)
    ctx.close()
