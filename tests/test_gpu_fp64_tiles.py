"""FP64 products, Gram and masked update at the edges of their tiles (8 x 4 and 16 x 8 outputs, 32
reduction steps; 8 x 32 outputs in the update) against the FP64 oracle, element by element."""
import numpy as np
import pytest
import torch

import synth
from oracle import quaternion as Q
from tests._qutil import dev_rowmajor, dev_thin, host, small, small_to_np

pytestmark = pytest.mark.gpu
U64 = 2.0 ** -53


@pytest.fixture(scope="module")
def ctx():
    from paper_2507_13731_gb300 import build, qlr
    build.build()
    c = qlr.Context(0)
    yield c
    c.close()


# 2-row, tile-edge and one-past-edge sizes; the last two give enough tiles for 16 x 8
@pytest.mark.parametrize("m,n,l", [(2, 3, 1), (8, 32, 4), (9, 33, 5), (7, 65, 3), (401, 97, 113), (640, 31, 64)])
def test_fp64_products_at_tile_edges(ctx, m, n, l):
    from paper_2507_13731_gb300 import qlr
    A = synth.gaussian_qmat(31 + m, m, n)
    Ad = dev_rowmajor(A, "f64")
    for op, rin, rout in (("N", n, m), ("H", m, n)):
        X = synth.gaussian_qmat(32 + n, rin, l)
        Y = qlr.empty_thin(rout, l, torch.float64)
        qlr.qsketch(ctx, qlr.OP_N if op == "N" else qlr.OP_H, Ad, dev_thin(X, "f64"), Y, qlr.COMPUTE_F64)
        assert ctx.sync() == 0
        Aop = A if op == "N" else Q.qH(A)
        # 4 rin products per component, each rounded once when added: below 4 rin u sum |a| |x|
        assert np.all(Q.qnorm(host(Y) - Q.qmatmul(Aop, X)) <= 8 * rin * U64 * (Q.qnorm(Aop) @ Q.qnorm(X)))


@pytest.mark.parametrize("m,l", [(1, 1), (31, 4), (33, 5), (300, 15), (1000, 65), (97, 130)])
def test_fp64_gram_chunks(ctx, m, l):
    from paper_2507_13731_gb300 import qlr
    Y = synth.gaussian_qmat(41 + m, m, l)
    G = qlr.qgram(ctx, dev_thin(Y, "f64"), small(l))
    assert ctx.sync() == 0
    got, want = small_to_np(G), Q.qmatmul(Q.qH(Y), Y)
    bound = 8 * m * U64 * (Q.qnorm(Q.qH(Y)) @ Q.qnorm(Y))
    assert np.all(Q.qnorm(got - want) <= bound)
    assert np.array_equal(got, Q.qH(got))       # the full Hermitian matrix is written


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (8, 32, 8), (9, 33, 9), (70, 45, 3)])
def test_fp64_masked_update(ctx, m, n, k):
    from paper_2507_13731_gb300 import qlr
    M, U, V = (synth.gaussian_qmat(51 + i, *s) for i, s in enumerate([(m, n), (m, k), (n, k)]))
    S = np.linspace(2.0, 1.0, k)
    mask = (synth.uniform(55, m * n).reshape(m, n) < 0.5).astype(np.uint8)
    C = torch.full((4, m, n), np.nan, dtype=torch.float64, device="cuda")
    qlr.complete_update(ctx, dev_rowmajor(M, "f64"), torch.from_numpy(mask).cuda(), C, dev_thin(U, "f64"),
                        torch.from_numpy(S).cuda(), dev_thin(V, "f64"), k)
    assert ctx.sync() == 0
    X = Q.qmatmul(U * S[None, None, :], Q.qH(V))
    want = np.where(mask[None] != 0, M, X)
    err = Q.qnorm(host(C) - want)
    assert np.all(err[mask != 0] == 0.0)
    assert np.all(err <= 8 * (k + 1) * U64 * (Q.qnorm(U * S[None, None, :]) @ Q.qnorm(Q.qH(V))))
