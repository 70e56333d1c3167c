"""The tensor-core products of a tall FP32 operand (three BF16 splits per operand, six products): the
masked update and the QR's Q = Y R^{-1} at the edges of their tiles (128 rows, 32 columns, 16
reduction elements per MMA, 160 in the resident operand, chunks of 16 or 32)."""
import pytest
import torch

pytestmark = pytest.mark.gpu
TERMS = [[(0, 0, 1), (1, 1, 1), (2, 2, 1), (3, 3, 1)], [(1, 0, 1), (0, 1, -1), (3, 2, 1), (2, 3, -1)],
         [(2, 0, 1), (0, 2, -1), (1, 3, 1), (3, 1, -1)], [(3, 0, 1), (0, 3, -1), (2, 1, 1), (1, 2, -1)]]   # a conj(b)


@pytest.fixture(scope="module")
def ctx():
    from paper_2507_13731_gb300 import build, qlr
    build.build()
    c = qlr.Context(0)
    yield c
    c.close()


def _gauss(seed, *shape):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(*shape, generator=g, device="cuda")


def _mul_bh(U, V):
    """U V^H of quaternion matrices in FP64 planes."""
    return torch.stack([sum(s * (U[a] @ V[b].T) for a, b, s in t) for t in TERMS])


@pytest.mark.parametrize("m,n,k", [(4097, 3701, 1), (2049, 1900, 4), (1000, 3333, 5), (700, 613, 40), (613, 700, 41),
                                   (1000, 257, 64), (1000, 257, 65), (641, 129, 200), (500, 127, 256), (301, 200, 257)])
@pytest.mark.parametrize("in_place", [False, True])
def test_masked_update(ctx, m, n, k, in_place):
    from paper_2507_13731_gb300 import qlr
    U, V = (qlr.to_thin(_gauss(s, 4, r, k + 1)) for s, r in ((1, m), (2, n)))
    # singular values over six decades, rows of U over four
    S = torch.logspace(3, -3, k, dtype=torch.float64, device="cuda")
    U *= torch.logspace(-2, 2, m, device="cuda")[None, :, None]
    M = _gauss(3, 3, m, n)
    mask = (_gauss(4, m, n) < -0.5).to(torch.uint8)
    C = torch.full((4, m, n), float("nan"), device="cuda")
    src = M
    if in_place:
        C[0], C[1:] = 0, M
        src = C
    qlr.complete_update(ctx, src, mask, C, U, S, V, k)
    assert ctx.sync() == 0
    Us, Vd = U[:, :, :k].double() * S, V[:, :, :k].double()
    seen = mask.bool()
    want = torch.where(seen, torch.cat([torch.zeros_like(M[:1]), M]).double(), _mul_bh(Us, Vd))
    err = (C.double() - want).norm(dim=0)
    assert float(err[seen].max()) == 0.0
    # U S rounds once (2^-24); a chunk of 32 reduction elements loses at most a few ulps of its sum in the
    # tensor cores, and the chunks are added in FP32 (2^-24 each).  k = 257 runs in FP32.
    steps = -(-4 * k // 32) + 6 if k <= 256 else 2 * k
    bound = 2 * steps * 2.0 ** -23 * (Us.norm(dim=0) @ Vd.norm(dim=0).T)
    assert bool((err <= bound).all()), float((err / bound).max())


@pytest.mark.parametrize("m,l", [(40001, 25), (7001, 60), (6016, 64), (6019, 65), (2001, 110), (3000, 180), (700, 256),
                                 (700, 260)])
def test_cholqr_basis(ctx, m, l):
    from paper_2507_13731_gb300 import qlr
    Y = qlr.to_thin(_gauss(5, 4, m, l) * torch.logspace(0, -2, l, device="cuda"))
    Q, R = qlr.empty_thin(m, l), torch.empty(4, l, l, dtype=torch.float64, device="cuda")
    qlr.cholqr(ctx, Y, Q, R)
    assert ctx.sync() == 0
    Qh = Q.double().clone()
    Qh[1:] *= -1                      # conj(Q): conj(Q)^T Q through a conj(b) product of transposes
    G = _mul_bh(Qh.transpose(1, 2), Qh.transpose(1, 2))
    # a Q entry is a sum over at most 22 MMAs per accumulator (or l FP32 terms), relative to its row's
    # norm; Q^H Q differs from I by twice that over unit columns
    assert float((G - torch.eye(l, device="cuda") * torch.tensor([1., 0, 0, 0], device="cuda")[:, None, None]).abs().max()) < 1e-5
    Rt = R.transpose(1, 2)            # stored column-major: R[c, j, i]
    Rh = Rt.clone().transpose(1, 2)
    Rh[1:] *= -1                      # R^H, so that Q (R^H)^H = Q R
    err = (_mul_bh(Q.double(), Rh) - Y.double()).abs().max()
    assert float(err) < 1e-5 * float(Y.abs().max())


def test_masked_update_with_a_full_workspace(ctx):
    """A capturing stream cannot grow the workspace: the update runs all the same, in FP32."""
    from paper_2507_13731_gb300 import qlr
    m, n, k = 600, 500, 50
    s = torch.cuda.Stream()
    c = qlr.Context(0, s)
    U, V, S = qlr.to_thin(_gauss(1, 4, m, k)), qlr.to_thin(_gauss(2, 4, n, k)), torch.ones(k, dtype=torch.float64, device="cuda")
    M, mask, C = _gauss(3, 4, m, n), torch.zeros(m, n, dtype=torch.uint8, device="cuda"), torch.zeros(4, m, n, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        qlr.complete_update(c, M, mask, C, U, S, V, k)
    g.replay()
    torch.cuda.synchronize()
    want = _mul_bh(U.double(), V.double())
    assert float((C.double() - want).abs().max()) < 1e-5 * float(want.abs().max())
    c.close()
