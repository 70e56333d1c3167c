"""The tensor-core products of a tall FP32 operand at the ends of FP32's range: rows and columns far below
BF16's reach, infinities, NaN, sums next to the largest number.  FP32 multiply-adds are the measure."""
import pytest
import torch

from tests.test_gpu_tall_products import _gauss, _mul_bh, ctx  # noqa: F401

pytestmark = pytest.mark.gpu
M, N, K = 700, 613, 41            # m n k = 17.6e6: on the tensor cores
STEPS = -(-4 * K // 32) + 6       # as in test_gpu_tall_products: chunks of the sum, and the operands' roundings


def _operands():
    U, V = _gauss(1, 4, M, K), _gauss(2, 4, N, K)
    return U, V, torch.linspace(2, 1, K, dtype=torch.float64, device="cuda")


def _run(ctx, U, V, S):   # noqa: F811
    from paper_2507_13731_gb300 import qlr
    mask = torch.zeros(M, N, dtype=torch.uint8, device="cuda")
    C = torch.empty(4, M, N, device="cuda")
    qlr.complete_update(ctx, C, mask, C, qlr.to_thin(U), S, qlr.to_thin(V), K)
    assert ctx.sync() == 0
    return C.double(), _mul_bh(U.double() * S, V.double())


def _within(C, want, U, V, S):
    bound = 2 * STEPS * 2.0 ** -23 * ((U.double() * S).norm(dim=0).norm(dim=1)[:, None] * V.double().norm(dim=0).norm(dim=1)[None])
    err = (C - want).norm(dim=0)
    return bool((err <= bound).all()), float((err / bound).max())


@pytest.mark.parametrize("side", ["U", "V", "both", "S"])
@pytest.mark.parametrize("p", [-96, -104, -112, -118])
def test_small_rows(ctx, side, p):   # noqa: F811
    U, V, S = _operands()
    if side in ("U", "both"):
        U[:, ::3] *= 2.0 ** (p if side == "U" else p // 2)
    if side in ("V", "both"):
        V[:, ::7] *= 2.0 ** (p if side == "V" else p // 2)
    if side == "S":
        S = S * 2.0 ** p
    ok, worst = _within(*_run(ctx, U, V, S), U, V, S)
    assert ok, worst


@pytest.mark.parametrize("side", ["U", "V"])
@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
def test_not_finite(ctx, side, value):   # noqa: F811
    U, V, S = _operands()
    (U if side == "U" else V)[2, 130, 17] = value
    C, want = _run(ctx, U, V, S)
    hit = torch.zeros(M, N, dtype=torch.bool, device="cuda")
    if side == "U":
        hit[130] = True
    else:
        hit[:, 130] = True
    assert bool(torch.isfinite(want[:, ~hit]).all()) and not bool(torch.isfinite(want[:, hit]).any())
    assert torch.equal(torch.isnan(C), torch.isnan(want)) and torch.equal(C[:, hit].nan_to_num(), want[:, hit].float().double().nan_to_num())
    U[2, 130, 17] = V[2, 130, 17] = 0
    C[:, hit] = want[:, hit] = 0
    ok, worst = _within(C, want, U, V, S)
    assert ok, worst


def test_next_to_the_largest_number(ctx):   # noqa: F811
    U, V = torch.zeros(4, M, K, device="cuda"), torch.zeros(4, N, K, device="cuda")
    U[0, :, 3], V[0, :, 3] = 3.4e38, 0.5
    U[0, :, 4], V[0, :, 4] = 3.4e38, 0.498
    S = torch.ones(K, dtype=torch.float64, device="cuda")
    C, want = _run(ctx, U, V, S)
    assert bool((((C - want) / want[0].max()).abs() <= 2.0 ** -20).all())


def test_basis_of_a_matrix_with_small_rows(ctx):   # noqa: F811
    from paper_2507_13731_gb300 import qlr
    m, l = 7001, 64
    Y = _gauss(5, 4, m, l)
    Y[:, ::5] *= 2.0 ** -112
    Q, R = qlr.empty_thin(m, l), torch.empty(4, l, l, dtype=torch.float64, device="cuda")
    qlr.cholqr(ctx, qlr.to_thin(Y), Q, R)
    assert ctx.sync() == 0
    Rh = R.clone()                # stored column-major, R[c, j, i]: R^H before its conjugation
    Rh[1:] *= -1
    err = (_mul_bh(Q.double(), Rh) - Y.double()).norm(dim=0).norm(dim=1)
    # two products Q = Y R^{-1}, each a row's sum over at most 14 steps; R's condition number is below 2 and an
    # entry's bound holds l times in a row's norm
    assert bool((err <= 2 * 2 * 14 * 2.0 ** -23 * 2 * l ** 0.5 * Y.double().norm(dim=0).norm(dim=1)).all())
