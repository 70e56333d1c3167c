"""Tensor-core masked updates of rank <= 8 (one stage per tile) whose split over the SMs makes a CTA
begin on the last column tile of its rows: one of the two issuing warps then has no stage of those rows."""
import pytest
import torch

from tests.test_gpu_tall_products import _gauss, _mul_bh, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k", [(4096, 4200, 8), (1860, 2297, 8), (2297, 1860, 7), (4097, 3701, 2)])
def test_range_from_a_last_column_tile(ctx, m, n, k):   # noqa: F811
    from paper_2507_13731_gb300 import qlr
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ntiles, tiles = -(-m // 32), -(-n // 128) * -(-m // 32)
    cuts = [tiles * b // sms for b in range(sms + 1)]
    assert any(t0 % ntiles == ntiles - 1 and t1 > t0 + 1 for t0, t1 in zip(cuts, cuts[1:])) or sms not in (148, 152)
    U, V = qlr.to_thin(_gauss(1, 4, m, k)), qlr.to_thin(_gauss(2, 4, n, k))
    S = torch.linspace(2, 1, k, dtype=torch.float64, device="cuda")
    mask = torch.zeros(m, n, dtype=torch.uint8, device="cuda")
    want = _mul_bh(U.double() * S, V.double())
    # every row block of the tall operand far from its neighbours': a tile of stale rows stands out
    scale = 4.0 ** (torch.arange(n, device="cuda") // 128 % 3)
    Vs = qlr.to_thin(V * scale[None, :, None])
    bound = 2 * 8 * 2.0 ** -23 * ((U.double() * S).norm(dim=0) @ (Vs.double()).norm(dim=0).T)
    for _ in range(10):
        C = torch.full((4, m, n), float("nan"), device="cuda")
        qlr.complete_update(ctx, C, mask, C, U, S, Vs, k)
        assert ctx.sync() == 0
        err = (C.double() - want * scale).norm(dim=0)
        assert bool((err <= bound).all()), float((err / bound).max())
