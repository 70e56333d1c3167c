"""Core QSVDs on several streams at once, beside sketches that fill the GPU: the CTAs that replay a QSVD's
rotations wait for the ones that sweep, in whatever order the GPU places them."""
import pytest
import torch

from tests.test_gpu_tall_products import _gauss

pytestmark = pytest.mark.gpu


def test_core_qsvds_beside_each_other():
    from paper_2507_13731_gb300 import build, qlr
    build.build()
    jobs = []
    for i, (l, prec) in enumerate([(180, qlr.F32), (250, qlr.F32), (40, qlr.F32), (100, qlr.F64), (20, qlr.F64), (180, qlr.F32)]):
        s = torch.cuda.Stream()
        R = torch.triu(_gauss(i, 4, l, l)).transpose(1, 2).contiguous().double()
        out = [torch.empty(4, l, l, dtype=torch.float64, device="cuda") for _ in range(2)]
        jobs.append((qlr.Context(0, s), R, l, prec, out, torch.empty(l, dtype=torch.float64, device="cuda")))
    s = torch.cuda.Stream()
    c = qlr.Context(0, s)
    A, X, Y = _gauss(9, 4, 8192, 4096), qlr.to_thin(_gauss(10, 4, 4096, 110)), qlr.empty_thin(8192, 110)
    torch.cuda.synchronize()

    def run(j):
        ctx, R, l, prec, out, S = j
        qlr.qtsvd(ctx, R, l, out[0], S, out[1], prec)

    alone = []
    for j in jobs:
        run(j)
        assert j[0].sync() == 0
        alone.append((j[5].clone(), j[4][0].clone(), j[4][1].clone()))
    torch.cuda.synchronize()
    for _ in range(10):
        for j in jobs:
            qlr.qsketch(c, qlr.OP_N, A, X, Y)
            run(j)
    for j, want in zip(jobs, alone):
        assert j[0].sync() == 0
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip((j[5], *j[4]), want))
    assert c.sync() == 0
    for j in jobs:
        j[0].close()
    c.close()
