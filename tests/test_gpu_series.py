"""CholeskyQR2's second step by series (one cooperative launch): inputs whose second Gram matrix is I
exactly, near I and too far from I for the series, at sizes of one and several CTAs, eagerly and
replayed from a CUDA graph."""
import numpy as np
import pytest
import torch

import synth
from oracle import quaternion as Q
from oracle.qr import qr
from tests._qutil import dev_thin, host, small, small_to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", ["f32", "f64"])
@pytest.mark.parametrize("m,l", [(40, 1), (40, 2), (64, 17), (300, 64), (500, 130)])
@pytest.mark.parametrize("kind", ["identity", "spread", "ill"])
@pytest.mark.parametrize("graph", [False, True])
def test_cholqr2_series(dt, m, l, kind, graph):
    from paper_2507_13731_gb300 import build, qlr
    build.build()
    u = 2.0 ** -24 if dt == "f32" else 2.0 ** -53
    Y = np.zeros((4, m, l))
    if kind == "identity":
        Y[0, np.arange(l), np.arange(l)] = 1.0
    else:
        Y, _ = qr(synth.gaussian_qmat(3 + l, m, l))
        # ill: the first step leaves |E| ~ u kappa near the limit of the series or beyond it
        kappa = 1e2 if kind == "spread" else (2e5 if dt == "f32" else 1e7)
        V, _ = qr(synth.gaussian_qmat(4 + l, l, l))
        Y = Q.qmatmul(Y * np.logspace(0, -np.log10(kappa), l), Q.qH(V))
    s = torch.cuda.Stream()
    ctx = qlr.Context(0, s)
    Yd = dev_thin(Y, dt)
    Yh = host(Yd)
    Qd, R = qlr.empty_thin(m, l, Yd.dtype), small(l)
    ctx.reserve(qlr.workspace_size(m, max(l, 2), l, 0, 2, compute=qlr.COMPUTE_F64 if dt == "f64" else qlr.COMPUTE_AUTO))
    torch.cuda.synchronize()
    if graph:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            qlr.cholqr(ctx, Yd, Qd, R)
        for _ in range(2):
            Qd.fill_(float("nan"))
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
    else:
        qlr.cholqr(ctx, Yd, Qd, R)
    assert ctx.sync() == 0
    Qh, Rh = host(Qd), small_to_np(R)
    # every entry is a sum of l products of the working precision
    assert np.abs(Q.qmatmul(Q.qH(Qh), Qh) - Q.qeye(l)).max() <= 16 * (l + 4) * u
    assert np.abs(Q.qmatmul(Qh, Rh) - Yh).max() <= 16 * (l + 4) * u * np.abs(Yh).max()
    assert np.all(Rh[:, np.tril_indices(l, -1)[0], np.tril_indices(l, -1)[1]] == 0)
    ctx.close()
