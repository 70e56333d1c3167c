"""The core QSVD at the sizes where its kernels change: one CTA (1, 2, 3 or 4 rows a lane; FP32 below 57,
FP64 below 25), the cluster (1, 2, 4, 6 or 8 rows a lane) and the single-CTA form for cores too
large for either, against the FP64 adjoint's singular values."""
import numpy as np
import pytest
import torch

import synth
from oracle import quaternion as Q
from oracle.qr import qr
from tests._qutil import np_to_small, small, small_to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2507_13731_gb300 import build, qlr
    build.build()
    c = qlr.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("l,prec", [(l, 1) for l in (1, 2, 3, 16, 17, 32, 33, 48, 49, 56, 57, 64, 65, 128, 129, 192, 193,
                                                     256, 257)] +
                         [(l, 0) for l in (1, 2, 15, 16, 17, 24, 25, 32, 33, 64, 65)])
@pytest.mark.parametrize("kind", ["spread", "repeated", "deficient"])
def test_core_sizes(ctx, l, prec, kind):
    from paper_2507_13731_gb300 import qlr
    i = np.arange(l)
    sig = {"spread": 1.0 / (1 + i), "repeated": 2.0 - (i // 4 % 2), "deficient": np.where(i < (l + 1) // 2, 1.0 / (1 + i), 0.0)}[kind]
    U, _ = qr(synth.gaussian_qmat(7 + l, l, l))
    V, _ = qr(synth.gaussian_qmat(8 + l, l, l))
    R = Q.qmatmul(U * sig, Q.qH(V))
    k = max(1, l - 1)
    L, Rt, S = small(l, k), small(l, k), torch.zeros(k, dtype=torch.float64, device="cuda")
    qlr.qtsvd(ctx, np_to_small(R), k, L, S, Rt, prec)
    assert ctx.sync() == 0
    u = 2.0 ** -24 if prec == 1 else 2.0 ** -53
    # a pair counts as orthogonal below 8 sqrt(l) u, and each of its columns meets l others
    tol = 8 * np.sqrt(l) * u
    S, L, Rt = S.cpu().numpy(), small_to_np(L), small_to_np(Rt)
    want = np.sort(sig)[::-1][:k]
    np.testing.assert_allclose(S, want, atol=4 * l * u * sig.max())
    assert np.all(np.diff(S) <= tol * sig.max())
    on = want > 0                      # the right vectors of a zero singular value are not defined
    assert np.abs(Q.qmatmul(R, Rt) - L * S)[:, :, on].max() <= 2 * np.sqrt(l) * tol * sig.max()
    for X in (L, Rt[:, :, on]):
        assert np.abs(Q.qmatmul(Q.qH(X), X) - Q.qeye(X.shape[2])).max() <= 2 * np.sqrt(l) * tol
