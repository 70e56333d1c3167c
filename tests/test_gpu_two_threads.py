"""One context per host thread, each on its own stream: launches of the same kernels at different sizes."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


def test_contexts_in_two_threads():
    from paper_2507_13731_gb300 import build, qlr
    build.build()
    errors = []

    def work(l, seed):
        try:
            torch.cuda.set_device(0)
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                c = qlr.Context(0, s)
                g = torch.Generator(device="cuda")
                g.manual_seed(seed)
                A = torch.randn(4, 200, 160, generator=g, device="cuda")
                X = qlr.to_thin(torch.randn(4, 160, l, generator=g, device="cuda"))
                Y, Q = qlr.empty_thin(200, l), qlr.empty_thin(200, l)
                R = torch.empty(4, l, l, dtype=torch.float64, device="cuda")
                L, T = (torch.empty(4, l, l, dtype=torch.float64, device="cuda") for _ in range(2))
                S = torch.empty(l, dtype=torch.float64, device="cuda")
                first = None
                for _ in range(400):
                    qlr.qsketch(c, qlr.OP_N, A, X, Y)
                    qlr.cholqr(c, Y, Q, R)
                    qlr.qtsvd(c, R, l, L, S, T, qlr.F32)
                    if first is None:
                        assert c.sync() == 0
                        first = (Y.clone(), Q.clone(), S.clone())
                assert c.sync() == 0
                assert all(torch.equal(a, b) for a, b in zip(first, (Y, Q, S)))
                c.close()
        except Exception as e:   # noqa: BLE001
            errors.append((l, repr(e)))

    threads = [threading.Thread(target=work, args=(l, i)) for i, l in enumerate((17, 33, 48, 70))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
