"""The masked update keeps its operand splits apart from the workspace of the other calls: streams, graphs
captured before it, and what it refuses."""
import pytest
import torch

from tests.test_gpu_tall_products import _gauss

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2507_13731_gb300 import build
    build.build()


def _update_case(seed, m, n, k):
    from paper_2507_13731_gb300 import qlr
    U, V = qlr.to_thin(_gauss(seed, 4, m, k)), qlr.to_thin(_gauss(seed + 1, 4, n, k))
    S = torch.linspace(2, 1, k, dtype=torch.float64, device="cuda")
    return torch.empty(4, m, n, device="cuda"), torch.zeros(m, n, dtype=torch.uint8, device="cuda"), U, S, V, k


def _update(c, t):
    from paper_2507_13731_gb300 import qlr
    C, mask, U, S, V, k = t
    return qlr.complete_update(c, C, mask, C, U, S, V, k)


def _done(t):
    """A copy of a result of the context's stream."""
    torch.cuda.synchronize()
    return t.clone()


def _sketch_case(m, n, l):
    from paper_2507_13731_gb300 import qlr
    return _gauss(7, 4, m, n), qlr.to_thin(_gauss(8, 4, n, l)), qlr.empty_thin(m, l)


def test_update_beside_a_sketch_on_another_stream():
    from paper_2507_13731_gb300 import qlr
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    c = qlr.Context(0, s1)
    c.reserve(1 << 30)
    A, X, Y = _sketch_case(8192, 8192, 110)
    one, two = _update_case(1, 3000, 3000, 40), _update_case(3, 2000, 2500, 50)
    torch.cuda.synchronize()
    want_y = _done(qlr.qsketch(c, qlr.OP_N, A, X, Y))
    want1, want2 = _done(_update(c, one)), _done(_update(c, two))
    for _ in range(5):
        for t in (Y, one[0], two[0]):
            t.zero_()
        torch.cuda.synchronize()
        for _ in range(3):
            qlr.qsketch(c, qlr.OP_N, A, X, Y)
        c.set_stream(s2)
        _update(c, one)
        c.set_stream(s1)
        _update(c, two)
        qlr.qsketch(c, qlr.OP_N, A, X, Y)
        torch.cuda.synchronize()
        assert torch.equal(Y, want_y) and torch.equal(one[0], want1) and torch.equal(two[0], want2)
    c.close()


def test_update_after_a_capture_on_the_same_context():
    from paper_2507_13731_gb300 import qlr
    s = torch.cuda.Stream()
    c = qlr.Context(0, s)
    A, X, Y = _sketch_case(600, 500, 20)
    big = _update_case(5, 3000, 3000, 200)      # needs far more than the sketch's workspace
    torch.cuda.synchronize()
    want = _done(qlr.qsketch(c, qlr.OP_N, A, X, Y))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        qlr.qsketch(c, qlr.OP_N, A, X, Y)
    ref = _done(_update(c, big))
    Y.zero_()
    big[0].zero_()
    torch.cuda.synchronize()
    _update(c, big)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(Y, want) and torch.equal(big[0], ref)
    c.close()


def test_a_captured_update_does_not_depend_on_the_workspace():
    from paper_2507_13731_gb300 import qlr
    got = []
    for reserve in (0, 1 << 28):
        s = torch.cuda.Stream()
        c = qlr.Context(0, s)
        t = _update_case(9, 700, 613, 41)
        c.reserve(reserve)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            _update(c, t)
        g.replay()
        torch.cuda.synchronize()
        got.append(t[0].clone())
        c.close()
    assert torch.equal(*got)


@pytest.mark.parametrize("k", [0, 1])
def test_too_many_rows_are_refused(k):
    from paper_2507_13731_gb300 import qlr
    c = qlr.Context(0)
    c.reserve(1 << 28)
    C, mask, U, S, V, _ = _update_case(11, 65535 * 32 + 1, 8, 1)
    with pytest.raises(qlr.QlrError) as e:
        qlr.complete_update(c, C, mask, C, U, S, V, k)
    assert e.value.code == qlr.EUNSUPPORTED
    c.close()
