"""The W scratch of the tiled four-phonon path between captured and eager calls of one context: whatever runs
between two calls with the same arguments, both give the same bits."""
import numpy as np
import pytest

from synth import morse_system
from tests.helpers import make_engine

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SUB = [3, 11, 20]


def _engine(precision):
    return make_engine(morse_system(seed=3), (3, 3, 3), precision=precision, inject=False)


def _capture(fn):
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
        out = fn()
    torch.cuda.synchronize()
    return g, out


def _rates(e, mask):
    return e.rates(300.0, 0.1, mask, q_subset=SUB)


def _same(a, b):
    return all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("mask,other", [(12, 16), (16, 12), (8, 28)])
def test_captured_rates_beside_eager_calls(precision, mask, other):
    """mask's channels share a sign of W, so that the W of the call before could serve; other leaves another."""
    e = _engine(precision)
    dL = torch.ones((5, 6 * len(SUB)), dtype=torch.float64, device="cuda")
    ref = [x.clone() for x in _rates(e, mask)]
    ref_o = [x.clone() for x in _rates(e, other)]
    _rates(e, mask)
    g, out = _capture(lambda: _rates(e, mask))
    for between in (lambda: None, lambda: _rates(e, other), lambda: (_rates(e, mask), e.backward(dL))):
        between()
        for x in out:
            x.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert _same(out, ref)
    # eager calls beside replays that leave another W behind
    h, out_o = _capture(lambda: _rates(e, other))
    _rates(e, mask)
    h.replay()
    assert _same(_rates(e, mask), ref) and _same(out_o, ref_o)
    e.close()


@pytest.mark.parametrize("mask", [12, 16])
def test_captured_backward_beside_eager_rates(mask):
    e = _engine(0)
    dL = torch.tensor(np.random.default_rng(1).uniform(0.5, 1.5, (5, 6 * len(SUB))), device="cuda")
    _rates(e, mask)
    ref = [x.clone() for x in e.backward(dL)]
    rates = [x.clone() for x in _rates(e, mask)]
    g, out = _capture(lambda: e.backward(dL))
    for _ in range(2):
        assert _same(_rates(e, mask), rates)
        for x in out:
            x.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert _same(out, ref)
    e.close()


def test_captured_backward_keeps_its_scratch():
    """A larger W allowed after the capture: the graph's own buffer lives as long as the context."""
    e = _engine(0)
    dL = torch.tensor(np.random.default_rng(1).uniform(0.5, 1.5, (5, 6 * len(SUB))), device="cuda")
    e.set_mode_chunk(0, 4 * e.memory()["w_per_mode"])
    _rates(e, 28)
    ref = [x.clone() for x in e.backward(dL)]
    g, out = _capture(lambda: e.backward(dL))
    small = e.memory()["w_buffer"]
    e.set_mode_chunk(0, 0)
    rates = [x.clone() for x in _rates(e, 28)]
    assert e.memory()["w_buffer"] > small
    for _ in range(2):
        g.replay()
        torch.cuda.synchronize()
        assert _same(out, ref) and _same(_rates(e, 28), rates)
    e.close()
