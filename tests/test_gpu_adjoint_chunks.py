"""The FP64 gradient after rates that were chunked mode by mode, or with a W scratch of few modes: as fast as
after unchunked rates where the cap of the scratch allows it (it was 20 times slower with the chunks of the
rates; 3 leaves room for noise), and the same gradient in any case."""
import time

import numpy as np
import pytest

from synth import morse_system
from tests.helpers import make_engine

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _engine(mesh, chunk=0, w_modes=0):
    e = make_engine(morse_system(seed=3), mesh, precision=0, inject=False)
    e.set_mode_chunk(chunk, w_modes * e.memory()["w_per_mode"])
    return e


def _gradient(e, sub=None):
    nm = 6 * (e.nq if sub is None else len(sub))
    dL = torch.tensor(np.random.default_rng(1).uniform(0.5, 1.5, (5, nm)), device="cuda")
    e.rates(300.0, 0.1, 31, q_subset=sub)
    out = e.backward(dL)
    t = []
    for _ in range(3):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        e.backward(dL)
        torch.cuda.synchronize()
        t.append(time.perf_counter() - t0)
    return out, min(t)


def test_gradient_after_mode_by_mode_rates():
    ref, t_ref = _gradient(_engine((4, 4, 4)))
    out, t = _gradient(_engine((4, 4, 4), chunk=1))
    assert all(torch.equal(x, y) for x, y in zip(out, ref))
    assert t <= 3.0 * t_ref, (t, t_ref)


@pytest.mark.parametrize("mesh,sub,w_modes", [((3, 3, 3), None, 1), ((3, 3, 3), None, 25), ((3, 3, 3), [5, 7], 1),
                                              ((2, 3, 2), None, 9)])
def test_gradient_within_a_capped_scratch(mesh, sub, w_modes):
    """Many small chunks (the general adjoint: rounding only, 1e-12 of the largest entry), few and larger ones."""
    ref, _ = _gradient(_engine(mesh), sub)
    e = _engine(mesh, w_modes=w_modes)
    out, _ = _gradient(e, sub)
    assert e.memory()["w_buffer"] <= w_modes * e.memory()["w_per_mode"]
    assert torch.equal(out[0], ref[0])
    assert (out[1] - ref[1]).abs().max() <= 1e-12 * ref[1].abs().max()


def test_shared_w_after_memory_was_short():
    """++ and +- share W where there is memory for H beside it.  A gradient without that memory does without, and the
    next one with it takes it again; the same bits either way."""
    e = _engine((8, 8, 8))
    sub = [7, 100, 200, 300]
    dL = torch.ones((5, 24), dtype=torch.float64, device="cuda")
    e.rates(300.0, 0.1, 12, q_subset=sub)
    e.backward(dL)
    h = 24 * e.memory()["w_per_mode"]
    assert e.memory()["w_buffer"] == h
    ref = e.backward(dL)[1].clone()
    full = e.memory()["total"]
    e.close()
    e = _engine((8, 8, 8))
    e.rates(300.0, 0.1, 12, q_subset=sub)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    rest = torch.empty(torch.cuda.mem_get_info()[0] - h // 2, dtype=torch.uint8, device="cuda")
    assert torch.equal(e.backward(dL)[1], ref)
    assert e.memory()["total"] == full - h
    del rest
    torch.cuda.empty_cache()
    assert torch.equal(e.backward(dL)[1], ref)
    assert e.memory()["total"] == full
    e.close()
