"""Which force constants the triangular partner domains are used for: those whose leg-exchange symmetry holds to
rounding (3ph-, the FP64 gradient) or to 1e-12 (4ph rates), with one stored cluster for each exchanged one."""
import numpy as np
import pytest

import oracle
from synth import morse_system
from tests.helpers import assert_close, make_engine, modes_of
from tests.test_gpu_rates3 import _check

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _evaluated(sysm, ch):
    e = make_engine(sysm, (4, 4, 4), inject=False)
    e.rates(300.0, 0.3, 1 << ch)
    st = e.stats()
    e.close()
    return st["evaluated"][ch], st["kept"][ch]


def test_nearly_symmetric_phi3_takes_the_rectangle():
    """An asymmetry of 9e-13 of max |Φ3| moves 3ph- by 8e-10 where soft modes weigh it (the half domain counts one
    of |V(λ', λ'')|² and |V(λ'', λ')|² twice); the oracle's sum is the rectangular one."""
    sysm = morse_system(seed=3)
    phi, mx = sysm[2].phi, np.abs(sysm[2].phi).max()
    exact, noise = phi.copy(), np.random.default_rng(0).uniform(-0.5, 0.5, phi.shape)
    phi[:] = exact * (1 + 2e-16 * np.sign(noise))                       # rounding only
    n, kept = _evaluated(sysm, 1)
    assert n < kept
    phi[:] = exact + 9e-13 * mx * noise
    n, kept = _evaluated(sysm, 1)
    assert n == kept
    _check(sysm, (1, 1, 127), [3, 60], 4.0, False)


def test_repeated_cluster_takes_the_rectangle():
    """One Φ4 cluster stored twice, its leg-exchanged ones once: V is not symmetric though every stored tensor has
    its transposed partner.  Rates and gradient against the oracle (1e-10, 1e-8 as elsewhere)."""
    c, p2, p3, p4 = morse_system(seed=3)
    legs = [[(a, *x) for a, x in zip(at[1:], cell.tolist())] for at, cell in zip(p4.atoms.tolist(), p4.cells)]
    k = next(i for i, x in enumerate(legs) if x[0] != x[1] and x[1] != x[2])
    for name in ("atoms", "cells", "phi"):
        setattr(p4, name, np.concatenate([getattr(p4, name), getattr(p4, name)[k:k + 1]]))
    mesh, q = (3, 2, 2), [4]
    prob = oracle.Problem(c, p2, p3, p4, mesh, sigma=0.3)
    G, WP, CNT = prob.rates(modes_of(q, 6), channel_mask=28)
    assert CNT.sum() > 0
    e = make_engine((c, p2, p3, p4), mesh, prob=prob)
    g, wp, cnt = (x.cpu().numpy() for x in e.rates(300.0, 0.3, 28, q_subset=q))
    assert np.array_equal(cnt, CNT)
    assert_close(g[2:], G[2:], 1e-10, what="gamma")
    assert_close(wp[2:], WP[2:], 1e-10, what="wp")
    dL = np.random.default_rng(2).uniform(0.5, 1.5, (5, 6))
    dL[:2] = 0.0
    d4 = e.backward(torch.tensor(dL, device="cuda"))[1].cpu().numpy()
    assert_close(d4.reshape(-1), prob.grad(modes_of(q, 6), dL)[1].reshape(-1), 1e-8, floor_frac=1e-9, what="dphi4")
    e.close()


@pytest.mark.parametrize("call", ["rates", "static", "backward"])
def test_replays_after_the_symmetry_is_gone(call):
    """Captured with symmetric force constants, replayed with ones that are not (and back): as the eager call then,
    to the bit."""
    c, p2, p3, p4 = morse_system(seed=3)
    rng = np.random.default_rng(4)
    broken = [p.phi + 0.1 * np.abs(p.phi).max() * rng.normal(size=p.phi.shape) for p in (p3, p4)]
    e = make_engine((c, p2, p3, p4), (3, 3, 3), inject=False)
    sub = [3, 11, 20]
    dL = torch.tensor(rng.uniform(0.5, 1.5, (5, 18)), device="cuda")
    run = {"rates": lambda: e.rates(300.0, 0.3, 3, q_subset=sub),
           "static": lambda: e.rates_static(300.0, 0.3, 3, sub),
           "backward": lambda: e.backward(dL)}[call]
    e.rates(300.0, 0.3, 31, q_subset=sub)
    run()
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
        out = run()
    for phi3, phi4 in (broken, (p3.phi, p4.phi), broken):
        e.update_anharmonic(phi3, phi4)
        g.replay()
        torch.cuda.synchronize()
        got = [x.clone() for x in out]
        assert all(torch.equal(x, y) for x, y in zip(got, run()))
    e.close()
