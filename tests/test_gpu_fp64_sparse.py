"""FP64 tile kernel where few units have a kept process: W is fetched with a unit's first entry, in whichever
round of q'' that is.  Against the general kernel (fc4_rates_static; counts exact, 1e-10)."""
import numpy as np
import pytest

from synth import morse_system
from tests.helpers import assert_close, make_engine

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("mesh,sigma", [((8, 8, 9), 0.0005), ((8, 8, 9), 0.01), ((1, 40, 27), 0.002), ((3, 3, 3), 0.02)])
def test_first_entry_in_any_round(mesh, sigma):
    n = int(np.prod(mesh))
    e = make_engine(morse_system(seed=3), mesh, precision=0, inject=False)
    q = [n // 3, n - 2]
    g, wp, cnt = (x.cpu().numpy() for x in e.rates(300.0, sigma, 28, q_subset=q))
    G, WP, CNT = (x.cpu().numpy() for x in e.rates_static(300.0, sigma, 28, q))
    assert CNT.sum() and np.array_equal(cnt, CNT)
    assert_close(g[2:], G[2:], 1e-10, what="gamma")
    assert_close(wp[2:], WP[2:], 1e-10, what="wp")
    e.close()


def test_window_without_entries_costs_no_w():
    """With nothing kept FP64 does the window sweep of mixed precision at half its blocks per SM: at most twice
    the time (all modes of 3^3, ++; the fetch of W made it more)."""
    from paper_2510_00518_gb300 import Engine
    t = []
    for precision in (0, 1):
        e = Engine(*morse_system(seed=3), (3, 3, 3), precision=precision, timing=True)
        out, ms = None, []
        for _ in range(20):
            out = e.rates(300.0, 1e-9, 4, out=out)
            ms.append(e.timings()["4ph++"])
        assert int(out[2].sum()) == 0
        t.append(np.median(ms[5:]))
        e.close()
    print("ms", t)
    assert t[0] <= 2.0 * t[1], t


@pytest.mark.parametrize("mesh,sigma,adaptive", [((3, 3, 3), 0.1, False), ((5, 4, 3), 1.0, True)])
def test_one_atom(mesh, sigma, adaptive):
    """Cells of one atom (three blocks per SM) against the oracle."""
    import oracle
    from tests.helpers import modes_of
    from tests.test_gpu_adaptive_list import _system
    prob = oracle.Problem(*_system(1), mesh, sigma=sigma, sigma_adaptive=adaptive)
    e = make_engine(_system(1), mesh, precision=0, prob=prob)
    q = [1, int(np.prod(mesh)) - 1]
    G, WP, CNT = prob.rates(modes_of(q, 3), channel_mask=28)
    g, wp, cnt = (x.cpu().numpy() for x in e.rates(300.0, sigma, 28, q_subset=q, adaptive=adaptive))
    assert CNT[2:].sum() > 0 and np.array_equal(cnt, CNT)
    assert_close(g[2:], G[2:], 1e-10, what="gamma")
    assert_close(wp[2:], WP[2:], 1e-10, what="wp")
    e.close()
