"""General four-phonon kernel (cells of more than two atoms) at the edges of its item passes: several
pieces of W (more clusters than one piece holds), entries beyond one sub-batch, every block size,
fixed and adaptive σ, FP64 and mixed, against the oracle (counts exact, Γ and WP 1e-10 / 1e-4)."""
import numpy as np
import pytest

import oracle
from synth import diamond_crystal, morse_ifcs, random_cluster_ifcs, supercell_crystal
from tests.helpers import assert_close, make_engine, modes_of

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _system(atoms, n_random=0):
    c = supercell_crystal(diamond_crystal(), atoms // 2, np.linspace(15.0, 80.0, atoms))
    p2, p3, p4 = morse_ifcs(c, seed=4)
    if n_random:
        p4 = random_cluster_ifcs(c, 4, n_random, seed=7, scale=3.0)
    return c, p2, p3, p4


@pytest.mark.parametrize("atoms,mesh,n_random,sigma,adaptive,threads", [
    (4, (3, 2, 2), 0, 0.3, False, 128), (4, (4, 4, 5), 30, 0.05, False, 64), (4, (2, 3, 2), 350, 1.0, True, 96),
    (6, (2, 2, 1), 0, 0.2, False, 128), (8, (2, 1, 1), 0, 0.5, False, 96), (8, (3, 2, 1), 40, 1.5, True, 64)])
def test_general_kernel_edges(atoms, mesh, n_random, sigma, adaptive, threads):
    sysm = _system(atoms, n_random)
    prob = oracle.Problem(*sysm, mesh, sigma=sigma, sigma_adaptive=adaptive)
    q = [int(np.prod(mesh)) - 1]
    G, WP, CNT = prob.rates(modes_of(q, 3 * atoms), channel_mask=28)
    assert CNT.sum() > 0
    for precision, tol in ((0, 1e-10), (1, 1e-4)):
        e = make_engine(sysm, mesh, precision=precision, prob=prob, block_threads=threads)
        g, wp, cnt = (x.cpu().numpy() for x in e.rates(300.0, sigma, 28, q_subset=q, adaptive=adaptive))
        assert np.array_equal(cnt, CNT)
        floor = 1e-12 if precision == 0 else 1e-6
        assert_close(g[2:], G[2:], tol, floor_frac=floor, what="gamma")
        assert_close(wp[2:], WP[2:], tol, floor_frac=floor, what="wp")
        e.close()
