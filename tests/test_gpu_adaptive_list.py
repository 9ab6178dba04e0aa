"""Adaptive ++ and -- by the candidate list (cells of one and two atoms, FP64 and mixed): rounds of 128
and 256 points just short of full, full and just over, windows that keep hardly anything and nearly
everything (the list at its longest), against the oracle: counts exact, Γ and WP 1e-10 (FP64) and 1e-4
(mixed) as for the other kernels."""
import numpy as np
import pytest

import oracle
from synth import diamond_crystal, morse_ifcs, random_cluster_ifcs, supercell_crystal
from tests.helpers import assert_close, make_engine, modes_of

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _system(atoms):
    c = supercell_crystal(diamond_crystal(), 1)
    if atoms == 2:
        return (c,) + morse_ifcs(c, seed=2)
    c.positions, c.masses = c.positions[:1], c.masses[:1]
    p2 = random_cluster_ifcs(c, 2, 6, seed=1, scale=0.5)
    p2.atoms = np.concatenate([p2.atoms, [[0, 0]]]).astype(np.int32)
    p2.cells = np.concatenate([p2.cells, np.zeros((1, 1, 3))]).astype(np.int32)
    p2.phi = np.concatenate([p2.phi, [np.diag([10.0, 40.0, 160.0]).reshape(-1)]])
    return c, p2, random_cluster_ifcs(c, 3, 10, seed=2), random_cluster_ifcs(c, 4, 20, seed=3)


@pytest.mark.parametrize("atoms,mesh,scale", [
    (2, (3, 2, 1), 30.0), (2, (5, 5, 5), 0.05), (2, (4, 4, 8), 8.0), (2, (3, 5, 9), 1.0), (2, (4, 8, 8), 0.3),
    (1, (5, 3, 17), 2.0), (1, (4, 5, 13), 20.0), (1, (8, 8, 4), 0.1)])
def test_adaptive_candidate_list(atoms, mesh, scale):
    sysm = _system(atoms)
    prob = oracle.Problem(*sysm, mesh, sigma=scale, sigma_adaptive=True)
    q = [int(np.prod(mesh)) - 2]
    G, WP, CNT = prob.rates(modes_of(q, 3 * atoms), channel_mask=20)
    for precision, tol, floor in ((0, 1e-10, 1e-12), (1, 1e-4, 1e-6)):
        e = make_engine(sysm, mesh, precision=precision, prob=prob)
        g, wp, cnt = (x.cpu().numpy() for x in e.rates(300.0, scale, 20, q_subset=q, adaptive=True))
        e.close()
        assert np.array_equal(cnt, CNT)
        if CNT.sum():
            assert_close(g[[2, 4]], G[[2, 4]], tol, floor_frac=floor, what="gamma")
            assert_close(wp[[2, 4]], WP[[2, 4]], tol, floor_frac=floor, what="wp")
