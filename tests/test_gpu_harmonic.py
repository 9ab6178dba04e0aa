"""Device harmonic solution for every share of its block: matrix entries over the threads, rows of A and
U over the lanes (more rows than lanes from 6 atoms up), clusters of a velocity sum over 42 to 5 parts
(fewer clusters than parts, and many more).  Residuals and velocities of the device's own eigenvectors
against the dynamical matrix in FP64: a few hundred roundings, bar 1e-12 of the largest sum of
magnitudes."""
import numpy as np
import pytest

import oracle
from synth import diamond_crystal, morse_ifcs, random_cluster_ifcs, supercell_crystal
from tests.helpers import make_engine

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _system(atoms):
    base = diamond_crystal()
    if atoms % 2 == 0:
        c = supercell_crystal(base, atoms // 2, np.linspace(12.0, 90.0, atoms))
        return (c,) + morse_ifcs(c, seed=1)
    c = supercell_crystal(base, (atoms + 1) // 2)
    c.positions, c.masses = c.positions[:atoms], np.linspace(20.0, 50.0, atoms)
    p2 = random_cluster_ifcs(c, 2, 3 * atoms, seed=1, scale=0.05)
    p2.atoms = np.concatenate([p2.atoms, [[a, a] for a in range(atoms)]]).astype(np.int32)
    p2.cells = np.concatenate([p2.cells, np.zeros((atoms, 1, 3))]).astype(np.int32)
    p2.phi = np.concatenate([p2.phi, [(1 + 0.3 * a) * np.diag([2.0, 8.0, 30.0]).reshape(-1) for a in range(atoms)]])
    return c, p2, random_cluster_ifcs(c, 3, 5, seed=2), random_cluster_ifcs(c, 4, 5, seed=3)


@pytest.mark.parametrize("atoms", [1, 2, 3, 5, 6, 8])
def test_harmonic_solution(atoms):
    sysm = _system(atoms)
    c, p2 = sysm[:2]
    mesh = (3, 2, 5)
    e = make_engine(sysm, mesh, inject=False)
    om, vel, ev = e.get_modes()
    e.close()
    nb = 3 * atoms
    qs = oracle.q_cart(c.lattice, mesh)
    for q in range(len(qs)):
        D, dD = oracle.dynamical_matrix(c, p2, qs[q])
        D = 0.5 * (D + D.conj().T)
        size = np.linalg.norm(D)
        E, w = ev[q], om[q * nb:(q + 1) * nb]
        assert np.abs(E.conj().T @ E - np.eye(nb)).max() <= 1e-12
        A = E.conj().T @ D @ E
        lam = np.real(np.diag(A))
        assert np.abs(A - np.diag(lam)).max() <= 1e-12 * size
        assert np.all(np.diff(lam) >= -1e-12 * size)
        for j in range(3 if q == 0 else 0, nb):
            assert abs(w[j] ** 2 / oracle.EIG_TO_RADPS2 - lam[j]) <= 1e-12 * size
            a = np.abs(E[:, j])
            for x in range(3):
                f = oracle.EIG_TO_RADPS2 / (2.0 * w[j])
                ref = np.real(np.conj(E[:, j]) @ dD[x] @ E[:, j]) * f
                bar = sum(float(a[3 * i:3 * i + 3] @ np.abs(p.reshape(3, 3)) @ a[3 * k:3 * k + 3]) *
                          np.linalg.norm(R[0] @ c.lattice) / np.sqrt(c.masses[i] * c.masses[k])
                          for (i, k), R, p in zip(p2.atoms, p2.cells, p2.phi)) * f
                assert abs(vel[q * nb + j, x] - ref) <= 1e-12 * (bar + 1e-300)
