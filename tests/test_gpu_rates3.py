"""Three-phonon kernels at the edges of their spans of partner points (512 for cells of up to two
atoms) and of their rounds of 128 points or processes, for every branch grouping of the window and with
a Φ3 that has no leg-exchange symmetry, against the FP64 oracle.

Counts are exact.  Γ and WP are sums whose terms have both signs once the window is wide (at (1, 1, 127)
with σ = 4 THz a soft mode's terms cancel 6800-fold), so the FP64 bar of 1e-10 applies to the sum of
the terms' magnitudes: a term is ~500 rounded operations, ~6e-14 of itself at worst, on either side."""
import numpy as np
import pytest

import oracle
from synth import diamond_crystal, morse_ifcs, morse_system, random_cluster_ifcs, supercell_crystal
from tests.helpers import make_engine, modes_of

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _magnitudes(prob, q0, j0, ch, T=300.0):
    """Σ |γ| and Σ |w| of one mode and channel."""
    s = 1 if ch == 0 else -1
    nb, na, mesh, p3 = prob.nb, prob.nb // 3, np.array(prob.mesh), prob.phi3
    if q0 == 0 and j0 < 3:
        return 0.0, 0.0
    g = oracle.q_coords(prob.mesh)
    q2 = (g[q0] + s * g) % mesh @ np.array([1, mesh[0], mesh[0] * mesh[1]])
    w, E = prob.modes.omega.reshape(-1, nb), prob.modes.evec
    n = oracle.occupations(prob.modes.omega, T).reshape(-1, nb)
    with np.errstate(divide="ignore"):
        iw = np.where(w > 0, 1 / w, 0.0)
    e1 = (E if s > 0 else E.conj()).reshape(-1, na, 3, nb)
    e2, el = E[q2].conj().reshape(-1, na, 3, nb), E[q0][:, j0].reshape(na, 3)
    V = np.zeros((len(g), nb, nb), complex)
    for (a, b, c), cell, phi in zip(p3.atoms, p3.cells, p3.phi):
        A = np.einsum("a,abc->bc", el[a], phi.reshape(3, 3, 3)) / np.sqrt(np.prod(prob.crystal.masses[[a, b, c]]))
        ph = np.exp(2j * np.pi * ((s * g * cell[0] - (g[q0] + s * g) * cell[1]) / mesh).sum(1))
        V += ph[:, None, None] * np.einsum("qbj,bc,qck->qjk", e1[:, b], A, e2[:, c], optimize=True)
    w1, w2 = w[:, :, None], w[q2][:, None, :]
    d = (w[q0, j0] + w1) - w2 if ch == 0 else w[q0, j0] - (w1 + w2)
    if prob.sigma_adaptive:
        v = prob.modes.vel.reshape(-1, nb, 3) @ oracle.reciprocal(prob.crystal.lattice).T / mesh
        sg = prob.sigma * np.sqrt(((v[:, :, None] - v[q2][:, None]) ** 2).sum(-1) / 6)
    else:
        sg = np.full(d.shape, 2.0 * np.pi * prob.sigma)
    keep = (np.abs(d) <= 2 * sg) & (sg > 1e-9) & (w1 > 0) & (w2 > 0)
    f = n[:, :, None] - n[q2][:, None, :] if ch == 0 else (1 + n[:, :, None] + n[q2][:, None, :]) / 2
    sg = np.where(keep, sg, 1.0)
    wt = np.where(keep, f * np.exp(-(d / sg) ** 2) / (sg * np.sqrt(np.pi)), 0.0)
    wt = np.abs(wt * iw[q0, j0] * iw[:, :, None] * iw[q2][:, None, :])
    return oracle.C3 / len(g) * (wt * np.abs(V) ** 2).sum(), wt.sum() / len(g)


def _check(system, mesh, q, sigma, adaptive):
    prob = oracle.Problem(*system, mesh, sigma=sigma, sigma_adaptive=adaptive)
    e = make_engine(system, mesh, prob=prob)
    G, WP, CNT = prob.rates(modes_of(q, e.nb), channel_mask=3)
    mag = np.array([[_magnitudes(prob, k, j, ch) for k in q for j in range(e.nb)] for ch in (0, 1)])
    g, wp, cnt = (x.cpu().numpy() for x in e.rates(300.0, sigma, 3, q_subset=q, adaptive=adaptive))
    assert np.array_equal(cnt, CNT)
    assert (np.abs(g - G)[:2] <= 1e-10 * mag[..., 0]).all()
    assert (np.abs(wp - WP)[:2] <= 1e-10 * mag[..., 1]).all()
    F = np.random.default_rng(0).normal(size=(e.nq * e.nb, 3))
    if e.n_atoms <= 2:
        d = e.bte_offdiag(300.0, sigma, torch.from_numpy(F).cuda(), 3, q_subset=q, adaptive=adaptive).cpu().numpy()
        off = prob.bte_offdiag(F, modes_of(q, e.nb), channel_mask=3)
        # Δ sums terms of both signs: 1e-10 of the largest component
        assert np.abs(d - off).max() <= 1e-10 * np.abs(off).max()
    e.close()


@pytest.mark.parametrize("mesh", [(1, 1, 1), (1, 1, 127), (8, 4, 4), (3, 43, 1), (16, 16, 1), (1, 1, 256), (8, 8, 8), (8, 8, 9)])
@pytest.mark.parametrize("sigma,adaptive", [(0.1, False), (4.0, False), (1.0, True)])
def test_span_and_queue_edges(mesh, sigma, adaptive):
    n = int(np.prod(mesh))
    _check(morse_system(seed=3), mesh, sorted({0, n // 2, n - 1}), sigma, adaptive)


@pytest.mark.parametrize("atoms", [1, 3, 4, 6, 8])
def test_branch_groupings(atoms):
    base = diamond_crystal()
    if atoms % 2:
        c = supercell_crystal(base, 2)
        c.positions, c.masses = c.positions[:atoms], np.array([20.0, 35.0, 50.0])[:atoms]
        # generic clusters; the harmonic part is made positive by strong on-site springs
        p2 = random_cluster_ifcs(c, 2, 12, seed=1, scale=0.1)
        p2.atoms = np.concatenate([p2.atoms, [[a, a] for a in range(atoms)]]).astype(np.int32)
        p2.cells = np.concatenate([p2.cells, np.zeros((atoms, 1, 3))]).astype(np.int32)
        p2.phi = np.concatenate([p2.phi, [(1 + 0.3 * a) * np.diag([2.0, 8.0, 30.0]).reshape(-1) for a in range(atoms)]])
        p3, p4 = random_cluster_ifcs(c, 3, 40, seed=2), random_cluster_ifcs(c, 4, 10, seed=3)
    else:
        c = supercell_crystal(base, atoms // 2, np.linspace(12.0, 90.0, atoms))
        p2, p3, p4 = morse_ifcs(c, seed=1)
    _check((c, p2, p3, p4), (5, 3, 9), [0, 77][:2 if atoms < 6 else 1], 0.5 if atoms > 2 else 2.0, False)


def test_broken_leg_exchange_takes_the_rectangle():
    """3ph- evaluates one process of a swapped pair only where Φ3 is symmetric in legs 1 and 2."""
    c, p2, p3, p4 = morse_system(seed=3)
    e = make_engine((c, p2, p3, p4), (4, 4, 4))
    e.rates(300.0, 0.3, 3)
    st = e.stats()
    assert st["evaluated"][0] == st["kept"][0] and st["evaluated"][1] < st["kept"][1]
    e.close()
    p3.phi[5, 7] += 0.3 * np.abs(p3.phi).max()
    _check((c, p2, p3, p4), (4, 4, 4), [0, 9], 0.3, False)
    e = make_engine((c, p2, p3, p4), (4, 4, 4))
    e.rates(300.0, 0.3, 3)
    st = e.stats()
    assert np.array_equal(st["evaluated"][:2], st["kept"][:2])
    e.update_anharmonic(phi3=morse_system(seed=3)[2].phi)
    e.rates(300.0, 0.3, 3)
    assert e.stats()["evaluated"][1] < st["kept"][1]
    e.close()


@pytest.mark.parametrize("atoms", [2, 4])
def test_bits_do_not_depend_on_the_chunk_or_the_subset(atoms):
    """Γ and WP of a mode to the bit, whatever modes share its chunk or its call, on a mesh whose points fill
    several warps of a block."""
    sysm = morse_system(seed=3) if atoms == 2 else \
        (lambda c: (c,) + morse_ifcs(c, seed=1))(supercell_crystal(diamond_crystal(), 2, np.linspace(12.0, 90.0, 4)))
    e = make_engine(sysm, (7, 6, 7), inject=False)
    ref = [x.cpu().numpy() for x in e.rates(300.0, 0.2, 3)]
    for chunk in (1, 3, 50):
        e.set_mode_chunk(chunk, 0)
        for x, y in zip(e.rates(300.0, 0.2, 3), ref):
            assert np.array_equal(x.cpu().numpy(), y)
    e.set_mode_chunk(0, 0)
    nb = 3 * atoms
    for q in ([5], [293, 17, 100]):
        rows = modes_of(q, nb)
        for x, y in zip(e.rates(300.0, 0.2, 3, q_subset=q), ref):
            assert np.array_equal(x.cpu().numpy(), y[:, rows])
    e.close()
