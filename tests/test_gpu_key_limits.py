"""Φ3 and Φ4 lists whose clusters nearly all have a key (leg atoms and cell difference) of their own, up to the
shared memory of the kernels and beyond it."""
import numpy as np
import pytest

from synth import morse_system, random_cluster_ifcs
from tests.helpers import make_engine

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _system(n3, seed=5):
    c, p2, p3, p4 = morse_system(seed=3)
    return c, p2, random_cluster_ifcs(c, 3, n3, seed=seed, max_cell=6), p4


def test_a_refused_call_leaves_no_error_behind():
    from paper_2510_00518_gb300 import FC4Error
    e = make_engine(_system(2000), (2, 2, 2), inject=False)
    f = make_engine(_system(20), (2, 2, 2), inject=False)
    for _ in range(2):
        with pytest.raises(FC4Error):
            e.rates(300.0, 0.1, 3)
        assert torch.isfinite(f.rates(300.0, 0.1, 3)[0]).all()
        with pytest.raises(FC4Error):
            e.rates(300.0, 0.1, 3)
        make_engine(_system(20), (2, 2, 2), inject=False).close()


@pytest.mark.parametrize("atoms,n3,mesh,sigma,adaptive", [
    (2, 900, (3, 2, 3), 1.0, False), (2, 1500, (2, 3, 2), 2.0, False), (2, 1545, (2, 3, 2), 1.0, True),
    (2, 1600, (2, 3, 2), 2.0, False), (1, 1530, (3, 3, 2), 3.0, False), (4, 1500, (2, 2, 1), 1.0, False)])
def test_rates_with_many_keys(atoms, n3, mesh, sigma, adaptive):
    """Against the oracle at the bars of the other three-phonon tests: one copy of G in the pair kernel (to 1500
    keys), then the kernel of the larger cells, with a short queue at its own limit."""
    from synth import diamond_crystal, morse_ifcs, supercell_crystal
    from tests.test_gpu_rates3 import _check
    if atoms == 2:
        sysm = _system(n3)
    elif atoms == 4:
        c = supercell_crystal(diamond_crystal(), 2, np.linspace(12.0, 90.0, 4))
        p2, p3, p4 = morse_ifcs(c, seed=1)
        sysm = c, p2, random_cluster_ifcs(c, 3, n3, seed=5, max_cell=6), p4
    else:
        c = supercell_crystal(diamond_crystal(), 1)
        c.positions, c.masses = c.positions[:1], c.masses[:1]
        p2 = random_cluster_ifcs(c, 2, 6, seed=1, scale=0.5)
        p2.atoms = np.concatenate([p2.atoms, [[0, 0]]]).astype(np.int32)
        p2.cells = np.concatenate([p2.cells, np.zeros((1, 1, 3))]).astype(np.int32)
        p2.phi = np.concatenate([p2.phi, [np.diag([10.0, 40.0, 160.0]).reshape(-1)]])
        sysm = c, p2, random_cluster_ifcs(c, 3, n3, seed=5, max_cell=9), random_cluster_ifcs(c, 4, 5, seed=6)
    _check(sysm, mesh, [1, int(np.prod(mesh)) - 1], sigma, adaptive)


@pytest.mark.parametrize("atoms,n3,mesh,sigma,adaptive", [
    (2, 640, (3, 3, 2), 1.0, False), (2, 690, (3, 3, 2), 1.0, False), (2, 1530, (3, 2, 2), 2.0, False),
    (2, 900, (4, 3, 2), 1.0, True), (4, 700, (2, 2, 1), 1.0, False), (4, 1400, (2, 2, 1), 1.0, False)])
def test_gradient_with_many_keys(atoms, n3, mesh, sigma, adaptive):
    """G and H in shared memory and, from 650 (two atoms) or 560 keys (four) on, in device memory.  L is quadratic
    in Φ3: L(Φ + Φ') - L(Φ - Φ') = 2 <dL/dΦ, Φ'> to the rounding of the two L (1e-10 of each, dL/dΓ > 0; the terms
    of an L are positive where 1 + n' + n'' weighs them, so 3ph- only)."""
    from synth import diamond_crystal, morse_ifcs, supercell_crystal
    if atoms == 2:
        sysm = _system(n3)
    else:
        c = supercell_crystal(diamond_crystal(), 2, np.linspace(12.0, 90.0, 4))
        p2, p3, p4 = morse_ifcs(c, seed=1)
        sysm = c, p2, random_cluster_ifcs(c, 3, n3, seed=5, max_cell=6), p4
    e = make_engine(sysm, mesh, precision=0, inject=False)
    n, nb = int(np.prod(mesh)), 3 * atoms
    sub = [1, n - 1]
    dL = torch.tensor(np.random.default_rng(3).uniform(0.5, 1.5, (5, nb * len(sub))), device="cuda")

    def loss():
        return float((dL * e.rates(300.0, sigma, 2, q_subset=sub, adaptive=adaptive)[0]).sum())

    assert loss() > 0.0
    d3 = e.backward(dL)[0].clone()
    assert torch.equal(d3, e.backward(dL)[0])
    phi, rng = sysm[2].phi, np.random.default_rng(5)
    for k in (0, n3 // 2, n3 - 1, None):
        step = rng.normal(size=phi.shape)
        if k is not None:
            step[np.arange(n3) != k] = 0.0
        L = []
        for sgn in (1, -1):
            e.update_anharmonic(phi3=phi + sgn * step)
            L.append(loss())
        e.update_anharmonic(phi3=phi)
        got = float((d3.cpu().numpy() * step).sum())
        assert abs((L[0] - L[1]) / 2 - got) <= 1e-10 * (abs(L[0]) + abs(L[1])), (k, L, got)
    e.close()


def _few_keys(n4):
    """n4 distinct Φ4 clusters, all with legs 2 and 3 in one cell: four keys."""
    from synth.morse import IFC
    c, p2, p3, _ = morse_system(seed=3)
    rng = np.random.default_rng(8)
    legs = {(*rng.integers(0, 2, 4), *rng.integers(-4, 5, 6)) for _ in range(n4 + 50)}
    legs = np.array(sorted(tuple(int(x) for x in v) for v in legs)[:n4])
    cells = np.stack([legs[:, 4:7], legs[:, 7:], legs[:, 7:]], 1)
    return c, p2, p3, IFC(4, legs[:, :4].astype(np.int32), cells.astype(np.int32), rng.normal(size=(n4, 81)))


@pytest.mark.parametrize("n4", [960, 1000, 1028])
def test_mixed_rates_with_many_clusters_of_few_keys(n4):
    """W by columns and, from 969 to 1028 clusters of four keys, with Ψ in shared memory, against the general kernel (counts
    exact, the mixed bar of 1e-4)."""
    e = make_engine(_few_keys(n4), (3, 3, 2), precision=1, inject=False)
    assert e.info()["n_keys"] == 4
    q = [4, 11]
    g, wp, cnt = (x.cpu().numpy() for x in e.rates(300.0, 0.3, 28, q_subset=q))
    G, WP, CNT = (x.cpu().numpy() for x in e.rates_static(300.0, 0.3, 28, q))
    assert CNT.sum() and np.array_equal(cnt, CNT)
    for x, y in ((g, G), (wp, WP)):
        assert np.abs(x[2:] - y[2:]).max() <= 1e-4 * np.abs(y[2:]).max()
    e.close()


def test_gradient_where_the_w_of_the_tiled_path_does_not_fit():
    """600 clusters: mixed rates, then the FP64 gradient of that call; its tiled form would need a W kernel that does
    not fit, the general one takes it.  Against the mixed gradient (1e-4 of the largest entry)."""
    e = make_engine(_few_keys(600), (3, 2, 2), precision=1, inject=False)
    dL = torch.tensor(np.random.default_rng(1).uniform(0.5, 1.5, (5, 6)), device="cuda")
    e.rates(300.0, 0.3, 28, q_subset=[5])
    ref = e.backward(dL)[1].clone()
    e.set_precision(0)
    got = e.backward(dL)[1]
    assert (got - ref).abs().max() <= 1e-4 * ref.abs().max()
    e.close()
