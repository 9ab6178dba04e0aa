"""Gradient with respect to Φ3 on meshes whose points need more than 16 bits.

L = Σ dL/dΓ Γ is quadratic in Φ3, so L(Φ + Φ') - L(Φ - Φ') = 2 <dL/dΦ, Φ'> up to the rounding of the two L
(1e-10 of each, the FP64 bar; dL/dΓ > 0, so L has no cancellation between modes)."""
import numpy as np
import pytest

from synth import diamond_crystal, morse_ifcs, morse_system, supercell_crystal
from tests.helpers import make_engine

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("atoms,mesh,sigma,adaptive", [(2, (41, 41, 40), 0.1, False), (2, (64, 32, 33), 0.5, True),
                                                       (4, (64, 64, 17), 0.02, False)])
def test_backward_above_65536_points(atoms, mesh, sigma, adaptive):
    if atoms == 2:
        sysm = morse_system(seed=6)
    else:
        c = supercell_crystal(diamond_crystal(), atoms // 2, np.linspace(12.0, 90.0, atoms))
        sysm = (c,) + morse_ifcs(c, seed=1)
    n, nb = int(np.prod(mesh)), 3 * atoms
    assert n > 1 << 16
    e = make_engine(sysm, mesh, precision=0, inject=False)
    sub = [n - 7]
    dL = torch.tensor(np.random.default_rng(3).uniform(0.5, 1.5, (5, nb)), device="cuda")

    def loss():
        return float((dL * e.rates(300.0, sigma, 3, q_subset=sub, adaptive=adaptive)[0]).sum())

    assert loss() > 0.0
    # the kept processes reach partner points on both sides of 65536
    q1 = np.concatenate([e.processes(ch, sub[0] * nb + nb - 1) for ch in (0, 1)]) // (nb * nb)
    assert q1.min() < 1 << 16 <= q1.max()
    loss()
    d3 = e.backward(dL)[0].cpu().numpy()
    phi = sysm[2].phi
    rng = np.random.default_rng(5)
    for k in (0, len(phi) // 2, len(phi) - 1):
        step = np.zeros_like(phi)
        step[k] = rng.normal(size=27) * np.abs(phi).max()
        L = []
        for sgn in (1, -1):
            e.update_anharmonic(phi3=phi + sgn * step)
            L.append(loss())
        e.update_anharmonic(phi3=phi)
        assert abs((L[0] - L[1]) / 2 - (d3 * step).sum()) <= 1e-10 * (abs(L[0]) + abs(L[1])), (k, L)
    e.close()
