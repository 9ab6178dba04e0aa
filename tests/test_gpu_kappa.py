"""κ's multi-block sum at the edges of its blocks of 64 modes and beyond its 608 blocks (38912 modes),
against the oracle (1e-12: sums of positive terms, each ~100 rounded operations)."""
import numpy as np
import pytest

import oracle
from synth import morse_system
from tests.helpers import make_engine

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("mesh", [(1, 1, 1), (1, 2, 5), (1, 1, 11), (8, 8, 8), (12, 24, 24)])
def test_kappa_blocks(mesh):
    sysm = morse_system(seed=2)
    prob = oracle.Problem(*sysm, mesh)
    e = make_engine(sysm, mesh, prob=prob)
    g = np.exp(np.random.default_rng(1).normal(-3.0, 1.0, size=(5, e.nq * e.nb)))
    g[:, ::7] = 0.0                                     # skipped modes
    gd = torch.tensor(g, device="cuda")
    k = [e.kappa(300.0, gd, 21).cpu().numpy() for _ in range(3)]
    ref = oracle.kappa(sysm[0], prob.modes, 300.0, g[[0, 2, 4]].sum(0), mesh)
    assert np.array_equal(k[0], k[1]) and np.array_equal(k[0], k[2])
    assert np.abs(k[0] - ref).max() <= 1e-12 * np.abs(ref).max()
    back = e.kappa_backward(300.0, gd, torch.eye(3, dtype=torch.float64, device="cuda"), 21).cpu().numpy()
    # Σ_λ Γ_λ dκ/dΓ_λ = -tr κ (κ is homogeneous of degree -1 in Γ)
    assert abs((back * g).sum() + np.trace(ref)) <= 1e-12 * abs(np.trace(ref))
    assert not back[1].any() and not back[3].any()


def test_kappa_overlapping_streams():
    """Calls of one context that overlap, on more streams than the scratch has slots for eager calls, and
    beside replays of captured ones (more captures than slots: the last run on one block): each equals the
    call alone, to the bit where the blocks are the same."""
    sysm = morse_system(seed=2)
    e = make_engine(sysm, (12, 24, 24), inject=False)
    g = torch.tensor(np.exp(np.random.default_rng(1).normal(-3.0, 1.0, size=(5, e.nq * e.nb))), device="cuda")
    T = [100.0 + 10.0 * i for i in range(28)]
    ref = [e.kappa(t, g, 31).cpu().numpy() for t in T]
    streams = [torch.cuda.Stream() for _ in range(12)]
    torch.cuda.synchronize()
    graphs = []
    for i, t in enumerate(T):
        gr = torch.cuda.CUDAGraph()
        with torch.cuda.graph(gr, stream=streams[i % 12], capture_error_mode="thread_local"):
            out = e.kappa(t, g, 31)
        graphs.append((gr, out))
    for _ in range(4):
        eager = []
        for i, t in enumerate(T):
            with torch.cuda.stream(streams[i % 12]):
                eager.append(e.kappa(t, g, 31))
            with torch.cuda.stream(streams[(i + 5) % 12]):
                graphs[i][0].replay()
        torch.cuda.synchronize()
        for i, r in enumerate(ref):
            assert np.array_equal(eager[i].cpu().numpy(), r)
            if i < 24:
                assert np.array_equal(graphs[i][1].cpu().numpy(), r)
            else:
                assert np.abs(graphs[i][1].cpu().numpy() - r).max() <= 1e-12 * np.abs(r).max()
