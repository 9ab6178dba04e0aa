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
