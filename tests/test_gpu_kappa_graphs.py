"""Captured κ: the bits of the eager call however many captures a context has seen, on every number of thread
groups and cluster blocks, and with executable graphs of one capture side by side."""
import ctypes

import numpy as np
import pytest

from synth import morse_system
from tests.helpers import make_engine

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _system(mesh):
    e = make_engine(morse_system(seed=2), mesh, inject=False)
    g = torch.tensor(np.exp(np.random.default_rng(1).normal(-3.0, 1.0, size=(5, e.nq * e.nb))), device="cuda")
    return e, g


def _ok(status):
    assert status == 0, status


class _Graph:
    """A captured κ call as a plain CUDA graph, which can be instantiated several times."""

    def __init__(self, e, T, g):
        self.cu = ctypes.CDLL("libcuda.so.1")
        self.out = torch.empty(9, dtype=torch.float64, device="cuda")
        self.graph, self.execs = ctypes.c_void_p(), []
        s = torch.cuda.Stream()
        torch.cuda.synchronize()
        _ok(self.cu.cuStreamBeginCapture_v2(ctypes.c_void_p(s.cuda_stream), 1))          # thread-local
        e.kappa(T, g, 31, out=self.out, stream=s)
        _ok(self.cu.cuStreamEndCapture(ctypes.c_void_p(s.cuda_stream), ctypes.byref(self.graph)))

    def instantiate(self):
        x = ctypes.c_void_p()
        _ok(self.cu.cuGraphInstantiateWithFlags(ctypes.byref(x), self.graph, ctypes.c_ulonglong(0)))
        self.execs.append(x)

    def launch(self, i, stream):
        _ok(self.cu.cuGraphLaunch(self.execs[i], ctypes.c_void_p(stream.cuda_stream)))

    def close(self):
        for x in self.execs:
            _ok(self.cu.cuGraphExecDestroy(x))
        _ok(self.cu.cuGraphDestroy(self.graph))


@pytest.mark.parametrize("mesh", [(1, 1, 1), (1, 1, 11), (1, 5, 17), (1, 2, 43), (1, 6, 57), (3, 5, 91), (1, 7, 196), (12, 24, 24)])
def test_captured_equals_eager(mesh):
    """1, 2, 8, 9, 33, 128, 129 and 608 groups."""
    e, g = _system(mesh)
    ref = e.kappa(300.0, g, 31).reshape(9).clone()
    gr = _Graph(e, 300.0, g)
    gr.instantiate()
    gr.out.zero_()
    torch.cuda.synchronize()
    gr.launch(0, torch.cuda.Stream())
    torch.cuda.synchronize()
    assert torch.equal(gr.out, ref)
    gr.close()
    e.close()


def test_many_captures():
    e, g = _system((6, 6, 6))
    ref = e.kappa(300.0, g, 31).clone()
    for _ in range(40):
        s, gr = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(gr, stream=s, capture_error_mode="thread_local"):
            out = e.kappa(300.0, g, 31)
        gr.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
        del gr
    e.close()


def test_executables_of_one_capture_side_by_side():
    e, g = _system((16, 16, 16))
    ref = e.kappa(300.0, g, 31).reshape(9).clone()
    gr = _Graph(e, 300.0, g)
    streams = [torch.cuda.Stream() for _ in range(4)]
    for _ in streams:
        gr.instantiate()
    torch.cuda.synchronize()
    for _ in range(50):
        gr.out.zero_()
        torch.cuda.synchronize()
        for i, s in enumerate(streams):
            gr.launch(i, s)
        torch.cuda.synchronize()
        assert torch.equal(gr.out, ref)
    gr.close()
    e.close()
