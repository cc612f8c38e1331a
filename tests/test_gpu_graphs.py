"""An FP64 apply captured by a program into a graph of its own: the graph has
kernel nodes only, so that it can be instantiated several times, cloned and put
into another graph, and its work space lives as long as any of these."""
import ctypes
import glob

import pytest
import torch

from paper_1012_3615_gb300 import Brillouin, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    for name in ["libcudart.so.13", "libcudart.so"] + sorted(glob.glob("/usr/local/cuda/lib64/libcudart.so*")):
        try:
            return ctypes.CDLL(name)
        except OSError:
            pass
    pytest.skip("no shared CUDA runtime")


def _p(v=None):
    return ctypes.c_void_p(v)


def test_captured_apply_many_executables(gpu, rt):
    L = (8, 6, 6, 8)
    op = Brillouin(L)
    op.build_hops(torch.as_tensor(synth.random_su3_links(L, 0.3, 81), device=gpu))
    x = torch.as_tensor(synth.gaussian_spinor(L, 6, 82), device=gpu)
    want = [op.apply(op.apply(x[r:r + 1], m0=0.1), m0=0.1) for r in range(6)]
    static, mid, out = (torch.zeros_like(x[:1]) for _ in range(3))
    stream = torch.cuda.Stream()

    def capture():
        torch.cuda.synchronize()
        s, g = _p(stream.cuda_stream), _p()
        with torch.cuda.stream(stream):
            assert rt.cudaStreamBeginCapture(s, 1) == 0
            op.apply(static, m0=0.1, out=mid)
            op.apply(mid, m0=0.1, out=out)
            assert rt.cudaStreamEndCapture(s, ctypes.byref(g)) == 0
        return g

    def replay(e, r):
        static.copy_(x[r:r + 1])
        out.zero_()
        torch.cuda.synchronize()
        assert rt.cudaGraphLaunch(e, _p(stream.cuda_stream)) == 0
        torch.cuda.synchronize()
        assert torch.equal(out, want[r])

    def instantiate(g):
        e = _p()
        assert rt.cudaGraphInstantiate(ctypes.byref(e), g, ctypes.c_ulonglong(0)) == 0
        return e

    g = capture()
    e1, e2 = instantiate(g), instantiate(g)
    outer, node = _p(), _p()
    assert rt.cudaGraphCreate(ctypes.byref(outer), 0) == 0
    assert rt.cudaGraphAddChildGraphNode(ctypes.byref(node), outer, None, ctypes.c_size_t(0), g) == 0
    assert rt.cudaGraphDestroy(g) == 0
    e3 = instantiate(outer)
    assert rt.cudaGraphDestroy(outer) == 0
    for r, e in enumerate((e1, e2, e3)):
        replay(e, r)
    for e in (e1, e2):
        assert rt.cudaGraphExecDestroy(e) == 0
    # captures that come and go, while e3 keeps its work space
    for r in range(4):
        g = capture()
        e = instantiate(g)
        assert rt.cudaGraphDestroy(g) == 0
        replay(e, r)
        replay(e3, 5 - r)
        assert rt.cudaGraphExecDestroy(e) == 0
    assert rt.cudaGraphExecDestroy(e3) == 0
