"""The convolution behind kernels that let their dependents in early (it is
launched as a programmatic dependent of the kernel before it): it reads what
that kernel writes last, however long it runs on, with a second dependency on
another stream, issued directly and captured into a graph."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from gpu_util import conv_case, np_words, oracle_conv_nhwc, oracle_requant_pack
from paper_1809_10572_gb300 import build, samd

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def early_release(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("early") / "libearly.so")
    r = subprocess.run([build.nvcc()] + build.ARCH + ["-shared", "-Xcompiler", "-fPIC", "-o", so,
                                                      os.path.join(HERE, "early_release.cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    fn = ctypes.CDLL(so).early_release
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong, ctypes.c_ulonglong, ctypes.c_void_p]
    fn.restype = ctypes.c_int

    def call(src, dst, ns, stream):
        assert fn(src.data_ptr(), dst.data_ptr(), src.numel(), ns, stream.cuda_stream) == 0

    return call


class Layer:
    """A layer whose activations a kernel writes at its end."""

    def __init__(self, shape, ba, bw, seed):
        a_v, w_v, self.src, w_w, fa, fw = conv_case(shape, ba, False, bw, True, seed)
        self.fo = samd.fmt(8, True)
        self.shift = 5
        self.conv = samd.PreparedConv(w_w, shape, fa, fw, self.fo)
        self.act = torch.zeros_like(self.src)
        self.out = self.conv.outputs(want_acc=False)[1]
        self.want = oracle_requant_pack(oracle_conv_nhwc(a_v, w_v, shape), self.shift, self.fo)
        self.conv(self.src, None, self.out, self.shift)  # kernel attributes, outside any capture
        torch.cuda.synchronize()
        self.clear()

    def clear(self):
        self.act.zero_()
        self.out.zero_()

    def run(self, stream):
        self.conv(self.act, None, self.out, self.shift, stream=stream)

    def check(self):
        assert np.array_equal(np_words(self.out, 32), self.want)


# 1.3 s is more than any wait of the convolution may take.
@pytest.mark.parametrize("shape,ba,bw", [(samd.ConvShape(2, 64, 14, 14, 64), 4, 4),
                                         (samd.ConvShape(2, 200, 9, 8, 264), 6, 2)],
                         ids=lambda v: f"K{v.K}" if isinstance(v, samd.ConvShape) else None)
def test_conv_waits_for_a_kernel_that_let_it_in_early(samd_lib, early_release, shape, ba, bw):
    layer = Layer(shape, ba, bw, 5)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    early_release(layer.src, layer.act, 1_300_000_000, s)
    layer.run(s)
    torch.cuda.synchronize()
    assert samd.samd_device_status() == samd.SAMD_OK
    layer.check()


def fork_and_join(early_release, a, b, c, main, side):
    """a on main and b on side behind kernels of their own; c on main behind a
    and, by an event, behind the kernel on side that writes c's input after b."""
    side.wait_stream(main)
    early_release(a.src, a.act, 300_000, main)
    a.run(main)
    early_release(b.src, b.act, 600_000, side)
    b.run(side)
    early_release(c.src, c.act, 2_000_000, side)
    main.wait_stream(side)
    c.run(main)


@pytest.mark.parametrize("captured", (False, True))
def test_conv_with_two_dependencies(samd_lib, early_release, captured):
    layers = [Layer(samd.ConvShape(2, 64, 14, 14, 64), 4, 4, 6), Layer(samd.ConvShape(2, 40, 9, 8, 48, R=1, S=1, pad=0), 6, 3, 7),
              Layer(samd.ConvShape(2, 200, 9, 8, 264), 4, 4, 8)]
    main, side = torch.cuda.Stream(), torch.cuda.Stream()
    main.wait_stream(torch.cuda.current_stream())
    if captured:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=main):
            fork_and_join(early_release, *layers, main, side)
    for _ in range(3):
        for l in layers:
            l.clear()
        torch.cuda.synchronize()
        if captured:
            graph.replay()
        else:
            fork_and_join(early_release, *layers, main, side)
        torch.cuda.synchronize()
        for l in layers:
            l.check()
    assert samd.samd_device_status() == samd.SAMD_OK
