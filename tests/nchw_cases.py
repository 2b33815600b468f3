"""NCHW layers whose route is part of what they test: (shape, activation bits
and sign, weight bits and sign, word bits, output bits or 0), for the
wide-multiply engine and for the tensor cores. tests/test_plan_cpu.py checks
that each takes its route with the workspace that
samd_conv2d_workspace_size asks for; tests/test_gpu_nchw.py runs them."""
import itertools

from paper_1809_10572_gb300 import samd

# Few input channels against the output's: kernel rows of 3, 4 and 5 taps,
# one row and several, rows of several 31-segment chunks.
ENGINE = [(s, ba, sa, bw, sw, wb, fo) for s, (ba, sa, bw, sw), wb, fo in itertools.product(
    (samd.ConvShape(1, 2, 4, 50, 40), samd.ConvShape(2, 3, 5, 70, 64), samd.ConvShape(1, 1, 1, 301, 8, R=1, S=3, pad=1),
     samd.ConvShape(1, 2, 5, 33, 48, R=3, S=4, pad=0)),
    ((4, True, 4, True), (2, True, 2, True), (5, False, 3, True), (3, True, 5, False), (1, True, 1, True)), (32, 64), (0, 4))]
ENGINE += [(samd.ConvShape(1, 3, 6, 41, 64, R=5, S=5, pad=2), b, True, b, True, 32, fo) for b in (1, 2) for fo in (0, 2)]

# Enough input channels: e4m3 and fp16 operands, several channel blocks
# (K > 256), split weight digits in one block and in two (K > 128).
TENSOR = [(s, ba, sa, bw, sw, wb, fo) for s, (ba, sa, bw, sw), wb, fo in itertools.product(
    (samd.ConvShape(1, 40, 4, 50, 3), samd.ConvShape(1, 320, 5, 20, 300)),
    ((4, True, 4, True), (2, True, 2, True), (4, False, 4, True)), (32, 64), (0, 5))]
TENSOR += [(samd.ConvShape(1, 320, 5, 20, 300, R=2, S=2, pad=0), 5, False, 3, True, 32, 6),
           (samd.ConvShape(1, 320, 5, 20, 300, R=2, S=2, pad=0), 8, False, 6, True, 64, 0),
           (samd.ConvShape(2, 640, 4, 17, 24, R=3, S=1, pad=0), 8, False, 8, True, 32, 8),
           (samd.ConvShape(1, 640, 5, 20, 150, R=3, S=1, pad=0), 8, False, 8, True, 32, 8)]
