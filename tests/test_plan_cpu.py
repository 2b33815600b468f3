"""The convolution planner on the host (no GPU): tests/plan_check.cu
compiles conv2d.cu's planning code with the kernel launchers stubbed and
checks every plan over a grid of shapes and formats against the
shared-memory, TMEM and layout limits."""
import os
import subprocess
import tempfile

import pytest

import nchw_cases
from paper_1809_10572_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run_host_program(name, stdin=""):
    """Compiles tests/<name>.cu for the host and runs it."""
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not available")
    with tempfile.TemporaryDirectory(prefix="samd_plan_") as tmp:
        exe = os.path.join(tmp, name)
        cmd = [nvcc] + build.ARCH + ["-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "include"),
                                     os.path.join(ROOT, "tests", name + ".cu"), "-o", exe, "-lcuda"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-2000:]
        return subprocess.run([exe], capture_output=True, text=True, timeout=600, input=stdin)


def test_nchw_cases_take_their_routes():
    cases = nchw_cases.ENGINE + nchw_cases.TENSOR
    lines = [" ".join(map(str, (s.N, s.C, s.H, s.W, s.K, s.R, s.S, s.pad, ba, int(sa), bw, int(sw), wb, fo)))
             for s, ba, sa, bw, sw, wb, fo in cases]
    r = run_host_program("nchw_route", "\n".join(lines) + "\n")
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.split() == ["engine"] * len(nchw_cases.ENGINE) + ["tensor"] * len(nchw_cases.TENSOR)


def test_every_plan_fits_and_does_not_overlap():
    r = run_host_program("plan_check")
    assert r.returncode == 0, r.stdout[-2000:]
    assert "bad 0" in r.stdout
    # the grid reaches every planning mode
    for mode in ("halo", "segmented", "e4m3", "resident", "two-half", "four-part", "window gather",
                 "staged epilogue", "flat epilogue", "filter-row stages", "int32 stage", "pooled"):
        count = int(r.stdout.split(mode)[1].split()[0].strip("(),"))
        assert count > 0, (mode, r.stdout)


@pytest.mark.parametrize("N,H,W,R,S,pad", [(2, 3, 4, 3, 3, 1), (3, 1, 1, 3, 3, 1), (2, 5, 4, 5, 5, 2), (2, 4, 3, 3, 3, 2),
                                           (2, 4, 5, 2, 2, 1), (2, 4, 5, 3, 5, 1), (2, 6, 5, 3, 3, 0), (1, 3, 3, 5, 5, 4)])
def test_shared_padding_grid_reads_what_two_sided_padding_reads(N, H, W, R, S, pad):
    """The planner's virtual grid keeps pad columns on one side of a row and
    pad rows on one side of an image (pad < R, S): the position one tap row or
    column on always holds the input value that tap reads, or padding."""
    assert pad < R and pad < S
    Hv, Wp = H + pad, W + pad
    Ho, Wo = H + 2 * pad - R + 1, W + 2 * pad - S + 1
    assert Ho <= Hv and Wo <= Wp
    for n in range(N):
        for oh in range(Ho):
            for ow in range(Wo):
                for r in range(R):
                    for s in range(S):
                        ih, iw = oh + r - pad, ow + s - pad
                        want = (n, ih, iw) if 0 <= ih < H and 0 <= iw < W else None
                        v = (n * Hv + oh) * Wp + ow + r * Wp + s
                        img, rem = divmod(v, Hv * Wp)
                        gh, gw = rem // Wp - pad, rem % Wp - pad
                        got = (img, gh, gw) if img < N and 0 <= gh < H and 0 <= gw < W else None
                        assert got == want
