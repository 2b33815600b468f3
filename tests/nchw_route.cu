// Host-only: which way samd_conv2d takes NCHW layers with the workspace that
// samd_conv2d_workspace_size asks for. Reads layers from standard input, one a
// line (N C H W K R S pad, activation bits and sign, weight bits and sign, word
// bits, output lane bits or 0), and prints "tensor", "engine" or "refused".
// Compiled and run by tests/test_plan_cpu.py.
#include "../paper_1809_10572_gb300/csrc/conv2d.cu"
#include "../paper_1809_10572_gb300/csrc/widemul.cu"
#include "conv_stubs.cuh"

namespace samd {
cudaError_t launch_pack(samd_fmt, const int8_t *, void *, int64_t, int64_t, cudaStream_t) { return cudaErrorInvalidValue; }
}  // namespace samd

#include <cstdio>

int main() {
  using namespace samd;
  int v[14];
  for (;;) {
    for (int i = 0; i < 14; ++i)
      if (scanf("%d", &v[i]) != 1) return i == 0 ? 0 : 1;
    const samd_conv_desc d{v[0], v[1], v[2], v[3], v[4], v[5], v[6], 1, v[7], SAMD_NCHW};
    const uint8_t wb = static_cast<uint8_t>(v[12]);
    const samd_fmt fa{(uint8_t)v[8], (uint8_t)v[9], 0, wb}, fw{(uint8_t)v[10], (uint8_t)v[11], 0, wb};
    const samd_fmt fo{(uint8_t)v[13], 0, 0, v[13] ? wb : (uint8_t)0};
    size_t ws = 0;
    conv::Plan p;
    NchwBuffers b;
    if (conv2d_nchw_check(&d, fa, fw, fo, &ws) != SAMD_OK)
      puts("refused");
    else
      puts(nchw_on_tensor_cores(&d, fa, fw, fo, ws, p, b) ? "tensor" : "engine");
  }
}
