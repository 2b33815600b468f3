// Stand-ins for the kernel launchers and the SM count, for host-only programs
// that include conv2d.cu (nothing is launched).
#pragma once

#define SAMD_STUB(name)                                                                                      \
  namespace samd {                                                                                           \
  namespace conv {                                                                                           \
  cudaError_t name(bool, const CUtensorMap &, const ConvArgs &, bool, dim3, size_t, cudaStream_t) {          \
    return cudaErrorInvalidValue;                                                                            \
  }                                                                                                          \
  }                                                                                                          \
  }
SAMD_STUB(launch_conv_f16_w32_b1) SAMD_STUB(launch_conv_f16_w32_b2) SAMD_STUB(launch_conv_f16_w32_b3)
SAMD_STUB(launch_conv_f16_w32_b4) SAMD_STUB(launch_conv_f16_w32_b5) SAMD_STUB(launch_conv_f16_w32_b6)
SAMD_STUB(launch_conv_f16_w32_b7) SAMD_STUB(launch_conv_f16_w32_b8) SAMD_STUB(launch_conv_f16_w64_b1)
SAMD_STUB(launch_conv_f16_w64_b2) SAMD_STUB(launch_conv_f16_w64_b3) SAMD_STUB(launch_conv_f16_w64_b4)
SAMD_STUB(launch_conv_f16_w64_b5) SAMD_STUB(launch_conv_f16_w64_b6) SAMD_STUB(launch_conv_f16_w64_b7)
SAMD_STUB(launch_conv_f16_w64_b8) SAMD_STUB(launch_conv_f8_w32_b1) SAMD_STUB(launch_conv_f8_w32_b2)
SAMD_STUB(launch_conv_f8_w32_b3) SAMD_STUB(launch_conv_f8_w32_b4) SAMD_STUB(launch_conv_f8_w32_b5)
SAMD_STUB(launch_conv_f8_w64_b1) SAMD_STUB(launch_conv_f8_w64_b2) SAMD_STUB(launch_conv_f8_w64_b3)
SAMD_STUB(launch_conv_f8_w64_b4) SAMD_STUB(launch_conv_f8_w64_b5)

namespace samd {
int sm_count() { return 152; }  // defined in samd_api.cu, not linked here
}  // namespace samd
