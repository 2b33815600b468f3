// Host-only check of the convolution planner (conv2d.cu's make_plan,
// layout_ok and place_acc_stage) over a grid of shapes and formats: every plan
// it accepts, plain, with int32 rows staged, or pooled, fits the shared-memory
// and TMEM limits, its regions follow one another without overlap, and a
// pooled plan reads the prepared weights of the plain one. Compiled and run by
// tests/test_plan_cpu.py; the kernel launchers are replaced by stubs (nothing
// is launched).
#include "../paper_1809_10572_gb300/csrc/conv2d.cu"

#include "conv_stubs.cuh"

namespace samd {
// the NCHW path lives in widemul.cu, not linked here
samd_status conv2d_nchw_check(const samd_conv_desc *, samd_fmt, samd_fmt, samd_fmt, size_t *) { return SAMD_EUNSUP; }
samd_status conv2d_nchw(const samd_conv_desc *, samd_fmt, const void *, samd_fmt, const void *, int32_t *, samd_fmt,
                        void *, int, void *, size_t, cudaStream_t) {
  return SAMD_EUNSUP;
}
}  // namespace samd

#include <cstdio>

namespace {
using namespace samd;

// Operand stages, weight stages, packed staging, epilogue stage, barriers, one
// after the other; sizes are counted again here, not taken from layout_ok.
bool regions_ok(const conv::Plan &p, const samd_conv_desc &d, samd_fmt fo) {
  const size_t no = p.halo ? p.hbufs : p.stages_a, ng = 2;
  const size_t weights = static_cast<size_t>(p.stages) * p.tgroup * p.mma_n * p.row_bytes;
  size_t epi = 0;
  if (p.e_flat) epi = 8 * 32 * 4 * static_cast<size_t>(words_per_row(fo, d.K));  // 32 whole rows a warp
  if (p.e_stage && epi < 8 * 32 * 33 * 4) epi = 8 * 32 * 33 * 4;                 // 32 words of 32 rows, 33 apart
  if (epi < 8 * 4 * static_cast<size_t>(p.e_words)) epi = 8 * 4 * static_cast<size_t>(p.e_words);
  if (p.pool) epi = 256 * 4 * static_cast<size_t>(p.pool_pitch);
  const size_t bars = 8 * (2 * p.stages + 2 * no + 7) + 4;
  bool ok = no * p.op_stride <= p.off_b && p.off_b + weights <= p.off_g && p.off_g + ng * p.g_stride <= p.off_e &&
            p.off_e + epi <= p.off_bar && 1023 + p.off_bar + bars <= p.smem_bytes && p.smem_bytes <= 227 * 1024;
  // a streamed stage is a tile or a filter row of them; resident weights are all there
  ok = ok && (p.tgroup == 1 || (p.halo && !p.b_resident && p.tgroup == d.S)) &&
       (!p.b_resident || (p.nblocks == 1 && p.stages == p.nchunks)) && p.nchunks % p.tgroup == 0;
  if (p.pool) {
    // whole row pairs of a tile, their words within a staged row, windows within the buffer
    const int words = static_cast<int>(words_per_row(fo, p.NBc));
    ok = ok && p.hv <= 2 && p.pool_rows * p.Wp <= 128 * p.hv && p.pool_rows % 2 == 0 && p.pool_nw == words &&
         p.pool_pitch >= words && p.pool_tpi * p.pool_rows >= p.Ho && (p.pool_tpi - 1) * p.pool_rows < p.Ho;
  }
  return ok && conv::layout_ok(p);
}
}  // namespace

int main() {
  long long flat = 0, rows = 0, accs = 0, pools = 0;
  long long n = 0, bad = 0, halo = 0, seg = 0, fp8 = 0, res = 0, unsup = 0, hv2 = 0, win = 0, estg = 0, hv4 = 0;
  const int Cs[] = {1, 3, 16, 24, 64, 96, 128, 256, 512, 1024};
  const int Ks[] = {1, 16, 40, 64, 96, 128, 256, 300, 512, 1024};
  const int HWs[] = {1, 2, 7, 14, 28, 56, 224};
  for (int wb : {32, 64})
    for (int ba = 1; ba <= 8; ++ba)
      for (int sa = 0; sa < 2; ++sa)
        for (int bw = 1; bw <= 8; bw += (bw < 2 ? 1 : 2))
          for (int sw = 0; sw < 2; ++sw)
            for (int C : Cs)
              for (int K : Ks)
                for (int hw : HWs)
                  for (int rs : {1, 3, 5})
                    for (int st : {1, 2}) {
                      if (rs > hw + 2) continue;
                      samd_conv_desc d{hw >= 112 ? 16 : 2, C, hw, hw, K, rs, rs, st, rs / 2, SAMD_NHWC};  // batch 16 for large images (four-part tiles)
                      samd_fmt fa{(uint8_t)ba, (uint8_t)sa, 0, (uint8_t)wb};
                      samd_fmt fw{(uint8_t)bw, (uint8_t)sw, 0, (uint8_t)wb};
                      for (int fob : {0, 3, 4, 6}) {
                        samd_fmt fo{(uint8_t)fob, 0, 0, 32};
                        conv::Plan p;
                        const samd_status s = conv::make_plan(&d, fa, fw, fo, p);
                        ++n;
                        if (s != SAMD_OK) {
                          ++unsup;
                          continue;
                        }
                        if (p.M == 0) continue;
                        bool ok = regions_ok(p, d, fo);
                        if (p.halo) {
                          ++halo;
                          if (p.nseg > 1) ++seg;
                          const int maxrow = (d.R - 1) * p.row_step + (d.S - 1) + 128 * p.hv - 1;
                          const int srow = (p.WC * wb / 8 + 15) / 16 * 16;
                          ok = ok && maxrow < p.nseg * p.seg_rows &&
                               p.nseg * p.seg_rows * static_cast<long long>(p.row_bytes) <= p.op_stride &&
                               static_cast<long long>(p.nseg) * p.seg_rows * srow <= p.g_stride;
                        } else {
                          // gather staging: a producer group's ring of kGatherDepth x 128 rows
                          const int chunk_bytes = p.WC * wb / 8;
                          const int srow = (chunk_bytes + 15) / 16 * 16;
                          ok = ok && p.g_row >= srow && p.g_row % 16 == 0 &&
                               p.g_stride >= static_cast<uint32_t>(conv::kGatherDepth * conv::BM * p.g_row);
                          if (p.gather_win) {
                            ++win;
                            // (channel chunk, tap) chunks, each inside one pixel
                            ok = ok && p.g_row >= srow + 16 && (p.g_row / 16) % 2 == 1 &&
                                 p.nchunks == p.nck * p.taps && p.nck * p.WC >= p.wpr && (p.nck - 1) * p.WC < p.wpr;
                          }
                        }
                        if (p.fp8) ++fp8;
                        if (p.b_resident) ++res;
                        if (p.hv == 2) ++hv2;
                        if (p.hv == 4) ++hv4;
                        ok = ok && p.tmem_cols <= 512 && 2 * p.hv * p.mma_n <= static_cast<int>(p.tmem_cols);
                        if (p.e_stage) {
                          ++estg;
                          ok = ok && (fob == 3 || fob == 5 || fob == 6) && p.off_e + conv::kEpiStageBytes <= p.off_bar;
                        }
                        if (p.e_flat) ++flat;
                        if (p.tgroup > 1) ++rows;
                        conv::Plan q = p;
                        if (conv::place_acc_stage(q)) {
                          ++accs;
                          ok = ok && q.e_words >= 32 * conv::kEpiPitch && q.e_words >= p.e_words && regions_ok(q, d, fo);
                        }
                        if (fob == 4 && conv::make_plan(&d, fa, fw, fo, q, true) == SAMD_OK) {
                          ++pools;
                          ok = ok && q.pool && regions_ok(q, d, fo) && p.halo && q.Kpad == p.Kpad && q.mma_n == p.mma_n &&
                               q.NBc == p.NBc && q.nblocks == p.nblocks && q.fp8 == p.fp8 && q.split == p.split;
                        }
                        if (!ok && ++bad < 10)
                          printf("BAD C%d K%d hw%d rs%d st%d a%d%d w%d%d wb%d fo%d: smem %zu stages %d sta %d\n", C, K,
                                 hw, rs, st, ba, sa, bw, sw, wb, fob, p.smem_bytes, p.stages, p.stages_a);
                      }
                    }
  printf("plans %lld, bad %lld, unsupported %lld, halo %lld (segmented %lld), e4m3 %lld, resident %lld, "
         "two-half %lld, four-part %lld, window gather %lld, staged epilogue %lld, "
         "flat epilogue %lld, filter-row stages %lld, int32 stage %lld, pooled %lld\n",
         n, bad, unsup, halo, seg, fp8, res, hv2, hv4, win, estg, flat, rows, accs, pools);
  return bad != 0;
}
