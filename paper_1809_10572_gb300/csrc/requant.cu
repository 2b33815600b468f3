// requant.cu -- lane-wise requantize into another format:
// out = clamp_fo(floor(x / 2^shift)) (not in the paper; the step between
// layers of different precision).
//
// Spacer-free 32-bit words: a thread takes whole periods of the two lane
// grids, lcm(L_in, L_out) lanes, so that every lane's word and bit position
// are compile-time on both sides; 64-bit words whose lane widths divide 32
// are such words, two to each. A lane costs four operations: two extract and
// shift it, one adds the offset of a signed output, clamps to its range and
// to zero (viaddmin with relu), one inserts it; the offset is taken off a
// whole word by flipping its lanes' top bits. Bound by HBM where both formats
// have at most eight lanes a word, by the integer pipe for narrower lanes.
// 2^26 signed 8-bit lanes to unsigned 4-bit ones, 32-bit words: 139 us with
// one thread per output word that divided and switched for each lane, now
// 18.6 us (5.4 TB/s).
//
// Every other pair of formats (spacers, 64-bit words of 3, 5, 6 or 7 bits,
// words of different width) takes one thread per output word that walks the
// input lanes from one exact multiply-high division.
#include "samd_internal.cuh"

namespace samd {
namespace {

constexpr int kThreads = 256;

struct LaneFmt {
  int bits, is_signed, lane_w, L;
};

LaneFmt lane_fmt(samd_fmt f) { return LaneFmt{f.bits, f.is_signed, f.bits + f.spacer, lanes_per_word(f)}; }

// x / d and the remainder for x < 2^63, 1 <= d <= 64: the multiply-high by
// floor(2^64 / d) is the quotient or one less (d = 1: the quotient less one
// for x > 0).
__device__ __forceinline__ int64_t div_small(int64_t x, int d, uint64_t recip, int *rem) {
  int64_t q = static_cast<int64_t>(__umul64hi(static_cast<uint64_t>(x), recip));
  int64_t r = x - q * d;
  if (r >= d) {
    r -= d;
    ++q;
  }
  *rem = static_cast<int>(r);
  return q;
}

// Output word w: lanes [w L_out, min((w + 1) L_out, n)).
template <typename WI, typename WO>
__device__ __forceinline__ WO requant_word(const LaneFmt &fa, const WI *a, const LaneFmt &fo, int64_t w, int64_t n,
                                           int shift, uint64_t recip) {
  const uint32_t ma = (1u << fa.bits) - 1, mo = (1u << fo.bits) - 1;
  const int lo = lane_lo(fo.bits, fo.is_signed), hi = lane_hi(fo.bits, fo.is_signed);
  const int64_t e0 = w * fo.L;
  if (e0 >= n) return 0;  // the high half of a last 64-bit word
  const int cnt = n - e0 < fo.L ? static_cast<int>(n - e0) : fo.L;
  int li;
  const WI *p = a + div_small(e0, fa.L, recip, &li);
  WI cur = *p;
  int pos = li * fa.lane_w;
  WO word = 0;
  for (int l = 0; l < cnt; ++l) {
    if (li == fa.L) {
      cur = *++p;
      li = pos = 0;
    }
    const int v = lane_value(static_cast<uint32_t>(cur >> pos) & ma, fa.bits, fa.is_signed) >> shift;
    word |= static_cast<WO>(static_cast<uint32_t>(clamp_int(v, lo, hi)) & mo) << (l * fo.lane_w);
    ++li;
    pos += fa.lane_w;
  }
  return word;
}

template <typename WI, typename WO>
__global__ void __launch_bounds__(kThreads)
    requant_lane_kernel(LaneFmt fa, const WI *a, LaneFmt fo, WO *out, int64_t n, int64_t nwords_out, int shift,
                        uint64_t recip) {
  for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < nwords_out;
       w += (int64_t)gridDim.x * blockDim.x)
    out[w] = requant_word<WI, WO>(fa, a, fo, w, n, shift, recip);
}

constexpr int gcd_c(int a, int b) { return b == 0 ? a : gcd_c(b, a % b); }

// The lanes one thread takes: the period of the two grids, four of them where
// that makes both sides whole 16-byte vectors of at most 128 lanes.
template <int BA, int BO>
struct Period {
  static constexpr int LA = 32 / BA, LO = 32 / BO;
  static constexpr int E = LA / gcd_c(LA, LO) * LO;
  static constexpr int G = E * 4 <= 128 ? 4 : 1;
  static constexpr int kLanes = E * G, IW = kLanes / LA, OW = kLanes / LO;
};

template <int N>
__device__ __forceinline__ void load_words(const uint32_t *p, uint32_t (&w)[N]) {
  if constexpr (N % 4 == 0) {
#pragma unroll
    for (int i = 0; i < N / 4; ++i) {
      const uint4 q = __ldcs(reinterpret_cast<const uint4 *>(p) + i);
      w[4 * i] = q.x, w[4 * i + 1] = q.y, w[4 * i + 2] = q.z, w[4 * i + 3] = q.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) w[i] = __ldcs(p + i);
  }
}

template <int N>
__device__ __forceinline__ void store_words(uint32_t *p, const uint32_t (&w)[N]) {
  if constexpr (N % 4 == 0) {
#pragma unroll
    for (int i = 0; i < N / 4; ++i)
      __stcs(reinterpret_cast<uint4 *>(p) + i, make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]));
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) __stcs(p + i, w[i]);
  }
}

// `shift` is at most BA - 1; keep: the bits an unsigned lane has left after
// the whole shift (0 from BA on; signed lanes are 0 or -1 from BA - 1 on).
// off: half the range of a signed output, else 0; flip: the output lanes' top
// bits if it is signed, else 0. The lanes past the last whole period take the
// word form.
template <int BA, int BO, bool SA>
__global__ void __launch_bounds__(kThreads)
    requant32_kernel(const uint32_t *a, uint32_t *out, int64_t nperiods, int64_t n, int64_t nwords_out, int shift,
                     uint32_t keep, int whole_shift, int off, uint32_t flip, uint64_t recip) {
  using P = Period<BA, BO>;
  constexpr int omax = (1 << BO) - 1;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x, t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  for (int64_t t = t0; t < nperiods; t += stride) {
    uint32_t in[P::IW], w[P::OW];
    load_words(a + t * P::IW, in);
#pragma unroll
    for (int j = 0; j < P::OW; ++j) w[j] = 0;
#pragma unroll
    for (int e = 0; e < P::kLanes; ++e) {
      constexpr int LA = P::LA, LO = P::LO;
      const uint32_t x = in[e / LA];
      const int p = (e % LA) * BA;
      const int v = SA ? static_cast<int>(x << (32 - BA - p)) >> (32 - BA + shift)
                       : static_cast<int>((x >> (p + shift)) & keep);
      w[e / LO] += static_cast<uint32_t>(__viaddmin_s32_relu(v, off, omax)) << ((e % LO) * BO);
    }
#pragma unroll
    for (int j = 0; j < P::OW; ++j) w[j] ^= flip;
    store_words(out + t * P::OW, w);
  }
  const LaneFmt fa{BA, SA, BA, P::LA}, fo{BO, off != 0, BO, P::LO};
  for (int64_t w = nperiods * P::OW + t0; w < nwords_out; w += stride)
    out[w] = requant_word<uint32_t, uint32_t>(fa, a, fo, w, n, whole_shift, recip);
}

uint64_t recip_of(int d) { return d == 1 ? ~0ull : static_cast<uint64_t>((static_cast<unsigned __int128>(1) << 64) / d); }

template <int BA, int BO, bool SA>
cudaError_t launch32(const uint32_t *a, uint32_t *out, int64_t n, int64_t nwords_out, int shift, bool so,
                     cudaStream_t s) {
  using P = Period<BA, BO>;
  const int64_t nperiods = n / P::kLanes;
  const uint32_t keep = shift < BA ? ((1u << BA) - 1) >> shift : 0u;
  uint32_t flip = 0;
  if (so)
    for (int i = 0; i < P::LO; ++i) flip |= 1u << (i * BO + BO - 1);
  const int64_t work = nperiods > 0 ? nperiods : nwords_out;
  requant32_kernel<BA, BO, SA><<<resident_grid<requant32_kernel<BA, BO, SA>>(work, kThreads), kThreads, 0, s>>>(
      a, out, nperiods, n, nwords_out, shift < BA ? shift : BA - 1, keep, shift, so ? 1 << (BO - 1) : 0, flip,
      recip_of(P::LA));
  return cudaGetLastError();
}

template <int BA, bool SA>
cudaError_t dispatch_out(int bo, bool so, const uint32_t *a, uint32_t *out, int64_t n, int64_t nwo, int shift,
                         cudaStream_t s) {
  switch (bo) {
    case 1: return launch32<BA, 1, SA>(a, out, n, nwo, shift, so, s);
    case 2: return launch32<BA, 2, SA>(a, out, n, nwo, shift, so, s);
    case 3: return launch32<BA, 3, SA>(a, out, n, nwo, shift, so, s);
    case 4: return launch32<BA, 4, SA>(a, out, n, nwo, shift, so, s);
    case 5: return launch32<BA, 5, SA>(a, out, n, nwo, shift, so, s);
    case 6: return launch32<BA, 6, SA>(a, out, n, nwo, shift, so, s);
    case 7: return launch32<BA, 7, SA>(a, out, n, nwo, shift, so, s);
    case 8: return launch32<BA, 8, SA>(a, out, n, nwo, shift, so, s);
    default: return cudaErrorInvalidValue;
  }
}

bool pow2_bits(samd_fmt f) { return (f.bits & (f.bits - 1)) == 0; }

template <typename WI, typename WO>
cudaError_t lane_dispatch(samd_fmt fa, const void *a, samd_fmt fo, void *out, int64_t n, int shift, cudaStream_t s) {
  const int64_t nwo = words_per_row(fo, n);
  requant_lane_kernel<WI, WO><<<resident_grid<requant_lane_kernel<WI, WO>>(nwo, kThreads), kThreads, 0, s>>>(
      lane_fmt(fa), static_cast<const WI *>(a), lane_fmt(fo), static_cast<WO *>(out), n, nwo, shift,
      recip_of(lanes_per_word(fa)));
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_requant(samd_fmt fa, const void *a, samd_fmt fo, void *out, int64_t n, int shift, cudaStream_t s) {
  // 64-bit words of 1, 2, 4 or 8 bits are pairs of 32-bit words
  const bool halves = fa.word_bits == 64 && fo.word_bits == 64 && pow2_bits(fa) && pow2_bits(fo);
  if (fa.spacer == 0 && fo.spacer == 0 && ((fa.word_bits == 32 && fo.word_bits == 32) || halves)) {
    const uint32_t *pa = static_cast<const uint32_t *>(a);
    uint32_t *po = static_cast<uint32_t *>(out);
    const bool so = fo.is_signed != 0;
    const int64_t nwo = words_per_row(fo, n) * (halves ? 2 : 1);
    switch (fa.bits * 2 + (fa.is_signed ? 1 : 0)) {
#define SAMD_RQ(B)                                                              \
  case 2 * B: return dispatch_out<B, false>(fo.bits, so, pa, po, n, nwo, shift, s);  \
  case 2 * B + 1: return dispatch_out<B, true>(fo.bits, so, pa, po, n, nwo, shift, s);
      SAMD_RQ(1) SAMD_RQ(2) SAMD_RQ(3) SAMD_RQ(4) SAMD_RQ(5) SAMD_RQ(6) SAMD_RQ(7) SAMD_RQ(8)
#undef SAMD_RQ
      default: return cudaErrorInvalidValue;
    }
  }
  if (fa.word_bits == 32 && fo.word_bits == 32) return lane_dispatch<uint32_t, uint32_t>(fa, a, fo, out, n, shift, s);
  if (fa.word_bits == 32) return lane_dispatch<uint32_t, uint64_t>(fa, a, fo, out, n, shift, s);
  if (fo.word_bits == 32) return lane_dispatch<uint64_t, uint32_t>(fa, a, fo, out, n, shift, s);
  return lane_dispatch<uint64_t, uint64_t>(fa, a, fo, out, n, shift, s);
}

}  // namespace samd
