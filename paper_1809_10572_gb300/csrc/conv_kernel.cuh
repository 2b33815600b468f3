// conv_kernel.cuh -- the persistent tcgen05 convolution kernel (device code
// shared by the translation units that instantiate it).
//
// The paper's DNN convolution (section 7, Fig. 12, direct-sum2d) is
//   acc[n][k][ho][wo] = sum_{c,r,s} act[n][c][ho*st-p+r][wo*st-p+s] * wt[k][c][r][s].
// Here it is the GEMM D[M x K] = A[M x Kg] * B[K x Kg]^T with M = N*Ho*Wo
// output pixels and a reduction index Kg running over (tap, packed word,
// lane). Activations and weights stay packed in HBM and L2 and are widened
// only in shared memory, right before the MMA (the "unpack to the native
// type" baseline of section 7, moved on-chip).
//
// Exactness. sm_103a has no integer MMA, so lanes are widened to a float
// type whose every value in play is an exact integer, and the fp32
// accumulators hold exact integers while every partial sum stays below 2^24:
//   e4m3 (kind::f8f6f4, K = 32 per MMA) when |a| <= 16 and |w| <= 16 (lane
//        widths up to 4 bits, and signed 5-bit lanes); half the shared-memory
//        bytes of fp16 per product, twice the tensor rate;
//   fp16 (kind::f16, K = 16 per MMA) otherwise: every integer of [-128, 255].
// The A operand holds its integers times a power of two (op_exp), so the
// accumulators do too; that changes no exactness.
// When R*S*C*max|a|*max|w| reaches 2^24 (wide weights over many taps), the
// fp16 weights are split into two 4-bit digits w = 16*hi + lo stacked along
// the MMA's N; the epilogue forms 16*hi + lo in int32.
//
// Both operand types use rows of 64 reduction positions: 128-byte rows with
// the 128-byte swizzle (fp16) or 64-byte rows with the 64-byte swizzle
// (e4m3). An MMA consumes 32 bytes of a row either way, so the descriptors
// advance by the same 32 bytes per MMA.
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>

#include <cstring>
#include <type_traits>
#include <utility>

#include "samd_internal.cuh"
#include "tc_ptx.cuh"

namespace samd {
namespace conv {

constexpr int BM = 128;  // output pixels per tile = MMA M = TMEM lanes
constexpr int BK = 64;   // reduction positions per chunk = one operand row
constexpr uint64_t kWaitLimitNs = 1000000000ull;  // 1 s
constexpr int kGatherDepth = 4;                    // packed chunks in flight per producer thread
constexpr int kProdWarps = 8;                      // operand producers
constexpr int kEpiWarps = 8;                       // epilogue
constexpr int kProdThreads = 32 * kProdWarps;
// HALO: packed staging slots. Gathers run one item ahead of the widening: the
// producers finish a tile's operands microseconds before its MMAs start, and
// the sweep step measured 6% slower with four slots.
constexpr int kHaloGatherSlots = 2;
constexpr int kMaxHaloRows = 1024;                 // of one tile (kMaxHaloRows / kProdThreads rows per producer thread)
constexpr int kThreads = 32 * (2 + kProdWarps + kEpiWarps);
constexpr int kFirstEpiWarp = 2 + kProdWarps;
// Optional epilogue staging (ConvArgs::e_stage): per epilogue warp 32 words of
// 32 rows, kEpiPitch words apart (odd, so that 32 lanes writing one word of
// their own rows hit 32 banks).
constexpr int kEpiPitch = 33;
constexpr uint32_t kEpiStageBytes = kEpiWarps * 32 * kEpiPitch * 4;

template <bool FP8>
struct OpTraits {
  static constexpr int kRowBytes = FP8 ? 64 : 128;  // one row of BK positions
  static constexpr int kKPerMma = FP8 ? 32 : 16;
  static constexpr uint32_t kTileBytes = BM * kRowBytes;
  // 16-byte chunk c of row r (rows kRowBytes apart from a 1024-byte-aligned base)
  __device__ static __forceinline__ int swz(int r, int c) { return FP8 ? (c ^ ((r >> 1) & 3)) : (c ^ (r & 7)); }
  __device__ static __forceinline__ uint64_t desc(uint32_t saddr) {
    return FP8 ? ptx::sw64_kmajor_desc(saddr) : ptx::sw128_kmajor_desc(saddr);
  }
};

__host__ __device__ constexpr bool pair16(int bits) { return bits == 1 || bits == 2 || bits == 4 || bits == 8; }

// The lane of a packed word held by reduction position `pos` (0 <= pos < L)
// of that word. For lane widths dividing 16, positions 2p and 2p+1 hold
// lanes p and p + 16/bits of the same 32-bit half, which sit exactly 16 bits
// apart, so one masked shift widens both at once. Other widths keep lane
// order. A and B use the same map, so the dot products are unchanged.
__host__ __device__ constexpr int kpos_lane(int bits, int pos) {
  if (pair16(bits)) {
    int g = 32 / bits, half = pos / g, jj = pos % g;
    return half * g + jj / 2 + (jj & 1) * (g / 2);
  }
  return pos;
}

// A's operand elements are the lanes' own bits where that is a number: the
// subnormal and first normal binade of a float format are linear in its
// encoding, so the byte v (0..16) is v * 2^-9 in e4m3 and the half-word v
// (0..2047) is v * 2^-24 in fp16. Widening an unsigned lane is then a shift
// and a mask, without a table, a bias or a conversion. The accumulators hold
// exact multiples of 2^-kOpExp (the same 24 bits of an integer sum, scaled by
// a power of two) and the epilogue's scale takes the factor back. Signed
// lanes are sign and magnitude in e4m3; in fp16 they are widened through the
// mantissa of 1024.0 to their own value (exponent 0).
__host__ __device__ constexpr int op_exp(bool is_signed, bool fp8) { return fp8 ? 9 : (is_signed ? 0 : 24); }

// Orders of the e4m3 positions of a 32-bit half-word of 1-, 2- and 4-bit
// lanes; A and B use the same one. By masks (unsigned lanes, signed 4-bit
// lanes): word x >> (BITS k) keeps one lane of every byte, so position 4k + b
// is lane b * 8 / BITS + k. By permutes (signed 1- and 2-bit lanes, whose
// nibbles select from a table): even then odd lanes for 2 bits, lanes k,
// k + 4, ... for 1 bit.
__host__ __device__ constexpr bool mask8(int bits, bool is_signed) {
  return bits == 4 || (!is_signed && (bits == 1 || bits == 2));
}
__host__ __device__ constexpr bool prmt8(int bits, bool is_signed) { return is_signed && (bits == 1 || bits == 2); }
__host__ __device__ constexpr int kpos_lane_mask32(int bits, int p) { return (p % 4) * (8 / bits) + p / 4; }
__host__ __device__ constexpr int kpos_lane_prmt32(int bits, int p) {
  return bits == 2 ? 2 * (p % 4 + 4 * ((p / 4) % 2)) + p / 8 : 4 * (p % 8) + p / 8;
}
// The lane of an activation word held by reduction position `pos` for the
// operand type in use.
__host__ __device__ constexpr int kpos_lane_op(int bits, bool is_signed, bool fp8, int pos) {
  if (fp8 && (mask8(bits, is_signed) || prmt8(bits, is_signed))) {
    const int g = 32 / bits, half = pos / g, p = pos % g;
    return half * g + (mask8(bits, is_signed) ? kpos_lane_mask32(bits, p) : kpos_lane_prmt32(bits, p));
  }
  return kpos_lane(bits, pos);
}

// e4m3 code of v * 2^-9 (|v| <= 16): sign and magnitude.
__host__ __device__ constexpr uint32_t e4m3_code(int v) { return v < 0 ? 0x80u | static_cast<uint32_t>(-v) : static_cast<uint32_t>(v); }
__host__ __device__ constexpr uint32_t e4m3_table4(int v0, int v1, int v2, int v3) {
  return e4m3_code(v0) | (e4m3_code(v1) << 8) | (e4m3_code(v2) << 16) | (e4m3_code(v3) << 24);
}

// prmt.b32 in its default mode: byte i of the result is byte (c_i & 7) of
// {b, a}, or, when bit 3 of selector nibble c_i is set, that byte's sign bit
// repeated eight times.
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

struct ConvArgs {
  const void *act;
  int32_t *acc_out;
  void *packed_out;
  // NCHW outputs (nchw = 1): acc_out is [N][K][Ho][Wo], and q8_out (or null)
  // receives the requantized lane patterns one per byte in the same order
  int nchw;
  uint8_t *q8_out;
  int *status;  // sticky SAMD_ETIMEOUT record of this device
  int N, C, H, W, K, R, S, stride, pad, Ho, Wo;
  long long M;
  int wpr;          // activation words per pixel
  int nchunks;      // weight tiles per output tile
  int NBc;          // output channels per channel block
  int n_mma;        // NBc rounded up to 16
  int mma_n;        // MMA N: n_mma, or 2 * n_mma with split weight digits
  int split;        // 1: accumulator columns [0, n_mma) hold hi digits, [n_mma, 2 n_mma) lo digits
  int stages;       // weight stages in flight (or resident tiles)
  int tgroup;       // weight tiles of a stage: a filter row's (HALO, streamed weights) or 1
  int stages_a;     // GATHER: A tiles in flight
  int b_resident;   // 1: all weight tiles of the layer stay in shared memory
  long long grid_m; // 128-position tiles along the output
  int nblocks;      // channel blocks
  int gather_vec;   // AGather::vec
  int gather_win;   // AGather::issue_win (chunks that are not aligned 16-byte vectors); chunk = (channel chunk, tap)
  int g_row;        // GATHER staging row pitch in bytes
  int hbufs;        // HALO: widened halo buffers (2 or 3); item k goes to buffer k mod hbufs
  long long act_bytes;  // bytes of the activation tensor (the windows stop at its end)
  uint32_t tmem_cols;
  int out_bits, out_signed, out_lane_w, out_L, out_word64, out_wpr;
  int out_fast;     // output lanes per word when they divide 32 (whole words per 32 channels), else 0
  int shift;
  float acc_scale;  // an accumulator times acc_scale is its integer sum (2^op_exp)
  float out_scale;  // acc_scale * 2^-shift
  int fast_req;     // |acc| / 2^shift < 2^22: requantize through floor_scaled_biased
  int fast_acc;     // |acc| < 2^22: int32 outputs through floor_scaled_biased
  // HALO (stride 1): virtual output grid of N x Hv x Wp positions. A tile of
  // 128 consecutive positions v0.. reads nseg segments of the input grid:
  // segment g holds seg_used rows starting at virtual row v0 + g * Wp and
  // occupies seg_rows rows of the halo buffer; tap (r, s) reads the 128 rows
  // starting at halo row r * row_step + s.
  int Hv, Wp;
  int nseg, seg_rows, seg_used, row_step;
  int nck;   // channel chunks per pixel (ceil(wpr / WC))
  int full;  // AUnpack FULL: one chunk holds all the pixel's words
  int hv;    // tile of hv parts of 128 output positions (1, 2, or 4 for e4m3 halo layers)
  int taps;  // R * S
  FastDiv fd_plane, fd_wp;  // / (Hv * Wp), / Wp
  FastDiv fd_seg;           // / seg_rows
  FastDiv fd_wo, fd_ho;     // output pixel index -> (n, oh, ow)
  FastDiv fd_howo;          // output pixel index -> (n, pixel of the image)
  FastDiv fd_gm;            // tile -> (channel block, position tile)
  // shared memory carve-up (bytes from the 1024-byte-aligned base)
  uint32_t op_stride;  // one halo buffer or one A tile
  uint32_t off_b, b_bytes, off_g, g_stride, off_e, off_bar;
  int e_stage;  // 1: kEpiStageBytes at off_e stage 32 words of each 3/5/6-bit packed row (epilogue_row_words)
  int e_flat;   // 1: 32 whole rows per epilogue warp at off_e instead (one channel block)
  int acc_stage;  // 1: int32 rows are staged too, 32 words of each (epilogue_row_acc)
  int e_words;    // words of an epilogue warp's stage
  int early;    // 1: the next kernel of the stream may be set up while this one drains
  // Fused 2x2 max-pool (pool = 1; halo layers): tile mt is pool_rows output
  // rows (pool_rows / 2 row pairs) of one image from an even row on, at
  // virtual position img * Hv * Wp + g * pool_rows * Wp (img = mt / tiles
  // per image, g its remainder). The epilogue warps that drain a tile pack
  // its rows into the pool_pitch-word rows of their buffer at off_e (pool_nw
  // words of the channel block per row) and write only the lane-wise maxima
  // of the 2x2 windows, rows of (N, Ho / 2, Wo / 2) pixels, to packed_out.
  int pool, pool_rows, pool_nw, pool_pitch;
  FastDiv fd_tpi;          // tiles per image
  FastDiv fd_pnw, fd_wo2;  // / pool_nw, / (Wo / 2)
};

// First position, in the padded virtual grid N x Hv x Wp, of tile mt of a
// halo layer (tiles of bmt consecutive positions, or pooled tiles of whole
// row pairs).
__device__ __forceinline__ uint32_t tile_first_pos(const ConvArgs &args, uint32_t mt, int bmt) {
  if (!args.pool) return mt * static_cast<uint32_t>(bmt);
  const uint32_t img = fdiv(mt, args.fd_tpi);
  const uint32_t g = mt - img * args.fd_tpi.d;
  return img * args.fd_plane.d + g * static_cast<uint32_t>(args.pool_rows * args.Wp);
}

__device__ __forceinline__ uint32_t hsub2_bits(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

// Four lane patterns of `BITS` bits, one per byte, as signed e4m3 codes:
// negative patterns (top bit set) become their magnitude with the sign bit.
template <int BITS>
__device__ __forceinline__ uint32_t sign_magnitude4(uint32_t e) {
  const uint32_t n = (e >> (BITS - 1)) & 0x01010101u;       // 1 in the bytes of negative lanes
  return ((e ^ (n * ((1u << BITS) - 1))) + n) + n * 0x80u;  // 2^BITS - e: bytes stay below 2^7
}

// Widening of one 64-position row of the A operand (one pixel, one chunk).
// A chunk is WC whole words. FULL (lanes per word not dividing 64, at most
// 64 channels in ceil(64 / L) words): one chunk holds all the pixel's words
// and its 64 positions are channels 0..63 -- the last word's lanes past 64
// are padding; otherwise WC = floor(64 / L) and positions past WC * L are
// zero.
template <typename W, int BITS, bool SIGNED, bool FP8, bool FULL = false>
struct AUnpack {
  static constexpr int WB = WordTraits<W>::kBits;
  static constexpr int L = WB / BITS;
  static constexpr int WC = FULL ? (BK + L - 1) / L : BK / L;  // packed words per chunk
  static constexpr int KUSED = FULL ? BK : WC * L;             // positions holding lanes; the rest are zero
  static constexpr uint32_t LM = (1u << BITS) - 1;
  static constexpr uint32_t OFF = SIGNED ? (1u << (BITS - 1)) : 0u;  // offset-binary zero
  static constexpr uint32_t BIAS = 0x6400u + OFF;                   // fp16 bits of 1024 + OFF
  static constexpr uint32_t BIAS2 = BIAS | (BIAS << 16);

  static constexpr W sign_mask() {
    W m = 0;
    for (int i = 0; i < L; ++i) m |= W(1) << (i * BITS + BITS - 1);
    return m;
  }

  template <int POS>
  __device__ static __forceinline__ uint32_t field(W w) {
    return static_cast<uint32_t>(w >> (kpos_lane(BITS, POS) * BITS)) & LM;
  }

  // Two fp16 operand elements. Unsigned lanes: their bits. Signed lanes: a
  // pattern v in offset binary becomes 1024 + v by or-ing it into the
  // mantissa of 1024.0; subtracting 1024 + OFF leaves the lane's value
  // exactly. A zero word (padding) therefore widens to zeros.
  __device__ static __forceinline__ uint32_t half2(uint32_t t) {
    if constexpr (SIGNED) return hsub2_bits(t | 0x64006400u, BIAS2);
    return t;
  }
  template <int P>
  __device__ static __forceinline__ uint32_t pair(const W (&w)[WC]) {
    constexpr int j0 = 2 * P, j1 = 2 * P + 1;
    if constexpr (j0 >= KUSED) {
      return 0u;
    } else if constexpr (pair16(BITS)) {
      constexpr int q = j0 / L, pos = j0 % L, g = 32 / BITS, half = pos / g;
      constexpr int lane0 = kpos_lane(BITS, pos) - half * g;
      const uint32_t x = static_cast<uint32_t>(w[q] >> (half * 32));
      return half2((x >> (lane0 * BITS)) & (LM | (LM << 16)));
    } else {
      const uint32_t v0 = field<j0 % L>(w[j0 / L]);
      uint32_t v1 = OFF;
      if constexpr (j1 < KUSED) v1 = field<j1 % L>(w[j1 / L]);
      return half2(v0 | (v1 << 16));
    }
  }

  template <int... P>
  __device__ static __forceinline__ void pairs(const W (&w)[WC], uint32_t (&h)[32],
                                               std::integer_sequence<int, P...>) {
    ((h[P] = pair<P>(w)), ...);
  }

  // The e4m3 bytes of the lanes of one 32-bit half-word of 1-, 2- or 4-bit
  // lanes, in reduction order (32 / BITS bytes into out[0 .. 8 / BITS)).
  static constexpr bool kWordwise = FP8 && (mask8(BITS, SIGNED) || prmt8(BITS, SIGNED));
  __device__ static __forceinline__ void bytes_of_half(uint32_t x, uint32_t *out) {
    if constexpr (mask8(BITS, SIGNED)) {
#pragma unroll
      for (int k = 0; k < 8 / BITS; ++k) {
        out[k] = (x >> (BITS * k)) & (LM * 0x01010101u);
        if constexpr (SIGNED) out[k] = sign_magnitude4<BITS>(out[k]);
      }
    } else if constexpr (BITS == 2) {
      constexpr uint32_t t = e4m3_table4(0, 1, -2, -1);
      const uint32_t se = x & 0x33333333u, so = (x >> 2) & 0x33333333u;
      out[0] = prmt(t, 0u, se);
      out[1] = prmt(t, 0u, se >> 16);
      out[2] = prmt(t, 0u, so);
      out[3] = prmt(t, 0u, so >> 16);
    } else {
      constexpr uint32_t t = e4m3_table4(0, -1, 0, 0);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t sk = (x >> k) & 0x11111111u;
        out[2 * k] = prmt(t, 0u, sk);
        out[2 * k + 1] = prmt(t, 0u, sk >> 16);
      }
    }
  }

  // Four e4m3 operand elements, positions 4 P .. 4 P + 3 in lane order (3-
  // and 5-bit lanes).
  template <int P>
  __device__ static __forceinline__ uint32_t quad(const W (&w)[WC]) {
    const uint32_t e = lane_at<4 * P>(w) | (lane_at<4 * P + 1>(w) << 8) | (lane_at<4 * P + 2>(w) << 16) |
                       (lane_at<4 * P + 3>(w) << 24);
    if constexpr (SIGNED) return sign_magnitude4<BITS>(e);
    return e;
  }
  template <int J>
  __device__ static __forceinline__ uint32_t lane_at(const W (&w)[WC]) {
    if constexpr (J < KUSED)
      return static_cast<uint32_t>(w[J / L] >> ((J % L) * BITS)) & LM;
    else
      return 0u;
  }
  template <int... P>
  __device__ static __forceinline__ void quads(const W (&w)[WC], uint32_t (&b)[16], std::integer_sequence<int, P...>) {
    ((b[P] = quad<P>(w)), ...);
  }

  // Widen one pixel's chunk and store it as row `row` of a swizzled K-major
  // operand whose rows are OpTraits::kRowBytes apart.
  __device__ static __forceinline__ void unpack_row(W (&w)[WC], uint8_t *tile, int row) {
    using T = OpTraits<FP8>;
    uint8_t *rp = tile + row * T::kRowBytes;
    if constexpr (FP8) {
      uint32_t b[16];
      if constexpr (kWordwise) {
        constexpr int kHalves = WB / 32, kPer = 8 / BITS;  // 32-bit words of e4m3 bytes per half-word
#pragma unroll
        for (int q = 0; q < WC; ++q)
#pragma unroll
          for (int hh = 0; hh < kHalves; ++hh)
            bytes_of_half(static_cast<uint32_t>(w[q] >> (32 * hh)), b + (q * kHalves + hh) * kPer);
      } else {
        quads(w, b, std::make_integer_sequence<int, 16>{});
      }
#pragma unroll
      for (int c = 0; c < 4; ++c)
        *reinterpret_cast<uint4 *>(rp + (T::swz(row, c) << 4)) = make_uint4(b[4 * c], b[4 * c + 1], b[4 * c + 2], b[4 * c + 3]);
    } else {
      if constexpr (SIGNED) {
#pragma unroll
        for (int q = 0; q < WC; ++q) w[q] ^= sign_mask();
      }
      uint32_t h[32];
      pairs(w, h, std::make_integer_sequence<int, 32>{});
#pragma unroll
      for (int c = 0; c < 8; ++c)
        *reinterpret_cast<uint4 *>(rp + (T::swz(row, c) << 4)) =
            make_uint4(h[4 * c], h[4 * c + 1], h[4 * c + 2], h[4 * c + 3]);
    }
  }
};

// Bytes of one pixel-chunk row in the packed staging buffers (a multiple of 16).
template <typename W, int WC>
struct Staging {
  static constexpr int kBytes = WC * static_cast<int>(sizeof(W));
  static constexpr int kRowBytes = (kBytes + 15) / 16 * 16;
  // widest cp.async that divides a whole chunk held by one pixel
  static constexpr int kVec = kBytes % 16 == 0 ? 16 : (kBytes % 8 == 0 ? 8 : static_cast<int>(sizeof(W)));
};

// Copies a pixel-chunk of kBytes from `src` (vector-aligned) to staging with
// cp.async; nbytes = 0 zero-fills it.
template <typename W, int WC>
__device__ __forceinline__ void stage_chunk(uint32_t dst, const char *src, uint32_t valid) {
  using St = Staging<W, WC>;
#pragma unroll
  for (int v = 0; v < St::kBytes / St::kVec; ++v) {
    if constexpr (St::kVec == 16)
      ptx::cp_async_16(dst + 16 * v, src + 16 * v, valid ? 16u : 0u);
    else if constexpr (St::kVec == 8)
      ptx::cp_async_8(dst + 8 * v, src + 8 * v, valid ? 8u : 0u);
    else
      ptx::cp_async_4(dst + 4 * v, src + 4 * v, valid ? 4u : 0u);
  }
}

// Reads a staged pixel-chunk back into words.
template <typename W, int WC>
__device__ __forceinline__ void load_staged(const uint8_t *src, W (&cur)[WC]) {
  using St = Staging<W, WC>;
#pragma unroll
  for (int v = 0; v < St::kRowBytes / 16; ++v) {
    const uint4 q4 = *reinterpret_cast<const uint4 *>(src + 16 * v);
    const uint32_t tw[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
    for (int kq = 0; kq < 4; ++kq) {
      const int byte = 16 * v + 4 * kq;
      if (byte < St::kBytes) {
        if constexpr (sizeof(W) == 4) {
          cur[byte / 4] = tw[kq];
        } else if ((kq & 1) == 0) {
          cur[byte / 8] = static_cast<W>(tw[kq]) | (static_cast<W>(tw[kq + 1]) << 32);
        }
      }
    }
  }
}

// 16-byte pieces that cover one chunk from the 16-byte boundary at or below
// its first byte (the chunk then starts o bytes into the staged row, o < 16).
template <typename W, int WC>
constexpr int kWinPieces = (WC * static_cast<int>(sizeof(W)) + 15) / 16 + 1;

// Reads a chunk staged through its 16-byte window (AGather::issue_win): the
// chunk starts o4 32-bit units into the row; words from nw on are zero.
template <typename W, int WC>
__device__ __forceinline__ void load_window(const uint8_t *row, int o4, int nw, W (&cur)[WC]) {
  constexpr int kU = WC * static_cast<int>(sizeof(W)) / 4;  // 32-bit units of a chunk
  constexpr int kV = (kU + 3 + 3) / 4;                       // 16-byte reads covering kU + 3 units
  static_assert(kV <= kWinPieces<W, WC>, "the window holds every unit read");
  uint32_t u[4 * kV];
#pragma unroll
  for (int v = 0; v < kV; ++v) {
    const uint4 q = *reinterpret_cast<const uint4 *>(row + 16 * v);
    u[4 * v] = q.x, u[4 * v + 1] = q.y, u[4 * v + 2] = q.z, u[4 * v + 3] = q.w;
  }
  // shift down by o4 units: by one unit, then by two
  uint32_t s1[kU + 2];
#pragma unroll
  for (int i = 0; i < kU + 2; ++i) s1[i] = (o4 & 1) ? u[i + 1] : u[i];
  const int nu = nw * static_cast<int>(sizeof(W)) / 4;
#pragma unroll
  for (int i = 0; i < kU; ++i) {
    uint32_t x = (o4 & 2) ? s1[i + 2] : s1[i];
    if (i >= nu) x = 0u;
    if constexpr (sizeof(W) == 4)
      cur[i] = x;
    else if (i & 1)
      cur[i / 2] |= static_cast<W>(x) << 32;
    else
      cur[i / 2] = x;
  }
}

// Gathers one output pixel's operand chunks (implicit im2col): chunk (j, r, q)
// is channel chunk j, the words [j WC, min((j + 1) WC, wpr)), of the input
// pixel under tap (r, q); taps outside the image are zero-filled (source size
// 0). The position of the chunk is kept by counters that advance one chunk at
// a time, in the order of the reduction: taps inside channel chunks (windows)
// or channel chunks inside taps (whole 16-byte vectors).
template <typename W, int WC>
struct AGather {
  const W *act;
  int H, W_, wpr, R, S, nck;
  bool win;
  bool row_valid;
  int ih0, iw0, pix0;    // input pixel under tap (0, 0) of this thread's output pixel
  int j = 0, r = 0, q = 0;

  // Next chunk; true after the output tile's last one.
  __device__ __forceinline__ bool advance() {
    if (!win) {
      if (++j < nck) return false;
      j = 0;
    }
    if (++q < S) return false;
    q = 0;
    if (++r < R) return false;
    r = 0;
    if (!win) return true;
    if (++j < nck) return false;
    j = 0;
    return true;
  }

  __device__ __forceinline__ const W *chunk(bool &valid) const {
    valid = row_valid && static_cast<unsigned>(ih0 + r) < static_cast<unsigned>(H) &&
            static_cast<unsigned>(iw0 + q) < static_cast<unsigned>(W_);
    return act + (static_cast<long long>(pix0 + r * W_ + q) * wpr + j * WC);
  }

  // A chunk that is a whole number of aligned 16-byte vectors.
  __device__ __forceinline__ void issue(uint32_t dst) const {
    bool valid;
    const W *src = chunk(valid);
    stage_chunk<W, WC>(dst, reinterpret_cast<const char *>(valid ? src : act), valid ? 1u : 0u);
  }

  // Any other chunk is copied as the 16-byte pieces of the aligned window
  // around it, so that every copy is 16 bytes wide whatever the pixel's
  // alignment. Pieces past the chunk are zero-filled; a piece that reaches
  // past the end of the activation tensor (act_end) copies only the bytes
  // before it. Returns the chunk's offset into the staged row in 32-bit units
  // (load_window). act is 16-byte aligned.
  __device__ __forceinline__ int issue_win(uint32_t dst, uintptr_t act_end) const {
    const int nw = wpr - j * WC < WC ? wpr - j * WC : WC;
    bool valid;
    const W *px = chunk(valid);
    const uintptr_t a = valid ? reinterpret_cast<uintptr_t>(px) : reinterpret_cast<uintptr_t>(act);
    const uintptr_t a0 = a & ~static_cast<uintptr_t>(15);
    const uintptr_t end = a + static_cast<uintptr_t>(nw) * sizeof(W);
#pragma unroll
    for (int v = 0; v < kWinPieces<W, WC>; ++v) {
      const uintptr_t pa = a0 + 16u * v;
      uint32_t n = 0;
      if (valid && pa < end) n = act_end - pa < 16 ? static_cast<uint32_t>(act_end - pa) : 16u;
      ptx::cp_async_16(dst + 16 * v, n ? reinterpret_cast<const void *>(pa) : static_cast<const void *>(act), n);
    }
    return static_cast<int>((a - a0) >> 2);
  }
};

// Packs 32 requantized lane patterns (zero past `cnt`) into 32 / LO words of
// LO lanes each and stores them; LO divides 32, so every word of the
// 32-channel group is whole.
template <int LO, typename WO>
__device__ __forceinline__ void pack_regs(const uint32_t (&y)[32], int lane_w, int cnt, WO *dst) {
  constexpr int NW = 32 / LO;  // words of this 32-channel group
  WO w[NW];
#pragma unroll
  for (int k = 0; k < NW; ++k) {
    w[k] = 0;
#pragma unroll
    for (int l = 0; l < LO; ++l) w[k] |= static_cast<WO>(y[k * LO + l]) << (l * lane_w);
  }
  constexpr int kWordBytes = static_cast<int>(sizeof(WO));
  if (cnt == 32 && (NW * kWordBytes) % 16 == 0 && (reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
#pragma unroll
    for (int v = 0; v < NW * kWordBytes / 16; ++v) {
      uint4 q;
      memcpy(&q, reinterpret_cast<const uint8_t *>(w) + 16 * v, 16);
      reinterpret_cast<uint4 *>(dst)[v] = q;
    }
  } else {
#pragma unroll
    for (int k = 0; k < NW; ++k)
      if (k * LO < cnt) dst[k] = w[k];
  }
}

constexpr int32_t kMagicBits = 0x4B400000;  // encoding of 1.5 * 2^23

// floor(acc * scale) + 1.5 * 2^23 as the encoding of a float: with rounding
// toward minus infinity the fma result, which lies in [2^23, 2^24) where the
// unit in the last place is 1, is exactly floor(acc * scale) + 1.5 * 2^23
// while |acc * scale| < 2^22 (scale = 2^-shift makes acc * scale exact).
// The encoding is then kMagicBits + floor(acc * scale), monotonic in it.
__device__ __forceinline__ int32_t floor_scaled_biased(float acc, float scale) {
  float r;
  asm("fma.rm.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(acc), "f"(scale), "f"(12582912.0f));
  return __float_as_int(r);
}

// Packs lane patterns into words of L lanes one channel at a time (any L):
// the running word `cur` receives lane nl at bit sh and is stored when full.
template <typename WO>
struct RowPacker {
  WO *dst;
  WO cur = 0;
  int nl = 0, sh = 0;
  __device__ __forceinline__ void put(uint32_t y, int L, int lw) {
    cur |= static_cast<WO>(y) << sh;
    sh += lw;
    if (++nl == L) {
      *dst++ = cur;
      cur = 0;
      sh = 0;
      nl = 0;
    }
  }
  __device__ __forceinline__ void flush() {
    if (nl) *dst = cur;
  }
};

// One requantized lane as an offset pattern: clamp_fo(floor(acc / 2^shift))
// plus half the range of a signed format (0 for an unsigned one), by one fma
// and one add-clamp: `addend` takes the fma's bias off and adds the offset,
// min with the largest pattern, relu for the smallest. Flipping the top bits
// of a word's signed lanes then gives their two's complement.
__device__ __forceinline__ uint32_t requant_lane(uint32_t acc, float scale, int32_t addend, int32_t omax) {
  return static_cast<uint32_t>(__viaddmin_s32_relu(floor_scaled_biased(__uint_as_float(acc), scale), addend, omax));
}
__device__ __forceinline__ constexpr int32_t requant_addend(int bits, bool is_signed) {
  return (is_signed ? 1 << (bits - 1) : 0) - kMagicBits;
}

// Requantizes columns FIRST .. FIRST + 15 of a 32-column group into the
// group's words of 32 / OB offset patterns.
template <int OB, bool OS, int FIRST, int NH>
__device__ __forceinline__ void pack_16(const uint32_t (&r)[16], uint32_t (&h)[NH], float scale) {
  constexpr int LH = 32 / OB;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int c = FIRST + k;
    const uint32_t v = requant_lane(r[k], scale, requant_addend(OB, OS), (1 << OB) - 1) << ((c % LH) * OB);
    h[c / LH] = c % LH == 0 ? v : h[c / LH] + v;
  }
}

// What the epilogue of a row works on: rows are output pixels (m; ~0 for a
// row outside the output, which only skips the stores), nvalid the channels
// of this block from ch0 on. The first, store-free pass asks for one column
// group only (warm).
struct EpiRow {
  uint32_t taddr;   // TMEM address of the warp's rows, first column
  uint32_t m;
  int ch0, nvalid;
  __device__ __forceinline__ bool valid() const { return m != ~0u; }
};
__device__ __forceinline__ EpiRow epi_row(const ConvArgs &args, uint32_t taddr, uint32_t m, int nb, bool warm) {
  EpiRow e{taddr, m, nb * args.NBc, 0};
  e.nvalid = args.K - e.ch0 < args.NBc ? args.K - e.ch0 : args.NBc;
  if (warm) {
    e.m = ~0u;
    e.nvalid = 1;
  }
  return e;
}

// Epilogue of one accumulator row of a channel block: fp32 accumulators ->
// exact integers -> optional int32 store, optional requantize-and-pack.
// Called by whole warps. tcgen05.ld is collective, and lanes make or skip
// their stores by their own row: a __syncwarp before the next load converges
// the warp (nothing else would guarantee it), or, in the loops that it would
// slow down (epilogue_row_words: ResNet-50 56x56 block 123 -> 128 us;
// epilogue_row_acc), the stores are predicated and the warp never branches
// apart.
//
// Formats with spacers or 64-bit words of 3, 5, 6 or 7 bits: packed output
// only, no split digits, |acc| / 2^shift < 2^22.
template <typename WO>
__device__ __forceinline__ void epilogue_row_fast(const ConvArgs &args, const EpiRow &e) {
  const int32_t addend = requant_addend(args.out_bits, args.out_signed != 0), omax = (1 << args.out_bits) - 1;
  const uint32_t flip = args.out_signed ? 1u << (args.out_bits - 1) : 0u;
  const float scale = args.out_scale;
  const int L = args.out_L, lw = args.out_lane_w;
  RowPacker<WO> pk;
  WO *const row = static_cast<WO *>(args.packed_out) + (static_cast<long long>(e.m) * args.out_wpr + e.ch0 / L);
  pk.dst = row;
  for (int col = 0; col < e.nvalid; col += 32) {
    __syncwarp();
    // the block's MMA columns are a multiple of 16; past them, which may be
    // past this CTA's tensor memory, the first ones are read again
    uint32_t y[32];
    ptx::tmem_ld_32x32b_x16(e.taddr + col, y);
    ptx::tmem_ld_32x32b_x16(e.taddr + (col + 16 < args.n_mma ? col + 16 : 0), y + 16);
    ptx::tmem_wait_ld(y);
    const int cnt = e.nvalid - col < 32 ? e.nvalid - col : 32;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      y[k] = requant_lane(y[k], scale, addend, omax) ^ flip;
      if (k >= cnt) y[k] = 0u;
    }
    if (!e.valid()) continue;
    if (args.out_fast) {  // L divides 32: whole words per 32-channel group
      WO *dst = row + col / L;
      switch (args.out_fast) {
        case 4:
          if constexpr (sizeof(WO) == 4) pack_regs<4>(y, lw, cnt, dst);
          break;
        case 8: pack_regs<8>(y, lw, cnt, dst); break;
        case 16: pack_regs<16>(y, lw, cnt, dst); break;
        default: pack_regs<32>(y, lw, cnt, dst); break;
      }
    } else {
#pragma unroll
      for (int k = 0; k < 32; ++k)
        if (k < cnt) pk.put(y[k], L, lw);
    }
  }
  if (!args.out_fast && e.valid()) pk.flush();
}

// The fast epilogue for output lanes of OB = 1, 2, 4, 7 or 8 bits without
// spacers (7 only in 32-bit words): the words of a 32-channel group are built
// 32 bits at a time (for OB dividing 32 a 64-bit word is its two 32-bit
// halves, low half first, so the bytes are the same) with compile-time
// shifts: three operations a lane.
template <int OB, bool OS>
__device__ __forceinline__ void epilogue_row_spec(const ConvArgs &args, const EpiRow &e) {
  constexpr int LH = 32 / OB;  // lanes per 32-bit half-word (a divisor of 32: OB = 1, 2, 4, 7, 8)
  constexpr int NH = 32 / LH;  // half-words per 32-channel group
  static_assert(32 % LH == 0, "whole half-words per 32-channel group");
  constexpr uint32_t flip = OS ? LaneMsb<uint32_t, OB>::kValue : 0u;
  const float scale = args.out_scale;
  // 32-bit half-words of this row: output channel c sits in half-word c / LH
  uint32_t *row32 = reinterpret_cast<uint32_t *>(static_cast<uint8_t *>(args.packed_out) +
                                                 static_cast<size_t>(e.m) * args.out_wpr * (args.out_word64 ? 8 : 4)) +
                    e.ch0 / LH;
  // 4-bit lanes: two 32-channel groups make one 32-byte store (a warp's
  // 32-byte rows then cover whole 128-byte lines, in the L1 data path the
  // MMAs' operand reads share)
  const bool pair32 = NH == 4 && e.nvalid % 64 == 0 && (reinterpret_cast<uintptr_t>(row32) & 31) == 0;
  uint32_t p0 = 0, p1 = 0, p2 = 0, p3 = 0;
  // 16 columns are packed while the next 16 are on their way (the block's MMA
  // columns are a multiple of 16; past them the first ones are read again)
  uint32_t ra[16], rb[16];
  auto load = [&](int col, uint32_t (&r)[16]) {
    ptx::tmem_ld_32x32b_x16(e.taddr + (col < args.n_mma ? col : 0), r);
  };
  __syncwarp();
  load(0, ra);
  ptx::tmem_wait_ld(ra);
  for (int col = 0; col < e.nvalid; col += 32) {
    __syncwarp();
    const int cnt = e.nvalid - col < 32 ? e.nvalid - col : 32;
    uint32_t h[NH];
    load(col + 16, rb);
    pack_16<OB, OS, 0>(ra, h, scale);
    ptx::tmem_wait_ld(rb);
    load(col + 32, ra);
    pack_16<OB, OS, 16>(rb, h, scale);
#pragma unroll
    for (int j = 0; j < NH; ++j) h[j] ^= flip;
    ptx::tmem_wait_ld(ra);
    if constexpr (NH == 4) {
      if (pair32) {
        if ((col & 32) == 0) {
          p0 = h[0], p1 = h[1], p2 = h[2], p3 = h[3];
        } else if (e.valid()) {
          ptx::st_global_v8(row32 + (col - 32) / LH, p0, p1, p2, p3, h[0], h[1], h[2], h[3]);
        }
        continue;
      }
    }
    if (!e.valid()) continue;
    uint32_t *dst = row32 + col / LH;
    if (cnt < 32) {  // the last group of a channel count that is not a multiple of 32
#pragma unroll
      for (int j = 0; j < NH; ++j) {
        const int c0 = j * LH;  // first channel of half-word j
        if (c0 < cnt) {
          const int nl = cnt - c0 < LH ? cnt - c0 : LH;
          dst[j] = nl == LH ? h[j] : (h[j] & ((1u << (nl * OB)) - 1));
        }
      }
    } else if constexpr (NH == 8) {
      if ((reinterpret_cast<uintptr_t>(dst) & 31) == 0) {
        // one 32-byte store per row: with 32-byte rows a warp writes whole lines
        ptx::st_global_v8(dst, h[0], h[1], h[2], h[3], h[4], h[5], h[6], h[7]);
      } else if ((reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
        reinterpret_cast<uint4 *>(dst)[0] = make_uint4(h[0], h[1], h[2], h[3]);
        reinterpret_cast<uint4 *>(dst)[1] = make_uint4(h[4], h[5], h[6], h[7]);
      } else {
#pragma unroll
        for (int j = 0; j < NH; ++j) dst[j] = h[j];
      }
    } else if constexpr (NH % 4 == 0) {
      if ((reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
#pragma unroll
        for (int v = 0; v < NH / 4; ++v)
          reinterpret_cast<uint4 *>(dst)[v] = make_uint4(h[4 * v], h[4 * v + 1], h[4 * v + 2], h[4 * v + 3]);
      } else {
#pragma unroll
        for (int j = 0; j < NH; ++j) dst[j] = h[j];
      }
    } else if constexpr (NH == 2) {
      if ((reinterpret_cast<uintptr_t>(dst) & 7) == 0)
        *reinterpret_cast<uint2 *>(dst) = make_uint2(h[0], h[1]);
      else
        dst[0] = h[0], dst[1] = h[1];
    } else {
      dst[0] = h[0];
    }
  }
  // a last 64-bit word of which only the low half-word holds channels
  const int nhalf = (e.nvalid + LH - 1) / LH;
  if (args.out_word64 && (nhalf & 1) && e.valid()) row32[nhalf] = 0u;
}

// The fast epilogue for 32-bit output words whose L = 32 / OB lanes do not
// divide 32 (OB = 3, 5, 6: L = 10, 6, 5): two or four words (20 or 24 columns)
// at a time, the next ones' columns on their way meanwhile, loaded in pieces that never reach past the block's MMA columns.
// The loop's body is small on purpose: unrolled over the 160 or 96 columns
// after which word boundaries repeat on a 32-column grid, the two or so warps
// of a scheduler spent most of their time fetching it (2700 instructions a
// row of 256 6-bit channels at 0.2 a cycle).
//
// Rows leave in one of three ways. Flat (e_flat: one channel block): the
// warp's valid rows are consecutive output pixels, so their words are one
// contiguous run; they are staged side by side and copied with 16-byte
// accesses. By rows (e_stage): 32 words of each row are staged at a time and
// written row by row. Else each thread stores its own row's words.
template <int OB, bool OS>
__device__ __forceinline__ void epilogue_row_words(const ConvArgs &args, const EpiRow &e, uint32_t *stg) {
  constexpr int L = 32 / OB;
  constexpr int kWords = L == 10 ? 2 : 4;      // words of a group
  constexpr int kCols = kWords * L;            // 20 or 24 columns
  constexpr int kPiece = L == 6 ? 8 : 4;       // columns of one TMEM load; divides 16, as the block's MMA columns are
  constexpr int32_t addend = requant_addend(OB, OS), omax = (1 << OB) - 1;
  constexpr uint32_t flip = OS ? LaneMsb<uint32_t, OB>::kValue : 0u;
  static_assert(kCols % kPiece == 0, "whole pieces");
  const int lane = threadIdx.x & 31;
  const float scale = args.out_scale;
  const int nwords = (e.nvalid + L - 1) / L;
  const int last_lanes = e.nvalid - (nwords - 1) * L;
  const uint32_t last_mask = (1u << (last_lanes * OB)) - 1;  // L * OB <= 30 bits
  uint32_t *const out = static_cast<uint32_t *>(args.packed_out);
  uint32_t *const own = out + (static_cast<size_t>(e.m) * args.out_wpr + e.ch0 / L);
  const unsigned vmask = __ballot_sync(0xffffffffu, e.valid());
  const bool flat = args.e_flat != 0, by_rows = args.e_stage != 0;
  uint32_t *const mine = flat ? stg + __popc(vmask & ((1u << lane) - 1)) * nwords : stg + lane * kEpiPitch;
  auto load = [&](int c0, uint32_t (&r)[kCols]) {
    if (c0 + kCols <= args.n_mma) {  // a whole group: two loads (each takes the warp about 27 cycles)
      ptx::tmem_ld_32x32b_x16(e.taddr + c0, r);
      if constexpr (kCols == 20)
        ptx::tmem_ld_32x32b_x4(e.taddr + c0 + 16, r + 16);
      else
        ptx::tmem_ld_32x32b_x8(e.taddr + c0 + 16, r + 16);
      return;
    }
#pragma unroll
    for (int q = 0; q < kCols; q += kPiece) {
      const int col = c0 + q < args.n_mma ? c0 + q : 0;  // past the last column: any, not stored
      if constexpr (kPiece == 4)
        ptx::tmem_ld_32x32b_x4(e.taddr + col, r + q);
      else
        ptx::tmem_ld_32x32b_x8(e.taddr + col, r + q);
    }
  };
  // rows of a multiple of four words are staged 16 bytes at a time (13 such
  // pieces a row of 256 6-bit channels: an odd number, so no bank conflicts)
  const bool vec4 = kWords == 4 && flat && (nwords & 3) == 0;
  uint32_t *const to = flat ? mine : own;
  auto group = [&](int c0, int w0, const uint32_t (&r)[kCols]) {
    uint32_t w[kWords];
#pragma unroll
    for (int j = 0; j < kWords; ++j) {
      w[j] = 0;
#pragma unroll
      for (int l = 0; l < L; ++l) w[j] += requant_lane(r[j * L + l], scale, addend, omax) << (l * OB);
      w[j] ^= flip;
      if (w0 + j == nwords - 1) w[j] &= last_mask;  // the row's last, partial word
    }
    if (by_rows) {
#pragma unroll
      for (int j = 0; j < kWords; ++j) mine[(w0 + j) & 31] = w[j];
    } else if (vec4) {
      if constexpr (kWords == 4) ptx::st_v4_if(e.valid(), to + w0, w[0], w[1], w[2], w[3]);
    } else {
#pragma unroll
      for (int j = 0; j < kWords; ++j) ptx::st_if(e.valid() && w0 + j < nwords, to + w0 + j, w[j]);
    }
    if (by_rows && (((w0 + kWords) & 31) == 0 || c0 + kCols >= e.nvalid)) {
      __syncwarp();
      const int wb = w0 & ~31;  // first word of this flush
      const bool has = wb + lane < nwords;
#pragma unroll 4
      for (int rr = 0; rr < 32; ++rr) {
        const uint32_t mr = __shfl_sync(0xffffffffu, e.m, rr);
        if (has && mr != ~0u)
          out[static_cast<size_t>(mr) * args.out_wpr + e.ch0 / L + wb + lane] = stg[rr * kEpiPitch + lane];
      }
      __syncwarp();
    }
  };
  // the next group's columns are on their way while one is packed
  uint32_t ra[kCols], rb[kCols];
  load(0, ra);
  ptx::tmem_wait_ld(ra);
  for (int c0 = 0, w0 = 0; c0 < e.nvalid; c0 += 2 * kCols, w0 += 2 * kWords) {
    load(c0 + kCols, rb);
    group(c0, w0, ra);
    ptx::tmem_wait_ld(rb);
    if (c0 + kCols >= e.nvalid) break;
    load(c0 + 2 * kCols, ra);
    group(c0 + kCols, w0 + kWords, rb);
    ptx::tmem_wait_ld(ra);
  }
  if (flat && vmask != 0u) {
    __syncwarp();
    const uint32_t m0 = __shfl_sync(0xffffffffu, e.m, __ffs(vmask) - 1);
    uint32_t *const dst = out + static_cast<size_t>(m0) * args.out_wpr;
    const int total = __popc(vmask) * nwords;
    int i = 0;
    if ((reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
      i = total & ~3;
#pragma unroll 4
      for (int k = 4 * lane; k < i; k += 128)
        *reinterpret_cast<uint4 *>(dst + k) = *reinterpret_cast<const uint4 *>(stg + k);
    }
    for (int k = i + lane; k < total; k += 32) dst[k] = stg[k];
    __syncwarp();
  }
}

// The exact integers of 16 accumulator columns (split digits: 16 hi + lo).
__device__ __forceinline__ void exact_16(const ConvArgs &args, uint32_t taddr, int (&v)[16]) {
  uint32_t r[16];
  ptx::tmem_ld_32x32b_x16(taddr, r);
  ptx::tmem_wait_ld(r);
  if (args.split) {
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = 16 * __float2int_rn(__uint_as_float(r[k]) * args.acc_scale);
    ptx::tmem_ld_32x32b_x16(taddr + args.n_mma, r);
    ptx::tmem_wait_ld(r);
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] += __float2int_rn(__uint_as_float(r[k]) * args.acc_scale);
  } else if (args.fast_acc) {  // |acc| < 2^22: the exact integer from the float's encoding
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = floor_scaled_biased(__uint_as_float(r[k]), args.acc_scale) - kMagicBits;
  } else {
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = __float2int_rn(__uint_as_float(r[k]) * args.acc_scale);
  }
}

// int32 outputs: whole sectors of a thread's own row where rows are whole
// sectors; otherwise 32 columns of the warp's rows are staged (acc_stage) and
// written row by row, 32 consecutive words a store, or, without room for
// that, one word at a time. (So do the later channel blocks of whole-sector
// rows beside 3- and 6-bit packed ones: their first channel is a multiple of
// 10 or 5, and the stage is planned by K alone.) 29 x 51 x 140 positions of 262 channels (217 MB),
// with 3-bit packed rows: 451 us one word at a time, 242 this way.
__device__ __forceinline__ void epilogue_row_acc(const ConvArgs &args, const EpiRow &e, uint32_t *stg) {
  const bool vec_ok = args.K % 4 == 0 && e.ch0 % 4 == 0;
  const bool vec8_ok = args.K % 8 == 0 && e.ch0 % 8 == 0 && (reinterpret_cast<uintptr_t>(args.acc_out) & 31) == 0;
  const int lane = threadIdx.x & 31;
  uint32_t *const row = reinterpret_cast<uint32_t *>(args.acc_out) + (static_cast<size_t>(e.m) * args.K + e.ch0);
  for (int col = 0; col < e.nvalid; col += 16) {
    int v[16];
    exact_16(args, e.taddr + col, v);
    const int cnt = e.nvalid - col < 16 ? e.nvalid - col : 16;
    if (args.acc_stage) {
#pragma unroll
      for (int k = 0; k < 16; ++k) stg[lane * kEpiPitch + (col & 16) + k] = static_cast<uint32_t>(v[k]);
      if ((col & 16) == 0 && col + 16 < e.nvalid) continue;
      __syncwarp();
      const int c = (col & ~31) + lane;
      const bool has = c < e.nvalid;
#pragma unroll 4
      for (int rr = 0; rr < 32; ++rr) {
        const uint32_t mr = __shfl_sync(0xffffffffu, e.m, rr);
        if (has && mr != ~0u)
          args.acc_out[static_cast<size_t>(mr) * args.K + e.ch0 + c] = static_cast<int32_t>(stg[rr * kEpiPitch + lane]);
      }
      __syncwarp();
      continue;
    }
    uint32_t *dst = row + col;
    if (cnt == 16 && vec8_ok) {
#pragma unroll
      for (int k = 0; k < 16; k += 8)
        ptx::st_global_v8_if(e.valid(), dst + k, v[k], v[k + 1], v[k + 2], v[k + 3], v[k + 4], v[k + 5], v[k + 6], v[k + 7]);
    } else if (cnt == 16 && vec_ok) {
#pragma unroll
      for (int k = 0; k < 16; k += 4) ptx::st_v4_if(e.valid(), dst + k, v[k], v[k + 1], v[k + 2], v[k + 3]);
    } else {
#pragma unroll
      for (int k = 0; k < 16; ++k) ptx::st_if(e.valid() && k < cnt, dst + k, v[k]);
    }
  }
}

// Packed rows that the fast forms do not take (split digits, |acc| / 2^shift
// of 2^22 and more), 16 columns at a time.
template <typename WO>
__device__ __forceinline__ void epilogue_row_general(const ConvArgs &args, const EpiRow &e) {
  const int lo = lane_lo(args.out_bits, args.out_signed), hi = lane_hi(args.out_bits, args.out_signed);
  const uint32_t omask = (1u << args.out_bits) - 1;
  const int L = args.out_L, lw = args.out_lane_w;
  RowPacker<WO> pk;
  pk.dst = static_cast<WO *>(args.packed_out) + (static_cast<long long>(e.m) * args.out_wpr + e.ch0 / L);
  for (int col = 0; col < e.nvalid; col += 16) {
    int v[16];
    __syncwarp();
    exact_16(args, e.taddr + col, v);
    if (!e.valid()) continue;
    const int cnt = e.nvalid - col < 16 ? e.nvalid - col : 16;
#pragma unroll
    for (int k = 0; k < 16; ++k)
      if (k < cnt) pk.put(static_cast<uint32_t>(clamp_int(v[k] >> args.shift, lo, hi)) & omask, L, lw);
  }
  if (e.valid()) pk.flush();
}

// NCHW outputs: the 32 rows of a warp are neighbouring pixels, so for one
// channel their int32 sums, or their requantized bytes, are neighbours in
// memory and each store covers whole sectors.
__device__ __forceinline__ void epilogue_row_nchw(const ConvArgs &args, const EpiRow &e) {
  const int lo = lane_lo(args.out_bits, args.out_signed), hi = lane_hi(args.out_bits, args.out_signed);
  const uint32_t omask = (1u << args.out_bits) - 1;
  const uint32_t howo = args.fd_howo.d;
  const uint32_t img = e.valid() ? fdiv(e.m, args.fd_howo) : 0u;
  const size_t base = (static_cast<size_t>(img) * args.K + e.ch0) * howo + (e.m - img * howo);
  for (int col = 0; col < e.nvalid; col += 16) {
    int v[16];
    __syncwarp();
    exact_16(args, e.taddr + col, v);
    if (!e.valid()) continue;
    const int cnt = e.nvalid - col < 16 ? e.nvalid - col : 16;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      if (k >= cnt) break;
      const size_t at = base + static_cast<size_t>(col + k) * howo;
      if (args.acc_out) args.acc_out[at] = v[k];
      if (args.q8_out) args.q8_out[at] = static_cast<uint8_t>(static_cast<uint32_t>(clamp_int(v[k] >> args.shift, lo, hi)) & omask);
    }
  }
}

__device__ __forceinline__ void epilogue_row(const ConvArgs &args, const EpiRow &e, uint32_t *estage) {
  __syncwarp();  // the stores of the part before
  if (args.nchw) {
    epilogue_row_nchw(args, e);
    return;
  }
  // int32 sums and packed rows are two passes over the accumulator (reading it
  // again costs less than packing by the general form)
  if (args.acc_out) epilogue_row_acc(args, e, estage);
  if (!args.packed_out) return;
  const bool fast = !args.split && args.fast_req;
  if (fast && args.out_lane_w == args.out_bits && (!args.out_word64 || (args.out_bits & (args.out_bits - 1)) == 0)) {
    switch (args.out_bits * 2 + (args.out_signed ? 1 : 0)) {
      case 2: epilogue_row_spec<1, false>(args, e); return;
      case 3: epilogue_row_spec<1, true>(args, e); return;
      case 4: epilogue_row_spec<2, false>(args, e); return;
      case 5: epilogue_row_spec<2, true>(args, e); return;
      case 6: epilogue_row_words<3, false>(args, e, estage); return;
      case 7: epilogue_row_words<3, true>(args, e, estage); return;
      case 8: epilogue_row_spec<4, false>(args, e); return;
      case 9: epilogue_row_spec<4, true>(args, e); return;
      case 10: epilogue_row_words<5, false>(args, e, estage); return;
      case 11: epilogue_row_words<5, true>(args, e, estage); return;
      case 12: epilogue_row_words<6, false>(args, e, estage); return;
      case 13: epilogue_row_words<6, true>(args, e, estage); return;
      case 14: epilogue_row_spec<7, false>(args, e); return;
      case 15: epilogue_row_spec<7, true>(args, e); return;
      case 16: epilogue_row_spec<8, false>(args, e); return;
      case 17: epilogue_row_spec<8, true>(args, e); return;
      default: break;
    }
  }
  if (args.out_word64) {
    if (fast)
      epilogue_row_fast<uint64_t>(args, e);
    else
      epilogue_row_general<uint64_t>(args, e);
  } else {
    if (fast)
      epilogue_row_fast<uint32_t>(args, e);
    else
      epilogue_row_general<uint32_t>(args, e);
  }
}

// A role's wait on one of the kernel's barriers. A role whose wait gives up
// (false) stops: the loader at once, the others at the end of their tile or a
// few items, filling and releasing every stage in step until there (with
// undefined values). The others' waits then give up in turn, within one poll
// of the failure's being recorded, and the kernel ends with what was in flight
// drained.
__device__ __forceinline__ bool role_wait(uint32_t bar, uint32_t parity, int *status, uint64_t limit_ns = kWaitLimitNs) {
  return ptx::mbar_wait(bar, parity, status, static_cast<int>(SAMD_ETIMEOUT), limit_ns);
}

// The same by a whole warp, every lane polling for itself: one answer for all,
// and the warp is converged again behind it (the collective tcgen05.ld needs
// that).
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, int *status, uint64_t limit_ns = kWaitLimitNs) {
  return __all_sync(0xffffffffu, role_wait(bar, parity, status, limit_ns));
}

// The epilogue warps' meeting point of a pooled tile: every warp of the
// tile's group arrives on `bar` once its part of the step is done, then
// waits, bounded, for the phase. (One that gives up goes on to the end of its
// tile: what it reads and writes there is in bounds, and undefined.)
__device__ __forceinline__ void epi_group_sync(uint32_t bar, uint32_t &phase, int *status) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) ptx::mbar_arrive(bar);
  (void)warp_wait(bar, phase & 1u, status);
  ++phase;
}

// Epilogue of one pooled tile for output lanes of OB = 1, 2, 4 or 8 bits
// (32-bit words, no spacers), called by each warp of the tile's group of
// gw warps (gi = this warp's index in it) for its 32 rows:
// requantize and pack the row (tile row trow) into the pool buffer, free the
// accumulator, meet the other epilogue warps, then write the lane-wise max of
// every 2x2 window of the tile's row pairs (the maximum commutes with the
// monotone requantize, so this is the pool of the requantized output), and
// meet again before the buffer is reused.
template <int OB, bool OS>
__device__ __noinline__ void epilogue_pool_tile(const ConvArgs &args, uint32_t taddr, int trow, uint32_t mt, int nb,
                                                uint32_t *pbuf, uint32_t acc_empty, uint32_t group_bar,
                                                uint32_t &phase, int *status, int gw, int gi) {
  constexpr int LH = 32 / OB;  // lanes per word
  constexpr int NH = 32 / LH;  // words per 32 channels
  constexpr uint32_t flip = OS ? LaneMsb<uint32_t, OB>::kValue : 0u;
  const int ch0 = nb * args.NBc;
  const int nvalid = args.K - ch0 < args.NBc ? args.K - ch0 : args.NBc;
  const int nw = (nvalid + LH - 1) / LH;  // this block's words of a row (<= pool_nw; fewer in a last, partial block)
  const int pitch = args.pool_pitch;
  const float scale = args.out_scale;
  uint32_t *prow = pbuf + trow * pitch;
  // 16 columns are packed while the next 16 are on their way
  uint32_t ra[16], rb[16];
  auto load = [&](int col, uint32_t (&r)[16]) {
    ptx::tmem_ld_32x32b_x16(taddr + (col < args.n_mma ? col : 0), r);
  };
  load(0, ra);
  ptx::tmem_wait_ld(ra);
  for (int col = 0; col < nvalid; col += 32) {
    const int cnt = nvalid - col < 32 ? nvalid - col : 32;
    uint32_t h[NH];
    load(col + 16, rb);
    pack_16<OB, OS, 0>(ra, h, scale);
    ptx::tmem_wait_ld(rb);
    load(col + 32, ra);
    pack_16<OB, OS, 16>(rb, h, scale);
#pragma unroll
    for (int j = 0; j < NH; ++j) {
      uint32_t w = h[j] ^ flip;
      const int wi = col / LH + j;
      // lanes past the block's channels are zero
      const int nl = cnt - j * LH;
      if (nl < LH) w &= nl > 0 ? (1u << (nl * OB)) - 1 : 0u;
      if (wi < nw) prow[wi] = w;
    }
    ptx::tmem_wait_ld(ra);
  }
  ptx::tc_fence_before();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) ptx::mbar_arrive(acc_empty);
  epi_group_sync(group_bar, phase, status);
  // the 2x2 windows of this tile's row pairs
  const uint32_t img = fdiv(mt, args.fd_tpi);
  const int g = static_cast<int>(mt - img * args.fd_tpi.d);
  const int Ho2 = args.Ho / 2, Wo2 = args.Wo / 2, q = args.pool_rows / 2;
  const int q_here = Ho2 - g * q < q ? Ho2 - g * q : q;
  const int total = q_here * Wo2 * args.pool_nw;
  uint32_t *out = static_cast<uint32_t *>(args.packed_out) + ch0 / LH;
  const int Wp = args.Wp;
#pragma unroll 2
  for (int idx = 32 * gi + static_cast<int>(threadIdx.x & 31); idx < total; idx += 32 * gw) {
    const int pix = static_cast<int>(fdiv(static_cast<uint32_t>(idx), args.fd_pnw)), w = idx - pix * args.pool_nw;
    if (w >= nw) continue;  // a last block of fewer words
    const int i = static_cast<int>(fdiv(static_cast<uint32_t>(pix), args.fd_wo2)), j = pix - i * Wo2;
    const uint32_t *b0 = pbuf + (2 * i * Wp + 2 * j) * pitch + w;
    const uint32_t top = swar_lane_max<uint32_t, OB>(b0[0], b0[pitch], flip);
    const uint32_t bot = swar_lane_max<uint32_t, OB>(b0[Wp * pitch], b0[(Wp + 1) * pitch], flip);
    const long long orow = (static_cast<long long>(img) * Ho2 + g * q + i) * Wo2 + j;
    out[orow * args.out_wpr + w] = swar_lane_max<uint32_t, OB>(top, bot, flip);
  }
  epi_group_sync(group_bar, phase, status);
}

__device__ __forceinline__ void epilogue_pool_dispatch(const ConvArgs &args, uint32_t taddr, int trow, uint32_t mt,
                                                       int nb, uint32_t *pbuf, uint32_t acc_empty, uint32_t group_bar,
                                                       uint32_t &phase, int *status, int gw, int gi) {
#define SAMD_POOL_TILE(OB, OS) \
  epilogue_pool_tile<OB, OS>(args, taddr, trow, mt, nb, pbuf, acc_empty, group_bar, phase, status, gw, gi)
  switch (args.out_bits * 2 + (args.out_signed ? 1 : 0)) {
    case 2: SAMD_POOL_TILE(1, false); return;
    case 3: SAMD_POOL_TILE(1, true); return;
    case 4: SAMD_POOL_TILE(2, false); return;
    case 5: SAMD_POOL_TILE(2, true); return;
    case 8: SAMD_POOL_TILE(4, false); return;
    case 9: SAMD_POOL_TILE(4, true); return;
    case 16: SAMD_POOL_TILE(8, false); return;
    default: SAMD_POOL_TILE(8, true); return;
  }
#undef SAMD_POOL_TILE
}

// Issues the MMAs of `n` consecutive taps of a filter row, KS k-steps each
// and one MMA per 128-row part of the tile (HV = 1, 2, 4): part h accumulates
// into d + h * dn from A rows 128 h on (a + h * ah). Tap t reads weight tile
// t (b advances by b_step16) and the A operand one row further on. Descriptors
// advance in 16-byte units of their start-address field. Run by the whole
// warp on uniform values; the leader lane issues.
template <bool FP8, int HV, int KS>
__device__ __forceinline__ void issue_row(uint32_t leader, uint32_t d, uint32_t dn, uint64_t a, uint64_t ah, uint64_t b,
                                          uint32_t idesc, int n, uint32_t a_row16, uint32_t b_step16, uint32_t acc) {
  for (int t = 0; t < n; ++t) {
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
#pragma unroll
      for (int h = 0; h < HV; ++h) {
        const uint32_t accumulate = ks == 0 ? acc : 1u;
        if constexpr (FP8)
          ptx::mma_f8(leader, d + h * dn, a + h * ah + 2 * ks, b + 2 * ks, idesc, accumulate);
        else
          ptx::mma_f16(leader, d + h * dn, a + h * ah + 2 * ks, b + 2 * ks, idesc, accumulate);
      }
    }
    acc = 1;
    a += a_row16;
    b += b_step16;
  }
}

// ---- the persistent convolution kernel ----------------------------------------
//
// One CTA per SM loops over output tiles (tile = blockIdx.x + i * gridDim.x;
// tile = nb * grid_m + mt: channel block nb, position tile mt of 128 * HV
// positions; with HV = 2 or 4 each k-step issues one MMA per 128-row part,
// so the parts share every synchronization). Eighteen warps with fixed
// roles, connected by mbarrier rings:
//   warp 0      TMEM allocation; lane 0 streams weight tiles with TMA. When
//               the layer has one channel block and all its weight tiles fit,
//               they are loaded once and stay resident.
//   warp 1      issues tcgen05.mma (one elected lane) into one of two TMEM
//               accumulators, so tile i+1 accumulates while the epilogue
//               drains tile i.
//   warps 2-9   operand producers.
//               HALO: for each (tile, channel chunk) the halo rows the tile
//               needs are gathered with cp.async and widened once into one of
//               two or three halo buffers; every tap reads the halo through a
//               descriptor shifted by r * row_step + s rows.
//               GATHER: each thread gathers its pixel's packed words (implicit
//               im2col, zero padding) through a cp.async ring and widens them
//               into a ring of A tiles; with HV = 1 two groups of four warps
//               take alternate (tile, chunk) items, with HV = 2 the two groups
//               fill the two halves of every item. Chunks that are not whole
//               16-byte vectors are copied as 16-byte windows.
//   warps 10-17 epilogue: tcgen05.ld, exact integers, optional int32 store,
//               optional requantize-and-pack. HV = 1: warps 10-13 drain
//               accumulator 0 (the CTA's even tiles), warps 14-17
//               accumulator 1; HV = 2: warps 10-13 drain the first half and
//               14-17 the second half of every tile; HV = 4 (halo layers on
//               e4m3 operands): warps 10-13 drain parts 0 and 1, 14-17 parts
//               2 and 3. Warp w reads the TMEM lanes of quadrant w % 4. A
//               first, store-free pass over the first tile fetches the
//               epilogue's code early. Pooled tiles (ConvArgs::pool) are
//               drained, requantized and pooled by the warps of a group.
// Every wait is bounded; a role whose wait gives up records SAMD_ETIMEOUT and
// stops (role_wait).
template <typename W, int BITS, bool SIGNED, bool HALO, bool FP8, bool FULL, int HV>
__global__ void __launch_bounds__(kThreads, 1) conv_kernel(const __grid_constant__ CUtensorMap tmap_b,
                                                           const ConvArgs args) {
  using U = AUnpack<W, BITS, SIGNED, FP8, FULL>;
  constexpr int BMT = BM * HV;  // output positions per tile
  using T = OpTraits<FP8>;
  constexpr int WC = U::WC;
  using St = Staging<W, WC>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));

  const int STB = args.stages;  // weight stages in flight (or resident tiles)
  const bool resident = args.b_resident != 0;
  const uint32_t b_bytes = args.b_bytes;
  uint8_t *sOp = smem;  // HALO: hbufs halo buffers; GATHER: stages_a A tiles
  uint8_t *sB = smem + args.off_b;
  uint8_t *sG = smem + args.off_g;  // packed staging
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + args.off_bar);
  // barriers: full_b[STB] empty_b[STB] opfull[NO] opempty[NO] accfull[2] accempty[2] drain group[2]
  const int NO = HALO ? args.hbufs : args.stages_a;
  uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(bars + 2 * STB + 2 * NO + 7);
  auto full_b = [&](int s) { return ptx::smem_addr(bars + s); };
  auto empty_b = [&](int s) { return ptx::smem_addr(bars + STB + s); };
  auto opfull = [&](int s) { return ptx::smem_addr(bars + 2 * STB + s); };
  auto opempty = [&](int s) { return ptx::smem_addr(bars + 2 * STB + NO + s); };
  auto accfull = [&](int a) { return ptx::smem_addr(bars + 2 * STB + 2 * NO + a); };
  auto accempty = [&](int a) { return ptx::smem_addr(bars + 2 * STB + 2 * NO + 2 + a); };
  const uint32_t drain_bar = ptx::smem_addr(bars + 2 * STB + 2 * NO + 4);
  // the epilogue warps of a pooled tile: all eight (two-half tiles), or the
  // four of epilogue set g (one-half tiles, group_bar(g))
  auto group_bar = [&](int g) { return ptx::smem_addr(bars + 2 * STB + 2 * NO + 5 + g); };

  int *const status = args.status;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // No global read precedes the setup barrier: a failure recorded by an
  // earlier launch is seen by the first wait that has to wait.
  if (warp == 0) {
    ptx::tmem_alloc(ptx::smem_addr(tmem_holder), args.tmem_cols);
    ptx::tmem_relinquish();
  }
  if (threadIdx.x == 32) {
    for (int s = 0; s < STB; ++s) {
      ptx::mbar_init(full_b(s), 1);
      ptx::mbar_init(empty_b(s), 1);
    }
    for (int s = 0; s < NO; ++s) {
      ptx::mbar_init(opfull(s), (HALO || HV == 2) ? kProdWarps : kProdWarps / 2);
      ptx::mbar_init(opempty(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      ptx::mbar_init(accfull(a), 1);
      ptx::mbar_init(accempty(a), HV >= 2 ? kEpiWarps : kEpiWarps / 2);  // the warps that drain accumulator a
    }
    ptx::mbar_init(drain_bar, 1);
    for (int g = 0; g < 2; ++g) ptx::mbar_init(group_bar(g), HV >= 2 ? kEpiWarps : kEpiWarps / 2);
    ptx::fence_barrier_init();
  }
  __syncwarp();  // every warp reaches the barrier converged (bar.sync counts whole warps)
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;

  // fewer than 2^31 tiles, and a CTA's last step stays below 2^31 + gridDim.x (checked on the host)
  const uint32_t total_tiles = static_cast<uint32_t>(args.grid_m) * static_cast<uint32_t>(args.nblocks);
  const uint32_t first_tile = blockIdx.x, tile_step = gridDim.x;
  const int nchunks = args.nchunks;  // weight tiles per output tile

  if (warp == 0) {
    if (lane == 0) {
      // ---- weight tiles ----
      ptx::prefetch_tmap(&tmap_b);
      ptx::grid_dependency_wait();  // the prepared weights
      int quiet = 0;  // the waits below end only when the copies land (or time out)
      if (resident) {
        for (int c = 0; c < nchunks; ++c) {
          ptx::mbar_arrive_expect_tx(full_b(c), b_bytes);
          ptx::tma_load_2d(ptx::smem_addr(sB + c * b_bytes), &tmap_b, c * BK, 0, full_b(c));
        }
        // the CTA does not exit with a copy in flight, whatever the other roles do
        for (int c = 0; c < nchunks; ++c) ptx::mbar_wait_bounded(full_b(c), 0, &quiet, kWaitLimitNs);
      } else {
        // Ring position and round parity advance by increments (a 64-bit
        // division by the runtime ring size costs this thread about as much
        // as the rest of the step).
        int s = 0, loaded = 0;  // loaded: tiles issued so far, counted up to the ring's size
        uint32_t par = 1;       // parity of the previous round's release
        // A stage is armed again when its copies have landed and the MMAs have
        // released it. (Those waited for the copies too, unless that wait gave
        // up; a barrier armed twice in one phase would be lost.)
        bool ok = true;
        for (uint32_t tile = first_tile; ok && tile < total_tiles; tile += tile_step) {
          const int row0 = static_cast<int>(fdiv(tile, args.fd_gm)) * args.mma_n;
          for (int c = 0; c < nchunks; c += args.tgroup) {
            if (loaded == STB) {
              ok = role_wait(full_b(s), par, status) && role_wait(empty_b(s), par, status);
              if (!ok) break;
            } else {
              ++loaded;
            }
            ptx::mbar_arrive_expect_tx(full_b(s), args.tgroup * b_bytes);
            const uint32_t dst = ptx::smem_addr(sB) + s * args.tgroup * b_bytes;
            for (int g = 0; g < args.tgroup; ++g)
              ptx::tma_load_2d(dst + g * b_bytes, &tmap_b, (c + g) * BK, row0, full_b(s));
            if (++s == STB) {
              s = 0;
              par ^= 1;
            }
          }
        }
        // the CTA does not exit with a copy in flight: the ring's last round,
        // oldest first (slots q < s were filled in this round, whose full
        // phase has parity par ^ 1, the others in the round before)
        for (int k = 0; k < loaded; ++k) {
          int q = loaded == STB ? s + k : k;
          if (q >= STB) q -= STB;
          ptx::mbar_wait_bounded(full_b(q), q < s ? par ^ 1u : par, &quiet, kWaitLimitNs / 10);
        }
      }
    }
  } else if (warp == 1) {
    // ---- MMA issue ----
    // The whole warp runs this loop on warp-uniform values; each tcgen05.mma
    // and tcgen05.commit is predicated on one lane (the same one throughout,
    // whose operations a commit tracks). Running the loop in one thread, or
    // the issue behind a branch on that lane, turns every descriptor into a
    // per-thread value that has to be moved to the uniform datapath before
    // each MMA, which costs more than the MMA.
    const uint32_t leader = ptx::elect_one() ? 1u : 0u;
    const uint32_t idesc = ptx::idesc_f16_f32(BM, args.mma_n);
    // A wait that gives up ends the loop behind its tile: an exit at the wait,
    // or a leader that depends on it, costs the loop its uniform registers
    // (sweep step 122 -> 139 us).
    bool gave_up = false;
    auto wait = [&](uint32_t bar, uint32_t parity) {
      if (!role_wait(bar, parity, status)) gave_up = true;
    };
    // Ring positions advance by increments (no division in this loop).
    int sb = 0, so = 0;
    uint32_t bpar = 0, opar = 0;
    const uint32_t sOp_addr = ptx::smem_addr(sOp);
    const int nops = HALO ? args.nck : nchunks;  // operand stages per tile
    // filter rows and taps a row of one operand stage, and how far the A
    // operand moves on behind a row of taps
    const int frows = HALO ? args.R : 1, ftaps = HALO ? args.S : 1;
    const int tgroup = args.tgroup;
    const uint32_t b_step16 = b_bytes >> 4, b_stage16 = static_cast<uint32_t>(tgroup) * b_step16;
    const uint64_t bdesc0 = T::desc(ptx::smem_addr(sB));
    constexpr uint32_t a_row16 = T::kRowBytes / 16;  // one operand row in descriptor units
    constexpr uint64_t a_half16 = static_cast<uint64_t>(BM) * a_row16;  // from one 128-row part's A rows to the next
    const uint32_t dn = static_cast<uint32_t>(args.mma_n);          // the second half's accumulator columns
    const uint32_t a_skip16 = HALO ? static_cast<uint32_t>(args.row_step - args.S) * a_row16 : 0u;
    // The first wait's limit counts from here on, not from the launch: the
    // kernel before this one may run on long after it let this one in.
    ptx::grid_dependency_wait();
    if (resident)  // resident weights: wait for all of them once
      for (int c = 0; c < nchunks; ++c) wait(full_b(c), 0);
    uint32_t i = 0;
    for (uint32_t tile = first_tile; tile < total_tiles; tile += tile_step, ++i) {
      const int a = static_cast<int>(i & 1);
      if (i >= 2) wait(accempty(a), ((i >> 1) - 1) & 1u);
      ptx::tc_fence_after();  // the epilogue's reads of this accumulator are complete
      const uint32_t tmem_d = tmem_base + static_cast<uint32_t>(a * HV * args.mma_n);
      uint32_t acc = 0;
      int jt = 0, jc = 0;  // window gather: tap and channel chunk of item j
      for (int j = 0; j < nops; ++j) {
        wait(opfull(so), opar);
        // words of the packed chunk: channel chunk j (halo) or jc (window
        // gather) of a pixel; the chunks of a vector gather are whole
        int words = WC;
        if (HALO) {
          words = args.wpr - j * WC;
        } else if (args.gather_win) {
          words = args.wpr - jc * WC;
          if (++jt == args.taps) {
            jt = 0;
            ++jc;
          }
        }
        if (words > WC) words = WC;
        int npos = words * U::L;
        if (npos > BK) npos = BK;  // FULL: the last word's lanes past 64 are padding
        const int ksteps = (npos + T::kKPerMma - 1) / T::kKPerMma;
        // No tcgen05 fence here: the operands arrived through the async proxy
        // (TMA, or stores fenced with fence.proxy.async before the producers'
        // arrive), which the mbarrier wait already orders.
        const uint64_t a0 = T::desc(sOp_addr + so * args.op_stride);
        auto run = [&](auto ksteps_c) {
          constexpr int KS = decltype(ksteps_c)::value;
          uint64_t a_r = a0;
          if (resident) {
            uint64_t b_r = bdesc0 + static_cast<uint32_t>(j * frows * ftaps) * b_step16;
            auto all_taps = [&](uint32_t who) {
              for (int r = 0; r < frows; ++r) {
                issue_row<FP8, HV, KS>(who, tmem_d, dn, a_r, a_half16, b_r, idesc, ftaps, a_row16, b_step16, acc);
                acc = 1;
                a_r += static_cast<uint32_t>(ftaps) * a_row16 + a_skip16;
                b_r += static_cast<uint32_t>(ftaps) * b_step16;
              }
            };
            // MMAs of up to 64 columns (48 cycles) are the one case where the
            // predicate costs more than the branch: VGG-16 conv2, back to
            // back, 39.1 us with the predicate, 35.0 with the branch; conv4
            // (128 columns) 27.6 and 30.7
            if (args.mma_n <= 64) {
              if (leader) all_taps(1u);
              __syncwarp();
              acc = 1;
            } else {
              all_taps(leader);
            }
          } else {
            // Streamed weights: a stage holds tgroup tiles, a whole filter row
            // where three such stages fit, so that one wait and one commit
            // serve its MMAs and not one tap's.
            for (int r = 0; r < frows; ++r) {
              for (int q = 0; q < ftaps; q += tgroup) {
                wait(full_b(sb), bpar);
                issue_row<FP8, HV, KS>(leader, tmem_d, dn, a_r, a_half16, bdesc0 + static_cast<uint32_t>(sb) * b_stage16,
                                       idesc, tgroup, a_row16, b_step16, acc);
                ptx::mma_commit(leader, empty_b(sb));
                acc = 1;
                a_r += static_cast<uint32_t>(tgroup) * a_row16;
                if (++sb == STB) {
                  sb = 0;
                  bpar ^= 1;
                }
              }
              a_r += a_skip16;
            }
          }
        };
        if constexpr (FP8) {
          if (ksteps == 2)
            run(std::integral_constant<int, 2>{});
          else
            run(std::integral_constant<int, 1>{});
        } else {
          switch (ksteps) {
            case 4: run(std::integral_constant<int, 4>{}); break;
            case 3: run(std::integral_constant<int, 3>{}); break;
            case 2: run(std::integral_constant<int, 2>{}); break;
            default: run(std::integral_constant<int, 1>{}); break;
          }
        }
        ptx::mma_commit(leader, opempty(so));  // the stage is free once these MMAs complete
        if (++so == NO) {
          so = 0;
          opar ^= 1;
        }
      }
      ptx::mma_commit(leader, accfull(a));
      if (__any_sync(0xffffffffu, gave_up)) break;
    }
    ptx::mma_commit(leader, drain_bar);
    __syncwarp();
    if (lane == 0) {
      int quiet = 0;
      ptx::mbar_wait_bounded(drain_bar, 0, &quiet, kWaitLimitNs);
    }
    __syncwarp();
  } else if (warp < kFirstEpiWarp) {
    // ---- operand producers ----
    const int t = threadIdx.x - 64;  // 0 .. kProdThreads - 1
    const W *act = static_cast<const W *>(args.act);
    ptx::grid_dependency_wait();  // the activations
    bool gave_up = false;  // looked at behind a tile, or a few items: a vote on every item costs time
    if constexpr (HALO) {
      const int halo_rows = args.nseg * args.seg_rows;
      // Input pixels of this thread's halo rows in the tile being gathered
      // (-1: padding), found once per tile and used for every channel chunk.
      constexpr int kRowsPerThread = kMaxHaloRows / kProdThreads;
      int pix[kRowsPerThread];
      auto locate = [&](uint32_t tile) {
        const uint32_t mt = tile - fdiv(tile, args.fd_gm) * args.fd_gm.d;
        const uint32_t v0 = tile_first_pos(args, mt, BMT);
#pragma unroll
        for (int r = 0; r < kRowsPerThread; ++r) {
          const uint32_t hr = static_cast<uint32_t>(t + r * kProdThreads);
          const uint32_t g = fdiv(hr, args.fd_seg);  // rows past a segment's used ones are read by no tap
          const uint32_t u = v0 + hr + g * static_cast<uint32_t>(args.Wp - args.seg_rows);
          const uint32_t img = fdiv(u, args.fd_plane);
          const uint32_t rem = u - img * args.fd_plane.d;
          const uint32_t ihp = fdiv(rem, args.fd_wp);
          const int ih = static_cast<int>(ihp) - args.pad;
          const int iw = static_cast<int>(rem - ihp * args.fd_wp.d) - args.pad;
          const bool valid = static_cast<int>(img) < args.N && static_cast<unsigned>(ih) < static_cast<unsigned>(args.H) &&
                             static_cast<unsigned>(iw) < static_cast<unsigned>(args.W);
          pix[r] = valid ? (static_cast<int>(img) * args.H + ih) * args.W + iw : -1;
        }
      };
      // items k = (tile i, channel chunk j), in the MMA's order
      auto gather = [&](int j, int slot) {
        const uint32_t dst0 = ptx::smem_addr(sG + slot * args.g_stride);
        const int nw = args.wpr - j * WC;  // words of the chunk; lanes past them meet zero weights
#pragma unroll
        for (int r = 0; r < kRowsPerThread; ++r) {
          const int hr = t + r * kProdThreads;
          if (hr >= halo_rows) break;
          const bool valid = pix[r] >= 0;
          const W *px = valid ? act + (static_cast<long long>(pix[r]) * args.wpr + j * WC) : act;
          const uint32_t dst = dst0 + hr * St::kRowBytes;
          if (args.gather_vec) {
            stage_chunk<W, WC>(dst, reinterpret_cast<const char *>(px), valid ? 1u : 0u);
          } else {
#pragma unroll
            for (int q = 0; q < WC; ++q) {
              if (q >= nw) break;
              if constexpr (sizeof(W) == 8)
                ptx::cp_async_8(dst + 8 * q, px + (valid ? q : 0), valid ? 8u : 0u);
              else
                ptx::cp_async_4(dst + 4 * q, px + (valid ? q : 0), valid ? 4u : 0u);
            }
          }
        }
      };
      auto advance = [&](uint32_t &tile, int &j) {
        if (++j == args.nck) {
          j = 0;
          tile += tile_step;
        }
      };
      // Packed staging is a ring of kHaloGatherSlots = D slots: item k is gathered
      // into slot k mod D, D - 1 items before it is widened. Each iteration
      // commits exactly one cp.async group (empty past the last item), so
      // waiting until at most D - 1 groups are pending means item k landed.
      // A thread reads back only the rows it gathered itself, so refilling
      // the slot it finished with one item earlier needs no barrier.
      constexpr int D = kHaloGatherSlots;
      uint32_t gtile = first_tile;  // issue side
      int gj = 0, gslot = 0;
      auto issue = [&]() {
        if (gtile < total_tiles) {
          if (gj == 0) locate(gtile);
          gather(gj, gslot);
        }
        ptx::cp_async_commit();
        advance(gtile, gj);
        if (++gslot == D) gslot = 0;
      };
      for (int d = 0; d + 1 < D; ++d) issue();
      uint32_t ctile = first_tile;  // widening side
      int cj = 0, cslot = 0;
      int hb = 0;           // halo buffer of item k
      bool reused = false;  // buffers are in their second or a later round
      uint32_t hpar = 1;    // parity of the previous round's release
      while (ctile < total_tiles) {
        issue();
        ptx::cp_async_wait<D - 1>();  // item k of this thread's rows has landed
        if (reused && !role_wait(opempty(hb), hpar, status)) gave_up = true;
        const uint8_t *stg = sG + cslot * args.g_stride;
        for (int hr = t; hr < halo_rows; hr += kProdThreads) {
          W cur[WC];
          load_staged<W, WC>(stg + hr * St::kRowBytes, cur);
          U::unpack_row(cur, sOp + hb * args.op_stride, hr);
        }
        ptx::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(opfull(hb));
        advance(ctile, cj);
        if (cj == 0 && __any_sync(0xffffffffu, gave_up)) break;
        if (++cslot == D) cslot = 0;
        if (++hb == NO) {
          hb = 0;
          reused = true;
          hpar ^= 1;
        }
      }
      ptx::cp_async_wait<0>();
    } else {
      // GATHER: with one-half tiles group grp (four warps) takes items grp,
      // grp + 2, ...; with two-half tiles both groups take every item, group
      // grp filling rows 128 grp .. 128 grp + 127. A thread owns one row.
      const int grp = t / BM;
      const int row = (HV == 2 ? grp * BM : 0) + t % BM;  // row of the A tile
      constexpr int kItemStep = HV == 2 ? 1 : 2;
      const bool win = args.gather_win != 0;
      AGather<W, WC> g;
      g.act = act;
      g.H = args.H;
      g.W_ = args.W;
      g.wpr = args.wpr;
      g.R = args.R;
      g.S = args.S;
      g.nck = args.nck;
      g.win = win;
      auto set_tile = [&](uint32_t tile) {
        const uint32_t mt = tile - fdiv(tile, args.fd_gm) * args.fd_gm.d;
        const uint32_t m = mt * BMT + row;
        g.row_valid = m < static_cast<uint64_t>(args.M);
        const uint32_t mm = g.row_valid ? m : 0u;
        const uint32_t tq = fdiv(mm, args.fd_wo);
        const uint32_t nq = fdiv(tq, args.fd_ho);
        g.iw0 = static_cast<int>(mm - tq * args.fd_wo.d) * args.stride - args.pad;
        g.ih0 = static_cast<int>(tq - nq * args.fd_ho.d) * args.stride - args.pad;
        g.pix0 = (static_cast<int>(nq) * args.H + g.ih0) * args.W + g.iw0;
      };
      const uint32_t g_row = static_cast<uint32_t>(args.g_row);  // staging row pitch
      const uint32_t kSlotBytes = BM * g_row;
      const uint32_t slot0 = ptx::smem_addr(sG) + grp * (kGatherDepth * kSlotBytes) + (t % BM) * g_row;
      const uintptr_t act_end = reinterpret_cast<uintptr_t>(args.act) + static_cast<uintptr_t>(args.act_bytes);
      uint32_t o4s = 0;  // window offsets of the kGatherDepth slots, 2 bits each
      // Items (tile, chunk) are counted, not divided: the issue side runs
      // kGatherDepth of this group's items ahead of the consume side.
      uint32_t itile = first_tile;
      auto step = [&]() {
        if (g.advance()) itile += tile_step;
      };
      if (HV == 1 && grp == 1) step();
      if (itile < total_tiles) set_tile(itile);
      auto issue_next = [&](int slot) {
        if (itile < total_tiles) {
          if (win) {
            const int o4 = g.issue_win(slot0 + slot * kSlotBytes, act_end);
            o4s = (o4s & ~(3u << (2 * slot))) | (static_cast<uint32_t>(o4) << (2 * slot));
          } else {
            g.issue(slot0 + slot * kSlotBytes);
          }
          const uint32_t prev = itile;
          step();
          if (kItemStep == 2) step();
          if (itile != prev && itile < total_tiles) set_tile(itile);
        }
        ptx::cp_async_commit();
      };
#pragma unroll 1
      for (int d = 0; d < kGatherDepth; ++d) issue_next(d);
      const long long items = static_cast<long long>((total_tiles - first_tile + tile_step - 1) / tile_step) * nchunks;
      int slot = 0;
      int ct = 0, cj = 0;   // windows: tap and channel chunk of the item consumed next
      auto cstep = [&]() {
        if (++ct == args.taps) {
          ct = 0;
          if (++cj == args.nck) cj = 0;
        }
      };
      int sa = 0;           // A tile of the item
      bool reused = false;  // the A tiles are in their second or a later round
      uint32_t apar = 1;    // parity of the previous round's release
      if (HV == 1 && grp == 1) {
        cstep();
        sa = 1;
      }
      for (long long k = HV == 2 ? 0 : grp; k < items; k += kItemStep) {
        ptx::cp_async_wait<kGatherDepth - 1>();
        W cur[WC];
        const uint8_t *srow = sG + grp * (kGatherDepth * kSlotBytes) + slot * kSlotBytes + (t % BM) * g_row;
        if (win) {
          const int wi = cj * WC;
          const int nw = args.wpr - wi < WC ? args.wpr - wi : WC;
          load_window<W, WC>(srow, static_cast<int>((o4s >> (2 * slot)) & 3u), nw, cur);
          cstep();
          if (kItemStep == 2) cstep();
        } else {
          load_staged<W, WC>(srow, cur);
        }
        if (reused && !role_wait(opempty(sa), apar, status)) gave_up = true;
        U::unpack_row(cur, sOp + sa * args.op_stride, row);
        ptx::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(opfull(sa));
        issue_next(slot);  // refill the slot just read
        if (++slot == kGatherDepth) {
          slot = 0;
          if (__any_sync(0xffffffffu, gave_up)) break;
        }
        sa += kItemStep;
        if (sa >= NO) {
          sa -= NO;
          reused = true;
          apar ^= 1;
        }
      }
      ptx::cp_async_wait<0>();
    }
    // what is left of this CTA is its last MMAs and rows: the next kernel of
    // the stream may be set up where there is room
    if (args.early) ptx::grid_dependents_launch();
  } else {
    // ---- epilogue ----
    // One-half tiles: warp set `set` drains accumulator `set`, i.e. the CTA's
    // tiles i with i % 2 == set. Two-half tiles: both sets drain every tile,
    // set `set` its half `set`. Warp w reads the TMEM lanes of quadrant w % 4.
    const int quad = warp & 3;
    const int set = (warp - kFirstEpiWarp) / 4;
    uint32_t *const estage =
        reinterpret_cast<uint32_t *>(smem + args.off_e) + (warp - kFirstEpiWarp) * args.e_words;
    const int row = quad * 32 + lane;
    constexpr int kTileStep = HV >= 2 ? 1 : 2;
    // parts of 128 rows of a tile this warp drains: set `set` takes parts
    // set * kParts .. set * kParts + kParts - 1 (HV = 2: its half; HV = 4:
    // two of the four parts); with HV = 1 the sets take alternate tiles
    constexpr int kParts = HV == 4 ? 2 : 1;
    uint32_t i = HV >= 2 ? 0 : set;
    // The first pass over the first tile runs with its stores off and without
    // waiting for the accumulator (whatever it reads is discarded): the row
    // epilogue is the largest code of the kernel, and this way its
    // instructions are fetched while the first tile is being computed rather
    // than after it.
    bool warm = true;
    bool pooled = false;
    if constexpr (HALO && HV <= 2) {
      if (args.pool) {
        // pooled tiles (no warm-up pass): two-half tiles are drained and
        // pooled by all eight epilogue warps, one-half tiles by the four of
        // the set that drains them (alternate tiles, own buffer and barrier)
        pooled = true;
        ptx::grid_dependency_wait();
        constexpr int gw = HV == 2 ? kEpiWarps : kEpiWarps / 2;
        const int gi = HV == 2 ? warp - kFirstEpiWarp : warp - kFirstEpiWarp - 4 * set;
        uint32_t *const pbuf = reinterpret_cast<uint32_t *>(smem + args.off_e) + (HV == 2 ? 0 : set * BM * args.pool_pitch);
        const uint32_t gbar = group_bar(HV == 2 ? 0 : set);
        constexpr int kStep = HV == 2 ? 1 : 2;
        uint32_t gphase = 0;
        uint32_t ip = HV == 2 ? 0 : set;
        for (uint32_t tile = first_tile + (HV == 2 ? 0 : set) * tile_step; tile < total_tiles;
             tile += kStep * tile_step, ip += kStep) {
          const int acc_i = HV == 2 ? static_cast<int>(ip & 1) : set;
          if (!warp_wait(accfull(acc_i), (ip >> 1) & 1u, status)) break;
          ptx::tc_fence_after();
          const uint32_t nbu = fdiv(tile, args.fd_gm);
          const uint32_t mt = tile - nbu * args.fd_gm.d;
          const uint32_t taddr = tmem_base + static_cast<uint32_t>((acc_i * HV + (HV == 2 ? set : 0)) * args.mma_n) +
                                 (static_cast<uint32_t>(quad * 32) << 16);
          epilogue_pool_dispatch(args, taddr, (HV == 2 ? set * BM : 0) + row, mt, static_cast<int>(nbu), pbuf,
                                 accempty(acc_i), gbar, gphase, status, gw, gi);
        }
      }
    }
    for (uint32_t tile = first_tile + (HV >= 2 ? 0 : set) * tile_step; !pooled && tile < total_tiles;) {
      const int acc_i = HV >= 2 ? static_cast<int>(i & 1) : set;  // accumulator of this tile
      bool ok = true;
      if (!warm) {
        ok = warp_wait(accfull(acc_i), (i >> 1) & 1u, status);
        ptx::tc_fence_after();
      }
      const uint32_t nbu = fdiv(tile, args.fd_gm);
      const int nb = static_cast<int>(nbu);
      const uint32_t mt = tile - nbu * args.fd_gm.d;
#pragma unroll 1
      for (int hh = 0; hh < kParts; ++hh) {
        const int part = HV >= 2 ? set * kParts + hh : 0;
        bool valid;
        uint32_t m;
        const int trow = part * BM + row;  // row of the tile
        if (HALO) {
          const uint32_t v = tile_first_pos(args, mt, BMT) + trow;
          const uint32_t img = fdiv(v, args.fd_plane);
          const uint32_t rem = v - img * args.fd_plane.d;
          const uint32_t oh = fdiv(rem, args.fd_wp);
          const uint32_t ow = rem - oh * args.fd_wp.d;
          valid = static_cast<int>(img) < args.N && static_cast<int>(oh) < args.Ho && static_cast<int>(ow) < args.Wo;
          m = (img * args.Ho + oh) * args.Wo + ow;
        } else {
          m = mt * BMT + trow;
          valid = m < static_cast<uint64_t>(args.M);
        }
        const uint32_t taddr = tmem_base + static_cast<uint32_t>((acc_i * HV + part) * args.mma_n) +
                               (static_cast<uint32_t>(quad * 32) << 16);
        epilogue_row(args, epi_row(args, taddr, valid ? m : ~0u, nb, warm), estage);
      }
      if (warm) {
        warm = false;
        ptx::grid_dependency_wait();  // earlier readers of the outputs
        continue;
      }
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(accempty(acc_i));
      if (!ok) break;
      tile += kTileStep * tile_step;
      i += kTileStep;
    }
  }

  __syncwarp();
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, args.tmem_cols);
  }
}

// cudaFuncSetAttribute once per (kernel, device); defined in conv2d.cu.
cudaError_t ensure_smem_attr(const void *kern, size_t smem);

// FULL variants exist only for lane counts that do not divide 64.
__host__ __device__ constexpr bool needs_full(int word_bits, int bits) { return 64 % (word_bits / bits) != 0; }

template <typename W, int BITS, bool SIGNED, bool FP8>
cudaError_t launch_conv(const CUtensorMap &tmap, const ConvArgs &args, bool halo, dim3 grid, size_t smem,
                        cudaStream_t s) {
  constexpr bool kHasFull = needs_full(WordTraits<W>::kBits, BITS);
  using K = void (*)(const CUtensorMap, const ConvArgs);
  K kern;
  if (args.hv == 2)
    kern = halo ? conv_kernel<W, BITS, SIGNED, true, FP8, false, 2> : conv_kernel<W, BITS, SIGNED, false, FP8, false, 2>;
  else
    kern = halo ? conv_kernel<W, BITS, SIGNED, true, FP8, false, 1> : conv_kernel<W, BITS, SIGNED, false, FP8, false, 1>;
  if constexpr (kHasFull) {
    if (args.full && args.hv == 2)
      kern = halo ? conv_kernel<W, BITS, SIGNED, true, FP8, true, 2> : conv_kernel<W, BITS, SIGNED, false, FP8, true, 2>;
    else if (args.full)
      kern = halo ? conv_kernel<W, BITS, SIGNED, true, FP8, true, 1> : conv_kernel<W, BITS, SIGNED, false, FP8, true, 1>;
  }
  // four-part tiles: halo layers on e4m3 operands only (planned so)
  if constexpr (FP8) {
    if (args.hv == 4) {
      if (!halo) return cudaErrorInvalidValue;
      kern = conv_kernel<W, BITS, SIGNED, true, FP8, false, 4>;
      if constexpr (kHasFull)
        if (args.full) kern = conv_kernel<W, BITS, SIGNED, true, FP8, true, 4>;
    }
  } else {
    if (args.hv == 4) return cudaErrorInvalidValue;
  }
  cudaError_t e = ensure_smem_attr(reinterpret_cast<const void *>(kern), smem);
  if (e != cudaSuccess) return e;
  // Launched as a programmatic dependent of the kernel before it in the
  // stream: barriers, tensor memory and the epilogue's code are set up while
  // that one drains; every role waits (grid_dependency_wait) before it reads
  // or writes global memory, or waits for another role.
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kern, tmap, args);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// Launchers, one per (operand type, activation word width, lane width), each
// compiled from conv_inst.cu in its own unit.
using LaunchFn = cudaError_t (*)(bool is_signed, const CUtensorMap &tmap, const ConvArgs &args, bool halo, dim3 grid,
                                 size_t smem, cudaStream_t s);
#define SAMD_CONV_LAUNCHER(name) \
  cudaError_t name(bool is_signed, const CUtensorMap &tmap, const ConvArgs &args, bool halo, dim3 grid, size_t smem, \
                   cudaStream_t s);
#define SAMD_CONV_LAUNCHERS(t, wb)                                                                          \
  SAMD_CONV_LAUNCHER(launch_conv_##t##_w##wb##_b1) SAMD_CONV_LAUNCHER(launch_conv_##t##_w##wb##_b2)        \
  SAMD_CONV_LAUNCHER(launch_conv_##t##_w##wb##_b3) SAMD_CONV_LAUNCHER(launch_conv_##t##_w##wb##_b4)        \
  SAMD_CONV_LAUNCHER(launch_conv_##t##_w##wb##_b5)
SAMD_CONV_LAUNCHERS(f16, 32)
SAMD_CONV_LAUNCHERS(f16, 64)
SAMD_CONV_LAUNCHERS(f8, 32)
SAMD_CONV_LAUNCHERS(f8, 64)
SAMD_CONV_LAUNCHER(launch_conv_f16_w32_b6)
SAMD_CONV_LAUNCHER(launch_conv_f16_w32_b7)
SAMD_CONV_LAUNCHER(launch_conv_f16_w32_b8)
SAMD_CONV_LAUNCHER(launch_conv_f16_w64_b6)
SAMD_CONV_LAUNCHER(launch_conv_f16_w64_b7)
SAMD_CONV_LAUNCHER(launch_conv_f16_w64_b8)
#undef SAMD_CONV_LAUNCHERS
#undef SAMD_CONV_LAUNCHER

}  // namespace conv
}  // namespace samd
