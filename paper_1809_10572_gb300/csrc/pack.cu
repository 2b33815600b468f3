// pack.cu -- int8 bytes <-> packed b-bit lanes (section 2.1 of the paper:
// b-bit lanes laid side by side in a scalar word; section 7: unpacking to
// the native 8-bit type).
//
// Layouts:
//   - one row, or rows of whole words, of spacer-free 32-bit words: a thread
//     moves four words with the widest aligned vectors (pack32_*, unpack32_*);
//     64-bit words whose lane width divides 32 are pairs of such words, except
//     where a thread packs a 64-bit word faster (pack64_word_kernel);
//   - spacer formats of 16 and more lanes a word are packed by a thread a word
//     (pack_generic_kernel);
//   - anything else (rows that end inside a word, 64-bit words of 3, 5, 6 or
//     7 bits, spacer bits, and the few words the vector kernels leave): the
//     bytes of a tile of consecutive words are one contiguous run, staged in
//     shared memory with 16-byte accesses (pack_rows_kernel,
//     unpack_rows_kernel).
// All forms produce the same canonical words.
#include "samd_internal.cuh"

namespace samd {
namespace {

constexpr int kThreads = 256;

// Largest power of two dividing n, capped at 16: the vector width in bytes
// for moving L consecutive bytes that start at a multiple of L.
__host__ __device__ constexpr int vec_bytes(int n) {
  return (n % 16 == 0) ? 16 : (n % 8 == 0) ? 8 : (n % 4 == 0) ? 4 : (n % 2 == 0) ? 2 : 1;
}

// Load/store NB consecutive 32-bit chunks with VB-byte vectors (VB >= 4,
// address VB-aligned).
template <int VB, int NB>
__device__ __forceinline__ void load_chunks(const void *src, uint32_t (&c)[NB]) {
  if constexpr (VB == 16) {
#pragma unroll
    for (int v = 0; v < NB / 4; ++v) {
      const uint4 t = __ldcs(reinterpret_cast<const uint4 *>(src) + v);
      c[4 * v] = t.x, c[4 * v + 1] = t.y, c[4 * v + 2] = t.z, c[4 * v + 3] = t.w;
    }
  } else if constexpr (VB == 8) {
#pragma unroll
    for (int v = 0; v < NB / 2; ++v) {
      const uint2 t = __ldcs(reinterpret_cast<const uint2 *>(src) + v);
      c[2 * v] = t.x, c[2 * v + 1] = t.y;
    }
  } else {
#pragma unroll
    for (int v = 0; v < NB; ++v) c[v] = __ldcs(reinterpret_cast<const uint32_t *>(src) + v);
  }
}

template <int VB, int NB>
__device__ __forceinline__ void store_chunks(void *dst, const uint32_t (&c)[NB]) {
  if constexpr (VB == 16) {
#pragma unroll
    for (int v = 0; v < NB / 4; ++v)
      __stcs(reinterpret_cast<uint4 *>(dst) + v, make_uint4(c[4 * v], c[4 * v + 1], c[4 * v + 2], c[4 * v + 3]));
  } else if constexpr (VB == 8) {
#pragma unroll
    for (int v = 0; v < NB / 2; ++v) __stcs(reinterpret_cast<uint2 *>(dst) + v, make_uint2(c[2 * v], c[2 * v + 1]));
  } else {
#pragma unroll
    for (int v = 0; v < NB; ++v) __stcs(reinterpret_cast<uint32_t *>(dst) + v, c[v]);
  }
}

__device__ __forceinline__ uint32_t bfe_u32(uint32_t x, int pos, int len) {
  uint32_t r;
  asm("bfe.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(x), "r"(pos), "r"(len));
  return r;
}
__device__ __forceinline__ uint32_t bfe_s32(uint32_t x, int pos, int len) {
  uint32_t r;
  asm("bfe.s32 %0, %1, %2, %3;" : "=r"(r) : "r"(x), "r"(pos), "r"(len));
  return r;
}
__device__ __forceinline__ uint32_t bfi_b32(uint32_t src, uint32_t into, int pos, int len) {
  uint32_t r;
  asm("bfi.b32 %0, %1, %2, %3, %4;" : "=r"(r) : "r"(src), "r"(into), "r"(pos), "r"(len));
  return r;
}

// ---- single-row (or whole-word rows) 32-bit words: four words per thread ----
//
// A thread packs 4 consecutive words (one 16-byte store) from 4L consecutive
// bytes read with the widest aligned vector that divides 4L. For 1-, 4- and
// 8-bit lanes whole groups of lanes move at once:
//   b = 1: (x & 0x01010101) * 0x01020408 >> 24 gathers the low bits of four
//          bytes into a nibble (the partial products never meet below bit 24);
//   b = 4: x | x >> 4 puts nibble pairs in bytes 0 and 2 of each 32-bit chunk,
//          and one byte permute (PRMT) joins two chunks into a word;
//   b = 8: the bytes are the word.
// Other widths insert lane by lane with compile-time shifts.
template <int BITS>
__device__ __forceinline__ uint32_t pack_word32(const uint32_t *c) {  // c: the L bytes of the word as L/4 chunks
  constexpr int L = 32 / BITS;
  if constexpr (BITS == 8) {
    return c[0];
  } else if constexpr (BITS == 4) {
    const uint32_t a = c[0] & 0x0F0F0F0Fu, b = c[1] & 0x0F0F0F0Fu;
    return __byte_perm(a | (a >> 4), b | (b >> 4), 0x6420);
  } else if constexpr (BITS == 1) {
    uint32_t w = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) w |= (((c[i] & 0x01010101u) * 0x01020408u) >> 24) << (4 * i);
    return w;
  } else {
    (void)L;
    return 0u;  // not used: other widths take pack_lanes
  }
}

template <int BITS, int NB>
__device__ __forceinline__ void pack_lanes(const uint32_t (&in)[NB], uint32_t (&w)[4]) {
  constexpr int L = 32 / BITS;
  constexpr uint32_t M = (1u << BITS) - 1;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    uint32_t word = 0;
#pragma unroll
    for (int l = 0; l < L; ++l) {
      const int e = k * L + l;
      word = bfi_b32(in[e / 4] >> (8 * (e % 4)), word, l * BITS, BITS);
      (void)M;
    }
    w[k] = word;
  }
}

// A warp packs 32 consecutive quads of words. Its 32 x 4L input bytes are one
// contiguous block, read with consecutive 16-byte loads into shared memory
// (rows padded by 16 bytes), from where each lane takes its own 4L bytes.
template <int BITS>
__global__ void __launch_bounds__(kThreads) pack32_staged_kernel(const int8_t *__restrict__ src,
                                                                 uint32_t *__restrict__ dst, int64_t nwarp_tiles) {
  constexpr int L = 32 / BITS;
  constexpr int IB = 4 * L;  // input bytes per lane
  constexpr int NB = IB / 4;
  constexpr int ROW = IB + 16;
  constexpr int TILE16 = 2 * IB;
  __shared__ __align__(16) uint8_t stage[kThreads / 32][32 * ROW];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  uint8_t *my = stage[wib];
  const int64_t warps_total = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t wt = blockIdx.x * (int64_t)(blockDim.x >> 5) + wib; wt < nwarp_tiles; wt += warps_total) {
    const uint4 *in16 = reinterpret_cast<const uint4 *>(src + wt * 32 * IB);
#pragma unroll
    for (int p = lane; p < TILE16; p += 32) {
      const uint4 t = __ldcs(in16 + p);
      const uint32_t tw[4] = {t.x, t.y, t.z, t.w};
      const int byte = p * 16, r = byte / IB, off = byte - r * IB;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int b = off + 4 * k, rr = r + b / IB, oo = b - (b / IB) * IB;
        *reinterpret_cast<uint32_t *>(my + rr * ROW + oo) = tw[k];
      }
    }
    __syncwarp();
    uint32_t in[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) in[i] = *reinterpret_cast<const uint32_t *>(my + lane * ROW + 4 * i);
    __syncwarp();
    uint32_t w[4];
    if constexpr (BITS == 1 || BITS == 4 || BITS == 8) {
#pragma unroll
      for (int k = 0; k < 4; ++k) w[k] = pack_word32<BITS>(in + k * (L / 4));
    } else {
      pack_lanes<BITS, NB>(in, w);
    }
    __stcs(reinterpret_cast<uint4 *>(dst) + wt * 32 + lane, make_uint4(w[0], w[1], w[2], w[3]));
  }
}

// Lanes of 2 bits and more read their 4L bytes directly (at most 64 bytes a
// lane; the L1 cache merges a warp's neighbouring lines).
template <int BITS>
__global__ void __launch_bounds__(kThreads) pack32_vec_kernel(const int8_t *__restrict__ src, uint32_t *__restrict__ dst,
                                                              int64_t nquads) {
  constexpr int L = 32 / BITS;
  constexpr int IB = 4 * L;
  constexpr int VB = vec_bytes(IB);
  constexpr int NB = IB / 4;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nquads; q += (int64_t)gridDim.x * blockDim.x) {
    uint32_t in[NB];
    load_chunks<VB, NB>(src + q * IB, in);
    uint32_t w[4];
    if constexpr (BITS == 4 || BITS == 8) {
#pragma unroll
      for (int k = 0; k < 4; ++k) w[k] = pack_word32<BITS>(in + k * (L / 4));
    } else {
      pack_lanes<BITS, NB>(in, w);
    }
    __stcs(reinterpret_cast<uint4 *>(dst) + q, make_uint4(w[0], w[1], w[2], w[3]));
  }
}

// One row, or rows of whole words, of 64-bit words of 1, 2, 5 and 6 bits: a
// thread packs one word from its L bytes, read with the widest aligned
// vectors. 2^28 lanes, against pairs of 32-bit words (1 and 2 bits) and
// pack_rows_kernel (5 and 6): 49.6 us and 51.2, 51.6 and 55.8, 80.2 and 95.2,
// 97.0 and 110. (At 3 and 7 bits, whose L is odd, that one is the faster: 119
// and 87, 136 and 115.)
template <int VB> struct Vec;
template <> struct Vec<16> { using T = uint4; };
template <> struct Vec<4> { using T = uint32_t; };
template <> struct Vec<2> { using T = uint16_t; };

template <int BITS>
__global__ void __launch_bounds__(kThreads) pack64_word_kernel(const int8_t *__restrict__ src,
                                                               uint64_t *__restrict__ dst, int64_t nwords, int64_t n) {
  constexpr int L = 64 / BITS, VB = vec_bytes(L);
  constexpr uint64_t mask = (1u << BITS) - 1;
  using T = typename Vec<VB>::T;
  for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < nwords; w += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e0 = w * L;
    uint64_t word = 0;
    if (n - e0 >= L) {
      const T *const p = reinterpret_cast<const T *>(src + e0);
      uint8_t buf[L];
#pragma unroll
      for (int v = 0; v < L / VB; ++v) {
        const T t = __ldg(p + v);
        const uint8_t *const b = reinterpret_cast<const uint8_t *>(&t);
#pragma unroll
        for (int j = 0; j < VB; ++j) buf[v * VB + j] = b[j];
      }
#pragma unroll
      for (int i = 0; i < L; ++i) word |= (buf[i] & mask) << (i * BITS);
    } else {
      for (int i = 0; i < static_cast<int>(n - e0); ++i) word |= (static_cast<uint8_t>(src[e0 + i]) & mask) << (i * BITS);
    }
    dst[w] = word;
  }
}

template <int BITS>
cudaError_t launch_pack64_words(const int8_t *src, uint64_t *dst, int64_t n, cudaStream_t s) {
  constexpr int L = 64 / BITS;
  const int64_t nwords = (n + L - 1) / L;
  pack64_word_kernel<BITS><<<grid_for(nwords, kThreads, sm_count() * 16), kThreads, 0, s>>>(src, dst, nwords, n);
  return cudaGetLastError();
}

// Spacer formats of 16 and more lanes a word: a thread packs a word from its
// bytes one at a time (pack_rows_kernel reads them from shared memory, 16 and
// more bytes from one thread to the next: 2^26 signed lanes with one spacer
// bit, 1 bit in 32-bit words 34.8 us and 38.9, in 64-bit words 59.7 and 65.6,
// 3 bits 36.9 and 41.0; with fewer lanes a word that one is 1.1 to 1.7 times
// as fast).
template <typename W>
__global__ void __launch_bounds__(kThreads) pack_generic_kernel(const int8_t *__restrict__ src, W *__restrict__ dst,
                                                                int64_t total_words, int64_t inner, int64_t wpr,
                                                                int bits, int lane_w, int L) {
  const W mask = (W(1) << bits) - 1;
  for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < total_words;
       w += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = w / wpr, wi = w - row * wpr;
    const int64_t e0 = row * inner + wi * L;
    const int64_t count = inner - wi * L < L ? inner - wi * L : L;
    W word = 0;
    for (int i = 0; i < count; ++i) word |= (W(static_cast<uint8_t>(src[e0 + i])) & mask) << (i * lane_w);
    dst[w] = word;
  }
}

// Unpack of 4 words per thread into 4L bytes, written with the widest aligned
// vector. b = 8: the word is its bytes. b = 4: the low and high nibbles of
// each byte are masked apart and interleaved by byte permutes; signed nibbles
// are extended by or-ing 0xF0 into bytes whose bit 3 is set
// ((x & 0x08080808) * 0x1E). b = 1: (nibble * 0x00204081) & 0x01010101
// spreads four bits into four bytes; signed 1-bit lanes are -bit (x 0xFF).
template <int BITS, bool SIGNED>
__device__ __forceinline__ void unpack_word32(uint32_t w, uint32_t *out) {  // out: L/4 chunks of 4 bytes
  constexpr int L = 32 / BITS;
  if constexpr (BITS == 8) {
    out[0] = w;
  } else if constexpr (BITS == 4) {
    uint32_t lo = w & 0x0F0F0F0Fu, hi = (w >> 4) & 0x0F0F0F0Fu;
    if constexpr (SIGNED) {
      lo |= (lo & 0x08080808u) * 0x1Eu;
      hi |= (hi & 0x08080808u) * 0x1Eu;
    }
    out[0] = __byte_perm(lo, hi, 0x5140);
    out[1] = __byte_perm(lo, hi, 0x7362);
  } else if constexpr (BITS == 1) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      uint32_t t = (((w >> (4 * i)) & 0xFu) * 0x00204081u) & 0x01010101u;
      if constexpr (SIGNED) t *= 0xFFu;
      out[i] = t;
    }
  } else if constexpr (BITS == 2) {
    // byte i of x takes bits 2i, 2i + 1 of eight: pairs first, then singles
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t x = (w >> (8 * i)) & 0xFFu;
      const uint32_t y = (x | (x << 12)) & 0x000F000Fu;
      uint32_t t = (y | (y << 6)) & 0x03030303u;
      if constexpr (SIGNED) t |= ((t >> 1) & 0x01010101u) * 0xFCu;
      out[i] = t;
    }
  } else {
#pragma unroll
    for (int j = 0; j < L / 4 + (L % 4 ? 1 : 0); ++j) out[j] = 0;
    (void)w;
  }
}

__device__ __forceinline__ void st_global_cs_v8(void *p, const uint32_t *c) {
  asm volatile("st.global.cs.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(c[0]), "r"(c[1]), "r"(c[2]),
               "r"(c[3]), "r"(c[4]), "r"(c[5]), "r"(c[6]), "r"(c[7])
               : "memory");
}

// Lanes of 2 and 4 bits: a quad of words fills whole 32-byte sectors of the
// output, so a thread stores its 4L bytes itself, 32 at a time; two quads a
// step, so that two loads are in flight. 51 M signed 4-bit lanes (77 MB
// moved): 16.4 us through shared memory, 16.1 this way; 2^28 2-bit lanes 59.6
// and 57.1. (1-bit lanes, 128 bytes a thread, 51.3 and 55.3: they stay with
// unpack32_vec_kernel.)
template <int BITS, bool SIGNED>
__global__ void __launch_bounds__(kThreads) unpack32_direct_kernel(const uint32_t *__restrict__ src,
                                                                   int8_t *__restrict__ dst, int64_t nquads) {
  constexpr int L = 32 / BITS, NC = L;  // 32-bit chunks of a quad's 4L bytes
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  auto expand = [&](const uint4 &v, int64_t q) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t c[NC];
#pragma unroll
    for (int k = 0; k < 4; ++k) unpack_word32<BITS, SIGNED>(w[k], c + k * (L / 4));
#pragma unroll
    for (int k = 0; k < NC; k += 8) st_global_cs_v8(dst + q * (4 * L) + 4 * k, c + k);
  };
  int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  for (; q + stride < nquads; q += 2 * stride) {
    const uint4 a = __ldcs(reinterpret_cast<const uint4 *>(src) + q);
    const uint4 b = __ldcs(reinterpret_cast<const uint4 *>(src) + q + stride);
    expand(a, q);
    expand(b, q + stride);
  }
  if (q < nquads) expand(__ldcs(reinterpret_cast<const uint4 *>(src) + q), q);
}

// A warp expands 32 consecutive quads of words; its 32 x 4L output bytes are
// one contiguous block. Each lane stages its 4L bytes in shared memory (rows
// padded by 16 bytes so the lanes' 16-byte writes spread over the banks),
// then the warp writes the block with consecutive 16-byte stores.
template <int BITS, bool SIGNED>
__global__ void __launch_bounds__(kThreads) unpack32_vec_kernel(const uint32_t *__restrict__ src,
                                                                int8_t *__restrict__ dst, int64_t nwarp_tiles) {
  constexpr int L = 32 / BITS;
  constexpr int OB = 4 * L;          // output bytes per lane
  constexpr int NC = OB / 4;
  constexpr int ROW = OB + 16;       // staged row pitch (16-byte aligned)
  constexpr int TILE16 = 2 * OB;     // 16-byte vectors per warp block (32 * OB / 16)
  __shared__ __align__(16) uint8_t stage[kThreads / 32][32 * ROW];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  uint8_t *my = stage[wib];
  const int64_t warps_total = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t wt = blockIdx.x * (int64_t)(blockDim.x >> 5) + wib; wt < nwarp_tiles; wt += warps_total) {
    const int64_t q = wt * 32 + lane;
    const uint4 v = __ldcs(reinterpret_cast<const uint4 *>(src) + q);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t c[NC];
    if constexpr (BITS == 1 || BITS == 2 || BITS == 4 || BITS == 8) {
#pragma unroll
      for (int k = 0; k < 4; ++k) unpack_word32<BITS, SIGNED>(w[k], c + k * (L / 4));
    } else {
#pragma unroll
      for (int i = 0; i < NC; ++i) c[i] = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int l = 0; l < L; ++l) {
          const int e = k * L + l;
          const uint32_t p = SIGNED ? bfe_s32(w[k], l * BITS, BITS) : bfe_u32(w[k], l * BITS, BITS);
          c[e / 4] = bfi_b32(p, c[e / 4], 8 * (e % 4), 8);
        }
    }
    // stage: lane's row holds its OB bytes (4-byte stores; OB may be 20 or 40)
#pragma unroll
    for (int i = 0; i < NC; ++i) *reinterpret_cast<uint32_t *>(my + lane * ROW + 4 * i) = c[i];
    __syncwarp();
    uint4 *out = reinterpret_cast<uint4 *>(dst + wt * 32 * OB);
#pragma unroll
    for (int p = lane; p < TILE16; p += 32) {
      const int byte = p * 16, r = byte / OB, off = byte - r * OB;  // 16-byte vector p of the block
      uint32_t t[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        // OB is a multiple of 4, so a 4-byte piece never straddles two rows
        const int b = off + 4 * k, rr = r + b / OB, oo = b - (b / OB) * OB;
        t[k] = *reinterpret_cast<const uint32_t *>(my + rr * ROW + oo);
      }
      __stcs(out + p, make_uint4(t[0], t[1], t[2], t[3]));
    }
    __syncwarp();
  }
}

template <typename W, int BITS, bool SIGNED>
__device__ __forceinline__ uint8_t lane_byte(W word, int i) {
  uint32_t p = static_cast<uint32_t>(word >> (i * BITS)) & ((1u << BITS) - 1);
  if (SIGNED) p = static_cast<uint32_t>(static_cast<int>(p << (32 - BITS)) >> (32 - BITS));
  return static_cast<uint8_t>(p);
}

// ---- any rows, any format ----------------------------------------------------
//
// Source bytes and packed words run in the same order, row after row, so the
// words [w0, w0 + T) of the array belong to one contiguous run of bytes. A
// block moves that run with 16-byte accesses (bytes at its ragged ends) and
// the words one per thread, coalesced, through shared memory; a thread turns
// the L bytes of a word, at any byte offset there, into the word or back.
// One thread per word moving its own bytes one at a time, as before, was
// bound by those accesses: 200704 rows of 64 6-bit lanes (23 MB moved) took
// 16.4 us to pack, now 10.2 (12.6 with 64-bit addressing in the tile and one
// wave of blocks that looped over the tiles).

// T words of L lanes: at most 16 KB of bytes, a few words per thread.
constexpr int tile_words(int L) { return L <= 12 ? 1024 : (L <= 24 ? 512 : 256); }
// The same for the forms of any format, whose L (at most 32) is known at run
// time.
__host__ __device__ constexpr int any_tile_words(int L) { return L <= 16 ? 1024 : 512; }

struct RowsArgs {
  int64_t inner;
  uint32_t total_words, wpr;
  int last_count;  // lanes of a row's last word
  int bits, is_signed, lane_w, L;  // for the forms of any format (BITS = 0)
  FastDiv fd_wpr;
};

// A tile of words [w0, w1) and its run of bytes: the run starts at byte b0 of
// the array, `lead` bytes past a 16-byte boundary, and is `bytes` long. Inside
// the tile everything is counted from the boundary in 32 bits.
struct RowsTile {
  uint32_t w0, w1, row0, wi0;
  int64_t b0;
  int lead, bytes;
  __device__ __forceinline__ RowsTile(const RowsArgs &a, uint32_t first, uint32_t tile, int L, const void *base)
      : w0(first), w1(a.total_words - first < tile ? a.total_words : first + tile) {
    row0 = fdiv(w0, a.fd_wpr);
    wi0 = w0 - row0 * a.wpr;
    b0 = row0 * a.inner + static_cast<int64_t>(wi0) * L;
    lead = static_cast<int>((reinterpret_cast<uintptr_t>(base) + static_cast<uintptr_t>(b0)) & 15u);
    int count;
    bytes = offset(a, w1 - 1, L, &count) - lead + count;
  }
  // Where word w's bytes start, and how many there are.
  __device__ __forceinline__ int offset(const RowsArgs &a, uint32_t w, int L, int *count) const {
    const uint32_t row = fdiv(w, a.fd_wpr), wi = w - row * a.wpr;
    *count = wi == a.wpr - 1 ? a.last_count : L;
    return lead + static_cast<int>((row - row0) * static_cast<uint32_t>(a.inner) + (wi - wi0) * static_cast<uint32_t>(L));
  }
  // Whether the 16 bytes at 16 v all belong to the run.
  __device__ __forceinline__ bool whole(int v) const { return 16 * v >= lead && 16 * v + 16 <= lead + bytes; }
};

// The low BITS bits of the four bytes of c, side by side.
template <int BITS>
__device__ __forceinline__ uint32_t pack_bytes4(uint32_t c) {
  constexpr uint32_t m = (1u << BITS) - 1;
  const uint32_t t = (c & (m * 0x00010001u)) | ((c & (m * 0x01000100u)) >> (8 - BITS));
  return (t & 0xFFFFu) | (t >> (16 - 2 * BITS) & ~0u << (2 * BITS));
}

template <typename W, int BITS>
__global__ void __launch_bounds__(kThreads) pack_rows_kernel(const int8_t *src, W *__restrict__ dst,
                                                             const RowsArgs a) {
  constexpr int kL = BITS ? WordTraits<W>::kBits / (BITS ? BITS : 1) : 0;
  constexpr int kBytes = BITS ? tile_words(kL) * kL : 16 * 1024;
  __shared__ __align__(16) uint8_t stage[kBytes + 48];  // 15 bytes before the run, reads up to 8 bytes past it
  const int L = BITS ? kL : a.L;
  const uint32_t tile = BITS ? tile_words(kL) : any_tile_words(L);
  for (uint32_t first = blockIdx.x * tile; first < a.total_words; first += gridDim.x * tile) {
    const RowsTile t(a, first, tile, L, src);
    const int8_t *const p = src + t.b0 - t.lead;
    const int nvec = (t.lead + t.bytes + 15) >> 4;
    for (int v = threadIdx.x; v < nvec; v += kThreads) {
      if (t.whole(v)) {
        *reinterpret_cast<uint4 *>(stage + 16 * v) = __ldcs(reinterpret_cast<const uint4 *>(p) + v);
      } else {
        for (int k = 16 * v; k < 16 * v + 16; ++k)
          if (k >= t.lead && k < t.lead + t.bytes) stage[k] = static_cast<uint8_t>(p[k]);
      }
    }
    __syncthreads();
    for (uint32_t w = t.w0 + threadIdx.x; w < t.w1; w += kThreads) {
      int count;
      const int off = t.offset(a, w, L, &count);
      const uint32_t *base = reinterpret_cast<const uint32_t *>(stage) + (off >> 2);
      const int sh = 8 * (off & 3);
      W word = 0;
      if constexpr (BITS != 0) {
        uint32_t lo = base[0];
#pragma unroll
        for (int k = 0; k < (kL + 3) / 4; ++k) {
          const uint32_t hi = base[k + 1];
          const uint32_t c = pack_bytes4<BITS ? BITS : 1>(__funnelshift_r(lo, hi, sh));
          lo = hi;
          word |= static_cast<W>(c) << (4 * k * BITS);  // lanes past the word's last fall off below
        }
        const int nb = count * BITS;
        if (nb < WordTraits<W>::kBits) word &= (W(1) << nb) - 1;
      } else {
        const uint32_t mask = (1u << a.bits) - 1;
        for (int i = 0; i < count; ++i) word |= static_cast<W>(stage[off + i] & mask) << (i * a.lane_w);
      }
      dst[w] = word;
    }
    __syncthreads();
  }
}

template <typename W, int BITS, bool SIGNED>
__global__ void __launch_bounds__(kThreads) unpack_rows_kernel(const W *__restrict__ src, int8_t *dst,
                                                               const RowsArgs a) {
  constexpr int kL = BITS ? WordTraits<W>::kBits / (BITS ? BITS : 1) : 0;
  constexpr int kBytes = BITS ? tile_words(kL) * kL : 16 * 1024;
  __shared__ __align__(16) uint8_t stage[kBytes + 32];
  const int L = BITS ? kL : a.L;
  const uint32_t tile = BITS ? tile_words(kL) : any_tile_words(L);
  for (uint32_t first = blockIdx.x * tile; first < a.total_words; first += gridDim.x * tile) {
    const RowsTile t(a, first, tile, L, dst);
    for (uint32_t w = t.w0 + threadIdx.x; w < t.w1; w += kThreads) {
      int count;
      const int off = t.offset(a, w, L, &count);
      const W word = __ldcs(src + w);
      if constexpr (BITS != 0) {
        if ((off & 3) == 0 && count == L) {
#pragma unroll
          for (int k = 0; k < kL / 4; ++k) {
            uint32_t c = 0;
#pragma unroll
            for (int l = 0; l < 4; ++l) c |= static_cast<uint32_t>(lane_byte<W, BITS ? BITS : 1, SIGNED>(word, 4 * k + l)) << (8 * l);
            *reinterpret_cast<uint32_t *>(stage + off + 4 * k) = c;
          }
#pragma unroll
          for (int i = kL / 4 * 4; i < kL; ++i) stage[off + i] = lane_byte<W, BITS ? BITS : 1, SIGNED>(word, i);
        } else {
#pragma unroll
          for (int i = 0; i < kL; ++i)
            if (i < count) stage[off + i] = lane_byte<W, BITS ? BITS : 1, SIGNED>(word, i);
        }
      } else {
        for (int i = 0; i < count; ++i) {
          const uint32_t p = static_cast<uint32_t>(word >> (i * a.lane_w)) & ((1u << a.bits) - 1);
          stage[off + i] = static_cast<uint8_t>(lane_value(p, a.bits, a.is_signed));
        }
      }
    }
    __syncthreads();
    int8_t *const p = dst + t.b0 - t.lead;
    const int nvec = (t.lead + t.bytes + 15) >> 4;
    for (int v = threadIdx.x; v < nvec; v += kThreads) {
      if (t.whole(v)) {
        __stcs(reinterpret_cast<uint4 *>(p) + v, *reinterpret_cast<const uint4 *>(stage + 16 * v));
      } else {
        for (int k = 16 * v; k < 16 * v + 16; ++k)
          if (k >= t.lead && k < t.lead + t.bytes) p[k] = static_cast<int8_t>(stage[k]);
      }
    }
    __syncthreads();
  }
}

template <int BITS>
cudaError_t launch_pack32_vec(const int8_t *src, uint32_t *dst, int64_t ntiles, cudaStream_t s) {
  if (BITS == 1)
    pack32_staged_kernel<BITS><<<resident_grid<pack32_staged_kernel<BITS>>(ntiles * 32, kThreads), kThreads, 0, s>>>(
        src, dst, ntiles);
  else
    pack32_vec_kernel<BITS><<<resident_grid<pack32_vec_kernel<BITS>>(ntiles * 32, kThreads), kThreads, 0, s>>>(
        src, dst, ntiles * 32);
  return cudaGetLastError();
}

template <int BITS, bool SIGNED>
cudaError_t launch_unpack32_vec(const uint32_t *src, int8_t *dst, int64_t ntiles, cudaStream_t s) {
  if constexpr (BITS == 2 || BITS == 4) {
    if ((reinterpret_cast<uintptr_t>(dst) & 31) == 0) {  // 32-byte stores (callers align to 16)
      const int grid = resident_grid<unpack32_direct_kernel<BITS, SIGNED>>(ntiles * 32, kThreads);
      unpack32_direct_kernel<BITS, SIGNED><<<grid, kThreads, 0, s>>>(src, dst, ntiles * 32);
      return cudaGetLastError();
    }
  }
  const int grid = resident_grid<unpack32_vec_kernel<BITS, SIGNED>>(ntiles * 32, kThreads);
  unpack32_vec_kernel<BITS, SIGNED><<<grid, kThreads, 0, s>>>(src, dst, ntiles);
  return cudaGetLastError();
}

constexpr int64_t kMostWords = int64_t(1) << 30;  // words of one rows launch (32-bit indexes)

RowsArgs rows_args(samd_fmt f, int64_t rows, int64_t inner) {
  RowsArgs a;
  const int64_t wpr = words_per_row(f, inner);
  a.inner = inner;
  a.total_words = static_cast<uint32_t>(rows * wpr);
  a.wpr = static_cast<uint32_t>(wpr);
  a.last_count = static_cast<int>(inner - (wpr - 1) * lanes_per_word(f));
  a.bits = f.bits;
  a.is_signed = f.is_signed;
  a.lane_w = f.bits + f.spacer;
  a.L = lanes_per_word(f);
  a.fd_wpr = make_fastdiv(a.wpr);
  return a;
}

template <auto Kernel, typename S, typename D>
cudaError_t launch_rows(const S *src, D *dst, const RowsArgs &a, int tile, cudaStream_t s) {
  // one tile per block: a block's load, barrier, store chain overlaps those of
  // the others on its SM, and the next block takes its place when it is done
  const int64_t tiles = (static_cast<int64_t>(a.total_words) + tile - 1) / tile;
  Kernel<<<grid_for(tiles, 1, 1 << 20), kThreads, 0, s>>>(src, dst, a);
  return cudaGetLastError();
}

template <typename W>
cudaError_t pack_rows(samd_fmt f, const int8_t *src, W *dst, int64_t rows, int64_t inner, cudaStream_t s) {
  const RowsArgs a = rows_args(f, rows, inner);
  if (f.spacer != 0) return launch_rows<pack_rows_kernel<W, 0>>(src, dst, a, any_tile_words(a.L), s);
  switch (f.bits) {
#define SAMD_PACK_CASE(B) \
  case B: return launch_rows<pack_rows_kernel<W, B>>(src, dst, a, tile_words(WordTraits<W>::kBits / B), s);
    SAMD_PACK_CASE(1) SAMD_PACK_CASE(2) SAMD_PACK_CASE(3) SAMD_PACK_CASE(4)
    SAMD_PACK_CASE(5) SAMD_PACK_CASE(6) SAMD_PACK_CASE(7) SAMD_PACK_CASE(8)
#undef SAMD_PACK_CASE
    default: return cudaErrorInvalidValue;
  }
}

template <typename W>
cudaError_t unpack_rows(samd_fmt f, const W *src, int8_t *dst, int64_t rows, int64_t inner, cudaStream_t s) {
  const RowsArgs a = rows_args(f, rows, inner);
  if (f.spacer != 0) return launch_rows<unpack_rows_kernel<W, 0, false>>(src, dst, a, any_tile_words(a.L), s);
  switch (f.bits * 2 + (f.is_signed ? 1 : 0)) {
#define SAMD_UNPACK_CASE(B)                                                                                           \
  case 2 * B:                                                                                                         \
    return launch_rows<unpack_rows_kernel<W, B, false>>(src, dst, a, tile_words(WordTraits<W>::kBits / B), s);        \
  case 2 * B + 1:                                                                                                     \
    return launch_rows<unpack_rows_kernel<W, B, true>>(src, dst, a, tile_words(WordTraits<W>::kBits / B), s);
    SAMD_UNPACK_CASE(1) SAMD_UNPACK_CASE(2) SAMD_UNPACK_CASE(3) SAMD_UNPACK_CASE(4)
    SAMD_UNPACK_CASE(5) SAMD_UNPACK_CASE(6) SAMD_UNPACK_CASE(7) SAMD_UNPACK_CASE(8)
#undef SAMD_UNPACK_CASE
    default: return cudaErrorInvalidValue;
  }
}

// Calls launch(first byte, first word, rows, inner) for slices of at most
// kMostWords words that together are the array: whole rows, or parts of one
// row of whole words.
template <typename F>
cudaError_t in_slices(samd_fmt f, int64_t rows, int64_t inner, const F &launch) {
  const int64_t L = lanes_per_word(f), wpr = words_per_row(f, inner);
  if (wpr <= kMostWords) {
    const int64_t step = kMostWords / wpr;
    for (int64_t r = 0; r < rows; r += step) {
      const cudaError_t e = launch(r * inner, r * wpr, rows - r < step ? rows - r : step, inner);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  for (int64_t r = 0; r < rows; ++r)
    for (int64_t w = 0; w < wpr; w += kMostWords) {
      const int64_t left = inner - w * L;
      const cudaError_t e = launch(r * inner + w * L, r * wpr + w, 1, left < kMostWords * L ? left : kMostWords * L);
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

// Words of the vector kernels' bulk (in 32-bit words): spacer-free rows of
// whole 32-bit words, or of whole 64-bit words whose lane width divides 32.
int64_t vec_tiles(samd_fmt f, int64_t rows, int64_t inner) {
  const int L = lanes_per_word(f);
  if (f.spacer != 0 || (rows != 1 && inner % L != 0)) return 0;
  if (f.word_bits == 64 && (f.bits & (f.bits - 1)) != 0) return 0;
  return rows * inner / (32 / f.bits) / 128;  // warp tiles of 32 quads of words
}

// Whether 64-bit words go by pack64_word_kernel.
bool word64_form(samd_fmt f, int64_t rows, int64_t inner) {
  return f.word_bits == 64 && f.spacer == 0 && (f.bits == 1 || f.bits == 2 || f.bits == 5 || f.bits == 6) &&
         (rows == 1 || inner % lanes_per_word(f) == 0);
}

template <typename W>
cudaError_t pack_dispatch(samd_fmt f, const int8_t *src, W *dst, int64_t rows, int64_t inner, cudaStream_t s) {
  if constexpr (sizeof(W) == 8)
    if (word64_form(f, rows, inner)) {
      const int64_t n = rows * inner;
      switch (f.bits) {
        case 1: return launch_pack64_words<1>(src, dst, n, s);
        case 2: return launch_pack64_words<2>(src, dst, n, s);
        case 5: return launch_pack64_words<5>(src, dst, n, s);
        default: return launch_pack64_words<6>(src, dst, n, s);
      }
    }
  if (f.spacer != 0 && lanes_per_word(f) >= 16) {
    const int64_t wpr = words_per_row(f, inner), total = rows * wpr;
    pack_generic_kernel<W><<<grid_for(total, kThreads, sm_count() * 16), kThreads, 0, s>>>(
        src, dst, total, inner, wpr, f.bits, f.bits + f.spacer, lanes_per_word(f));
    return cudaGetLastError();
  }
  const int64_t ntiles = vec_tiles(f, rows, inner);
  if (ntiles > 0) {
    cudaError_t e;
    uint32_t *d32 = reinterpret_cast<uint32_t *>(dst);
    switch (f.bits) {
      case 1: e = launch_pack32_vec<1>(src, d32, ntiles, s); break;
      case 2: e = launch_pack32_vec<2>(src, d32, ntiles, s); break;
      case 3: e = launch_pack32_vec<3>(src, d32, ntiles, s); break;
      case 4: e = launch_pack32_vec<4>(src, d32, ntiles, s); break;
      case 5: e = launch_pack32_vec<5>(src, d32, ntiles, s); break;
      case 6: e = launch_pack32_vec<6>(src, d32, ntiles, s); break;
      case 7: e = launch_pack32_vec<7>(src, d32, ntiles, s); break;
      default: e = launch_pack32_vec<8>(src, d32, ntiles, s); break;
    }
    if (e != cudaSuccess) return e;
    // what is left: fewer than 128 32-bit words of one row
    const int64_t done = ntiles * 128 * (32 / f.bits);
    src += done;
    dst += ntiles * 128 / (sizeof(W) / 4);
    inner = rows * inner - done;
    rows = 1;
    if (inner == 0) return cudaSuccess;
  }
  return in_slices(f, rows, inner, [&](int64_t b, int64_t w, int64_t r, int64_t n) {
    return pack_rows<W>(f, src + b, dst + w, r, n, s);
  });
}

template <typename W>
cudaError_t unpack_dispatch(samd_fmt f, const W *src, int8_t *dst, int64_t rows, int64_t inner, cudaStream_t s) {
  const int64_t ntiles = vec_tiles(f, rows, inner);
  if (ntiles > 0) {
    cudaError_t e;
    const uint32_t *s32 = reinterpret_cast<const uint32_t *>(src);
    switch (f.bits * 2 + (f.is_signed ? 1 : 0)) {
#define SAMD_UV(B)                                                                      \
  case 2 * B: e = launch_unpack32_vec<B, false>(s32, dst, ntiles, s); break;           \
  case 2 * B + 1: e = launch_unpack32_vec<B, true>(s32, dst, ntiles, s); break;
      SAMD_UV(1) SAMD_UV(2) SAMD_UV(3) SAMD_UV(4) SAMD_UV(5) SAMD_UV(6) SAMD_UV(7) SAMD_UV(8)
#undef SAMD_UV
      default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    const int64_t done = ntiles * 128 * (32 / f.bits);
    src += ntiles * 128 / (sizeof(W) / 4);
    dst += done;
    inner = rows * inner - done;
    rows = 1;
    if (inner == 0) return cudaSuccess;
  }
  return in_slices(f, rows, inner, [&](int64_t b, int64_t w, int64_t r, int64_t n) {
    return unpack_rows<W>(f, src + w, dst + b, r, n, s);
  });
}

}  // namespace

cudaError_t launch_pack(samd_fmt f, const int8_t *src, void *dst, int64_t rows, int64_t inner, cudaStream_t s) {
  if (f.word_bits == 32) return pack_dispatch<uint32_t>(f, src, static_cast<uint32_t *>(dst), rows, inner, s);
  return pack_dispatch<uint64_t>(f, src, static_cast<uint64_t *>(dst), rows, inner, s);
}

cudaError_t launch_unpack(samd_fmt f, const void *src, int8_t *dst, int64_t rows, int64_t inner, cudaStream_t s) {
  if (f.word_bits == 32)
    return unpack_dispatch<uint32_t>(f, static_cast<const uint32_t *>(src), dst, rows, inner, s);
  return unpack_dispatch<uint64_t>(f, static_cast<const uint64_t *>(src), dst, rows, inner, s);
}

}  // namespace samd
