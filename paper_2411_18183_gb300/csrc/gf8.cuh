// gf8.cuh -- signatures with byte symbols over GF(2^8) (Section 3.1: a symbol
// is a byte or a double byte).  Field polynomial P8 = x^8 + x^4 + x^3 + x^2 + 1,
// alpha_k = x^k (k = 1..4), symbol p_i = byte i:
//     sig8^k = sum_{i=0}^{l-1} b_i x^(k i),   component k in bits [8(k-1), 8k).
//
// The signature kernel's scheduling (sigkey.cuh) with this field's arithmetic.
// A key is a sequence of 32-bit words of four symbols, D_b(y) = sum_t bit_b(v_t)
// y^t for each bit position b = 8 c + e, and
//     sig8^k = sum_c x^(k c) sum_e x^e D_(8c+e)(x^(4k)).
// For k = 1, 2, 4 the points x^4, x^8, x^16 are conjugates of x, for k = 3
// x^12 is one of x^3; both minimal polynomials divide a trinomial, x^21 + x^10 +
// 1 and x^11 + x^5 + 1, so that the division in quotient form (quotient.cuh)
// takes one three-input XOR per word and divisor: 16 logic operations per
// 32-byte block for all four components.  At the end of a key the remainders
// are reduced to 8 coefficients modulo the minimal polynomials, still for all
// bit positions at once, and evaluated by Horner's rule; the key's start in its
// block leaves a factor x^(k a), taken off in the logarithm.
//
// 1M keys of 200-2000 bytes (1.1 GB): 1676 us with one thread per key and four
// bytes per table step, 215 us in this form (5.1 TB/s).  Relations of short keys
// still take a thread per key (by_thread).
#pragma once
#include <cstdint>

#include "sigkey.cuh"

namespace algsig {

constexpr uint32_t kPoly8 = 0x11Du;
constexpr int kOrder8 = 255;

__host__ __device__ __forceinline__ uint32_t gf8_times_x(uint32_t a) {
  a <<= 1;
  return (a & 0x100u) ? (a ^ kPoly8) : a;
}

// The reduction tables' entries {b x^8 mod P8 ^ b << 8, b x^16 mod P8 ^ b << 16} (as gf16.cuh's,
// one byte further down), and the logarithms: log[256], then antilog[512] (two periods)
__device__ uint2 g_red8[256];
constexpr int kLog8Bytes = 256 + 512;
__device__ uint4 g_log8[kLog8Bytes / 16];

// PRMT selectors: byte 1 or byte 2 of u into the index's byte 1
constexpr uint32_t kSel8 = 0x5514u;
constexpr uint32_t kSel16b = 0x5524u;

// u < 2^24 -> residue mod P8 (< 256)
template <class Cursor>
__device__ __forceinline__ uint32_t red8_24(uint32_t u, const Cursor& c) {
  return u ^ c.load(tab_index(u, c.off16, kSel8)) ^ c.load(tab_index(u, c.off24, kSel16b));
}
// u < 2^16 -> residue mod P8
template <class Cursor>
__device__ __forceinline__ uint32_t red8_16(uint32_t u, const Cursor& c) {
  return u ^ c.load(tab_index(u, c.off16, kSel8));
}

// Horner's rule on four bytes (b0 lowest) for all four components: a_k x^(4k) +
// b3 x^(3k) + b2 x^(2k) + b1 x^k + b0, at most 8 + 4 k bits before the reduction
template <class Cursor>
__device__ __forceinline__ void gf8_word(uint32_t w, uint32_t (&a)[4], const Cursor& rc) {
  const uint32_t b0 = w & 0xFFu, b1 = (w >> 8) & 0xFFu, b2 = (w >> 16) & 0xFFu, b3 = w >> 24;
  a[0] = red8_16((a[0] << 4) ^ (b3 << 3) ^ (b2 << 2) ^ (b1 << 1) ^ b0, rc);
  a[1] = red8_16((a[1] << 8) ^ (b3 << 6) ^ (b2 << 4) ^ (b1 << 2) ^ b0, rc);
  a[2] = red8_24((a[2] << 12) ^ (b3 << 9) ^ (b2 << 6) ^ (b1 << 3) ^ b0, rc);
  a[3] = red8_24((a[3] << 16) ^ (b3 << 12) ^ (b2 << 8) ^ (b1 << 4) ^ b0, rc);
}

struct Net8 {
  // Short keys, of which the signature kernel's work per key is more than a thread's work per byte: us, one key
  // per thread / staged, 4M keys of 16, 32, 48, 64 bytes 69 / 155, 99 / 155, 131 / 157, 161 / 157; half to one
  // and a half times 32, 40, 48 bytes 156 / 160, 177 / 160, 203 / 161.  Up to a key or so per thread of the device
  // both are bound by the launch.
  static constexpr uint64_t kThreadFrom = 100000;
  static constexpr uint32_t kThreadBelow = 50;
  static constexpr uint64_t kThreadMost = 1024;
  static constexpr int kPhases = 6;       // the rings of 24 and 16 words close together
  static constexpr int kShort = 0;
  static constexpr size_t kTabBytes = kLog8Bytes;
  __device__ __forceinline__ static const uint2* red_image() { return g_red8; }
  __device__ __forceinline__ static const uint4* tab_image() { return g_log8; }
  // Bytes [s, e) of a key; empty where s >= e
  struct Bytes {
    uint64_t s, e;
  };
  __device__ __forceinline__ static uint4 chunk(const uint8_t* __restrict__ arena, uint64_t at) {
    return __ldg(reinterpret_cast<const uint4*>(arena + at));
  }
  // the last 16-byte chunk of memory that holds one of them
  __device__ __forceinline__ static uint4 last_chunk(const uint8_t* __restrict__ arena, const Bytes& k) {
    return k.e > k.s ? chunk(arena, (k.e - 1) & ~15ull) : make_uint4(0, 0, 0, 0);
  }
  // Their signature's components by Horner's rule over words (realigned to byte s) from the last to the first,
  // 16 bytes of memory at a time; w: their last chunk, mt: lk_fill_masks' rows
  template <class Cursor>
  __device__ __forceinline__ static void by_words(uint32_t (&a)[4], const uint8_t* __restrict__ arena, const Bytes& k,
                                                  uint4 w, const uint4* mt, const Cursor& rc) {
    a[0] = a[1] = a[2] = a[3] = 0;
    if (k.e <= k.s) return;
    const uint32_t sh = 8u * ((uint32_t)k.s & 3u), w0 = ((uint32_t)k.s & 15u) >> 2;
    const uint4 m = mt[(((uint32_t)k.e - 1u) & 15u) + 1u];
    w.x &= m.x; w.y &= m.y; w.z &= m.z; w.w &= m.w;
    uint32_t above = 0;                                // the first word of the chunk above
    for (uint64_t at = (k.e - 1) & ~15ull;; at -= 16) {
      const bool first = at <= k.s;
      const uint4 below = first ? w : chunk(arena, at - 16);
      const uint32_t from = first ? w0 : 0u;           // the first chunk's words from byte s on
      gf8_word(__funnelshift_r(w.w, above, sh), a, rc);
      if (from <= 2u) gf8_word(__funnelshift_r(w.z, w.w, sh), a, rc);
      if (from <= 1u) gf8_word(__funnelshift_r(w.y, w.z, sh), a, rc);
      if (from == 0u) gf8_word(__funnelshift_r(w.x, w.y, sh), a, rc);
      if (first) break;
      above = w.x;
      w = below;
    }
  }
  // One key per thread.  The next key's last chunk and the offsets of the one after it are on their way
  // meanwhile.  A key of more than kThreadMost bytes, of which the places looked at showed none, is cut
  // into 32 pieces for the warp: piece p is worth x^(k p) times its own signature, p its first byte's place.
  template <class Cursor>
  __device__ __forceinline__ static void by_thread(const uint8_t* __restrict__ arena, const uint64_t* __restrict__ off,
                                                   uint64_t n, uint64_t* __restrict__ out, const uint4* mt,
                                                   const uint8_t* lg, const Cursor& rc) {
    auto key = [&](uint64_t i) { return i < n ? Bytes{__ldg(off + i), __ldg(off + i + 1)} : Bytes{0, 0}; };
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    Bytes k = key(i), k1 = key(i + stride);
    uint4 w = last_chunk(arena, k);
    for (; __any_sync(0xFFFFFFFFu, i < n); i += stride) {
      const Bytes k2 = key(i + 2 * stride);
      const uint4 w1 = last_chunk(arena, k1);
      const bool many = k.e - k.s > kThreadMost;
      uint32_t a[4];
      by_words(a, arena, many ? Bytes{0, 0} : k, w, mt, rc);
      for (uint32_t left = __ballot_sync(0xFFFFFFFFu, many); left; left &= left - 1u) {
        const int l = __ffs((int)left) - 1;
        const uint64_t s = __shfl_sync(0xFFFFFFFFu, k.s, l), e = __shfl_sync(0xFFFFFFFFu, k.e, l);
        const uint64_t each = ((e - s + 15) / 32 + 16) & ~15ull, from = (s & ~15ull) + (threadIdx.x & 31u) * each;
        const Bytes piece{max(s, from), min(e, from + each)};
        uint32_t b[4];
        by_words(b, arena, piece, last_chunk(arena, piece), mt, rc);
        const uint32_t at = (uint32_t)((piece.s - s) % kOrder8);
        uint32_t v = times_xe(lg, b[0], at) | times_xe(lg, b[1], 2u * at % kOrder8) << 8 |
                     times_xe(lg, b[2], 3u * at % kOrder8) << 16 | times_xe(lg, b[3], 4u * at % kOrder8) << 24;
        v = __reduce_xor_sync(0xFFFFFFFFu, v);
        if ((int)(threadIdx.x & 31u) == l) {
#pragma unroll
          for (int c = 0; c < 4; ++c) a[c] = (v >> (8 * c)) & 0xFFu;
        }
      }
      if (i < n) out[i] = (uint64_t)(a[0] | (a[1] << 8) | (a[2] << 16) | (a[3] << 24));
      k = k1;
      k1 = k2;
      w = w1;
    }
  }
  uint32_t p[24];                         // digits of the division by x^21 + x^10 + 1
  uint32_t q[16];                         // digits of the division by x^11 + x^5 + 1
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < 24; i++) p[i] = 0;
#pragma unroll
    for (int i = 0; i < 16; i++) q[i] = 0;
  }
  __device__ __forceinline__ void put(uint32_t (&st)[kLKState]) const {
#pragma unroll
    for (int i = 0; i < 24; i++) st[i] = p[i];
#pragma unroll
    for (int i = 0; i < 16; i++) st[24 + i] = q[i];
  }
  __device__ __forceinline__ void get(const uint32_t (&st)[kLKState]) {
#pragma unroll
    for (int i = 0; i < 24; i++) p[i] = st[i];
#pragma unroll
    for (int i = 0; i < 16; i++) q[i] = st[24 + i];
  }
  __device__ __forceinline__ void step(int ph, const uint32_t (&w)[8]) {
#pragma unroll
    for (int i = 7; i >= 0; --i) {
      const int s = 8 * (ph % 3) + i, z = 8 * (ph % 2) + i;
      p[s] = w[i] ^ p[(s + 21) % 24] ^ p[(s + 11) % 24];
      q[z] = w[i] ^ q[(z + 11) % 16] ^ q[(z + 6) % 16];
    }
  }
  // sum_i x^(4 k i) (b0 + x^k b1 + x^2k b2 + x^3k b3)(r_i) mod P8, b_c the bytes of r_i
  template <int K, class Cursor>
  __device__ __forceinline__ static uint32_t horner(uint32_t acc, uint32_t r, const Cursor& rc) {
    const uint32_t b0 = r & 0xFFu, b1 = (r >> 8) & 0xFFu, b2 = (r >> 16) & 0xFFu, b3 = r >> 24;
    const uint32_t u = (acc << (4 * K)) ^ b0 ^ (b1 * c_pow2[K]) ^ (b2 * c_pow2[2 * K]) ^ (b3 << (3 * K));
    return K <= 2 ? red8_16(u, rc) : red8_24(u, rc);   // below 2^(8 + 4 K)
  }
  // component value v at exponent e in [0, 255): x^e v
  __device__ __forceinline__ static uint32_t times_xe(const uint8_t* lg, uint32_t v, uint32_t e) {
    return v ? (uint32_t)lg[256u + lg[v] + e] : 0u;
  }
  template <class Cursor>
  __device__ __forceinline__ uint64_t finish(uint32_t a, const uint8_t* lg, const Cursor& rc) const {
    uint32_t r[21];
#pragma unroll
    for (int i = 0; i < 21; i++) r[i] = p[i] ^ (i >= 10 ? p[i >= 10 ? i - 10 : 0] : 0u);
#pragma unroll
    for (int i = 20; i >= 8; --i) {                    // x^8 = x^4 + x^3 + x^2 + 1
      r[i - 4] ^= r[i];
      r[i - 5] ^= r[i];
      r[i - 6] ^= r[i];
      r[i - 8] ^= r[i];
    }
    uint32_t v1 = 0, v2 = 0, v3 = 0, v4 = 0;
#pragma unroll
    for (int i = 7; i >= 0; --i) {
      v1 = horner<1>(v1, r[i], rc);
      v2 = horner<2>(v2, r[i], rc);
      v4 = horner<4>(v4, r[i], rc);
    }
    uint32_t t[11];
#pragma unroll
    for (int i = 0; i < 11; i++) t[i] = q[i] ^ (i >= 5 ? q[i >= 5 ? i - 5 : 0] : 0u);
#pragma unroll
    for (int i = 10; i >= 8; --i) {                    // y^8 = y^6 + y^5 + y^4 + y^2 + y + 1, y = x^3
      t[i - 2] ^= t[i];
      t[i - 3] ^= t[i];
      t[i - 4] ^= t[i];
      t[i - 6] ^= t[i];
      t[i - 7] ^= t[i];
      t[i - 8] ^= t[i];
    }
#pragma unroll
    for (int i = 7; i >= 0; --i) v3 = horner<3>(v3, t[i], rc);
    // the remainders are of the key's polynomial times x^21 (x^11 for component 3) in the words, x^a in the bytes
    const uint32_t e1 = 2u * kOrder8 - (a + 84u);      // a < 32
    const uint32_t s1 = times_xe(lg, v1, e1 % kOrder8), s2 = times_xe(lg, v2, 2u * e1 % kOrder8);
    const uint32_t s3 = times_xe(lg, v3, (2u * kOrder8 - 3u * (a + 44u)) % kOrder8);
    const uint32_t s4 = times_xe(lg, v4, 4u * e1 % kOrder8);
    return (uint64_t)(s1 | (s2 << 8) | (s3 << 16) | (s4 << 24));
  }
};

}  // namespace algsig
