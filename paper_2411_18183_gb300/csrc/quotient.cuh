// quotient.cuh -- the signature kernel's arithmetic for keys of more than a
// few blocks: polynomial division in quotient form.
//
// As in sigkey.cuh a key is a sequence of 32-bit words v_t (here the aligned
// words of memory, whatever the key's start), D_b(y) = sum_t bit_b(v_t) y^t for
// each of the 32 bit positions b, and all 32 polynomials are handled at once,
// bit b of a register belonging to D_b.  To evaluate the D_b at an element
// with minimal polynomial M they may be reduced modulo any multiple T of M.
// With T = x^N + sum_{j in J} x^j, dividing sum_t v_t x^(t+N) by T gives the
// quotient digits
//     q_t = v_t + sum_{j in J} q_(t+N-j),        t from the last word to 0,
// and the remainder R_i = sum_{j in J, j <= i} q_(i-j), i < N.  A step thus
// writes one register and reads |J| others: two three-input XORs per word when
// T has four or five terms, and nothing moves when the digits sit in a ring of
// registers indexed by t (the blocks' loop is unrolled over the ring).  The
// Horner step on the remainder (sigkey.cuh's xs_chunk) does the same division
// with the remainder as its state, where every step touches N registers.
//   components 1, 2, 4: T = P = x^16 + x^12 + x^3 + x + 1 (five terms);
//   component 3: the minimal polynomial of x^3 (equivalently x^6),
//     x^16 + x^12 + x^11 + x^9 + x^8 + x^4 + x^3 + x^2 + 1, has nine terms, but
//     divides T3 = x^23 + x^13 + x^8 + 1 (four).
// So a 32-byte block takes 32 logic operations for all four components,
// against 50 and the register moves of the remainder form.
//
// A key that starts at an odd byte has its symbols across the words.  Its
// stream shifted by one byte is w_t = (v_(t-1) >> 8) | (v_t << 24); division
// commutes with that (it acts on bit positions and shifts t), so the shift is
// made once, on the digits: q'_t = funnel(q_(t-1), q_t) after one more step
// with a zero word.  An even key takes the same step with q'_t = q_(t-1), so
// that every key's symbol i sits at symbol position s + i with
// s = floor(a / 2) + 2, a being the key's first byte in its block.
#pragma once
#include <cstdint>

namespace algsig {

// The last factor of component k, x^(-k s) times a constant, as a multiplication by
// x^(8 k h - E_k) (table 2 (k - 1) + h, h = 0 or 1) and one by x^(k j), j < 8,
// where 15 - floor(a / 2) = 8 h + j.
constexpr int kInvTables = 8;
constexpr int kInvEntries = kInvTables * 512;
// E_k for the quotient form: x^E_k times a component is what its remainder gives at floor(a / 2) = 15
constexpr int kQExp[4] = {49, 98, 189, 196};          // k (32 + 17) for k = 1, 2, 4; 6 * 23 + 3 * 17
// and for the remainder form (sigkey.cuh), which has no other factor
constexpr int kXExp[4] = {15, 30, 45, 60};

// Powers of two as operands the compiler cannot fold: a left shift by a constant
// is then an integer multiply, on the FMA pipe, beside the logic operations that
// fill the ALU pipe.
__constant__ uint32_t c_pow2[9] = {1u, 2u, 4u, 8u, 16u, 32u, 64u, 128u, 256u};

// One step of Horner's rule for component K: acc x^(2K) + lo + x^K hi (unreduced)
template <int K>
__device__ __forceinline__ uint32_t horner_pair(uint32_t acc, uint32_t lo, uint32_t hi) {
  return (acc * c_pow2[2 * K]) ^ lo ^ (hi * c_pow2[K]);
}

// Components 1, 2 and (NCOMP 4) 4: sum_i x^(2 k i) (lo16(r_i) + x^k hi16(r_i))
// mod P by Horner over i, each 32-bit accumulator reduced before it would overflow
template <int NCOMP, int N, class Cursor>
__device__ __forceinline__ void components_124(const uint32_t (&r)[N], uint32_t (&v)[4], const Cursor& rc) {
  uint32_t a1 = 0, a2 = 0, a4 = 0;
#pragma unroll
  for (int i = N - 1; i >= 0; --i) {
    const uint32_t lo = r[i] & 0xFFFFu, hi = r[i] >> 16;
    const int m = N - i;
    a1 = horner_pair<1>(a1, lo, hi);
    if (m % 8 == 0 || i == 0) a1 = red32(a1, rc);
    a2 = horner_pair<2>(a2, lo, hi);
    if (m % 4 == 0 || i == 0) a2 = red32(a2, rc);
    if constexpr (NCOMP == 4) {
      a4 = horner_pair<4>(a4, lo, hi);
      if (m % 2 == 0 || i == 0) a4 = red32(a4, rc);
    }
  }
  v[0] = a1;
  v[1] = a2;
  v[3] = a4;
}

// The packed signature from the components' values, a key that starts at byte a of its first block
template <int NCOMP, class Cursor>
__device__ __forceinline__ uint64_t place_components(const uint32_t (&v)[4], uint32_t a, const uint16_t* inv,
                                                     const Cursor& rc) {
  const uint32_t up = 15u - (a >> 1), j = up & 7u;
  const uint16_t* tab = inv + (up >> 3) * 512;
  const uint32_t s1 = red24(mulc(tab, v[0]) << j, rc);
  const uint32_t s2 = red32(mulc(tab + 1024, v[1]) << (2u * j), rc);
  uint64_t sig = (uint64_t)(s1 | (s2 << 16));
  if constexpr (NCOMP == 4) {
    const uint32_t s3 = red24(red32(mulc(tab + 2048, v[2]) << (2u * j), rc) << j, rc);
    const uint32_t s4 = red32(red32(mulc(tab + 3072, v[3]) << (2u * j), rc) << (2u * j), rc);
    sig |= (uint64_t)(s3 | (s4 << 16)) << 32;
  }
  return sig;
}

template <int NCOMP>
struct QNet {
  // blocks after which the rings are back at their first register: 16 words, 24 words, both
  static constexpr int kPhases = NCOMP == 4 ? 6 : 2;
  uint32_t p[16];                       // digits of the division by P, by t mod 16
  uint32_t q[NCOMP == 4 ? 24 : 1];      // digits of the division by T3, by t mod 24
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < 16; i++) p[i] = 0;
#pragma unroll
    for (int i = 0; i < (NCOMP == 4 ? 24 : 1); i++) q[i] = 0;
  }
  // the digits to and from a plain array
  template <int N>
  __device__ __forceinline__ void put(uint32_t (&st)[N]) const {
#pragma unroll
    for (int i = 0; i < 16; i++) st[i] = p[i];
#pragma unroll
    for (int i = 0; i < (NCOMP == 4 ? 24 : 1); i++) st[16 + i] = q[i];
  }
  template <int N>
  __device__ __forceinline__ void get(const uint32_t (&st)[N]) {
#pragma unroll
    for (int i = 0; i < 16; i++) p[i] = st[i];
#pragma unroll
    for (int i = 0; i < (NCOMP == 4 ? 24 : 1); i++) q[i] = st[16 + i];
  }
  // the words of block vb (words 8 vb + 7 down to 8 vb), ph = vb mod kPhases
  __device__ __forceinline__ void step(int ph, const uint32_t (&w)[8]) {
#pragma unroll
    for (int i = 7; i >= 0; --i) {
      const int s = 8 * (ph % 2) + i;
      p[s] = w[i] ^ p[s] ^ p[(s + 15) % 16] ^ p[(s + 13) % 16] ^ p[(s + 4) % 16];
      if constexpr (NCOMP == 4) {
        const int z = 8 * (ph % 3) + i;
        q[z] = w[i] ^ q[(z + 23) % 24] ^ q[(z + 15) % 24] ^ q[(z + 10) % 24];
      }
    }
  }
  // the signature of a key that starts at byte a of its first block, after block 0
  template <class Cursor>
  __device__ __forceinline__ uint64_t finish(uint32_t a, const uint16_t* inv, const Cursor& rc) const {
    const uint32_t sh = 8u * (a & 1u);
    uint32_t v[4];
    {
      uint32_t d[16], r[16];
      d[0] = __funnelshift_r(p[15] ^ p[14] ^ p[12] ^ p[3], p[0], sh);
#pragma unroll
      for (int i = 1; i < 16; i++) d[i] = __funnelshift_r(p[i - 1], p[i], sh);
#pragma unroll
      for (int i = 0; i < 16; i++)
        r[i] = d[i] ^ (i >= 1 ? d[i >= 1 ? i - 1 : 0] : 0u) ^ (i >= 3 ? d[i >= 3 ? i - 3 : 0] : 0u) ^
               (i >= 12 ? d[i >= 12 ? i - 12 : 0] : 0u);
      components_124<NCOMP>(r, v, rc);
    }
    if constexpr (NCOMP == 4) {
      uint32_t d[23];
      d[0] = __funnelshift_r(q[22] ^ q[14] ^ q[9], q[0], sh);
#pragma unroll
      for (int i = 1; i < 23; i++) d[i] = __funnelshift_r(q[i - 1], q[i], sh);
      uint32_t a3 = 0;
#pragma unroll
      for (int i = 22; i >= 0; --i) {
        const uint32_t r = d[i] ^ (i >= 8 ? d[i >= 8 ? i - 8 : 0] : 0u) ^ (i >= 13 ? d[i >= 13 ? i - 13 : 0] : 0u);
        a3 = horner_pair<3>(a3, r & 0xFFFFu, r >> 16);
        if ((23 - i) % 2 == 0 || i == 0) a3 = red32(a3, rc);
      }
      v[2] = a3;
    }
    return place_components<NCOMP>(v, a, inv, rc);
  }
};

}  // namespace algsig
