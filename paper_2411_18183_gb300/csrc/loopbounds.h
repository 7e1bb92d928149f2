// loopbounds.h -- loop bounds of the byte comparisons (the exact verification of
// every candidate pair that makes the join exact) and of the signature kernel's
// copies, shared by the device code and host-compiled checks of the bounds.
//
// A comparison of two len-byte keys counts in 32 bits from the aligned 16-byte
// chunk that holds the S key's first byte (that byte at offset sa < 16); the R
// key's bytes sit d < 16 bytes further.  The probe's (compare_some) goes by chunks:
// S chunk c against the R bytes [16 c + d, 16 c + d + 16), from the R chunks c and
// c + 1.  The comparison join's (warp_equal) takes steps of 1024 bytes, and every
// offset a step forms stays below
//     steps * 1024 + d + 16  <=  sa + len + 1023 + 15 + 16,
// which is below 2^32 for every len < kNarrowLen.  Longer keys are compared
// in 64-bit offsets.  The loop is counted in steps, so it ends by
// construction.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define ALGSIG_HD __host__ __device__ __forceinline__
#else
#define ALGSIG_HD inline
#endif

namespace algsig {

constexpr uint32_t kNarrowLen = 0xFFFFF000u;   // keys of 2^32 - 4096 bytes and more: 64-bit offsets

// 1024-byte steps of the 32-bit comparison of a key of len bytes (len < kNarrowLen)
// whose S copy starts at byte sa (< 16) of its aligned chunk
ALGSIG_HD uint32_t narrow_steps(uint32_t sa, uint32_t len) { return (uint32_t)(((uint64_t)sa + len + 1023u) >> 10); }

// the largest offset a step of that comparison forms, plus one (as a 64-bit
// value, so that a check can see whether it fits 32 bits); d < 16 is the R
// key's misalignment
ALGSIG_HD uint64_t narrow_offset_end(uint32_t sa, uint32_t len, uint32_t d) {
  return (uint64_t)narrow_steps(sa, len) * 1024u + d + 16u;
}

// Chunks of the probe's comparison of keys of len < kNarrowLen bytes: the S key
// ends at byte `end`, after nfull whole chunks and rem bytes of another.
ALGSIG_HD uint32_t narrow_end(uint32_t sa, uint32_t len) { return sa + len; }
// which of the two R chunks under whole S chunk c (below nfull), and under the
// partial one (rem > 0), hold a byte of the R key
ALGSIG_HD bool r_low(uint32_t c, uint32_t sa, uint32_t d) { return c > 0u || sa + d < 16u; }
ALGSIG_HD bool r_high(uint32_t c, uint32_t nfull, uint32_t rem, uint32_t d) { return c + 1u < nfull || rem + d > 0u; }
ALGSIG_HD bool r_low_partial(uint32_t nfull, uint32_t sa, uint32_t d) { return (nfull << 4) + 16u > sa + d; }
ALGSIG_HD bool r_high_partial(uint32_t rem, uint32_t d) { return 16u < rem + d; }

// Where a key of len > 0 bytes ends in the signature kernel's blocks of 32
// bytes (four to a step, two 16-byte chunks each), its first byte being byte
// a < 32 of block 0: it has `blocks` blocks, `full` of them with both chunks,
// and `rest` bytes of its last chunk (0: all 16).  Counted in blocks, so that
// every key below 2^32 blocks fits 32 bits (a key of 64 GiB has 2^32 chunks).
struct KeyEnd {
  uint32_t blocks, full, rest;
};
ALGSIG_HD KeyEnd key_end(uint32_t a, uint64_t len) {
  const uint64_t e = a + len, b = (e + 31) >> 5, f = (e + 15) >> 5;
  return {b < 0xFFFFFFFFull ? (uint32_t)b : 0xFFFFFFFFu, (uint32_t)f, (uint32_t)e & 15u};
}
// whether chunk q of eight of step s is the key's; have: `blocks` for the even chunks, `full` for the odd ones
ALGSIG_HD bool has_chunk(uint32_t s, uint32_t q, uint32_t have) { return 4u * s + (q >> 1) < have; }
// step of the key's last chunk, and its place of eight in it
ALGSIG_HD uint32_t last_step(uint32_t blocks) { return (blocks - 1u) >> 2; }
ALGSIG_HD uint32_t last_place(uint32_t blocks, uint32_t full) {
  return 2u * ((blocks - 1u) & 3u) + (full == blocks ? 1u : 0u);
}

}  // namespace algsig
