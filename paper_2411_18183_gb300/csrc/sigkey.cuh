// sigkey.cuh -- the signature kernel: one key per lane, keys grouped by
// length, components 1, 2 and 4 from a bit-sliced GF(2) Horner state.
//
// Arithmetic (Section 3.1: sig^k = sum_i p_i x^(k i), k = 1..4).  A key is
// read as 32-bit words v_t = p_{2t} | p_{2t+1} << 16 of its realigned stream
// (shifted by one byte when the key starts at an odd byte, so that symbols
// sit on 16-bit boundaries; word 0 starts at the key's first 32-byte block).
// Bit b of v_t is bit b of symbol 2t (b < 16) or bit b-16 of symbol 2t+1.
// For each of the 32 bit positions b ("planes") let
//     D_b(y) = sum_t bit_b(v_t) y^t,   a polynomial over GF(2).
// Then, with weights W_k(b) = x^b (b < 16) and x^(b - 16 + k) (b >= 16),
//     sig^k = sum_b W_k(b) D_b(x^(2k)).
// For k = 1, 2, 4 the exponent 2k is a power of two, and evaluating a GF(2)
// polynomial commutes with squaring (Frobenius): D_b(x^(2k)) = D_b(x)^(2k).
// So the 32 field elements S_b = D_b(x) determine components 1, 2 and 4.
// They are kept transposed ("bit-sliced"): register c_m holds, in bit b,
// coefficient m of S_b.  Horner's rule over the words, from the last to the
// first, S <- S * x + v_t, is then a fixed XOR network on the 16 registers
// (multiplication by x shifts the registers and folds c_15 back through
// x^16 = x^12 + x^3 + x + 1), 12 logic operations per 16 bytes for all 32
// planes at once.  At the end of the key,
//     sig^k = sum_m x^(2 k m) (lo16(c_m) + x^k hi16(c_m))   (mod P),
// since S_b^(2k) = sum_m c_m[b] x^(2 k m).  Component 3 (2k = 6 is not a power
// of two) has its own bit-sliced state over theta = x^1536, a Frobenius
// conjugate of x^3 (so D_b(x^6) is a fixed GF(2)-linear image of D_b(theta)),
// kept in a basis of GF(2^16) where its Horner step is 13 logic operations per
// 16 bytes; xs3_net.h (written by gen_xs3.py) holds that step and the map back
// to polynomial coordinates.  Groups whose keys have at most kLKShort blocks are
// computed this way; longer ones by the same evaluations in quotient form
// (quotient.cuh), 32 instead of 50 logic operations per block and about 70 more
// per key.
//
// Scheduling.  Each warp owns a range of keys with an equal share of the work
// (key bytes + a fixed cost per key; keys cut to a length come in bands, and keys'
// blocks are shared by their bytes) and walks it in windows of kLKWin keys.  A
// window's keys are sorted by length (unless all are short), and the warp computes them in groups of
// 32 consecutive sorted keys, one key per lane, so the lanes of a group have
// (nearly) the same amount of work.  Keys are taken in 32-byte blocks from the
// last to the first; the lanes of a group whose keys are shorter start later,
// so all lanes reach their first block in the group's last step and finish the
// signatures together.
//
// Loads.  A step is 4 blocks (128 bytes) of each of the group's keys.  The warp
// copies them into its shared-memory rows (one row per key) by 16-byte
// asynchronous copies, eight consecutive lanes to a key, so that a request
// covers up to a whole 128-byte line; then each lane reads its own row.  With
// every lane loading its own key's 32-byte blocks into registers instead, a
// warp load is 32 requests of one sector each, and keys of 256-1024 bytes stop
// at 4.2 TB/s whatever the arithmetic, the order of the keys or the bytes in
// flight (fixed-length keys, 5.1 TB/s); the copies alone reach 5.8 TB/s in the
// same order.  Steps are two or three ahead of the arithmetic, and the next
// group's first steps are requested before a group's signatures are finished.
// Copies are of the 16-byte chunks of a key's 32-byte blocks up to its last
// byte; nothing outside the arena's readable range is touched, and the rest of
// a row is zero-filled.
// Measured (signatures of 2M keys of 256-1024 bytes, 1.28 GB: 346 us with the
// register loads and the remainder form, 265 us now, 4.8 TB/s; 300k keys of
// 2048-8192 bytes, two components: 375 and 277 us; 4M keys of 32-128 bytes: 204
// and 181 us, bound by the arithmetic and the shared-memory wavefronts per key).
// In a batch the keys are the joins' row ranges back to back ("virtual
// rows"): the warps split them by work across the joins, and a window
// ends with its join's rows so that its keys are consecutive in the relation.
#pragma once
#include <cstdint>

#include "quotient.cuh"
#include "xs3_net.h"

namespace algsig {

// image of the shared-memory constant-multiply tables (quotient.cuh): those of
// the quotient form, then those of the remainder form; set up once per device
__device__ uint4 g_inv[4 * kInvEntries / 16];
// entries of the reduction tables (gf16.cuh): {T16[b], T24[b]}; set up once per device
__device__ uint2 g_red16[256];

// Kernel shapes: warps per block (one block per SM) and 32-byte blocks of each
// key in flight (a multiple of 4, one step).  The batch autotuner picks one per
// batch.  Shape 0 is the default of single relations.
struct LKShape {
  int warps, depth;
};
constexpr LKShape kLKShapes[] = {{16, 8}, {10, 12}, {8, 16}};
constexpr int kLKShapeCount = sizeof(kLKShapes) / sizeof(kLKShapes[0]);
constexpr int kLKWin = 256;                           // most keys of a sorting window
// A window whose keys have kLKNarrowFrom bytes or more on average is cut to
// kLKNarrowWin keys: neighbouring keys share a 128-byte line of DRAM, and with the
// larger window the line is often gone from L2 when the second key is read
// (2M keys of 256-1024 bytes: 1.47 GB read for 1.28 GB of keys, 283 against
// 271 us); for keys of 32-128 bytes the sort's share counts (197 against 205 us).
constexpr int kLKNarrowWin = 128;
constexpr uint64_t kLKNarrowFrom = 256;
// relations of this many keys and more are split over the warps by work (a
// search in the offsets); smaller ones by key count, which saves the search's
// dependent loads where they would be a large share of the kernel's time
constexpr uint64_t kLKSearchFrom = 1ull << 19;
// A key's work in key-byte equivalents is its length + kLKKeyCost: short keys
// cost their arithmetic (80 bytes as much as 240 of long ones), long ones their
// bytes.  The warps' shares are cut on it, so that a relation (or batch) that
// mixes short and long keys leaves no warp with far more work than the others
// (a batch of joins of 32-128, 256-1024 and 2048-8192 bytes: 1.51, 1.45, 1.39,
// 1.38 and 1.37 ms with 140, 170, 200, 240 and 300).
constexpr uint64_t kLKKeyCost = 256;

struct LKWarp {
  uint64_t woff[kLKWin + 2];       // offsets of the window's keys (woff[i] = off[wb + i]), i <= wn
  uint64_t full, rest_lo, rest_hi; // keys cut to a length: the end of the full bands, the warp's keys after them
  uint64_t pad;
  uint8_t order[kLKWin];           // window entries by block count
};
static_assert(kLKWin == 256, "the window sort: 8 entries and 8 bins per lane, entries in a byte");
constexpr int kLKStep = 4;                            // blocks per step
constexpr int kLKRow = 32 * kLKStep;                  // bytes of a key's row
constexpr int kLKPitch = 2 * kLKRow;                  // rows of two stages, or of a stage and a table, side by side
constexpr int kLKState = 40;                          // state registers of a key: 16 + 16 or 16 + 24
// groups of at most this many blocks take lk_short_blocks (at most one step; 4M keys of 32-128 bytes:
// 201, 199, 193 and 197 us with 0, 2, 3 and 4)
constexpr int kLKShort = 3;
// and windows whose keys all have at most as many are not sorted: a group's blocks beyond a key's own cost less
// than the sort, whose counters few bins share (us, 4M keys, two components, sorted / not: empty 95 / 81, 0-6 bytes
// 103 / 93, 12-36 108 / 99, equal ones of 64 104 / 89).  Asked of windows of kLKAsk bytes a key at most, and by the
// block length of items.
constexpr uint32_t kLKUnsorted = kLKShort, kLKAsk = 64;

// Shared memory: 256-byte lines of two halves.  The lower halves of the first
// 256 lines hold the reduction tables (16 copies of each entry).  A warp's
// stages are 32 rows each in one column of halves, one after the other: the
// upper halves beside the tables serve the first 8 / stages warps, the lines
// after them two warps side by side.  Then the constant-multiply tables, the
// byte masks and the warps' windows.
constexpr size_t kSmemLKMasks = 17 * 16;
constexpr size_t kSmemLKLook = 48;                    // an LKLook (not static: dynamic shared memory starts at 0x400)
constexpr uint32_t kLKStageBytes = 32 * kLKPitch;     // from one stage of a warp to the next
__host__ __device__ constexpr size_t lk_line_bytes(int warps, int depth) {
  const int stages = depth / kLKStep, beside = 8 / stages;
  return (size_t)256 * kLKPitch + (size_t)((warps > beside ? warps - beside : 0) + 1) / 2 * stages * kLKStageBytes;
}
template <class Net>
__host__ __device__ constexpr size_t lk_smem_bytes(int warps, int depth) {
  return lk_line_bytes(warps, depth) + Net::kTabBytes + kSmemLKMasks + kSmemLKLook + (size_t)warps * sizeof(LKWarp);
}
// byte offset of a warp's first stage
template <int kStages>
__device__ __forceinline__ uint32_t lk_stage_base(uint32_t w) {
  constexpr uint32_t kBeside = 8 / kStages;
  if (w < kBeside) return w * kStages * kLKStageBytes + kLKRow;
  const uint32_t j = w - kBeside;
  return 256u * kLKPitch + (j >> 1) * kStages * kLKStageBytes + (j & 1u) * kLKRow;
}

__device__ __forceinline__ void cp_async8(void* smem_dst, const void* gmem_src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(gmem_src) : "memory");
}
// the 16 bytes at src + s * step to shared memory; zeros (nothing read) where c >= n
__device__ __forceinline__ void cp_async16_below(uint32_t smem_dst, const uint8_t* src, uint32_t s, uint32_t step,
                                                 uint32_t c, uint32_t n) {
  asm volatile(
      "{\n.reg .pred p;\n.reg .u64 a;\n"
      "setp.ge.u32 p, %4, %5;\n"
      "mad.wide.u32 a, %2, %3, %1;\n"
      "cp.async.cg.shared.global [%0], [a], 16, p;\n}\n" ::"r"(smem_dst), "l"(src), "r"(s), "r"(step), "r"(c), "r"(n)
      : "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait_but() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts128(uint32_t addr, const uint4& v) {
  asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// Table cursors of the half-line tables (red32 and red24 of gf16.cuh): 16
// copies of each entry, lanes l and l + 16 share one.  Lookups take two bank
// cycles instead of one, 26 lookups of a pair per 32 keys, and the tables half
// the shared memory and half the time to copy.
template <bool AT400>
struct LKCursor {
  uint32_t tab, off16, off24;
  __device__ __forceinline__ explicit LKCursor(const uint8_t* smem) {
    tab = (uint32_t)__cvta_generic_to_shared(smem);
    off16 = 4u * (threadIdx.x & 15u);
    off24 = off16 + 64u;
  }
  __device__ __forceinline__ uint32_t load(uint32_t idx) const {
    if constexpr (!AT400) return lds32(tab + idx);
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+1024];" : "=r"(v) : "r"(idx));
    return v;
  }
};

// Bit-sliced Horner step over one 16-byte chunk (words v0..v3, v3 last in the
// key): S <- S x^4 + v3 x^3 + v2 x^2 + v1 x + v0, with x^16 = x^12 + x^3 + x + 1.
__device__ __forceinline__ void xs_chunk(uint32_t (&c)[16], uint32_t v0, uint32_t v1, uint32_t v2, uint32_t v3) {
  const uint32_t n0 = c[12] ^ v0;
  const uint32_t n1 = c[12] ^ c[13] ^ v1;
  const uint32_t n2 = c[13] ^ c[14] ^ v2;
  const uint32_t n3 = c[12] ^ c[14] ^ c[15] ^ v3;
  const uint32_t n4 = c[0] ^ c[13] ^ c[15];
  const uint32_t n5 = c[1] ^ c[14];
  const uint32_t n6 = c[2] ^ c[15];
  const uint32_t n12 = c[8] ^ c[12];
  const uint32_t n13 = c[9] ^ c[13];
  const uint32_t n14 = c[10] ^ c[14];
  const uint32_t n15 = c[11] ^ c[15];
  c[15] = n15; c[14] = n14; c[13] = n13; c[12] = n12;
  c[11] = c[7]; c[10] = c[6]; c[9] = c[5]; c[8] = c[4]; c[7] = c[3];
  c[6] = n6; c[5] = n5; c[4] = n4; c[3] = n3; c[2] = n2; c[1] = n1; c[0] = n0;
}

// Component 3 from its bit-sliced state: with p_i = the poly coordinate i of
// every D_b(x^6) (bit b), sum_i x^i (lo16(p_i) + x^3 hi16(p_i)) mod P, by
// Horner over i with a 32-bit accumulator reduced once on the way.
template <class Cursor>
__device__ __forceinline__ uint32_t xs3_component(const uint32_t (&c3)[16], const Cursor& rc) {
  uint32_t p[16];
  xs3_to_poly(c3, p);
  uint32_t acc = 0;
#pragma unroll
  for (int i = 15; i >= 0; --i) {
    acc = (acc * c_pow2[1]) ^ (p[i] & 0xFFFFu) ^ ((p[i] >> 16) * c_pow2[3]);   // degree <= 18 + (15 - i)
    if (i == 3) acc = red32(acc, rc);
  }
  return red32(acc, rc);
}

// The longest of 32 neighbouring keys, the mean of that over eight places of the
// relation, or the mean of all keys if that is more: what a thread per key waits
// for.  lk_look, by the whole block, of nine warps or more, puts together in shared
// memory what lk_seen gives after a barrier: a warp looks at a place.  (Of eight keys
// at four places it missed the long ones of a mixed relation often enough: 500k
// keys of 24 bytes, a tenth of 264, byte symbols 81 us by threads, 27 staged; with
// every warp looking at all eight places a call took 1 us longer.)
constexpr uint32_t kLKPlaces = 8;
struct LKLook {
  uint32_t longest[kLKPlaces], mean;
};
static_assert(sizeof(LKLook) <= kSmemLKLook, "the place for it");
__device__ __forceinline__ void lk_look(LKLook& l, const uint64_t* __restrict__ off, uint64_t n) {
  const uint32_t lane = threadIdx.x & 31u, p = threadIdx.x >> 5;
  if (p > kLKPlaces) return;                          // warp-uniform
  if (p == kLKPlaces) {
    if (lane == 0) l.mean = (uint32_t)min((__ldg(off + n) - __ldg(off)) / n, (uint64_t)0x10000000u);
    return;
  }
  const uint64_t i = min(n / (2 * kLKPlaces) * (2 * p + 1) / 32 * 32 + lane, n - 1);
  const uint32_t len = (uint32_t)min(__ldg(off + i + 1) - __ldg(off + i), (uint64_t)0x10000000u);
  const uint32_t longest = __reduce_max_sync(kFull, len);
  if (lane == 0) l.longest[p] = longest;
}
__device__ __forceinline__ uint32_t lk_seen(const LKLook& l) {
  uint32_t sum = 0;
#pragma unroll
  for (uint32_t p = 0; p < kLKPlaces; ++p) sum += l.longest[p] / kLKPlaces;
  return max(sum, l.mean);
}

// A lane's key in the current group.
struct LKKey {
  uint64_t kq;          // key index
  const uint8_t* base;  // 32-byte aligned address of the key's first block
  uint32_t nb;          // 32-byte blocks (0: empty key)
  uint32_t a;           // offset of the key's first byte in its first block (0..31)
  uint32_t full;        // of its blocks, those with both 16-byte chunks (loopbounds.h's key_end)
  uint32_t te;          // key bytes of its last chunk (0: all 16)
  bool valid;
};

// prefetch the offsets of the window starting at key wb (cp.async, one group)
__device__ __forceinline__ void lk_prefetch_window(LKWarp& W, const uint64_t* __restrict__ off, uint64_t wb,
                                                   uint64_t k_hi) {
  const uint32_t lane = threadIdx.x & 31u;
  if (wb < k_hi) {
    const uint64_t left = k_hi - wb;
    const uint32_t wn = left < (uint64_t)kLKWin ? (uint32_t)left : (uint32_t)kLKWin;   // (a window at most)
    for (uint32_t e = lane; e <= wn; e += 32) cp_async8(&W.woff[e], off + wb + e);
  }
  cp_async_commit();
}

// aligned 32-byte blocks that hold the key at absolute address abs
__device__ __forceinline__ uint32_t lk_blocks(uintptr_t abs, uint64_t len) {
  if (len == 0) return 0u;
  const uint64_t nb = ((abs & 31u) + len + 31) >> 5;
  return nb < 0xFFFFFFFFull ? (uint32_t)nb : 0xFFFFFFFFu;
}

// the window's entries as they come
__device__ __forceinline__ void lk_in_order(LKWarp& W) {
  const uint32_t lane = threadIdx.x & 31u, e = 0x08080808u * lane;
  reinterpret_cast<uint2*>(W.order)[lane] = make_uint2(0x03020100u + e, 0x07060504u + e);
  __syncwarp();
}

// order the window's entries by block count: a counting sort over the block
// counts (255 and more share the last bin; the order within a bin is
// arbitrary), so that each group of 32 consecutive entries has keys of
// nearly equal length.  rows: an empty stage, the first 8 rows of which hold
// the bins' counts.  (Short keys are bound by shared-memory wavefronts, 76 % of
// the peak for 4M keys of 32-128 bytes: with the bins moved eight words at a time
// and lk_copy_setup's rows in different banks that call takes 181 us, 197 before.)
template <bool ASK>
__device__ __forceinline__ void lk_sort_window(LKWarp& W, uint8_t* rows, uint32_t wn, uintptr_t arena,
                                               uint64_t cap_len) {
  const uint32_t lane = threadIdx.x & 31u;
  if (wn <= 32) {                                    // one group: nothing to balance
    lk_in_order(W);
    return;
  }
  constexpr int kPer = kLKWin / 32;                   // entries per lane
  auto blocks = [&](uint32_t i) -> uint32_t {
    const uint64_t ks = W.woff[i];
    return lk_blocks(arena + ks, min(W.woff[i + 1] - ks, cap_len));
  };
  if (ASK && min(W.woff[wn] - W.woff[0], cap_len * wn) <= kLKAsk * wn) {
    uint32_t most = 0;
#pragma unroll 1
    for (uint32_t i = lane; i < wn; i += 32) most = max(most, blocks(i));
    if (__reduce_max_sync(kFull, most) <= kLKUnsorted) {
      lk_in_order(W);
      return;
    }
  }
  auto count = [&](uint32_t b) -> uint32_t& {
    return reinterpret_cast<uint32_t*>(rows + (b >> 5) * kLKPitch)[b & 31u];
  };
  uint4* mine = reinterpret_cast<uint4*>(&count(8 * lane));   // the lane's 8 consecutive bins
  mine[0] = mine[1] = make_uint4(0, 0, 0, 0);
  __syncwarp();
  uint32_t bin[kPer], rank[kPer];
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const uint32_t i = lane + 32u * (uint32_t)j;
    bin[j] = 0;
    rank[j] = 0;
    if (i < wn) {
      bin[j] = min(blocks(i), 255u);
      rank[j] = atomicAdd(&count(bin[j]), 1u);
    }
  }
  __syncwarp();
  // exclusive prefix sum over the bins, 8 consecutive bins per lane
  const uint4 h0 = mine[0], h1 = mine[1];
  const uint32_t sum = h0.x + h0.y + h0.z + h0.w + h1.x + h1.y + h1.z + h1.w;
  uint32_t incl = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(kFull, incl, d);
    if (lane >= (uint32_t)d) incl += o;
  }
  const uint32_t b0 = incl - sum, b1 = b0 + h0.x + h0.y + h0.z + h0.w;
  __syncwarp();
  mine[0] = make_uint4(b0, b0 + h0.x, b0 + h0.x + h0.y, b0 + h0.x + h0.y + h0.z);
  mine[1] = make_uint4(b1, b1 + h1.x, b1 + h1.x + h1.y, b1 + h1.x + h1.y + h1.z);
  __syncwarp();
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const uint32_t i = lane + 32u * (uint32_t)j;
    if (i < wn) W.order[count(bin[j]) + rank[j]] = (uint8_t)i;
  }
  __syncwarp();
}

// group g of the window (wb: its first key) into the lanes; returns the
// group's block count (its longest key's, at least 1)
__device__ __forceinline__ uint32_t lk_load_group(LKKey& k, const LKWarp& W, uint64_t wb, uint32_t wn, uint32_t g,
                                                  const uint8_t* arena, uint64_t cap_len) {
  const uint32_t r = 32u * g + (threadIdx.x & 31u);
  k.valid = r < wn;
  k.kq = 0; k.base = arena; k.nb = 0; k.a = 0; k.full = 0; k.te = 0;
  if (k.valid) {
    const uint32_t i = W.order[r];
    const uint64_t ks = W.woff[i], len = min(W.woff[i + 1] - ks, cap_len);
    const uintptr_t abs = reinterpret_cast<uintptr_t>(arena) + ks;
    k.kq = wb + i;
    // blocks start on a 32-byte boundary (a DRAM sector each), but at the arena's first chunk where
    // that lies on an odd 16-byte boundary
    k.base = reinterpret_cast<const uint8_t*>(abs & ~(uintptr_t)31);
    if (k.base < arena) k.base += 16;
    k.a = (uint32_t)(abs - reinterpret_cast<uintptr_t>(k.base));
    if (len) {
      const KeyEnd e = key_end(k.a, len);
      k.nb = e.blocks;
      k.full = e.full;
      k.te = e.rest;
    }
  }
  const uint32_t G = __reduce_max_sync(kFull, k.nb);
  return G < 1u ? 1u : G;
}

// mask of the first e bytes of a chunk, e = 0..16
__device__ __forceinline__ void lk_fill_masks(uint4* mt) {
  for (int e = threadIdx.x; e <= 16; e += blockDim.x) {
    uint32_t m[4];
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const int r = e - 4 * j;
      m[j] = r <= 0 ? 0u : (r >= 4 ? ~0u : ((1u << (8 * r)) - 1u));
    }
    mt[e] = make_uint4(m[0], m[1], m[2], m[3]);
  }
}

// The copies of a group's steps: lane l copies chunk l % 8 of the rows of keys
// l / 8, l / 8 + 4, ..., whose addresses and ends it holds here.
struct LKCopy {
  const uint8_t* src[8];   // base + 16 (l % 8) of the key
  uint32_t have[8];        // the key's blocks that have such a chunk (has_chunk)
};

// chunk c of the lane's row at shared address row (the lane's swizzle folded in)
__device__ __forceinline__ uint32_t lk_chunk(uint32_t row, uint32_t c) { return row ^ (c << 4); }

// the group's keys to the lanes that copy them, through the empty stage at shared address st
__device__ __forceinline__ void lk_copy_setup(LKCopy& y, const LKKey& k, uint32_t st) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t b = reinterpret_cast<uint64_t>(k.base);
  __syncwarp();
  // (a row's place for it is the chunk of the row's number mod 8, so that neighbouring rows' are in different banks)
  sts128(st + kLKPitch * lane + ((lane & 7u) << 4), make_uint4((uint32_t)b, (uint32_t)(b >> 32), k.nb, k.full));
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t r = 4 * i + (lane >> 3);
    const uint4 v = lds128(st + kLKPitch * r + ((r & 7u) << 4));
    y.src[i] = reinterpret_cast<const uint8_t*>((uint64_t)v.x | ((uint64_t)v.y << 32)) + 16 * (lane & 7u);
    y.have[i] = lane & 1u ? v.w : v.z;
  }
  __syncwarp();
}

// request step s of the group's keys into the stage at shared address st
__device__ __forceinline__ void lk_copy_step(const LKCopy& y, uint32_t st, uint32_t s) {
  const uint32_t lane = threadIdx.x & 31u, q = lane & 7u, r = lane >> 3;
  const uint32_t c = 4u * s + (q >> 1);              // has_chunk
  // row 4 i + r, chunk q: its place is q ^ (row % 8), and row % 8 = 4 (i % 2) + r
  const uint32_t d0 = st + r * kLKPitch + ((q ^ r) << 4), d1 = st + r * kLKPitch + ((q ^ (r + 4u)) << 4);
#pragma unroll
  for (int i = 0; i < 8; ++i)
    cp_async16_below((i & 1 ? d1 : d0) + 4 * i * kLKPitch, y.src[i], s, kLKRow, c, y.have[i]);
}

// zero what is not the key's in the rows that hold its ends: the bytes after
// its last (in the step that holds it) and before its first (in step 0)
__device__ __forceinline__ void lk_trim(const LKKey& k, uint32_t row, uint32_t s, const uint4* mt) {
  if (k.te && last_step(k.nb) == s) {
    const uint32_t p = lk_chunk(row, last_place(k.nb, k.full));
    uint4 v = lds128(p);
    const uint4 m = mt[k.te];
    v.x &= m.x; v.y &= m.y; v.z &= m.z; v.w &= m.w;
    sts128(p, v);
  }
  if (s == 0) {
    const uint32_t p = lk_chunk(row, k.a >> 4);
    uint4 v = lds128(p);
    const uint4 m = mt[k.a & 15u];
    v.x &= ~m.x; v.y &= ~m.y; v.z &= ~m.z; v.w &= ~m.w;
    sts128(p, v);
    if (k.a >= 16u) sts128(lk_chunk(row, 0), make_uint4(0, 0, 0, 0));
  }
}

// block b (0..3) of the lane's row
__device__ __forceinline__ void lk_read(uint32_t (&w)[8], uint32_t row, int b) {
  const uint4 u = lds128(lk_chunk(row, 2 * b)), v = lds128(lk_chunk(row, 2 * b + 1));
  w[0] = u.x; w[1] = u.y; w[2] = u.z; w[3] = u.w;
  w[4] = v.x; w[5] = v.y; w[6] = v.z; w[7] = v.w;
}

// the Horner steps of one 32-byte block (its two chunks, the upper one first)
template <int NCOMP>
__device__ __forceinline__ void lk_block(const uint32_t (&w)[8], uint32_t sh, uint32_t& nxt0, uint32_t (&c)[16],
                                         uint32_t (&c3)[16]) {
  uint32_t v[8];
#pragma unroll
  for (int i = 0; i < 7; i++) v[i] = __funnelshift_r(w[i], w[i + 1], sh);
  v[7] = __funnelshift_r(w[7], nxt0, sh);
  nxt0 = w[0];
  xs_chunk(c, v[4], v[5], v[6], v[7]);
  xs_chunk(c, v[0], v[1], v[2], v[3]);
  if constexpr (NCOMP == 4) {
    xs3_chunk(c3, v[4], v[5], v[6], v[7]);
    xs3_chunk(c3, v[0], v[1], v[2], v[3]);
  }
}

// A key's signature from the Horner state of its blocks (values counted from
// the first block's start; the key starts floor(a / 2) symbols later).
template <int NCOMP, class Cursor>
__device__ __forceinline__ uint64_t lk_finish(const uint32_t (&st)[kLKState], uint32_t a, const uint16_t* inv,
                                              const Cursor& rc) {
  uint32_t c[16], c3[16], v[4];
#pragma unroll
  for (int i = 0; i < 16; i++) {
    c[i] = st[i];
    c3[i] = st[16 + i];
  }
  components_124<NCOMP>(c, v, rc);
  if constexpr (NCOMP == 4) v[2] = xs3_component(c3, rc);
  return place_components<NCOMP>(v, a, inv, rc);
}

// The state after a group of keys of at most kLKShort blocks, all of them in
// the row, by the Horner step on the remainders (lk_block): components 1, 2
// and 4's 16 registers, then component 3's.
template <int NCOMP>
__device__ __forceinline__ void lk_short_blocks(uint32_t (&st)[kLKState], const LKKey& k, uint32_t G, uint32_t row) {
  const uint32_t sh = 8u * (k.a & 1u);
  uint32_t nxt0 = 0;
  uint32_t c[16], c3[16];
#pragma unroll
  for (int i = 0; i < 16; i++) c[i] = c3[i] = 0;
#pragma unroll
  for (int vb = kLKShort - 1; vb >= 0; --vb) {
    if ((uint32_t)vb < G) {                           // warp-uniform
      uint32_t w[8];
      lk_read(w, row, vb);
      lk_block<NCOMP>(w, sh, nxt0, c, c3);
    }
  }
#pragma unroll
  for (int i = 0; i < 16; i++) {
    st[i] = c[i];
    st[16 + i] = c3[i];
  }
}

// What the kernel computes: signatures over GF(2^16) with two or four
// components.  A net names its shared-memory tables and has the digit rings and
// finish of the quotient form; kShort: groups of at most this many blocks take
// the remainder form; kThreadBelow: relations of more than kThreadFrom keys shorter
// than this (lk_seen) are signed by Net::by_thread, one key per thread.
template <int NCOMP>
struct Net16 : QNet<NCOMP> {
  static constexpr int kComponents = NCOMP;
  static constexpr int kShort = kLKShort;
  static constexpr uint32_t kThreadBelow = 0;         // (no way with a thread per key)
  static constexpr size_t kTabBytes = 4 * kInvEntries;
  __device__ __forceinline__ static const uint2* red_image() { return g_red16; }
  __device__ __forceinline__ static const uint4* tab_image() { return g_inv; }
  template <class Cursor>
  __device__ __forceinline__ uint64_t finish(uint32_t a, const uint8_t* tab, const Cursor& rc) const {
    return QNet<NCOMP>::finish(a, reinterpret_cast<const uint16_t*>(tab), rc);
  }
};
static_assert(lk_smem_bytes<Net16<4>>(16, 8) <= 232448 && lk_smem_bytes<Net16<4>>(10, 12) <= 232448 &&
                  lk_smem_bytes<Net16<4>>(8, 16) <= 232448,
              "the shapes' shared memory");

// The state after a group of longer keys, by division in quotient form
// (quotient.cuh): the digit rings, in st.  A stage is refilled with the step
// kStages further down once it is computed.  The loop is unrolled over three
// steps (12 blocks), after which the digit rings are at their first registers
// again.  base: shared address of the warp's first stage, row: of the lane's
// row in it; step s waits in stage s % kStages.
template <class Net, int kStages>
__device__ __forceinline__ void lk_long_blocks(uint32_t (&st)[kLKState], const LKKey& k, uint32_t G, const LKCopy& copy,
                                               uint32_t base, uint32_t row, const uint4* mt) {
  constexpr int P = Net::kPhases, U = 3;
  static_assert(U * kLKStep % P == 0, "the rings close over the unrolled steps");
  const uint32_t S = (G + kLKStep - 1) / kLKStep;
  Net net;
  net.clear();
  for (uint32_t s0 = (S - 1) / U * U;; s0 -= U) {
#pragma unroll
    for (int j = U - 1; j >= 0; --j) {
      const uint32_t s = s0 + (uint32_t)j;
      if (s < S) {                                    // warp-uniform
        const uint32_t at = (kStages == U ? (uint32_t)j : s % kStages) * kLKStageBytes;
        cp_async_wait_but<kStages - 1>();
        __syncwarp();
        lk_trim(k, row + at, s, mt);
        uint32_t w[2][8];                             // a block is read while the one above is computed
        lk_read(w[(kLKStep - 1) & 1], row + at, kLKStep - 1);
#pragma unroll
        for (int b = kLKStep - 1; b >= 0; --b) {
          if (b) lk_read(w[(b - 1) & 1], row + at, b - 1);
          // (warp-uniform: false only for the blocks above the longest key's last, in the group's first step)
          if (kLKStep * s + b < G) net.step((kLKStep * j + b) % P, w[b & 1]);
        }
        __syncwarp();
        if (s >= (uint32_t)kStages) lk_copy_step(copy, base + at, s - kStages);
        cp_async_commit();
      }
    }
    if (s0 == 0) break;
  }
  net.put(st);
}

// The window of at most `most` keys starting at key wb (keys below k_hi): returns its key
// count and sets *wa to its first row in the relation.  In a batch the keys are
// virtual rows (the joins' row ranges back to back) and a window ends with its
// join's rows, so that its keys are consecutive rows of the relation.
template <bool BATCH>
__device__ __forceinline__ uint32_t lk_window(const BatchJoin* __restrict__ J, int nj, int s_side, uint64_t wb,
                                              uint64_t k_hi, uint32_t most, uint64_t* wa) {
  uint64_t lim = k_hi;
  *wa = wb;
  if constexpr (BATCH) {
    const int j = s_side ? join_of_virtual<true>(J, nj, wb) : join_of_virtual<false>(J, nj, wb);
    const uint64_t b = s_side ? __ldg(&J[j].s_begin) : __ldg(&J[j].r_begin);
    const uint64_t e = s_side ? __ldg(&J[j].s_end) : __ldg(&J[j].r_end);
    const uint64_t v0 = s_side ? __ldg(&J[j].vs) : __ldg(&J[j].vr);
    *wa = b + (wb - v0);
    if (v0 + (e - b) < lim) lim = v0 + (e - b);
  }
  const uint64_t left = lim - wb;
  return left < (uint64_t)most ? (uint32_t)left : most;
}

// A warp's keys [lo, hi) of n (virtual rows of a batch side, or rows of a
// relation): equal counts of whole groups below kLKSearchFrom keys, for a group
// takes as long with one key as with 32 (100k keys of 64-256 bytes, 41 per warp:
// 14.9 us cut by keys, 11.7 us by groups; 300k keys of 256-1024 bytes, 123 per
// warp: 45.4 and 43.9 us; 100k keys of 2-8 KB: 120 and 102 us), else equal shares
// of the work, key bytes + kLKKeyCost per key (in a batch, over the joins' keys
// back to back).  Whole warp.
template <bool BATCH, int kWarps>
__device__ __forceinline__ void lk_warp_range(const BatchJoin* __restrict__ J, int nj, int s_side,
                                              const uint64_t* __restrict__ off, uint64_t n, uint64_t warp,
                                              uint64_t nwarps, uint64_t* lo, uint64_t* hi) {
  if (n <= 32 * nwarps) {                            // at most one group per warp
    const uint64_t u = (warp % kWarps) * (nwarps / kWarps) + warp / kWarps;   // neighbouring groups on different SMs
    *lo = 32 * u < n ? 32 * u : n;
    *hi = 32 * u + 32 < n ? 32 * u + 32 : n;
    return;
  }
  if (n < kLKSearchFrom) {
    const uint64_t groups = (n + 31) / 32;
    *lo = 32 * (groups * warp / nwarps);             // (64-bit products: a 128-bit division costs 1 us here)
    *hi = 32 * (groups * (warp + 1) / nwarps);
    if (*hi > n) *hi = n;
    return;
  }
  if constexpr (!BATCH) {
    // lanes 0 and 1 look for the two cuts by secant steps from the cut by count: where key lengths are
    // alike all along the relation two or three loads in sequence find a key whose start is off by less
    // than a 64th of a share, against five of the search's for each cut.  (A cut depends on its number
    // alone, so neighbouring warps agree on it.)
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t base = __ldg(off), total = __ldg(off + n) - base + kLKKeyCost * n;
    const uint64_t w = warp + (lane & 1u);
    const uint64_t t = (uint64_t)((unsigned __int128)total * w / nwarps);
    const double per = (double)total / (double)n;     // work per key, > 0
    uint64_t cut = (uint64_t)((unsigned __int128)n * w / nwarps);
    bool found = cut == 0 || cut >= n;
    for (int it = 0; it < 3 && !__all_sync(kFull, found); ++it) {
      if (!found) {
        const double d = (double)t - (double)(__ldg(off + cut) - base + kLKKeyCost * cut);
        if (fabs(d) * 64.0 * (double)nwarps <= (double)total) {
          found = true;
        } else {
          const double c = (double)cut + rint(d / per);
          cut = c <= 0.0 ? 0 : (c >= (double)n ? n : (uint64_t)c);
          if (cut == 0 || cut == n) cut = cut ? n - 1 : 1;   // (n is large here)
        }
      }
    }
    const uint64_t c0 = __shfl_sync(kFull, cut, 0), c1 = __shfl_sync(kFull, cut, 1);
    const bool f0 = __shfl_sync(kFull, (int)found, 0), f1 = __shfl_sync(kFull, (int)found, 1);
    auto search = [&](uint64_t v) -> uint64_t {
      return warp_lower_bound(off, n, base + (uint64_t)((unsigned __int128)total * v / nwarps), kLKKeyCost);
    };
    *lo = f0 ? c0 : search(warp);
    *hi = warp + 1 >= nwarps ? n : (f1 ? c1 : search(warp + 1));
  } else {
    const uint64_t total = s_side ? vcost_of_join<true>(J, nj, kLKKeyCost) : vcost_of_join<false>(J, nj, kLKKeyCost);
    auto cut = [&](uint64_t w) -> uint64_t {
      if (w == 0) return 0;
      if (w >= nwarps) return n;
      const uint64_t t = (uint64_t)((unsigned __int128)total * w / nwarps);
      if (t >= total) return n;
      return s_side ? vcut_in_join<true>(J, off, join_of_vcost<true>(J, nj, t, kLKKeyCost), t, kLKKeyCost)
                    : vcut_in_join<false>(J, off, join_of_vcost<false>(J, nj, t, kLKKeyCost), t, kLKKeyCost);
    };
    *lo = cut(warp);
    *hi = cut(warp + 1);
  }
}

// Keys of which only the first bytes are signed (a prefix join's): the work of a
// range of keys is not to be had from the offsets, and their lengths differ where
// the cap is above some.  So a warp takes kLKBand keys at a time, in bands of
// kLKBand keys per warp over the whole relation (bands' neighbours go to different
// SMs), and what is left, or a relation of less than two bands, in equal counts
// of whole groups.  A run of long keys is then spread over all warps.  (Join on
// prefixes of 4 KB of 2M keys of 64 bytes followed by 60k of 8 KB: 292 us, 836 with one
// range of equally many keys per warp.)
constexpr uint32_t kLKBand = 256;
template <int kWarps>
__device__ __forceinline__ void lk_first_band(LKWarp& W, uint64_t n, uint64_t warp, uint64_t nwarps, uint64_t* lo,
                                              uint64_t* hi) {
  const uint64_t place = (warp % kWarps) * (nwarps / kWarps) + warp / kWarps;
  const uint64_t band = kLKBand * nwarps, full = n < 2 * band ? 0 : n / band * band;
  const uint64_t groups = (n - full + 31) / 32;
  const uint64_t rest_lo = full + 32 * (groups * warp / nwarps);
  uint64_t rest_hi = full + 32 * (groups * (warp + 1) / nwarps);
  if (rest_hi > n) rest_hi = n;
  if ((threadIdx.x & 31u) == 0) {
    W.full = full;
    W.rest_lo = rest_lo;
    W.rest_hi = rest_hi;
  }
  *lo = full ? kLKBand * place : rest_lo;
  *hi = full ? kLKBand * (place + 1) : rest_hi;
}
// the warp's keys after its keys [.., hi); false: none
__device__ __forceinline__ bool lk_next_band(const LKWarp& W, uint64_t nwarps, uint64_t* lo, uint64_t* hi) {
  if (*hi > W.full) return false;
  *lo = *hi + kLKBand * (nwarps - 1);
  *hi = *lo + kLKBand;
  if (*lo >= W.full) {
    *lo = W.rest_lo;
    *hi = W.rest_hi;
  }
  return *lo < *hi;
}

// Keys cut into pieces: key i's pieces of `block` bytes (the last one shorter;
// one for an empty key) are items first[i] .. first[i + 1), first[keys] of them
// in all, and the kernel signs items instead of keys.  Consecutive items are
// consecutive bytes, so that an item ends where the next one starts.
struct LKItems {
  const uint64_t* first = nullptr;
  uint64_t keys = 0;
  uint32_t block = 0;
};

// Whether a relation's cumulative signatures are computed by items (or one key
// per thread or warp, prefix.cuh): a question of the keys' lengths, which only the
// device knows.  An item costs the finish of a signature whatever its length; a
// thread of its own follows a key at 90 instructions per 16 bytes, and a warp's 32
// take as long as their longest.  So what counts is the longest of neighbouring
// keys, the same for every warp of both kernels.  (By the mean length alone, from 128 bytes on, equal keys
// of 130-200 bytes took up to 1.4 times as long as with a thread each, and mixed
// ones of which a tenth are long half the speed they could have.)
// us, items / a thread per key, 500k keys at blocks of 32, 64, 256:
//   equal, 130 bytes    113 / 91     74 / 59     40 / 34
//   equal, 190 bytes    138 / 133    78 / 77     44 / 46
//   65-195 bytes        110 / 107    69 / 78     39 / 43
//   130-390 bytes       201 / 239   115 / 167    66 / 107
//   48, a tenth 528     101 / 176    62 / 129    47 / 99
// With one key or less per thread of the device the threads' latency is all that
// counts (60k equal keys of 190 bytes 28 / 25, 21 / 18, 12 / 13; of 400 bytes 46 / 44,
// 30 / 30, 21 / 21), but for so few that they do not fill it either.
// A warp per key (blocks of 16): 500k of 190 bytes 260 / 299, of 260 404 / 350; 16k of
// 96 bytes 19 / 17, 60k 27 / 40.
__device__ __forceinline__ bool by_items(LKLook& look, const uint64_t* __restrict__ off, uint64_t n, uint32_t block) {
  if (block < 32u) return n > 20000u && __ldg(off + n) - __ldg(off) < 192u * n;
  lk_look(look, off, n);
  __syncthreads();
  return lk_seen(look) >= (n >= (1u << 15) && n <= 5u << 15 ? 280u : 180u);
}

// A warp's items [lo, hi), whole groups of 32 but at the end, and a key at or
// before the one that holds item lo.  Up to a group per warp one group each;
// else equal shares of the work, the items' bytes + kLKKeyCost per item, for
// blocks of more than a few hundred bytes differ in length as keys do.  (2M keys
// of 64 bytes followed by 60k of 8 KB, with equally many items per warp instead:
// 820 us for blocks of 4 KB, 257 now; 500k keys of 200-2000 bytes unchanged.)  Both
// ends are searched for in the same loads, 32 keys at a time.
template <int kWarps>
__device__ __forceinline__ void lk_item_range(const uint64_t* __restrict__ off, const LKItems& it, uint64_t warp,
                                              uint64_t nwarps, uint64_t* lo, uint64_t* hi, uint64_t* key) {
  const uint64_t lane = threadIdx.x & 31u, n = it.keys, items = __ldg(it.first + n);
  if (items <= 32 * nwarps) {
    const uint64_t u = (warp % kWarps) * (nwarps / kWarps) + warp / kWarps;   // neighbouring groups on different SMs
    *lo = min(32 * u, items);
    *hi = min(32 * u + 32, items);
    *key = *lo < *hi ? warp_lower_bound(it.first, n, *lo + 1) - 1 : 0;
    return;
  }
  const uint64_t base = __ldg(off), total = __ldg(off + n) - base + kLKKeyCost * items;
  auto work = [&](uint64_t k) { return __ldg(off + k) - base + kLKKeyCost * __ldg(it.first + k); };   // before key k
  uint64_t t[2], a[2] = {0, 0}, b[2] = {n, n};       // the first key with more work before it than t: in [a, b]
  const uint64_t share = total / nwarps, rest = total - share * nwarps;
#pragma unroll
  for (int j = 0; j < 2; ++j)                        // total (warp + j) / nwarps
    t[j] = share * (warp + j) + (uint32_t)rest * (uint32_t)(warp + j) / (uint32_t)nwarps;
  while (a[0] < b[0] || a[1] < b[1]) {               // warp-uniform
    uint64_t step[2];
    bool before[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      step[j] = (b[j] - a[j] + 31) / 32;
      const uint64_t i = a[j] + lane * step[j];
      before[j] = i < b[j] && work(i) <= t[j];
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {                    // lanes 0..cnt - 1 are before t, the next one is not
      const uint64_t cnt = (uint64_t)__popc(__ballot_sync(kFull, before[j]));
      const uint64_t next = a[j] + cnt * step[j];
      if (cnt) a[j] = next - step[j] + 1;
      b[j] = min(next, b[j]);
    }
  }
  uint64_t cut[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const uint64_t k = a[j] ? a[j] - 1 : 0, f = __ldg(it.first + k);
    const uint64_t in = min((t[j] - work(k)) / (it.block + kLKKeyCost), __ldg(it.first + k + 1) - f);
    cut[j] = min((f + in + 31) / 32 * 32, items);
    if (j == 0) *key = k;
  }
  *lo = cut[0];
  *hi = warp + 1 >= nwarps ? items : cut[1];
}

// the starts of items [wb, wb + wn) and the end of the last one into the
// window; kb: a key at or before the one that holds item wb, moved on to the key
// that holds the last item; guess: keys to look at first, set to the keys the
// window took (whole warp).  The keys' first items and starts are copied into
// the empty stage at rows, up to 128 keys at a time (with 32 keys per wait and
// no copy the call took as long).
__device__ __forceinline__ void lk_item_window(LKWarp& W, uint8_t* rows, const uint64_t* __restrict__ off,
                                               const LKItems& it, uint64_t wb, uint32_t wn, uint64_t& kb,
                                               uint32_t& guess) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t we = wb + wn, k0 = kb;
  // key x of the batch: its first item and its start, in row x / 8
  auto pair = [&](uint32_t x) { return reinterpret_cast<uint64_t*>(rows + (x >> 3) * kLKPitch) + 2 * (x & 7u); };
  for (uint64_t kk = kb;;) {
    const uint32_t want = guess < 16u ? 16u : (guess > 128u ? 128u : guess);
    const uint32_t nk = it.keys - kk < want ? (uint32_t)(it.keys - kk) : want;
    for (uint32_t x = lane; x <= nk; x += 32) {
      cp_async8(pair(x), it.first + kk + x);
      cp_async8(pair(x) + 1, off + kk + x);
    }
    cp_async_commit();
    cp_async_wait_all();
    __syncwarp();
    bool done = false;
    for (uint32_t x0 = 0; x0 < nk && !done; x0 += 32) {
      const uint32_t x = x0 + lane;
      const bool have = x < nk;
      const uint64_t p0 = have ? pair(x)[0] : ~0ull, s = have ? pair(x)[1] : 0;
      const uint64_t p1 = have ? pair(x + 1)[0] : ~0ull;
      // the key's items in the window: [a, a + c)
      const uint64_t a = p0 > wb ? p0 : wb, z = p1 < we ? p1 : we;
      const uint32_t c = have && a < z ? (uint32_t)(z - a) : 0u;
      const bool many = c > 16u;
      for (uint32_t j = 0; __any_sync(kFull, !many && j < c); ++j)
        if (!many && j < c) W.woff[a - wb + j] = s + (a - p0 + j) * it.block;
      for (uint32_t m = __ballot_sync(kFull, many); m; m &= m - 1u) {
        const int l = __ffs((int)m) - 1;
        const uint32_t cl = __shfl_sync(kFull, c, l);
        const uint64_t al = __shfl_sync(kFull, a, l), pl = __shfl_sync(kFull, p0, l), sl = __shfl_sync(kFull, s, l);
        for (uint32_t j = lane; j < cl; j += 32) W.woff[al - wb + j] = sl + (al - pl + j) * it.block;
      }
      const bool last = c > 0u && z == we;             // one key at most
      if (last) W.woff[wn] = min(s + (we - p0) * it.block, pair(x + 1)[1]);
      const uint32_t lm = __ballot_sync(kFull, last);
      if (lm) {
        kb = kk + x0 + (uint64_t)(__ffs((int)lm) - 1);
        done = true;
      }
    }
    __syncwarp();
    kk += nk;
    if (done || kk >= it.keys) break;                  // (some key holds item we - 1)
  }
  guess = kb - k0 < 128u ? (uint32_t)(kb - k0) + 2u : 128u;
}

// A second relation that the same launch signs, with the blocks from `from` on
// (a join's S beside its R: one launch, and the two share the SMs where both
// are small).
struct LKSecond {
  const uint8_t* arena = nullptr;
  const uint64_t* off = nullptr;
  uint64_t n = 0;
  uint64_t* sig_out = nullptr;
  uint32_t from = 0xFFFFFFFFu;
};

// Whose signatures the kernel computes: of the rows of a relation, of the virtual
// rows of one side of a batch (s_side picks S, J and nj describe the joins, and
// sig_out is indexed by virtual row), of the first cap_len bytes of a relation's
// rows, or of the items of its rows.
enum class LKOf { kRows, kBatchRows, kPrefixes, kItems };

template <bool AT400, class Net, int kLKWarps, int kLKDepth, LKOf OF>
__global__ void __launch_bounds__(32 * kLKWarps, 1) sig_key_kernel(const uint8_t* __restrict__ arena,
                                                                const uint64_t* __restrict__ off, uint64_t n,
                                                                uint64_t* __restrict__ sig_out,
                                                                const BatchJoin* __restrict__ J, int nj, int s_side,
                                                                uint64_t cap, const LKItems items = LKItems(),
                                                                const LKSecond second = LKSecond()) {
  constexpr bool BATCH = OF == LKOf::kBatchRows, ITEMS = OF == LKOf::kItems, CAPPED = OF == LKOf::kPrefixes;
  const uint64_t cap_len = CAPPED ? cap : ~0ull;
  extern __shared__ __align__(128) uint8_t smem[];
  constexpr int kStages = kLKDepth / kLKStep;
  static_assert(kLKDepth % kLKStep == 0 && kStages >= 2 && (kStages == 3 || 8 % kStages == 0), "whole steps in flight");
  constexpr size_t kLines = lk_line_bytes(kLKWarps, kLKDepth);
  uint8_t* tab = smem + kLines;
  uint4* mt = reinterpret_cast<uint4*>(smem + kLines + Net::kTabBytes);
  LKLook& look = *reinterpret_cast<LKLook*>(smem + kLines + Net::kTabBytes + kSmemLKMasks);
  LKWarp* warps = reinterpret_cast<LKWarp*>(smem + kLines + Net::kTabBytes + kSmemLKMasks + kSmemLKLook);
  if constexpr (ITEMS) {
    if (!by_items(look, off, n, items.block)) return;
    asm volatile("griddepcontrol.launch_dependents;");   // prefix_rest_kernel, which waits where it has to
  }
  const int wib = threadIdx.x >> 5;
  const uint32_t lane = threadIdx.x & 31u;
  LKWarp& W = warps[wib];
  // the warp's keys and its first window's offsets first, so that their loads overlap the tables' copy
  uint32_t block = blockIdx.x, nblocks = gridDim.x;
  if constexpr (!BATCH && !ITEMS) {
    if (block >= second.from) {
      arena = second.arena;
      off = second.off;
      n = second.n;
      sig_out = second.sig_out;
      block -= second.from;
      nblocks -= second.from;
    } else if (second.from < nblocks) {
      nblocks = second.from;
    }
  }
  const uint64_t warp = (uint64_t)block * kLKWarps + wib;
  const uint64_t nwarps = (uint64_t)nblocks * kLKWarps;
  uint64_t k_lo, k_hi, kb = 0;                      // kb (items): the key of the window's first item
  uint32_t most = kLKWin;
  if constexpr (ITEMS) {
    if (items.block >= kLKNarrowFrom) most = kLKNarrowWin;
    lk_item_range<kLKWarps>(off, items, warp, nwarps, &k_lo, &k_hi, &kb);
  } else {
    if (CAPPED && lane == 0) W.full = 0;            // one range of keys
    if (CAPPED && n > 32 * nwarps)
      lk_first_band<kLKWarps>(W, n, warp, nwarps, &k_lo, &k_hi);
    else
      lk_warp_range<BATCH, kLKWarps>(J, nj, s_side, off, n, warp, nwarps, &k_lo, &k_hi);
  }
  if constexpr (Net::kThreadBelow > 0) {
    if (n > Net::kThreadFrom) lk_look(look, off, n);
  }
  uint64_t wb = k_lo, wa = 0;                       // the current window: first key, its row, key count
  uint32_t wn = k_lo < k_hi ? lk_window<BATCH>(J, nj, s_side, k_lo, k_hi, most, &wa) : 0u;
  if (wn && !ITEMS) lk_prefetch_window(W, off, wa, wa + wn);
  lk_fill_masks(mt);
  for (int i = threadIdx.x; i < (int)(Net::kTabBytes / 16); i += blockDim.x)
    reinterpret_cast<uint4*>(tab)[i] = Net::tab_image()[i];
  // the reduction tables: line b is 16 copies of one entry of b, then 16 of the other
  for (int i = threadIdx.x; i < 256 * 2; i += blockDim.x) {
    const uint2 e = __ldg(Net::red_image() + (i >> 1));
    const uint32_t v = i & 1 ? e.y : e.x;
    uint4* line = reinterpret_cast<uint4*>(smem + (i >> 1) * kLKPitch + (i & 1) * 64);
#pragma unroll
    for (int j = 0; j < 4; ++j) line[j] = make_uint4(v, v, v, v);
  }
  __syncthreads();
  const LKCursor<AT400> rc(smem);
  if constexpr (Net::kThreadBelow > 0) {
    if (n > Net::kThreadFrom && lk_seen(look) < Net::kThreadBelow) {
      cp_async_wait_all();
      Net::by_thread(arena, off, n, sig_out, mt, tab, rc);
      return;
    }
  }
  if (k_lo >= k_hi) return;

  uint8_t* stages = smem + lk_stage_base<kStages>((uint32_t)wib);
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(stages);
  const uint32_t row = base + lane * kLKPitch + ((lane & 7u) << 4);
  uint32_t g = 0, ng = 0, guess = 64;
  LKKey k, k2;
  LKCopy copy;
  // The warp's next group into k2, its first steps requested; returns its block count, 0 when there is
  // none.  The stages are empty and serve as scratch before they are filled.
  auto next_group = [&]() -> uint32_t {
    if (g == ng) {                                    // the next window, as prefetched
      if (ng) {
        wb += wn;
        if (wb >= k_hi && (!CAPPED || !lk_next_band(W, nwarps, &wb, &k_hi))) return 0u;
        wn = lk_window<BATCH>(J, nj, s_side, wb, k_hi, most, &wa);
      }
      g = 0;
      ng = (wn + 31) / 32;
      cp_async_wait_all();
      __syncwarp();
      if constexpr (ITEMS) lk_item_window(W, stages, off, items, wb, wn, kb, guess);
      if (!ITEMS && wn == (uint32_t)kLKWin && min((W.woff[wn] - W.woff[0]) / kLKWin, cap_len) >= kLKNarrowFrom) {
        wn = kLKNarrowWin;
        ng = kLKNarrowWin / 32;
      }
      if (ITEMS && items.block <= 32u * (kLKUnsorted - 1u))
        lk_in_order(W);
      else
        lk_sort_window<!ITEMS>(W, stages, wn, reinterpret_cast<uintptr_t>(arena), cap_len);
    }
    const uint32_t G2 = lk_load_group(k2, W, wb, wn, g, arena, cap_len);
    if (++g == ng) {                                  // the window's offsets are free: fetch the next ones
      __syncwarp();
      uint64_t nb = wb + wn, nh = k_hi, na;
      if (!ITEMS && (nb < nh || (CAPPED && lk_next_band(W, nwarps, &nb, &nh)))) {
        const uint32_t nn = lk_window<BATCH>(J, nj, s_side, nb, nh, most, &na);
        lk_prefetch_window(W, off, na, na + nn);
      }
    }
    lk_copy_setup(copy, k2, base);
    const uint32_t S = (G2 + kLKStep - 1) / kLKStep;
#pragma unroll
    for (uint32_t u = 0; u < (uint32_t)kStages; ++u) {
      if (u < S) lk_copy_step(copy, base + (S - 1 - u) % kStages * kLKStageBytes, S - 1 - u);
      cp_async_commit();
    }
    return G2;
  };
  for (uint32_t G2 = next_group(); G2;) {
    const uint32_t G = G2;
    k = k2;
    uint32_t st[kLKState];
    bool brief = false;
    if constexpr (Net::kShort > 0) {
      brief = G <= (uint32_t)Net::kShort;
      if (brief) {
        cp_async_wait_but<0>();
        __syncwarp();
        lk_trim(k, row, 0, mt);
        lk_short_blocks<Net::kComponents>(st, k, G, row);
        __syncwarp();
      }
    }
    if (!brief) lk_long_blocks<Net, kStages>(st, k, G, copy, base, row, mt);
    // the next group's first steps are in flight while this one's signatures are finished
    G2 = next_group();
    uint64_t sig = 0;
    if constexpr (Net::kShort > 0) {
      if (brief) sig = lk_finish<Net::kComponents>(st, k.a, reinterpret_cast<const uint16_t*>(tab) + kInvEntries, rc);
    }
    if (!brief) {
      Net net;
      net.get(st);
      sig = net.finish(k.a, tab, rc);
    }
    if (k.valid) sig_out[k.kq] = sig;
  }
  cp_async_wait_all();
}

}  // namespace algsig
