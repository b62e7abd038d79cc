// gmp_tile.cu - the decode kernel of libgmp for the default resolution
// (Gompresso-style, arXiv:1606.00519); gmp_decode.cu keeps the kernel whose
// 32-sequence groups and resolution rounds the statistics and the ablation of
// Sec. 5.1 are about.
//
// A pair of warps decodes a block in two phases:
//
//  Phase A, Huffman decoding (Sec. 3.2.1), the first warp: lane j decodes
//  sub-block j (lanes take j, j+32 for K > 32).  A lookup yields up to two
//  literals and the match length after them when their codes fit the table's
//  bits together, so that a sequence takes about one step.  Each sequence
//  becomes an 8-byte record with its literals inside {literal bytes, distance
//  | match length << 16 | literal count << 24}; a longer literal string takes
//  further records of 3 or 4 literals without a match.  In blocks of long
//  literal strings a step looks up to three times, and such records have 5 to 7
//  literals, in their first seven bytes.  Records go to the
//  pair's scratch slot.
//
//  Phase B, LZ77 decompression (Sec. 3.2.2): the first warp lays out groups of
//  64 records, two per lane, while the second writes the group before, 32
//  bytes at a time, one byte per lane (a tile).  The group's literal strings
//  and matches are segments; a bit per segment start and a population count
//  give each byte its segment, and the segment's entry the shared-memory
//  address its byte comes from: the output window, the literals, or the
//  staging of sources older than the window.  Tiles run in output order, so
//  that every byte below a tile is complete when the tile starts and no
//  resolution rounds are needed; four tiles whose sources all lie below the
//  first are written at once.  Sources inside the tile itself (rare) are
//  followed to the byte they repeat by pointer doubling over the warp's lanes.
//  So MRR and DE streams take the same path at the same speed.
//
//  Byte blocks (Gompresso/Byte, Sec. 3.1) run phase B on the stream's own
//  records, with each group's records checked before it is staged, in groups of
//  fewer records where they write more.
//
// What bounds it and what it measured (GB300, 152 SMs): the number of
// instructions with every SM full (2.4 warp instructions per byte of text,
// 61 % of the issue slots), and a block's chain of dependent ones on small
// launches.  The Huffman step without branches, records of 8 bytes with their
// literals inside and stored two at a time (single 8-byte stores cost 0.5 of
// 3.5 ms on 2 x 512 MiB of records; four at a time, whose register moves cost
// more than they save, 2 x 256 MiB of text 1.72 ms against 1.70), and tiles in
// place of per-sequence copies with resolution rounds: 2 x 512 MiB of records,
// MRR and DE in one launch, 4.53 -> 3.48 ms; 2 x 256 MiB of text 2.66 -> 2.15
// (before: gmp_decode.cu).
// A second warp for the writing, which doubles the warps on an SM in the same
// shared memory (16 blocks), and groups of 64 records instead of 32, whose
// layout and hand-over cost little more than one of 32: records 3.37 -> 2.90,
// text 2.08 -> 1.76, 1 GiB of Byte records 3.17 -> 1.90 (the pair alone, with
// groups of 32: 3.36, 2.08, 2.48).  64 registers a thread are what 32 warps
// leave; phase A spills a few of them.
// Every read of the compressed stream is bounds-checked; every loop over
// input data is bounded by sizes checked against the block header; corrupt
// input sets the caller's status word and abandons the block.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <type_traits>

#include "gmp.h"
#include "gmp_decode_common.h"
#include "gmp_internal.h"

namespace gmp {
namespace {

// ---------------------------------------------------------------------------
// Phase A tables.  Literal/length entry of an LLB-bit peek: bits 0-3 code
// bits consumed, 4-5 literals (0..2, in bytes 2 and 3), byte 1 the match (0
// none, else the length; as a signed byte -1 for the end symbol and -2 for
// lengths above the stream's longest match, which leave the fast path).  With an
// 11-bit table a prefix of 12-bit codes has kLongLL set and the two codes as
// 9-bit halves (bits 23-31 for a next bit of 0, 14-22 for 1): byte or match,
// bit 8 for a literal.  Offset entry: byte 0 holds 32 minus the bits of the
// code and its extra bits, byte 1 32 minus the extra bits, the upper half the
// distance base; a prefix of codes longer than the table's bits is kLongOff,
// and the canonical arrays decide (codes of 10 bits and more are about 0.3 %
// of a block's offsets).  No code: a base above every window.
constexpr uint32_t kLongLL = 1u << 7, kLongOff = 0xffffffffu;
constexpr uint32_t kNoOff = 0xffff2020u, kNoMatch = 0x2020u;

// The symbol's part of an entry: a literal's byte, or the match.
__device__ __forceinline__ uint32_t match_code(uint32_t sym, uint32_t max_match) {
  return sym == 256 ? 0xffu : sym - 254u > max_match ? 0xfeu : sym - 254u;
}
__device__ __forceinline__ uint32_t off_entry(uint32_t os, uint32_t len) {
  const uint32_t ne = os < 4 ? 0u : (os >> 1) - 1u;
  const uint32_t base = os < 4 ? os + 1u : ((2u | (os & 1u)) << ne) + 1u;
  return (base << 16) | ((32u - ne) << 8) | (32u - len - ne);
}

// Working space of the table build; overlaid by the bitstream ring.
struct BuildSmem {
  Canon cll;
  uint32_t run[2][16];
  uint16_t sorted_ll[N_LL + 1];
  uint8_t lens[N_LL + N_OFF + 3];
};

constexpr int kLLBits = 11, kOffBits = 9;  // a pair's tables
constexpr uint32_t kChunksAhead = 4;  // 16-byte bitstream chunks held per lane
struct TileSmemA {
  uint32_t ll[1 << kLLBits];
  uint32_t off[1 << kOffBits];
  union {
    uint32_t bits[32][4 * kChunksAhead];
    BuildSmem build;
  } u;
  Canon coff;
  uint16_t sorted_off[N_OFF + 2];
  uint32_t sb_bit[MAX_SUB + 1], sb_seq[MAX_SUB];
};

// Phase B.  The output window `buf` holds at least the last kHist output
// bytes and the group being written: it slides down (by a multiple of 16)
// when a group would not fit.
constexpr uint32_t kHist = 1024;
constexpr uint32_t kGroupRecs = 64;          // records of a group: two per lane, or half of them (Byte blocks: or
constexpr uint32_t kGroupMax = 32 * 68;  // fewer) if they write more than this (4 literals and a match of 64 per record)
constexpr uint32_t kBuf = 5840;
constexpr uint32_t kFlush = 512;    // output bytes per flush (one 16-byte store per lane)
constexpr uint32_t kFarChunks = 32 * 5;  // 16-byte chunks; a 64-byte source spans at most 5 aligned ones
constexpr uint32_t kLitStage = 8 * kGroupRecs;  // Huffman records, with their literals
// A group's staging: its literals, then its far chunks.  Byte groups share it as
// they need: a group is halved until both fit.
constexpr uint32_t kStage = kLitStage + 16 * kFarChunks;
constexpr uint32_t kMarkWords = (kGroupMax + 127) / 128 * 4;
struct TileSmemB {
  uint8_t stage[2][kStage];
  uint32_t seg[2][2 * kGroupRecs];
  uint32_t mark[2][kMarkWords];
  uint8_t buf[kBuf + 32];  // a last tile may write up to 31 bytes past its group
};
struct Window {
  uint32_t g0;       // output position of the next byte
  uint32_t cur;      // its place in buf
  uint32_t base;     // output position of buf[0] (a multiple of 16): g0 - cur
  uint32_t flushed;  // output bytes stored (a multiple of kFlush)
};
// What one warp reads of the caller's descriptors, index and block header and
// hands to the others that decode the block with it.
enum Work : uint32_t { kEnd, kSkip, kByte, kHuffman };
struct Job {
  BlockView view;
  uint8_t* out;
  uint32_t work, file;
};
// What the first warp of a pair hands to the second in phase B, group after
// group.
enum Step : uint32_t { kGroup, kDone, kAbandon };
struct StepMsg {
  uint32_t what, total, shift;  // of a group: its bytes, and what the window slides by before it
};
struct __align__(64) TileSmem {
  union {
    TileSmemA a;
    TileSmemB b;
  } u;
  uint32_t sb_out[MAX_SUB];  // sub-block output start
  uint32_t sb_cnt[MAX_SUB];  // its records
  Job job;
  int32_t result[3];  // of the parts of the table build
  StepMsg step[2];
};
static_assert(kBuf % 16 == 0 && sizeof(TileSmem) % 16 == 0, "16-byte copies");
static_assert(2 * (1023 + 65) <= kGroupMax && 2 * 1023 + 30 + 16 * 2 * 5 <= kStage, "any two records of a Byte block");
static_assert(kFarChunks >= 32 * 5, "any 32 records of a Huffman block");
static_assert(kGroupMax + kFlush + 80 + 16 + kGroupMax <= kBuf, "two groups of the longest matches");
static_assert(sizeof(TileSmem) * 4 + 1024 <= 57 * 1024, "16 pairs per SM in CTAs of 4");

// Both warps of a pair: 64 threads at the pair's hardware barrier (the kernel
// uses no __syncthreads).
__device__ __forceinline__ void pair_sync() {
  asm volatile("bar.sync %0, 64;" ::"r"(threadIdx.x >> 6) : "memory");
}

// First record of sub-block j, whose output starts at `out`: a record covers
// at least 3 bytes of output but for a sub-block's last one, and a corrupt
// stream may write two more; a multiple of 4, which keeps pairs of
// records 16-byte aligned.
__device__ __forceinline__ uint32_t rec_start(uint32_t out, uint32_t j) { return (out / 3 + 7 * j + 3) & ~3u; }

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t lds_u8(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts_u8(uint32_t a, uint32_t v) {
  asm volatile("st.shared.u8 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
// 16 bytes of shared memory, the first n copied, the others zeroed; `on` only.
__device__ __forceinline__ void cp_async16_if(uint32_t smem, const void* gmem, uint32_t n, bool on) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %3, 0;\n@p cp.async.cg.shared.global [%0], [%1], 16, %2;\n}\n" ::"r"(
                   smem),
               "l"(gmem), "r"(n), "r"((uint32_t)on)
               : "memory");
}
// A segment that starts at output byte `at` of its group: its bit in the words
// at `mark` and its entry; `on` only.
__device__ __forceinline__ void segment_if(uint32_t mark, uint32_t at, uint32_t entry_a, uint32_t entry, bool on) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n@p red.shared.or.b32 [%0], %1;\n@p st.shared.u32 [%2], %3;\n}\n" ::"r"(
          mark + ((at >> 3) & ~3u)),
      "r"(1u << (at & 31u)), "r"(entry_a), "r"(entry), "r"((uint32_t)on)
      : "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// One warp: the canonical arrays of a tree (C) and its symbols sorted by
// (length, symbol), from the code lengths.  Returns the number of used
// symbols, or -1 when the lengths do not form a complete prefix code of at
// most 12 bits and are not all zero.
__device__ int build_canon(Canon& C, uint32_t* run, uint16_t* sorted, const uint8_t* lens, int n) {
  const uint32_t lane = lane_id();
  if (lane < 16) { C.cnt[lane] = 0; run[lane] = 0; }
  __syncwarp();
  for (int base = 0; base < n; base += 32) {
    const int s = base + (int)lane;
    const uint32_t L = s < n ? lens[s] : 0u;
    const uint32_t m = __match_any_sync(FULL, L);
    if ((__ffs(m) - 1) == (int)lane) C.cnt[L] += __popc(m);
    __syncwarp();
  }
  uint32_t k = 0, code = 0, id = 0;  // every lane the same
  for (int L = 1; L <= LUT_BITS; L++) {
    const uint32_t c = C.cnt[L];
    if (lane == 0) {
      C.first[L] = code;
      C.idx[L] = id;
    }
    k += c << (LUT_BITS - L);
    id += c;
    code = (code + c) << 1;
  }
  const bool too_long = (C.cnt[13] | C.cnt[14] | C.cnt[15]) != 0;
  __syncwarp();
  if (too_long || (id != 0 && k != (uint32_t)LUT_SIZE)) return -1;
  for (int base = 0; base < n; base += 32) {
    const int s = base + (int)lane;
    const uint32_t L = s < n ? lens[s] : 0u;
    const uint32_t m = __match_any_sync(FULL, L);
    const uint32_t r = __popc(m & ((1u << lane) - 1u));
    if (L) sorted[C.idx[L] + run[L] + r] = (uint16_t)s;
    __syncwarp();
    if (r == 0) run[L] += __popc(m);
    __syncwarp();
  }
  return (int)id;
}

// Length of the code that a TB-bit left-justified value starts with (TB + 1
// when it is longer than TB); lim[L]: end of length L's range.
template <int TB>
__device__ __forceinline__ uint32_t code_length(const uint32_t (&lim)[TB + 1], uint32_t v) {
  uint32_t L = 1;
#pragma unroll
  for (int i = 1; i <= TB; i++) L += (v >= lim[i]) ? 1u : 0u;
  return L;
}

// The two lookup tables from the canonical arrays; threads t of n.
template <int TB>
__device__ __forceinline__ void fill_ll(uint32_t* lut, const Canon& C, const uint16_t* sorted, bool empty,
                                        uint32_t max_match, uint32_t t, uint32_t n) {
  uint32_t lim[TB + 1];
#pragma unroll
  for (int L = 1; L <= TB; L++) lim[L] = (C.first[L] + C.cnt[L]) << (TB - L);
  for (uint32_t e = t; e < (1u << TB); e += n) {
    const uint32_t v = __brev(e) >> (32 - TB);
    const uint32_t L = code_length<TB>(lim, v);
    uint32_t x;
    if (empty) {
      x = 0;
    } else if (L > (uint32_t)TB) {  // the prefix's two 12-bit codes
      const uint32_t i = C.idx[TB + 1] + 2 * v - C.first[TB + 1];
      auto half = [&](uint32_t s) { return s < 256 ? 256u | s : match_code(s, max_match); };
      x = kLongLL | (half(sorted[i]) << 23) | (half(sorted[i + 1]) << 14);
    } else {
      const uint32_t s = sorted[C.idx[L] + (v >> (TB - L)) - C.first[L]];
      if (s >= 256) {
        x = L | (match_code(s, max_match) << 8);
      } else {
        x = L | (1u << 4) | (s << 16);
        // the next code too, if it lies in the remaining bits
        const uint32_t v2 = (v << L) & ((1u << TB) - 1u);
        const uint32_t L2 = code_length<TB>(lim, v2);
        if (L + L2 <= (uint32_t)TB) {
          const uint32_t s2 = sorted[C.idx[L2] + (v2 >> (TB - L2)) - C.first[L2]];
          x = (L + L2) | (s << 16);
          x |= s2 < 256 ? (2u << 4) | (s2 << 24) : (1u << 4) | (match_code(s2, max_match) << 8);
        }
      }
    }
    lut[e] = x;
  }
}
template <int TB>
__device__ __forceinline__ void fill_off(uint32_t* lut, const Canon& C, const uint16_t* sorted, bool empty, uint32_t t,
                                         uint32_t n) {
  uint32_t lim[TB + 1];
#pragma unroll
  for (int L = 1; L <= TB; L++) lim[L] = (C.first[L] + C.cnt[L]) << (TB - L);
  for (uint32_t e = t; e < (1u << TB); e += n) {
    const uint32_t v = __brev(e) >> (32 - TB);
    const uint32_t L = code_length<TB>(lim, v);
    uint32_t x = kLongOff;
    if (empty) x = kNoOff;
    else if (L <= (uint32_t)TB) x = off_entry(sorted[C.idx[L] + (v >> (TB - L)) - C.first[L]], L);
    lut[e] = x;
  }
}

// Phase A of one lane's sub-block (whole warp calls; `act`: the lane has
// one).  The step is straight-line code: a lane that is done takes empty
// entries, and literal and match work run under selects (DENSE: the match's
// lookup is left out when no lane has one), so that the compiler
// can overlap a step's two table latencies with the record's arithmetic.  The
// lane's 16-byte bitstream chunks pass through a ring of four in shared
// memory, copied there by cp.async: asked for every second step, and at most
// 74 bits are taken in two steps (DENSE: every step, 61 bits), so that a chunk
// is not read before the third wait after it was asked for.
struct SubBlock {
  uint32_t pos, bits;      // first bit, size in bits
  uint32_t out, out_n;     // output start and size
  uint32_t seq, seq_n;     // first sequence and count
};
__device__ __forceinline__ void st_global_if(uint2* p, const uint2& v, bool on) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %3, 0;\n@p st.global.v2.u32 [%0], {%1, %2};\n}\n" ::"l"(p),
               "r"(v.x), "r"(v.y), "r"((uint32_t)on)
               : "memory");
}
__device__ __forceinline__ void st_global_16B_if(uint2* p, const uint2& a, const uint2& b, bool on) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %5, 0;\n@p st.global.v4.u32 [%0], {%1, %2, %3, %4};\n}\n" ::"l"(p),
               "r"(a.x), "r"(a.y), "r"(b.x), "r"(b.y), "r"((uint32_t)on)
               : "memory");
}
__device__ __forceinline__ int byte1_signed(uint32_t v) {
  int r;
  asm("prmt.b32 %0, %1, 0, 0x9991;" : "=r"(r) : "r"(v));
  return r;
}
__device__ __forceinline__ uint32_t shl_clamp(uint32_t v, uint32_t n) {  // 0 for n >= 32
  uint32_t r;
  asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));
  return r;
}
__device__ __forceinline__ uint32_t shr_clamp(uint32_t v, uint32_t n) {
  uint32_t r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));
  return r;
}
template <int LLB, int OFB, bool PAIR, bool DENSE>
__device__ __forceinline__ uint32_t huffman_lane(const uint32_t* ll_lut, const uint32_t* off_lut, const Canon& coff,
                                                 const uint16_t* sorted_off, const uint32_t* ring, const uint8_t* bs,
                                                 uint32_t n_chunks, bool act, bool empty, const SubBlock& sb,
                                                 uint32_t n_seq, uint32_t window, uint2* rec, int& err) {
  const uint32_t ring_s = smem_addr(ring);  // 64-byte aligned
  // bit positions are counted from 64, so that a position's word is the one
  // two ahead
  const uint32_t end = sb.pos + sb.bits + 64u, out_end = sb.out + sb.out_n, rec_cap = sb.out_n / 3 + 1;
  uint32_t outp = sb.out;              // output position of the current record
  uint32_t rem = act ? sb.seq_n : 0u;  // sequences to go
  if (rem && empty) {                  // no literal/length code at all
    err = GMP_STATUS_CORRUPT_SYMBOL;
    rem = 0;
  }
  auto chunk_in = [&](uint32_t c, bool ask) {
    const bool in = c < n_chunks;
    cp_async16_if(ring_s | ((c & (kChunksAhead - 1)) * 16u), bs + (in ? 16ull * c : 0ull), in ? 16u : 0u, ask);
  };
  uint32_t pos = sb.pos + 64u;
  uint32_t asked = (sb.pos >> 7) + kChunksAhead;  // chunks below it have been asked for
#pragma unroll
  for (uint32_t k = 0; k < kChunksAhead; k++) chunk_in((sb.pos >> 7) + k, rem != 0);
  cp_async_commit();
  cp_async_wait<0>();
  // the bitstream's word at pos and the two after it
  uint32_t w0 = 0, w1 = 0, w2 = 0;
  if (rem) {
    w0 = ring[(sb.pos >> 5) & 15u];
    w1 = ring[((sb.pos >> 5) + 1u) & 15u];
    w2 = ring[((sb.pos >> 5) + 2u) & 15u];
  }
  auto advance = [&](uint32_t n) {  // n < 32
    const uint32_t np = pos + n;
    const bool next = ((np ^ pos) & 32u) != 0;
    w0 = next ? w1 : w0;
    w1 = next ? w2 : w1;
    if (next) w2 = ring[(np >> 5) & 15u];
    pos = np;
  };
  std::conditional_t<DENSE, uint64_t, uint32_t> lits = 0;  // pending literals, ln8 bits
  uint32_t ln8 = 0, cnt = 0;
  uint2 q2 = make_uint2(0, 0), q3 = q2;  // PAIR: the last two records
  // the entry of a peek
  auto ll_of = [&](uint32_t pk) -> uint32_t {
    uint32_t e = ll_lut[pk & ((1u << LLB) - 1u)];
    if (LLB < LUT_BITS) {
      const uint32_t h = e >> (((pk >> LLB) & 1u) ? 14u : 23u);
      const uint32_t v = h & 255u, x = (h & 256u) ? (v << 16) | 28u : (v << 8) | 12u;
      e = (e & kLongLL) ? x : e;
    }
    return e;
  };
  auto off_long = [&](uint32_t pk2) -> uint32_t {
    const uint32_t x = decode_long<OFB>(coff, sorted_off, pk2 & (LUT_SIZE - 1));
    return x ? off_entry(x & 511u, x >> 9) : kNoOff;
  };
  bool odd = false;  // what the checks after a pair of steps look at
  auto one = [&]() {
    // a lookup, or up to three while they give literals alone and fewer than
    // six of them are pending
    int mc = 0;
#pragma unroll
    for (int k = 0; k < (DENSE ? 3 : 1); k++) {
      uint32_t e = ll_of(__funnelshift_r(w0, w1, pos));
      e = (k == 0 ? rem != 0 : mc == 0 && ln8 < 48u && rem != 0) ? e : 0u;
      mc = k == 0 ? byte1_signed(e) : mc + byte1_signed(e);
      advance(e & 15u);
      lits |= (decltype(lits))(e >> 16) << ln8;
      ln8 += (e >> 1) & 24u;
    }
    const uint32_t pk2 = __funnelshift_r(w0, w1, pos);
    uint32_t e2 = kNoMatch;
    if (!DENSE || __any_sync(FULL, mc > 0)) {
      e2 = off_lut[pk2 & ((1u << OFB) - 1u)];
      e2 = mc > 0 ? e2 : kNoMatch;
      if (OFB < LUT_BITS && __any_sync(FULL, e2 == kLongOff)) {
        if (e2 == kLongOff) e2 = off_long(pk2);
      }
    }
    const uint32_t s1 = e2 & 63u, s2 = __byte_perm(e2, 0, 0x4441);
    const uint32_t dist = (e2 >> 16) + shr_clamp(shl_clamp(pk2, s1), s2);
    advance(32u - s1);
    const uint32_t ml = (uint32_t)max(mc, 0), wpos = outp + (ln8 >> 3);
    odd = odd || mc < 0 || dist > min(window, wpos);
    if (DENSE) {
      // more literals than a match's record takes go out by themselves
      const bool wide = ln8 > 32u, match = mc != 0;
      st_global_if(rec + cnt, make_uint2((uint32_t)lits, (uint32_t)((uint64_t)lits >> 32) | (ln8 << 21)), wide);
      cnt += wide ? 1u : 0u;
      lits = wide ? 0u : lits;
      ln8 = wide ? 0u : ln8;
      st_global_if(rec + cnt, make_uint2((uint32_t)lits, dist | (ml << 16) | (ln8 << 21)), match);
      cnt += match ? 1u : 0u;
      outp = wide || match ? wpos + ml : outp;
      lits = match ? 0u : lits;
      ln8 = match ? 0u : ln8;
    } else {
      const bool emit = mc != 0 || ln8 >= 24u;
      const uint2 r = make_uint2((uint32_t)lits, dist | (ml << 16) | (ln8 << 21));
      if (PAIR) {
        q2 = emit ? q3 : q2;
        q3 = emit ? r : q3;
        cnt += emit ? 1u : 0u;
        st_global_16B_if(rec + (cnt - 2u), q2, q3, emit && (cnt & 1u) == 0);
      } else {
        st_global_if(rec + cnt, r, emit);
        cnt += emit ? 1u : 0u;
      }
      outp = emit ? wpos + ml : outp;
      lits = emit ? 0u : lits;
      ln8 = emit ? 0u : ln8;
    }
    rem -= mc != 0 ? 1u : 0u;
  };
  while (__any_sync(FULL, rem != 0)) {
    const uint32_t pos0 = pos, out0 = outp + (ln8 >> 3), rem0 = rem;
    odd = false;
    one();
    if (!DENSE) one();
    if (__any_sync(FULL, odd || pos > end || outp > out_end)) {
      // an end symbol or a corrupt stream: the step or pair of steps again, with
      // every check.  A lane that runs past its sub-block stops here, which bounds
      // the loop; literals past the sub-block's output are noticed when it ends.
      uint32_t p = pos0, o = out0, left = rem0;
      for (int k = 0; k < (DENSE ? 3 : 2) && left && !err && (!DENSE || p < pos); k++) {
        auto peek = [&]() {
          return __funnelshift_r(ring[((p >> 5) - 2u) & 15u], ring[((p >> 5) - 1u) & 15u], p);
        };
        const uint32_t e = ll_of(peek());
        const int mc = byte1_signed(e);
        p += e & 15u;
        o += (e >> 4) & 3u;
        if (mc > 0 || mc == -2) {
          const uint32_t pk2 = peek();
          uint32_t e2 = off_lut[pk2 & ((1u << OFB) - 1u)];
          if (OFB < LUT_BITS && e2 == kLongOff) e2 = off_long(pk2);
          const uint32_t s1 = e2 & 63u, ml = (uint32_t)mc;
          const uint32_t dist = (e2 >> 16) + shr_clamp(shl_clamp(pk2, s1), __byte_perm(e2, 0, 0x4441));
          p += 32u - s1;
          if (p > end) err = GMP_STATUS_BITSTREAM;
          else if (e2 == kNoOff || mc < 0) err = GMP_STATUS_CORRUPT_SYMBOL;
          else if (dist > window || dist > o) err = GMP_STATUS_BAD_OFFSET;
          else if (ml > out_end - min(o, out_end)) err = GMP_STATUS_OUTPUT_OVERRUN;
          o += ml;
          left--;
        } else if (p > end) {
          err = GMP_STATUS_BITSTREAM;
        } else if (mc < 0) {
          // the end symbol, which only closes the block's last sequence
          if (left != 1u || sb.seq + sb.seq_n != n_seq) err = GMP_STATUS_CORRUPT_SYMBOL;
          left--;
        }
      }
      if (err) rem = 0;
      cnt = min(cnt, rec_cap);
    }
    const bool ask = rem && ((pos - 64u) >> 7) + kChunksAhead > asked;
    chunk_in(asked, ask);
    asked += ask ? 1u : 0u;
    cp_async_commit();
    cp_async_wait<2>();
  }
  cp_async_wait<0>();
  if (PAIR && !DENSE && cnt <= rec_cap) {
    if (cnt & 1u) rec[cnt - 1u] = q3;  // not stored yet
  }
  outp += ln8 >> 3;
  if (!err && pos != end) err = GMP_STATUS_BITSTREAM;
  if (!err && outp != out_end) err = GMP_STATUS_OUTPUT_OVERRUN;
  return cnt;
}

// Whether a block's sequences are long strings of literals: more than 40 bits
// each, of which a match takes about 17 (text and CSV rows: 24 to 26 in all).  A
// step with one lookup decodes a literal or two in what a match takes too (1100
// blocks, us, step of one lookup / of three / gmp_decode.cu: 16 KiB of random
// bytes 3383 / 2010 / 2386; 64 KiB, 12 literals and a match of 9 per sequence
// 693 / 525 / 659, 31 literals 824 / 554 / 751).
__device__ __forceinline__ bool dense(const BlockView& V, uint32_t bs_off) {
  return (V.comp_bytes - bs_off) / 5u > V.n_seq;
}

// Sub-block table: prefix sums of bit sizes, output sizes and sequences over
// the K sub-blocks (one warp), with the totals checked in 64 bits, so that
// no wrapped 32-bit sum passes; sb_bit[K] is the last one's end.  The stream's
// table is read here only: sub_block() has the sizes that were checked, whatever
// a caller writes there meanwhile.  Returns a gmp_status.
__device__ int sub_block_table(const BlockView& V, uint64_t bits_avail, uint32_t* sb_bit, uint32_t* sb_out,
                               uint32_t* sb_seq) {
  const uint32_t lane = lane_id();
  uint32_t carry_bit = 0, carry_out = 0, carry_seq = 0;
  uint64_t tb = 0, to = 0, ts = 0;
  for (uint32_t base = 0; base < V.K; base += 32) {
    const uint32_t j = base + lane;
    uint32_t nb = 0, no = 0, ns = 0;
    if (j < V.K) {
      const uint8_t* e = V.B + 192 + 12 * j;
      nb = ld_u32_nc(e);
      no = ld_u32_nc(e + 4);
      ns = ld_u32_nc(e + 8);
    }
    const uint32_t ib = warp_incl_scan(nb), io = warp_incl_scan(no), is = warp_incl_scan(ns);
    if (j < V.K) {
      sb_bit[j] = carry_bit + ib - nb;
      sb_out[j] = carry_out + io - no;
      sb_seq[j] = carry_seq + is - ns;
    }
    carry_bit += __shfl_sync(FULL, ib, 31);
    carry_out += __shfl_sync(FULL, io, 31);
    carry_seq += __shfl_sync(FULL, is, 31);
    tb += nb;
    to += no;
    ts += ns;
  }
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) {
    tb += __shfl_xor_sync(FULL, tb, d);
    to += __shfl_xor_sync(FULL, to, d);
    ts += __shfl_xor_sync(FULL, ts, d);
  }
  if (lane == 0) sb_bit[V.K] = carry_bit;
  if (ts != V.n_seq || to != V.out_bytes) return GMP_STATUS_BAD_HEADER;
  return tb > bits_avail ? (int)GMP_STATUS_BITSTREAM : 0;
}
__device__ __forceinline__ SubBlock sub_block(const BlockView& V, const uint32_t* sb_bit, const uint32_t* sb_out,
                                              const uint32_t* sb_seq, uint32_t j) {
  if (j >= V.K) return SubBlock{0, 0, 0, 0, 0, 0};
  const bool last = j + 1 == V.K;
  return SubBlock{sb_bit[j], sb_bit[j + 1] - sb_bit[j], sb_out[j], (last ? V.out_bytes : sb_out[j + 1]) - sb_out[j],
                  sb_seq[j], (last ? V.n_seq : sb_seq[j + 1]) - sb_seq[j]};
}

__device__ __forceinline__ void unpack_lens(uint8_t* lens, const uint8_t* B, uint32_t t, uint32_t n) {
  for (uint32_t i = t; i < (uint32_t)(N_LL + N_OFF); i += n) {
    const uint32_t sym = i < (uint32_t)N_LL ? i : i - N_LL;
    const uint8_t v = __ldg(B + (i < (uint32_t)N_LL ? 8 : 168) + (sym >> 1));
    lens[i] = (sym & 1) ? (v >> 4) : (v & 15);
  }
}

// Phase A of one block by the warp pair; false: the block's status is set.
__device__ __forceinline__ bool huffman_block(TileSmem& S, const BlockView& V, int32_t* status, uint2* rec,
                                              uint32_t half) {
  const uint32_t lane = lane_id(), t = 32 * half + lane;
  TileSmemA& A = S.u.a;
  BuildSmem& T = A.u.build;
  const uint32_t bs_off = (192u + 12u * V.K + 15u) & ~15u;  // bitstream start within the block
  unpack_lens(T.lens, V.B, t, 64);
  pair_sync();
  if (half == 0) {
    const int r = build_canon(T.cll, T.run[0], T.sorted_ll, T.lens, N_LL);
    if (lane == 0) S.result[0] = r;
  } else {
    const int r = build_canon(A.coff, T.run[1], A.sorted_off, T.lens + N_LL, N_OFF);
    const int e = sub_block_table(V, (V.comp_bytes - bs_off) * 8ull, A.sb_bit, S.sb_out, A.sb_seq);
    if (lane == 0) {
      S.result[1] = r;
      S.result[2] = e;
    }
  }
  pair_sync();
  const int n_ll = S.result[0], n_off = S.result[1];
  int err = S.result[2] ? S.result[2] : n_ll < 0 || n_off < 0 ? (int)GMP_STATUS_BAD_HEADER : 0;
  if (err) {
    if (t == 0) set_status(status, err);
    return false;
  }
  fill_ll<kLLBits>(A.ll, T.cll, T.sorted_ll, n_ll == 0, V.max_match, t, 64);
  fill_off<kOffBits>(A.off, A.coff, A.sorted_off, n_off == 0, t, 64);
  pair_sync();  // the ring takes the build's place
  if (half == 0) {
    const uint8_t* bs = V.B + bs_off;
    const uint32_t n_chunks = (uint32_t)min((uint64_t)0xffffffffu, (V.comp_bytes - bs_off) / 16);
    for (uint32_t jb = 0; jb < V.K; jb += 32) {
      const uint32_t j = jb + lane;
      const SubBlock sb = sub_block(V, A.sb_bit, S.sb_out, A.sb_seq, j);
      auto decode = [&](auto is_dense) {
        return huffman_lane<kLLBits, kOffBits, true, decltype(is_dense)::value>(
            A.ll, A.off, A.coff, A.sorted_off, A.u.bits[lane], bs, n_chunks, j < V.K, n_ll == 0, sb, V.n_seq, V.window,
            rec + rec_start(sb.out, j), err);
      };
      const uint32_t cnt = dense(V, bs_off) ? decode(std::true_type()) : decode(std::false_type());
      if (j < V.K) S.sb_cnt[j] = cnt;
      // the status is the first damaged sub-block's
      const uint32_t bad = __ballot_sync(FULL, err != 0);
      if (bad) {
        if (lane == (uint32_t)__ffs(bad) - 1u) set_status(status, err);
        err = 1;
        break;
      }
    }
    if (lane == 0) S.result[0] = err;
  }
  pair_sync();  // the records are visible to the first warp, the tables' place is free
  return S.result[0] == 0;
}

// ---------------------------------------------------------------------------
// Phase B.
struct Group {
  uint32_t total, lits, shift;
  int err;
};

__device__ __forceinline__ void slide(uint8_t* buf, Window& w, uint32_t shift) {
  const uint32_t lane = lane_id();
  // ascending strips, each loaded whole before it is stored: a strip's
  // destination ends at or below every later strip's source
  const uint32_t n = w.cur - shift;
  for (uint32_t u = 0; u < n; u += 512u) {
    const uint32_t c = u + 16u * lane;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (c < n) v = *reinterpret_cast<const uint4*>(buf + shift + c);
    __syncwarp();
    if (c < n) *reinterpret_cast<uint4*>(buf + c) = v;
    __syncwarp();
  }
  w.cur -= shift;
  w.base += shift;
}

// Stores the output's whole rows up to w.g0; thread t of n.
__device__ __forceinline__ void flush(const uint8_t* buf, Window& w, uint8_t* out_blk, bool vec_ok, uint32_t t,
                                      uint32_t n) {
  if (w.g0 - w.flushed < kFlush) return;
  const uint32_t end = w.g0 & ~(kFlush - 1u);
  if (vec_ok) {
    for (uint32_t c = w.flushed + 16u * t; c < end; c += 16u * n)
      *reinterpret_cast<uint4*>(out_blk + c) = *reinterpret_cast<const uint4*>(buf + (c - w.base));
  } else {
    for (uint32_t c = w.flushed + t; c < end; c += n) out_blk[c] = buf[c - w.base];
  }
  w.flushed = end;
  __syncwarp();
}

// What is not flushed at the block's end.
__device__ __forceinline__ void flush_rest(const uint8_t* buf, const Window& w, uint8_t* out_blk, bool vec_ok,
                                           uint32_t t, uint32_t n) {
  uint32_t c = w.flushed;
  if (vec_ok) {
    for (uint32_t x = c + 16u * t; x + 16u <= w.g0; x += 16u * n)
      *reinterpret_cast<uint4*>(out_blk + x) = *reinterpret_cast<const uint4*>(buf + (x - w.base));
    c = w.g0 & ~15u;
  }
  for (c += t; c < w.g0; c += n) out_blk[c] = buf[c - w.base];
}

// A Byte group that does not fit the fast path: record after record, one
// warp copying each literal string and each match (window of `cap` bytes,
// `hist` of them kept).  The records, which were checked as a group, are read
// again here: every length is cut to what is left of the output and of the
// literals (up to lits_end), so that a record changed meanwhile stays in them.
__device__ __noinline__ void slow_group(uint8_t* buf, uint32_t cap, uint32_t hist, Window& w, const uint8_t* recs,
                                        uint32_t t0, uint32_t t1, const uint8_t* lits, const uint8_t* lits_end,
                                        uint8_t* out_blk, uint32_t out_bytes, bool vec_ok) {
  const uint32_t lane = lane_id();
  auto room = [&](uint32_t n) {
    if (w.cur + n > cap) slide(buf, w, (w.cur - hist) & ~15u);
  };
  for (uint32_t t = t0; t < t1; t++) {
    const uint32_t r = __shfl_sync(FULL, ld_u32_nc(recs + 4ull * t), 0), m = (r >> 10) & 63u, dist = (r >> 16) + 1u;
    uint32_t left = min(min(r & 1023u, out_bytes - w.g0), (uint32_t)min((uint64_t)1023u, (uint64_t)(lits_end - lits)));
    const uint32_t ml = m && dist <= w.g0 + left ? min(m + 2u, out_bytes - w.g0 - left) : 0u;
    while (left) {
      const uint32_t n = min(left, kFlush);
      room(n);
      for (uint32_t i = lane; i < n; i += 32) buf[w.cur + i] = __ldg(lits + i);
      __syncwarp();
      w.cur += n;
      w.g0 += n;
      lits += n;
      left -= n;
      flush(buf, w, out_blk, vec_ok, lane, 32);
    }
    if (ml) {
      room(ml);
      for (uint32_t i = lane; i < ml; i += 32) {
        // an overlapping copy repeats the dist bytes before it
        const uint32_t src = w.g0 - dist + (dist < ml ? i % dist : i);
        buf[w.cur + i] = src >= w.base ? buf[src - w.base] : (uint8_t)__ldcg(out_blk + src);
      }
      __syncwarp();
      w.cur += ml;
      w.g0 += ml;
      flush(buf, w, out_blk, vec_ok, lane, 32);
    }
  }
}

// The first warp of a pair reads the records and lays out group after group;
// the second writes them.
template <bool BYTE>
__device__ __forceinline__ void lay_out_block(TileSmem& SS, const BlockView& V, int32_t* status, const uint2* rec,
                                              uint8_t* out_blk) {
  TileSmemB& S = SS.u.b;
  const uint32_t lane = lane_id();
  const bool vec_ok = (((uintptr_t)out_blk) & 15u) == 0;
  const uint8_t* recs = V.B + 16;           // Byte blocks: the stream's records
  const uint8_t* lits = V.B + V.lit_off;    // and literals
  const uint32_t buf_a = smem_addr(S.buf);

  // the lane's two records of the group at i0: Huffman blocks {literals,
  // distance | match length << 16 | literal count << 24} of one sub-block,
  // Byte blocks {-, the stream's word}; zero past the end
  uint32_t j = 0, i0 = 0, n_j = 0;  // sub-block, record within it, its records (Byte: the block's)
  const uint2* rec_j = rec;
  if (BYTE) {
    n_j = V.n_seq;
  } else {
    while (j < V.K && (n_j = SS.sb_cnt[j]) == 0) j++;
    if (j < V.K) rec_j = rec + rec_start(SS.sb_out[j], j);
    else n_j = 0;
  }
  auto load = [&]() -> uint4 {
    const uint32_t i = i0 + 2 * lane;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (i < n_j) {
      // whole pairs: Byte blocks' records are followed by padding when their
      // number is odd, and a sub-block's have room for one more
      if (BYTE) {
        const uint2 u = __ldg(reinterpret_cast<const uint2*>(recs + 4ull * i));
        v.y = u.x;
        v.w = u.y;
      } else {
        v = __ldcg(reinterpret_cast<const uint4*>(rec_j + i));
      }
      if (i + 1u >= n_j) v.z = v.w = 0;
    }
    return v;
  };
  auto step = [&](uint32_t n) {  // past n records
    i0 += min(n, n_j - i0);
    if (i0 < n_j || BYTE) return;
    i0 = 0;
    n_j = 0;
    while (++j < V.K && (n_j = SS.sb_cnt[j]) == 0) {}
    if (j < V.K) rec_j = rec + rec_start(SS.sb_out[j], j);
  };

  // records of a group: as many as a group holds of the block's mean ones (16 KiB
  // blocks, 31 literals and a match of 9 per record, 1100 of them: 51 us; with the
  // groups that do not fit written record after record 362; gmp_decode.cu 86)
  uint32_t most = kGroupRecs;
  if (BYTE) {
    const uint32_t mean = V.out_bytes / max(V.n_seq, 1u);
    while (most > 2u && (uint64_t)most * mean > kGroupMax) most /= 2u;
  }
  uint4 r = load();
  // Lays out the next group (records r) at window w, its state before the
  // group, which follows one of `prev` bytes: segment starts and entries, far
  // sources and Byte literals staged by cp.async.
  auto prep = [&](const Window& w, uint32_t prev, uint32_t litpos, uint32_t stage) -> Group {
    Group G{0, 0, 0, 0};
    uint32_t lit_span = kLitStage;
    uint32_t ll[2], ml[2], dist[2];
    const uint4 own_recs = r;
#pragma unroll
    for (int k = 0; k < 2; k++) {
      const uint32_t y = k ? r.w : r.y;
      if (BYTE) {
        const uint32_t m = (y >> 10) & 63u;
        ll[k] = y & 1023u;
        ml[k] = m ? m + 2u : 0u;  // code 63 has no length; as 65 it fails the check below
        dist[k] = (y >> 16) + 1u;
      } else {
        ll[k] = y >> 24;
        ml[k] = ll[k] > 4u ? 0u : (y >> 16) & 255u;
        dist[k] = y & 0xffffu;
      }
    }
    // The second warp may still be writing the group before: everything up to
    // that one's start is complete, and stored but for a flush row.  Sources
    // older than the window must be stored, so this much stays in it.
    const uint32_t hist = max(kHist, prev + kFlush + 80u), near = min(w.cur, hist);
    uint32_t n = most, dst, segs, chunks, lit_at;
    if (BYTE && lane >= n / 2u) ll[0] = ll[1] = ml[0] = ml[1] = 0;
    for (;;) {
      // one scan gives output positions, segment numbers and places for the
      // chunks of sources that may be older than the window (in Byte blocks,
      // whose literal strings are longer, two scans)
      uint32_t own = 0, own_l = 0;
#pragma unroll
      for (int k = 0; k < 2; k++) {
        const uint32_t nc = ml[k] && dist[k] > near ? (ml[k] + 30u) >> 4 : 0u, ns = (ll[k] ? 1u : 0u) + (ml[k] ? 1u : 0u);
        own += ll[k] + ml[k] + (BYTE ? ns << 20 : (ns << 13) + (nc << 21));
        own_l += ll[k] + (nc << 16);
      }
      const uint32_t inc = warp_incl_scan(own), sum = __shfl_sync(FULL, inc, 31), ex = inc - own;
      uint32_t n_chunks;
      bool fits;
      if (BYTE) {
        const uint32_t inc_l = warp_incl_scan(own_l), sum_l = __shfl_sync(FULL, inc_l, 31), ex_l = inc_l - own_l;
        G.total = sum & 0xfffffu;
        G.lits = sum_l & 0xffffu;
        n_chunks = sum_l >> 16;
        dst = ex & 0xfffffu;
        segs = ex >> 20;
        chunks = ex_l >> 16;
        lit_at = (litpos & 15u) + (ex_l & 0xffffu);
        bool long_match = false, bad = false;
        uint32_t at = w.g0 + dst;
#pragma unroll
        for (int k = 0; k < 2; k++) {
          at += ll[k];
          long_match = long_match || ml[k] > V.max_match;
          bad = bad || (ml[k] > 0 && (dist[k] > V.window || dist[k] > at));
          at += ml[k];
        }
        G.err = 0;
        if (__any_sync(FULL, long_match)) G.err = GMP_STATUS_CORRUPT_SYMBOL;
        else if (__any_sync(FULL, bad)) G.err = GMP_STATUS_BAD_OFFSET;
        else if ((uint64_t)w.g0 + G.total > V.out_bytes || (uint64_t)litpos + G.lits > V.n_lit)
          G.err = GMP_STATUS_OUTPUT_OVERRUN;
        lit_span = ((litpos + G.lits + 15u) & ~15u) - (litpos & ~15u);
        fits = !G.err;
      } else {
        G.total = sum & 0x1fffu;
        n_chunks = sum >> 21;
        dst = ex & 0x1fffu;
        segs = (ex >> 13) & 255u;
        chunks = ex >> 21;
        lit_at = 16u * lane;
        fits = true;
      }
      fits = fits && G.total <= kGroupMax && lit_span + 16u * n_chunks <= kStage;
      if (fits) break;
      if (n == 2u) return G;  // (Byte blocks, a failed check: any two records fit)
      n /= 2u;
      if (lane >= n / 2u) ll[0] = ll[1] = ml[0] = ml[1] = 0;
    }
    // the records after this group are on their way while it is laid out
    step(n);
    r = load();
    G.shift = w.cur + G.total > kBuf ? (w.cur - hist) & ~15u : 0u;
    const uint32_t cur = w.cur - G.shift, base = w.base + G.shift;
    if (BYTE) {
      for (uint32_t c = 16u * lane; c < lit_span; c += 512u) cp_async16(S.stage[stage] + c, lits + (litpos & ~15u) + c);
    } else {
      *reinterpret_cast<uint4*>(S.stage[stage] + 16u * lane) = own_recs;
    }
    // segment starts
    uint32_t* mark = S.mark[stage];
    for (uint32_t x = lane; x < ((G.total + 127u) >> 7) * 4u; x += 32) mark[x] = 0;
    __syncwarp();
    // (predicated: with branches, of which every lane takes its own mix, 2 x 512
    // MiB of records 2.90 ms against 2.86, files of 256 MiB 1.30 against 1.27)
    const uint32_t lit_a = smem_addr(S.stage[stage]), mark_a = smem_addr(mark), far_a = lit_a + lit_span;
    uint32_t seg_a = smem_addr(S.seg[stage]) + 4u * segs;
#pragma unroll
    for (int k = 0; k < 2; k++) {
      const bool has_l = ll[k] != 0, has_m = ml[k] != 0;
      segment_if(mark_a, dst, seg_a, lit_a + lit_at - dst, has_l);
      seg_a += has_l ? 4u : 0u;
      dst += ll[k];
      lit_at += BYTE ? ll[k] : 8u;
      const uint32_t src = w.g0 + dst - dist[k], place = far_a + 16u * chunks;
      const bool is_far = has_m && src < base;
      segment_if(mark_a, dst, seg_a, is_far ? place + (src & 15u) - dst : buf_a + cur - dist[k], has_m);
      seg_a += has_m ? 4u : 0u;
      // sources older than the window
      if (vec_ok) {
        const uint8_t* g = out_blk + (src & ~15u);
        const uint32_t nc = is_far ? ((src & 15u) + ml[k] + 15u) >> 4 : 0u;
        cp_async16_if(place, g, 16, nc > 0);
        cp_async16_if(place + 16, g + 16, 16, nc > 1);
        if (__any_sync(FULL, nc > 2)) {
          cp_async16_if(place + 32, g + 32, 16, nc > 2);
          cp_async16_if(place + 48, g + 48, 16, nc > 3);
          cp_async16_if(place + 64, g + 64, 16, nc > 4);
        }
      } else if (is_far) {
        for (uint32_t i = 0; i < ml[k]; i++) sts_u8(place + (src & 15u) + i, __ldcg(out_blk + src + i));
      }
      chunks += has_m && dist[k] > near ? (ml[k] + 30u) >> 4 : 0u;
      dst += ml[k];
    }
    return G;
  };

  Window w{0, 0, 0, 0};
  uint32_t litpos = 0, prev = 0, stage = 0;
  auto tell = [&](uint32_t what, uint32_t total, uint32_t shift) {
    if (lane == 0) SS.step[stage] = StepMsg{what, total, shift};
    pair_sync();
    stage ^= 1u;
  };
  while (i0 < n_j) {
    const Group G = prep(w, prev, litpos, stage);
    if (BYTE && G.err) {
      if (lane == 0) set_status(status, G.err);
      tell(kAbandon, 0, 0);
      return;
    }
    cp_async_commit();
    cp_async_wait<0>();
    tell(kGroup, G.total, G.shift);
    w.g0 += G.total;
    w.base += G.shift;
    w.cur = w.g0 - w.base;
    prev = G.total;
    litpos += G.lits;
  }
  if ((w.g0 != V.out_bytes || (BYTE && litpos != V.n_lit)) && lane == 0) set_status(status, GMP_STATUS_OUTPUT_OVERRUN);
  tell(kDone, 0, 0);
}

// The second warp writes the groups, slides the window and stores whole rows
// of output.
__device__ __forceinline__ void write_block(TileSmem& SS, uint8_t* out_blk) {
  TileSmemB& S = SS.u.b;
  const uint32_t lane = lane_id(), le = (2u << lane) - 1u;
  const bool vec_ok = (((uintptr_t)out_blk) & 15u) == 0;
  const uint32_t buf_a = smem_addr(S.buf);

  // Writes the group's bytes at buf + cur, tile by tile.
  auto tiles = [&](uint32_t total, uint32_t cur, uint32_t stage) {
    const uint32_t* mark = S.mark[stage];
    const uint32_t* seg = S.seg[stage];
    uint32_t tile_a = buf_a + cur;  // shared address of the tile's first byte
    uint32_t before = 0xffffffffu;  // segments started before the tile, less one
    // the addresses of 128 bytes, a byte of each of four tiles per lane
    uint32_t a0, a1, a2, a3;
    auto look = [&](uint32_t t) {
      const uint4 m = *reinterpret_cast<const uint4*>(mark + (t >> 5));
      const uint32_t c0 = before + __popc(m.x), c1 = c0 + __popc(m.y), c2 = c1 + __popc(m.z), o = t + lane;
      a0 = seg[before + __popc(m.x & le)] + o;
      a1 = seg[c0 + __popc(m.y & le)] + o + 32u;
      a2 = seg[c1 + __popc(m.z & le)] + o + 64u;
      a3 = seg[c2 + __popc(m.w & le)] + o + 96u;
      before = c2 + __popc(m.w);
    };
    if (total) look(0);
    for (uint32_t t = 0; t < total; t += 128, tile_a += 128) {
      const uint32_t n = total - t;
      if (!__any_sync(FULL, max(max(a0, a1), max(a2, a3)) >= tile_a)) {
        // all 128 bytes at once; the next addresses are looked up meanwhile
        const uint32_t v0 = lds_u8(a0), v1 = lds_u8(a1), v2 = lds_u8(a2), v3 = lds_u8(a3);
        if (n > 128u) look(t + 128);
        sts_u8(tile_a + lane, v0);
        if (n > 32u) sts_u8(tile_a + 32u + lane, v1);
        if (n > 64u) sts_u8(tile_a + 64u + lane, v2);
        if (n > 96u) sts_u8(tile_a + 96u + lane, v3);
        __syncwarp();
        continue;
      }
      // a source inside its own tile is not written yet: follow it (to a
      // lower lane each time) to the address its byte comes from
      auto resolve = [&](uint32_t& a, uint32_t tile) {
        while (__any_sync(FULL, a >= tile)) {
          const uint32_t b = __shfl_sync(FULL, a, (a - tile) & 31u);
          if (a >= tile) a = b;
        }
      };
      if (__any_sync(FULL, a0 >= tile_a || a1 >= tile_a + 32u || a2 >= tile_a + 64u || a3 >= tile_a + 96u)) {
        resolve(a0, tile_a);
        if (n > 32u) resolve(a1, tile_a + 32u);
        if (n > 64u) resolve(a2, tile_a + 64u);
        if (n > 96u) resolve(a3, tile_a + 96u);
      }
      sts_u8(tile_a + lane, lds_u8(a0));
      __syncwarp();
      if (n > 32u) {
        sts_u8(tile_a + 32u + lane, lds_u8(a1));
        __syncwarp();
      }
      if (n > 64u) {
        sts_u8(tile_a + 64u + lane, lds_u8(a2));
        __syncwarp();
      }
      if (n > 96u) {
        sts_u8(tile_a + 96u + lane, lds_u8(a3));
        __syncwarp();
      }
      if (n > 128u) look(t + 128);
    }
  };

  Window w{0, 0, 0, 0};
  for (uint32_t stage = 0;; stage ^= 1u) {
    pair_sync();
    const StepMsg m = SS.step[stage];
    if (m.what == kGroup) {
      if (m.shift) slide(S.buf, w, m.shift);
      tiles(m.total, w.cur, stage);
      w.g0 += m.total;
      w.cur += m.total;
      flush(S.buf, w, out_blk, vec_ok, lane, 32);
    } else {
      if (m.what == kDone) flush_rest(S.buf, w, out_blk, vec_ok, lane, 32);
      return;
    }
  }
}

// Last file whose first item is <= item.
__device__ __forceinline__ uint32_t find_file(const KParams& P, uint64_t item) {
  uint32_t lo = 0, hi = P.n_files - 1;
  while (lo < hi) {
    const uint32_t mid = (lo + hi + 1) >> 1;
    if (P.item_start[mid] <= item) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// One warp: work item `item` of `total`, opened and checked, into J.  The warps
// that decode a block follow what it says and read none of this themselves: a
// caller could change it under the kernel, and warps that saw different values
// would miss each other at a barrier.
template <bool PIPE>
__device__ __forceinline__ void take_block(const KParams& P, uint64_t item, uint64_t total, Job& J) {
  const uint32_t lane = lane_id();
  uint32_t work = kEnd, file = 0;
  if (item < total) {
    uint64_t b = item;
    gmp_file_desc F = P.single;
    if (P.files) {
      file = find_file(P, item);
      b = item - P.item_start[file];
      F = P.files[file];
    }
    work = kSkip;
    int err = 0;
    if (!PIPE || !P.in_ready || wait_input(P.in_ready + file, P.abort_wait, P.gen, P.wait_ns)) {
      BlockView V;
      err = open_block(F, b, V);
      if (!err && !V.byte_fmt && (V.out_bytes > P.max_out || V.n_seq > P.max_seq)) err = GMP_STATUS_CAPACITY;
      if (!err) {
        work = V.byte_fmt ? kByte : kHuffman;
        if (lane == 0) {
          J.view = V;
          J.out = F.out + V.out_offset;
        }
      }
    } else {
      err = GMP_STATUS_INPUT_TIMEOUT;
    }
    if (err && lane == 0) set_status(P.status + file, err);
  }
  if (lane == 0) {
    J.work = work;
    J.file = file;
  }
}

// Of a pair of launches, a CTA per block and a pair of warps per block, the one
// that the route does not name returns at once.
__device__ __forceinline__ bool not_routed(const KParams& P, uint32_t mine) { return P.route && *P.route != mine; }

// Persistent kernel: warp pairs take blocks until none are left (the first one
// fixed and interleaved over the CTAs when P.spread, as in gmp_decode.cu).
template <bool PIPE>
__global__ void __launch_bounds__(1024, 1) tile_kernel(const KParams P) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const uint32_t pair = threadIdx.x >> 6, half = (threadIdx.x >> 5) & 1u, lane = lane_id(), pairs = blockDim.x >> 6;
  TileSmem& S = reinterpret_cast<TileSmem*>(smem_raw)[pair];
  uint2* rec = reinterpret_cast<uint2*>(P.scratch + ((uint64_t)blockIdx.x * pairs + pair) * P.slot_bytes);
  const uint64_t total = P.files ? P.item_start[P.n_files] : P.single.n_blocks;
  if (not_routed(P, kRoutePair)) return;
  bool first = P.spread != 0;
  for (;;) {
    if (half == 0) {
      unsigned long long item = (unsigned long long)pair * gridDim.x + blockIdx.x;
      if (!first) {
        if (lane == 0) item = (P.spread ? (unsigned long long)gridDim.x * pairs : 0ull) + atomicAdd(P.counter, 1ull);
        item = __shfl_sync(FULL, item, 0);
      }
      first = false;
      take_block<PIPE>(P, item, total, S.job);
    }
    pair_sync();
    const uint32_t work = S.job.work, file = S.job.file;
    if (work == kEnd) break;
    if (work != kSkip) {
      const BlockView& V = S.job.view;
      if (work == kByte || huffman_block(S, V, P.status + file, rec, half)) {
        if (half) write_block(S, S.job.out);
        else if (work == kByte) lay_out_block<true>(S, V, P.status + file, rec, S.job.out);
        else lay_out_block<false>(S, V, P.status + file, rec, S.job.out);
      }
    }
    if (PIPE && P.out_ready && half) {
      const uint64_t n = P.files ? P.files[file].n_blocks : P.single.n_blocks;
      block_done(P.done + file, P.out_ready + file, P.gen, n);
    }
    // the second warp is done with S.job before the first writes it again
    pair_sync();
  }
  if (PIPE && P.out_ready && half)
    pipeline_exit(P.exited, P.out_ready, P.gen, P.files ? P.n_files : 1u, gridDim.x * pairs);
}

// ---------------------------------------------------------------------------
// A block by a CTA of W warps, for launches with too few blocks to fill the
// GPU with a warp for each.  Phase A deals the sub-blocks out over the warps
// (fewer lanes per warp: fewer paths and table conflicts per step) with
// tables of 12 bits, which leave no long codes.  Phase B takes W groups at a
// time, a warp each.  The window holds everything a match may reach, so that
// nothing is staged.  The W groups' bytes (a wave) are written at once: each
// byte whose source lies below the wave is copied, the others note their
// source's place in the wave, and after a barrier follow it from byte to
// byte; a byte's note is replaced by its source's until that one is a value
// (pointer doubling), so that a chain of k copies takes about log2 k looks.
// What bounds it is latency: of a 256 KiB block of CSV rows' 0.31 ms with 16
// warps, about half is the chain of 1,000 Huffman steps in a lane (about 300
// cycles each), half 34 waves of four dependent parts (scan, lay out and copy,
// follow, flush).  One warp took 1.55 ms for it (a pair of warps now 1.0): 16 KiB 156 -> 51 us, 1 MiB of
// 64 KiB blocks 754 -> 195, 16 MiB of records 1554 -> 310, 64 MiB of text 1599
// -> 548, 128 MiB of Byte records 1541 -> 540.
// Literal bytes of a Byte block held: what 227 KB leave a CTA; the first kLitOver
// again at the end.  A wave's and the next one's fit.
__host__ __device__ constexpr uint32_t lit_ring(int W) { return W <= 8 ? 8192 : 32768; }
constexpr uint32_t kLitOver = 1024;
constexpr uint32_t kCoopRecs = 2;  // a lane's records of a group
constexpr uint32_t kCoopGroupMax = kCoopRecs * kGroupMax;
// most output bytes of a wave (a group of text or of CSV rows is about 520)
__host__ __device__ constexpr uint32_t wave_bytes(int W) { return 768 * W; }
__host__ __device__ constexpr uint32_t wave_lits(int W) {  // most literal bytes of a wave (Byte blocks)
  return lit_ring(W) / 2 - 16 < wave_bytes(W) ? lit_ring(W) / 2 - 16 : wave_bytes(W);
}
__host__ __device__ constexpr uint32_t coop_buf(int W) { return 32768 + 16 + wave_bytes(W) + (W <= 8 ? 4096 : 32768); }
constexpr uint32_t kFollow = 12;  // tiles followed at once
constexpr uint32_t kValue = 0x8000;  // note: bits 0-7 are the byte; else its source's place in the wave
static_assert(kCoopGroupMax <= wave_bytes(8) && wave_bytes(16) < kValue, "wave sizes");

struct CoopSmemA {
  uint32_t ll[LUT_SIZE], off[LUT_SIZE];
  uint32_t bits[MAX_SUB][4 * kChunksAhead];
  BuildSmem build;
  Canon coff;
  uint16_t sorted_off[N_OFF + 2];
  uint32_t sb_bit[MAX_SUB + 1], sb_seq[MAX_SUB];
};
template <int W>
struct CoopSmemB {
  uint32_t seg[W][64 * kCoopRecs];
  uint32_t mark[W][(kCoopGroupMax + 127) / 128 * 4];
  union {
    uint8_t huffman[W][256 * kCoopRecs];    // the records
    uint8_t ring[lit_ring(W) + kLitOver];  // Byte blocks
  } lits;
  uint16_t note[wave_bytes(W)];
  uint8_t buf[coop_buf(W) + 160];  // a last batch of tiles may read up to 127 bytes past the wave
};
template <int W>
struct __align__(64) CoopSmem {
  union {
    CoopSmemA a;
    CoopSmemB<W> b;
  } u;
  uint32_t sb_out[MAX_SUB], sb_cnt[MAX_SUB];
  uint32_t tot[2][W], tot_l[2][W];  // each group's output bytes; literal bytes of Byte blocks
  Window win;          // after a slow group
  int32_t result[3];   // of the parts of the table build
  uint32_t bad;        // lowest warp (Huffman: sub-block) << 8 | status of a failed check, else ~0
  Job job;
};

__device__ __forceinline__ uint32_t lds_u16(uint32_t a) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
  return v;
}

__device__ __forceinline__ void sts_u8_if(uint32_t a, uint32_t v, bool on) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %2, 0;\n@p st.shared.u8 [%0], %1;\n}\n" ::"r"(a), "r"(v),
               "r"((uint32_t)on)
               : "memory");
}
__device__ __forceinline__ void sts_u16_if(uint32_t a, uint32_t v, bool on) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %2, 0;\n@p st.shared.u16 [%0], %1;\n}\n" ::"r"(a),
               "h"((uint16_t)v), "r"((uint32_t)on)
               : "memory");
}

// Phase A of one block by the CTA; false: the block's status is set.
template <int W>
__device__ bool coop_huffman(CoopSmem<W>& S, const BlockView& V, int32_t* status, uint2* rec) {
  const uint32_t t = threadIdx.x, warp = t >> 5, lane = lane_id();
  CoopSmemA& A = S.u.a;
  BuildSmem& T = A.build;
  const uint32_t bs_off = (192u + 12u * V.K + 15u) & ~15u;  // bitstream start within the block
  if (t == 0) S.bad = ~0u;
  unpack_lens(T.lens, V.B, t, 32 * W);
  __syncthreads();
  if (warp < 3) {
    int r;
    if (warp == 0) r = sub_block_table(V, (V.comp_bytes - bs_off) * 8ull, A.sb_bit, S.sb_out, A.sb_seq);
    else if (warp == 1) r = build_canon(T.cll, T.run[0], T.sorted_ll, T.lens, N_LL);
    else r = build_canon(A.coff, T.run[1], A.sorted_off, T.lens + N_LL, N_OFF);
    if (lane == 0) S.result[warp] = r;
  }
  __syncthreads();
  const int n_ll = S.result[1], n_off = S.result[2];
  int err = S.result[0] ? S.result[0] : n_ll < 0 || n_off < 0 ? (int)GMP_STATUS_BAD_HEADER : 0;
  if (err) {
    if (t == 0) set_status(status, err);
    return false;
  }
  fill_ll<LUT_BITS>(A.ll, T.cll, T.sorted_ll, n_ll == 0, V.max_match, t, 32 * W);
  fill_off<LUT_BITS>(A.off, A.coff, A.sorted_off, n_off == 0, t, 32 * W);
  __syncthreads();
  const uint8_t* bs = V.B + bs_off;
  const uint32_t n_chunks = (uint32_t)min((uint64_t)0xffffffffu, (V.comp_bytes - bs_off) / 16);
  // warps of phase A: lanes spread over more warps meet fewer paths and bank
  // conflicts per step, but with several CTAs on an SM their instructions
  // count (64 MiB of text, 8 warps: 0.92 ms with 8 of them, 0.60 with 4)
  constexpr uint32_t HW = W == 16 ? 8 : 4;
  const uint32_t j = warp < HW ? lane * HW + warp : MAX_SUB;
  const SubBlock sb = sub_block(V, A.sb_bit, S.sb_out, A.sb_seq, j);
  auto decode = [&](auto is_dense) {
    return huffman_lane<LUT_BITS, LUT_BITS, false, decltype(is_dense)::value>(
        A.ll, A.off, A.coff, A.sorted_off, A.bits[min(j, (uint32_t)MAX_SUB - 1u)], bs, n_chunks, j < V.K, n_ll == 0,
        sb, V.n_seq, V.window, rec + rec_start(sb.out, j), err);
  };
  const uint32_t cnt = dense(V, bs_off) ? decode(std::true_type()) : decode(std::false_type());
  if (j < V.K) S.sb_cnt[j] = cnt;
  if (err) atomicMin(&S.bad, (j << 8) | (uint32_t)err);
  const bool bad = __syncthreads_or(err != 0);  // the records are visible to the whole CTA
  if (bad && t == 0) set_status(status, (int)(S.bad & 255u));  // the first damaged sub-block's
  return !bad;
}

template <int W, bool BYTE>
__device__ __forceinline__ void coop_lz(CoopSmem<W>& SS, const BlockView& V, int32_t* status, const uint2* rec,
                                        uint8_t* out_blk) {
  CoopSmemB<W>& S = SS.u.b;
  constexpr uint32_t NT = 32 * W, CB = coop_buf(W), kWave = wave_bytes(W), R = kCoopRecs, GR = 32 * R;
  constexpr uint32_t kLitRing = lit_ring(W), kLitWave = wave_lits(W);
  const uint32_t t = threadIdx.x, warp = t >> 5, lane = lane_id();
  const uint32_t le = (2u << lane) - 1u;
  const bool vec_ok = (((uintptr_t)out_blk) & 15u) == 0;
  const uint8_t* recs = V.B + 16;         // Byte blocks: the stream's records
  const uint8_t* lits = V.B + V.lit_off;  // and literals
  const uint32_t buf_a = smem_addr(S.buf), note_a = smem_addr(S.note);
  // kept below a wave: what a match reaches, and what is not flushed
  const uint32_t hist = max((V.window + 15u) & ~15u, kFlush);

  // groups of GR records of a sub-block; Byte blocks: of as many, a power of two,
  // as let every warp have its share of a wave (64 KiB blocks, 31 literals and a
  // match of 9 per record, groups of 64 and a ring of 4 KiB: one block 229 us, 700
  // of them 482; so 50 and 166; gmp_decode.cu 198 and 224).
  // i0: the warp's first record of sub-block j; Byte blocks: the lane's, past
  // every block for a lane without any.
  uint32_t n_groups, i0 = GR * warp, next = GR * W;
  if (BYTE) {
    const uint32_t mean = V.out_bytes / max(V.n_seq, 1u);
    uint32_t gr = GR;
    while (gr > 2u && (uint64_t)gr * mean > kWave / W) gr /= 2u;
    n_groups = V.n_seq / gr + (V.n_seq % gr ? 1u : 0u);
    i0 = R * lane < gr ? gr * warp + R * lane : 1u << 31;
    next = gr * W;
  } else {
    uint32_t g = 0;
    for (uint32_t j = lane; j < V.K; j += 32) g += (SS.sb_cnt[j] + GR - 1u) / GR;
    n_groups = __reduce_add_sync(FULL, g);
  }
  uint32_t j = 0, n_j = BYTE ? V.n_seq : SS.sb_cnt[0];
  const uint2* rec_j = rec;
  auto settle = [&]() {
    if constexpr (!BYTE) {
      if (i0 < n_j) return;
      while (j < V.K) {
        const uint32_t whole = (n_j + GR - 1u) / GR * GR;
        if (i0 < whole) break;
        i0 -= whole;
        j++;
        n_j = j < V.K ? SS.sb_cnt[j] : 0u;
      }
      if (j < V.K) rec_j = rec + rec_start(SS.sb_out[j], j);
    }
  };
  // the lane's R adjacent records: {literals, distance | match length << 16 |
  // literal count << 24}, Byte blocks {-, the stream's word}; zero past the end
  struct Recs {
    uint2 r[R];
  };
  auto load = [&]() -> Recs {
    const uint32_t i = BYTE ? i0 : i0 + R * lane;
    Recs x;
#pragma unroll
    for (uint32_t k = 0; k < R; k++) x.r[k] = make_uint2(0, 0);
    if (BYTE) {
#pragma unroll
      for (uint32_t k = 0; k < R; k++)
        if (i + k < n_j) x.r[k].y = ld_u32_nc(recs + 4ull * (i + k));
    } else {
      // whole pairs: a sub-block's records have room for one more
      if (i < n_j) {
        const uint4 v = __ldcg(reinterpret_cast<const uint4*>(rec_j + i));
        x.r[0] = make_uint2(v.x, v.y);
        if (i + 1u < n_j) x.r[R - 1] = make_uint2(v.z, v.w);
      }
    }
    return x;
  };
  rec_j = BYTE ? rec : rec + rec_start(SS.sb_out[0], 0);
  settle();
  Recs r = load();

  // Byte literals: a ring of kLitRing bytes filled at each wave's start for
  // the waves after it.  Each fill is a commit group of its own: the waits
  // before the barriers below cover committed copies only.
  uint32_t litpos = 0, lit_asked = 0;
  auto fill = [&]() {
    const uint32_t upto = min((V.n_lit + 15u) & ~15u, (litpos & ~15u) + kLitRing);
    for (uint32_t c = lit_asked + 16u * t; c < upto; c += 16u * NT) {
      const uint32_t at = c & (kLitRing - 1u);
      cp_async16(S.lits.ring + at, lits + c);
      if (at < kLitOver) cp_async16(S.lits.ring + kLitRing + at, lits + c);
    }
    cp_async_commit();
    lit_asked = max(lit_asked, upto);
  };
  if (t == 0) SS.bad = ~0u;
  if (BYTE) fill();

  Window w{0, 0, 0, 0};  // at the wave's start; the same in every thread
  for (uint32_t it = 0; it * W < n_groups; it++) {
    // lengths of the lane's records; one scan gives output positions and (from
    // bit 20) the number of the segments before
    uint32_t ll[R], ml[R], dist[R], own = 0, own_l = 0, inc_l = 0;
    if (!BYTE)
      *reinterpret_cast<uint4*>(S.lits.huffman[warp] + 8u * R * lane) =
          make_uint4(r.r[0].x, r.r[0].y, r.r[R - 1].x, r.r[R - 1].y);
#pragma unroll
    for (uint32_t k = 0; k < R; k++) {
      const uint32_t y = r.r[k].y;
      if (BYTE) {
        const uint32_t m = (y >> 10) & 63u;
        ll[k] = y & 1023u;
        ml[k] = m ? m + 2u : 0u;  // code 63 has no length; as 65 it fails the check below
        dist[k] = (y >> 16) + 1u;
      } else {
        ll[k] = y >> 24;
        ml[k] = ll[k] > 4u ? 0u : (y >> 16) & 255u;
        dist[k] = y & 0xffffu;
      }
      own += ll[k] + ml[k] + (ll[k] ? 1u << 20 : 0u) + (ml[k] ? 1u << 20 : 0u);
      own_l += ll[k];
    }
    const uint32_t inc = warp_incl_scan(own);
    const uint32_t dst0 = (inc - own) & 0xfffffu, seg0 = (inc - own) >> 20;
    const uint32_t total = __shfl_sync(FULL, inc, 31) & 0xfffffu;
    if (lane == 0) SS.tot[it & 1u][warp] = total;
    if (BYTE) {
      inc_l = warp_incl_scan(own_l);
      if (lane == 31) SS.tot_l[it & 1u][warp] = inc_l;
    }
    const uint32_t t_cur = i0;  // the group's (Byte blocks: the lane's) first record
    i0 += next;
    settle();
    r = load();
    if (BYTE) cp_async_wait<0>();
    __syncthreads();  // the wave before is complete, the totals are known
    const uint32_t T_i = lane < (uint32_t)W ? SS.tot[it & 1u][lane] : 0u;
    const uint32_t L_i = BYTE && lane < (uint32_t)W ? SS.tot_l[it & 1u][lane] : 0u;
    const bool slow_i = BYTE && (T_i > kCoopGroupMax || L_i > kLitWave);
    for (uint32_t lo = 0; lo < (uint32_t)W;) {
      // the wave: as many of the groups from lo on as fit, all of them as a rule
      uint32_t hi = W, sum = __reduce_add_sync(FULL, lane >= lo ? T_i : 0u);
      uint32_t sum_l = BYTE ? __reduce_add_sync(FULL, lane >= lo ? L_i : 0u) : 0u;
      bool slow = false;
      if (sum > kWave || (BYTE && (sum_l > kLitWave || __any_sync(FULL, slow_i)))) {
        const uint32_t s_t = warp_incl_scan(lane >= lo ? T_i : 0u), s_l = BYTE ? warp_incl_scan(lane >= lo ? L_i : 0u) : 0u;
        const uint32_t fit = __ballot_sync(FULL, lane >= lo && !slow_i && s_t <= kWave && s_l <= kLitWave);
        const uint32_t out = ~(fit >> lo);
        hi = min(lo + (out ? (uint32_t)__ffs(out) - 1u : 32u), (uint32_t)W);
        slow = hi == lo;
        if (slow) hi = lo + 1;
        sum = __shfl_sync(FULL, s_t, hi - 1);
        if (BYTE) sum_l = __shfl_sync(FULL, s_l, hi - 1);
      }
      const uint32_t pre = __reduce_add_sync(FULL, lane >= lo && lane < warp ? T_i : 0u);
      const uint32_t pre_l = BYTE ? __reduce_add_sync(FULL, lane >= lo && lane < warp ? L_i : 0u) : 0u;
      const bool mine = warp >= lo && warp < hi;
      if (lo) {
        if (BYTE) cp_async_wait<0>();
        __syncthreads();  // the wave before is complete
      }
      flush(S.buf, w, out_blk, vec_ok, t, NT);
      if (!slow && w.cur + sum > CB) {
        // strips as in slide(), every thread's loads before any store
        const uint32_t shift = (w.cur - hist) & ~15u, n = w.cur - shift;
        for (uint32_t u = 0; u < n; u += 16u * NT) {
          const uint32_t c = u + 16u * t;
          uint4 v = make_uint4(0, 0, 0, 0);
          if (c < n) v = *reinterpret_cast<const uint4*>(S.buf + shift + c);
          __syncthreads();
          if (c < n) *reinterpret_cast<uint4*>(S.buf + c) = v;
        }
        w.cur -= shift;
        w.base += shift;
        __syncthreads();
      }
      int err = 0;  // a group that fails its checks is neither laid out nor copied
      if (BYTE && mine) {
        bool long_match = false, far = false;
        uint32_t at = w.g0 + pre + dst0;
#pragma unroll
        for (uint32_t k = 0; k < R; k++) {
          at += ll[k];
          long_match = long_match || ml[k] > V.max_match;
          far = far || (ml[k] > 0 && (dist[k] > V.window || dist[k] > at));
          at += ml[k];
        }
        if (__any_sync(FULL, long_match)) err = GMP_STATUS_CORRUPT_SYMBOL;
        else if (__any_sync(FULL, far)) err = GMP_STATUS_BAD_OFFSET;
        else if ((uint64_t)w.g0 + pre + total > V.out_bytes ||
                 (uint64_t)litpos + pre_l + __shfl_sync(FULL, L_i, warp) > V.n_lit)
          err = GMP_STATUS_OUTPUT_OVERRUN;
        if (err && lane == 0) atomicMin(&SS.bad, (warp << 8) | (uint32_t)err);
      }
      if (BYTE && slow) {
        __syncthreads();
        if (SS.bad != ~0u) break;
        if (warp == lo) {
          Window x = w;
          const uint32_t t0 = __shfl_sync(FULL, t_cur, 0);
          slow_group(S.buf, CB, hist, x, recs, t0, min(t0 + next / W, V.n_seq), lits + litpos, lits + V.n_lit, out_blk,
                     V.out_bytes, vec_ok);
          if (lane == 0) SS.win = x;
        }
        __syncthreads();
        w = SS.win;
        litpos += sum_l;
        lit_asked = litpos & ~15u;
        fill();
        lo = hi;
        continue;
      }
      if (BYTE) fill();
      const uint32_t wave_a = buf_a + w.cur;
      if (mine && !err) {
        // segment starts and entries, as in lay_out_block
        uint32_t* mark = S.mark[warp];
        uint32_t* seg = S.seg[warp];
        for (uint32_t x = lane; x < ((total + 127u) >> 7) * 4u; x += 32) mark[x] = 0;
        __syncwarp();
        uint32_t at = dst0, n = seg0, lit_at = litpos + pre_l + inc_l - own_l;
#pragma unroll
        for (uint32_t k = 0; k < R; k++) {
          if (ll[k]) {
            atomicOr(mark + (at >> 5), 1u << (at & 31u));
            seg[n++] = (BYTE ? smem_addr(S.lits.ring) + (lit_at & (kLitRing - 1u))
                             : smem_addr(S.lits.huffman[warp]) + 8u * (R * lane + k)) -
                       at;
          }
          at += ll[k];
          lit_at += ll[k];
          if (ml[k]) {
            atomicOr(mark + (at >> 5), 1u << (at & 31u));
            seg[n++] = wave_a + pre - dist[k];
          }
          at += ml[k];
        }
        __syncwarp();
        uint32_t before = 0xffffffffu;  // segments started before the tile, less one
        for (uint32_t x = 0; x < total; x += 128) {
          const uint4 m = *reinterpret_cast<const uint4*>(mark + (x >> 5));
          const uint32_t c0 = before + __popc(m.x), c1 = c0 + __popc(m.y), c2 = c1 + __popc(m.z);
          const uint32_t o = x + lane;
          const uint32_t a0 = seg[before + __popc(m.x & le)] + o, a1 = seg[c0 + __popc(m.y & le)] + o + 32u;
          const uint32_t a2 = seg[c1 + __popc(m.z & le)] + o + 64u, a3 = seg[c2 + __popc(m.w & le)] + o + 96u;
          before = c2 + __popc(m.w);
          auto put = [&](uint32_t a, uint32_t at) {
            const bool in = at < total, follow = a >= wave_a;
            const uint32_t v = lds_u8(a);
            sts_u16_if(note_a + 2u * (pre + at), follow ? a - wave_a : kValue | v, in);
            sts_u8_if(wave_a + pre + at, v, in && !follow);
          };
          put(a0, o);
          put(a1, o + 32u);
          put(a2, o + 64u);
          put(a3, o + 96u);
        }
      }
      __syncthreads();  // every byte of the wave is written or noted
      if (BYTE && SS.bad != ~0u) break;
      if (mine) {
        for (uint32_t x = lane; x < total + lane; x += 32u * kFollow) {
          uint32_t v[kFollow], all = kValue, mine_to_write = 0;
#pragma unroll
          for (uint32_t i = 0; i < kFollow; i++) {
            const bool in = x + 32u * i < total;
            v[i] = lds_u16(in ? note_a + 2u * (pre + x + 32u * i) : note_a);
            v[i] = in ? v[i] : kValue;
            all &= v[i];
            mine_to_write |= (v[i] & kValue) ? 0u : 1u << i;
          }
          // a source's note may still be a place, but only one below it, and
          // the wave's lowest such byte always finds a value
          for (uint32_t spin = 0; __any_sync(FULL, !all); spin++) {
            if (spin == 1u << 20) {
              if (lane == 0) set_status(status, GMP_STATUS_MRR_NO_PROGRESS);
              break;
            }
            all = kValue;
#pragma unroll
            for (uint32_t i = 0; i < kFollow; i++) {
              const bool on = !(v[i] & kValue);
              const uint32_t n = lds_u16(on ? note_a + 2u * v[i] : note_a);
              v[i] = on ? n : v[i];
              all &= v[i];
              sts_u16_if(note_a + 2u * (pre + x + 32u * i), v[i], on);
            }
          }
#pragma unroll
          for (uint32_t i = 0; i < kFollow; i++) sts_u8_if(wave_a + pre + x + 32u * i, v[i], (mine_to_write >> i) & 1u);
        }
      }
      w.g0 += sum;
      w.cur += sum;
      litpos += sum_l;
      lo = hi;
    }
    if (BYTE && SS.bad != ~0u) break;
  }
  if (BYTE) cp_async_wait<0>();
  __syncthreads();
  if (BYTE && SS.bad != ~0u) {
    if (t == 0) set_status(status, (int)(SS.bad & 255u));
    return;
  }
  flush_rest(S.buf, w, out_blk, vec_ok, t, NT);
  if (t == 0 && (w.g0 != V.out_bytes || (BYTE && litpos != V.n_lit))) set_status(status, GMP_STATUS_OUTPUT_OVERRUN);
}

// Persistent kernel, a CTA of W warps per block.
template <int W, bool PIPE>
__global__ void __launch_bounds__(32 * W, W == 16 ? 1 : 3) coop_kernel(const KParams P) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  CoopSmem<W>& S = *reinterpret_cast<CoopSmem<W>*>(smem_raw);
  const uint32_t t = threadIdx.x;
  uint2* rec = reinterpret_cast<uint2*>(P.scratch + blockIdx.x * P.slot_bytes);
  const uint64_t total = P.files ? P.item_start[P.n_files] : P.single.n_blocks;
  if (not_routed(P, kRouteCoop)) return;
  for (bool first = P.spread != 0;; first = false) {
    if (t < 32) {
      unsigned long long item = blockIdx.x;
      if (!first) {
        if (t == 0) item = (P.spread ? gridDim.x : 0u) + atomicAdd(P.counter, 1ull);
        item = __shfl_sync(FULL, item, 0);
      }
      take_block<PIPE>(P, item, total, S.job);
    }
    __syncthreads();
    const uint32_t work = S.job.work, file = S.job.file;
    if (work == kEnd) break;
    int32_t* status = P.status + file;
    if (work != kSkip) {
      const BlockView V = S.job.view;
      if (work == kByte) coop_lz<W, true>(S, V, status, rec, S.job.out);
      else if (coop_huffman<W>(S, V, status, rec)) coop_lz<W, false>(S, V, status, rec, S.job.out);
    }
    if (PIPE && P.out_ready) __threadfence();
    __syncthreads();  // every thread's output is stored, and S.job free
    if (PIPE && P.out_ready && t < 32) {
      const uint64_t n = P.files ? P.files[file].n_blocks : P.single.n_blocks;
      block_done(P.done + file, P.out_ready + file, P.gen, n);
    }
  }
  if (PIPE && P.out_ready) pipeline_exit(P.exited, P.out_ready, P.gen, P.files ? P.n_files : 1u, gridDim.x * W);
}

}  // namespace

uint64_t tile_slot_bytes(uint64_t max_out) {
  // rec_start of the last sub-block and its records
  return ((max_out / 3 + 7ull * MAX_SUB + 8) * sizeof(uint2) + 255) & ~255ull;
}

// The shared memory limit is per kernel and process-wide: always the widest
// launch's, so that no host thread lowers it under another's launch.
static cudaError_t configure_tile() {
  const int lim = 16 * (int)sizeof(TileSmem);
  cudaError_t e = cudaFuncSetAttribute(tile_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(tile_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  return e;
}

cudaError_t tile_occupancy(int warps_per_cta, int* ctas_per_sm) {
  cudaError_t e = configure_tile();
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, tile_kernel<false>, warps_per_cta * 64,
                                                       warps_per_cta * sizeof(TileSmem));
}

cudaError_t launch_tile(const KParams& P, int grid, int warps_per_cta, bool pipe, cudaStream_t stream) {
  cudaError_t e = configure_tile();
  if (e != cudaSuccess) return e;
  const size_t smem = warps_per_cta * sizeof(TileSmem);
  if (pipe) tile_kernel<true><<<grid, warps_per_cta * 64, smem, stream>>>(P);
  else tile_kernel<false><<<grid, warps_per_cta * 64, smem, stream>>>(P);
  return cudaGetLastError();
}

template <int W>
static cudaError_t configure_coop() {
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(coop_kernel<W, false>, a, (int)sizeof(CoopSmem<W>));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(coop_kernel<W, true>, a, (int)sizeof(CoopSmem<W>));
  return e;
}

template <int W>
static cudaError_t coop(const KParams& P, int grid, bool pipe, cudaStream_t stream) {
  cudaError_t e = configure_coop<W>();
  if (e != cudaSuccess) return e;
  if (pipe) coop_kernel<W, true><<<grid, 32 * W, sizeof(CoopSmem<W>), stream>>>(P);
  else coop_kernel<W, false><<<grid, 32 * W, sizeof(CoopSmem<W>), stream>>>(P);
  return cudaGetLastError();
}

cudaError_t coop_occupancy(int warps, int* ctas_per_sm) {
  if (warps == 16) {
    const cudaError_t e = configure_coop<16>();
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, coop_kernel<16, false>, 512,
                                                         sizeof(CoopSmem<16>));
  }
  const cudaError_t e = configure_coop<8>();
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, coop_kernel<8, false>, 256, sizeof(CoopSmem<8>));
}

cudaError_t launch_coop(const KParams& P, int grid, int warps, bool pipe, cudaStream_t stream) {
  return warps == 16 ? coop<16>(P, grid, pipe, stream) : coop<8>(P, grid, pipe, stream);
}

}  // namespace gmp
