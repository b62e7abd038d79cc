// gmp_tile.cu - the decode kernel of libgmp for the default resolution
// (Gompresso-style, arXiv:1606.00519); gmp_decode.cu keeps the kernel whose
// 32-sequence groups and resolution rounds the statistics and the ablation of
// Sec. 5.1 are about.
//
// A warp decodes a block in two phases:
//
//  Phase A, Huffman decoding (Sec. 3.2.1): lane j decodes sub-block j (lanes
//  take j, j+32 for K > 32).  A lookup yields up to two literals and the
//  match length after them when their codes fit the table's bits together,
//  so that a sequence takes about one step.  Each sequence becomes an 8-byte
//  record with its literals inside {literal bytes, distance | match length
//  << 16 | literal count << 24}; a longer literal string takes further
//  records of 3 or 4 literals without a match.  Records go to the warp's
//  scratch slot.
//
//  Phase B, LZ77 decompression (Sec. 3.2.2): the warp takes 32 records per
//  group and writes the group's output 32 bytes at a time, one byte per lane
//  (a tile).  The group's literal strings and matches are segments; a bit
//  per segment start and a population count give each byte its segment, and
//  the segment's entry the shared-memory address its byte comes from: the
//  output window, the literals, or the staging of sources older than the
//  window.  Tiles run in output order, so that every byte below a tile is
//  complete when the tile starts and no resolution rounds are needed;
//  sources inside the tile itself (rare) are followed to the byte they
//  repeat by pointer doubling over the warp's lanes.  So MRR and DE streams
//  take the same path at the same speed.
//
//  Byte blocks (Gompresso/Byte, Sec. 3.1) run phase B on the stream's own
//  records, with each group's records checked before it is staged.
//
//
// What bounds it and what it measured (GB300, 152 SMs): with every SM full the
// integer pipe and the load/store unit (32 lanes reading and writing 32
// places), on small launches one warp's chain of dependent instructions.  The
// Huffman step without branches, records of 8 bytes with their literals
// inside and stored four at a time (single 8-byte stores cost 0.5 of 3.5 ms
// on 2 x 512 MiB of records), and tiles in place of per-sequence copies with
// resolution rounds: 2 x 512 MiB of records, MRR and DE in one launch, 4.53 ->
// 3.48 ms; 2 x 256 MiB of text 2.66 -> 2.15; 107 files of 256 MiB together
// 2.22 -> 1.73; one 64 MiB stream 1.95 -> 1.60 (before: gmp_decode.cu).
// Every read of the compressed stream is bounds-checked; every loop over
// input data is bounded by sizes checked against the block header; corrupt
// input sets the caller's status word and abandons the block.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include "gmp.h"
#include "gmp_decode_common.h"
#include "gmp_internal.h"

namespace gmp {
namespace {

// ---------------------------------------------------------------------------
// Phase A tables.  Literal/length entry of an LLB-bit peek: bits 0-3 code
// bits consumed (0 = no code), 4-5 literals (0..2, in bytes 2 and 3), byte 1
// the match (0 none, kEndCode the end symbol, else the length).  With an
// 11-bit table a prefix of 12-bit codes has kLongLL set and the two codes as
// halves (the upper one for a next bit of 0): byte or match in bits 0-7, bit
// 8 for a literal.  Offset entry:
// byte 0 holds 32 minus the bits of the code and its extra bits, byte 1 32
// minus the extra bits, the upper half the distance base; a prefix of codes
// longer than the table's bits is kLongOff, and the canonical arrays decide
// (codes of 10 bits and more are about 0.3 % of a block's offsets).  No code:
// a base that is above every window.
constexpr uint32_t kLongLL = 1u << 15, kLongOff = 0xffffffffu;
constexpr uint32_t kEndCode = 1;
constexpr uint32_t kNoOff = 0xffff2020u, kNoMatch = 0x2020u;

__device__ __forceinline__ uint32_t ll_entry(uint32_t sym, uint32_t len) {
  if (sym < 256) return len | (1u << 4) | (sym << 16);
  return len | ((sym == 256 ? kEndCode : sym - 254u) << 8);
}
__device__ __forceinline__ uint32_t off_entry(uint32_t os, uint32_t len) {
  const uint32_t ne = os < 4 ? 0u : (os >> 1) - 1u;
  const uint32_t base = os < 4 ? os + 1u : ((2u | (os & 1u)) << ne) + 1u;
  return (base << 16) | ((32u - ne) << 8) | (32u - len - ne);
}

// Working space of the table build; overlaid by the bitstream ring.
struct BuildSmem {
  Canon cll;
  uint32_t run[16];
  uint16_t sorted_ll[N_LL + 1];
  uint8_t lens[N_LL + N_OFF + 3];
};

constexpr int kLLBits = 11, kOffBits = 9;  // a warp's tables
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
  uint32_t sb_bit[MAX_SUB], sb_seq[MAX_SUB];
};

// Phase B.  The output window `buf` holds at least the last kHist output
// bytes and the group being written: it slides down (by a multiple of 16)
// when a group would not fit.
constexpr uint32_t kHist = 4096;
constexpr uint32_t kGroupMax = 32 * 68;  // 4 literals and a match of 64 per record
constexpr uint32_t kBuf = kHist + 16 + kGroupMax;
constexpr uint32_t kFlush = 512;    // output bytes per flush (one 16-byte store per lane)
constexpr uint32_t kFarSlot = 80;   // a 64-byte source spans at most 5 aligned 16-byte chunks
constexpr uint32_t kLitStage = 512; // a Byte group's literal run, with alignment
constexpr uint32_t kMarkWords = (kGroupMax + 127) / 128 * 4;
struct TileSmemB {
  uint8_t lit[2][kLitStage];
  uint8_t far[2][32][kFarSlot];
  uint32_t seg[2][64];
  uint32_t mark[2][kMarkWords];
  uint8_t buf[kBuf + 32];  // a last tile may write up to 31 bytes past its group
};
struct __align__(64) TileSmem {
  union {
    TileSmemA a;
    TileSmemB b;
  } u;
  uint32_t sb_out[MAX_SUB];  // sub-block output start
  uint32_t sb_cnt[MAX_SUB];  // its records
};
static_assert(kBuf % 16 == 0 && sizeof(TileSmem) % 16 == 0, "16-byte copies");
static_assert(sizeof(TileSmem) * 4 + 1024 <= 57 * 1024, "16 warps per SM in CTAs of 4");

// First record of sub-block j, whose output starts at `out`: a record covers
// at least 3 bytes of output but for a sub-block's last one; a multiple of 4,
// so that four records are 32-byte aligned.
__device__ __forceinline__ uint32_t rec_start(uint32_t out, uint32_t j) { return (out / 3 + 5 * j + 3) & ~3u; }

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
__device__ __forceinline__ void fill_ll(uint32_t* lut, const Canon& C, const uint16_t* sorted, bool empty, uint32_t t,
                                        uint32_t n) {
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
      auto half = [](uint32_t s) { return s < 256 ? 256u | s : s == 256 ? kEndCode : s - 254u; };
      x = kLongLL | (half(sorted[i]) << 16) | half(sorted[i + 1]);
    } else {
      const uint32_t s = sorted[C.idx[L] + (v >> (TB - L)) - C.first[L]];
      x = ll_entry(s, L);
      if (s < 256 && L < (uint32_t)TB) {
        // a literal: the next code too, if it lies in the remaining bits
        const uint32_t v2 = (v << L) & ((1u << TB) - 1u);
        const uint32_t L2 = code_length<TB>(lim, v2);
        if (L + L2 <= (uint32_t)TB) {
          const uint32_t s2 = sorted[C.idx[L2] + (v2 >> (TB - L2)) - C.first[L2]];
          x = (L + L2) | (s << 16);
          x |= s2 < 256 ? (2u << 4) | (s2 << 24) : (1u << 4) | ((s2 == 256 ? kEndCode : s2 - 254u) << 8);
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
// entries, and literal and match work run under selects, so that the compiler
// can overlap a step's two table latencies with the record's arithmetic.  The
// lane's 16-byte bitstream chunks pass through a ring of four in shared
// memory, copied there by cp.async: asked for every second step, and at most
// 74 bits are taken in two steps, so that a chunk is not read before the
// third wait after it was asked for.
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
__device__ __forceinline__ void st_global_32B_if(uint2* p, const uint2& a, const uint2& b, const uint2& c,
                                                 const uint2& d, bool on) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.u32 p, %9, 0;\n@p st.global.v8.u32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n}\n" ::"l"(
          p),
      "r"(a.x), "r"(a.y), "r"(b.x), "r"(b.y), "r"(c.x), "r"(c.y), "r"(d.x), "r"(d.y), "r"((uint32_t)on)
      : "memory");
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
template <int LLB, int OFB, bool QUAD>
__device__ __forceinline__ uint32_t huffman_lane(const uint32_t* ll_lut, const uint32_t* off_lut, const Canon& coff,
                                                 const uint16_t* sorted_off, const uint32_t* ring, const uint8_t* bs,
                                                 uint32_t n_chunks, bool act, const SubBlock& sb, uint32_t n_seq,
                                                 uint32_t window, uint32_t max_match, uint2* rec, int& err) {
  const uint32_t ring_s = smem_addr(ring);  // 64-byte aligned
  const uint32_t end = sb.pos + sb.bits, out_end = sb.out + sb.out_n, rec_cap = sb.out_n / 3 + 1;
  uint32_t outp = sb.out;                 // output position of the current record
  uint32_t rem = act ? sb.seq_n : 0u;     // sequences to go
  // the end symbol only closes the block's last sequence
  const uint32_t end_rem = sb.seq + sb.seq_n == n_seq ? 1u : 0u;
  auto chunk_in = [&](uint32_t c, bool ask) {
    const bool in = c < n_chunks;
    cp_async16_if(ring_s | ((c & (kChunksAhead - 1)) * 16u), bs + (in ? 16ull * c : 0ull), in ? 16u : 0u, ask);
  };
  // bit position, counted from 64 so that its word is the one two ahead
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
  uint32_t lits = 0, ln8 = 0, cnt = 0;
  uint2 q0 = make_uint2(0, 0), q1 = q0, q2 = q0, q3 = q0;  // QUAD: the last four records
  // what one step leaves for the checks
  struct Step {
    uint32_t L, mc, e2, ml, dist, wpos, pos, rem;
    bool bad;
  };
  auto one = [&]() -> Step {
    const uint32_t pk = __funnelshift_r(w0, w1, pos);
    uint32_t e = ll_lut[pk & ((1u << LLB) - 1u)];
    if (LLB < LUT_BITS) {
      const uint32_t h = e >> (((pk >> (LLB - 4)) & 16u) ^ 16u);
      const uint32_t v = h & 255u, x = (h & 256u) ? (v << 16) | 28u : (v << 8) | 12u;
      e = (e & kLongLL) ? x : e;
    }
    Step t;
    t.rem = rem;
    e = rem ? e : 0u;
    t.L = e & 15u;
    t.mc = __byte_perm(e, 0, 0x4441);
    advance(t.L);
    lits |= (e >> 16) << ln8;
    ln8 += (e >> 1) & 24u;
    const uint32_t pk2 = __funnelshift_r(w0, w1, pos);
    const bool match = t.mc > kEndCode;
    uint32_t e2 = off_lut[pk2 & ((1u << OFB) - 1u)];
    e2 = match ? e2 : kNoMatch;
    if (OFB < LUT_BITS && __any_sync(FULL, e2 == kLongOff)) {
      if (e2 == kLongOff) {
        const uint32_t x = decode_long<OFB>(coff, sorted_off, pk2 & (LUT_SIZE - 1));
        e2 = x ? off_entry(x & 511u, x >> 9) : kNoOff;
      }
    }
    t.e2 = e2;
    const uint32_t s1 = e2 & 63u, s2 = __byte_perm(e2, 0, 0x4441);
    t.dist = (e2 >> 16) + shr_clamp(shl_clamp(pk2, s1), s2);
    advance(32u - s1);
    t.pos = pos;
    t.ml = match ? t.mc : 0u;
    t.wpos = outp + (ln8 >> 3);
    // e2's base of kNoOff is above every window
    t.bad = (rem && t.L == 0) || pos > end + 64u || (t.mc == kEndCode && rem != end_rem) ||
            (match && (t.ml > max_match || t.dist > min(window, t.wpos) || t.wpos + t.ml > out_end));
    const bool emit = t.mc != 0 || ln8 >= 24u;
    const uint2 r = make_uint2(lits, t.dist | (t.ml << 16) | (ln8 << 21));
    // past the region only on a corrupt stream (caught below)
    if (QUAD) {
      q0 = emit ? q1 : q0;
      q1 = emit ? q2 : q1;
      q2 = emit ? q3 : q2;
      q3 = emit ? r : q3;
      cnt += emit ? 1u : 0u;
      st_global_32B_if(rec + (cnt - 4u), q0, q1, q2, q3, emit && (cnt & 3u) == 0 && cnt <= rec_cap);
    } else {
      st_global_if(rec + cnt, r, emit && cnt < rec_cap);
      cnt += emit ? 1u : 0u;
    }
    outp = emit ? t.wpos + t.ml : outp;
    lits = emit ? 0u : lits;
    ln8 = emit ? 0u : ln8;
    rem -= t.mc != 0 ? 1u : 0u;
    return t;
  };
  while (__any_sync(FULL, rem != 0)) {
    const Step t0 = one();
    const Step t1 = one();
    if (__any_sync(FULL, t0.bad || t1.bad)) {
      // a lane that runs past its sub-block stops here (this bounds the loop
      // on corrupt input); sizes are checked when the sub-block ends
      auto status = [&](const Step& t) {
        if (!t.bad || !t.rem || err) return;
        if (t.L == 0) err = GMP_STATUS_CORRUPT_SYMBOL;
        else if (t.pos > end + 64u) err = GMP_STATUS_BITSTREAM;
        else if (t.mc == kEndCode || t.e2 == kNoOff || t.ml > max_match) err = GMP_STATUS_CORRUPT_SYMBOL;
        else if (t.dist > window || t.dist > t.wpos) err = GMP_STATUS_BAD_OFFSET;
        else err = GMP_STATUS_OUTPUT_OVERRUN;
      };
      status(t0);
      status(t1);
      if (err) rem = 0;
    }
    const bool ask = rem && ((pos - 64u) >> 7) + kChunksAhead > asked;
    chunk_in(asked, ask);
    asked += ask ? 1u : 0u;
    cp_async_commit();
    cp_async_wait<2>();
  }
  cp_async_wait<0>();
  if (QUAD && cnt <= rec_cap) {
    const uint32_t n = cnt & 3u;  // records not stored yet
    if (n > 2) rec[cnt - 3u] = q1;
    if (n > 1) rec[cnt - 2u] = q2;
    if (n > 0) rec[cnt - 1u] = q3;
  }
  outp += ln8 >> 3;
  if (!err && pos != end + 64u) err = GMP_STATUS_BITSTREAM;
  if (!err && outp != out_end) err = GMP_STATUS_OUTPUT_OVERRUN;
  return cnt;
}

// Sub-block table: prefix sums of bit sizes, output sizes and sequences over
// the K sub-blocks (one warp), with the totals checked in 64 bits, so that
// no wrapped 32-bit sum passes.  Returns a gmp_status.
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
  if (ts != V.n_seq || to != V.out_bytes) return GMP_STATUS_BAD_HEADER;
  return tb > bits_avail ? (int)GMP_STATUS_BITSTREAM : 0;
}

__device__ __forceinline__ void unpack_lens(uint8_t* lens, const uint8_t* B, uint32_t t, uint32_t n) {
  for (uint32_t i = t; i < (uint32_t)(N_LL + N_OFF); i += n) {
    const uint32_t sym = i < (uint32_t)N_LL ? i : i - N_LL;
    const uint8_t v = __ldg(B + (i < (uint32_t)N_LL ? 8 : 168) + (sym >> 1));
    lens[i] = (sym & 1) ? (v >> 4) : (v & 15);
  }
}

// Phase A of one block by one warp; false: the block's status is set.
__device__ bool huffman_block(TileSmem& S, const BlockView& V, int32_t* status, uint2* rec) {
  const uint32_t lane = lane_id();
  TileSmemA& A = S.u.a;
  const uint32_t bs_off = (192u + 12u * V.K + 15u) & ~15u;  // bitstream start within the block
  int err = sub_block_table(V, (V.comp_bytes - bs_off) * 8ull, A.sb_bit, S.sb_out, A.sb_seq);
  if (err) {
    if (lane == 0) set_status(status, err);
    return false;
  }
  unpack_lens(A.u.build.lens, V.B, lane, 32);
  __syncwarp();
  BuildSmem& T = A.u.build;
  const int n_ll = build_canon(T.cll, T.run, T.sorted_ll, T.lens, N_LL);
  const int n_off = build_canon(A.coff, T.run, A.sorted_off, T.lens + N_LL, N_OFF);
  if (n_ll < 0 || n_off < 0) {
    if (lane == 0) set_status(status, GMP_STATUS_BAD_HEADER);
    return false;
  }
  fill_ll<kLLBits>(A.ll, T.cll, T.sorted_ll, n_ll == 0, lane, 32);
  fill_off<kOffBits>(A.off, A.coff, A.sorted_off, n_off == 0, lane, 32);
  __syncwarp();  // the ring takes the build's place
  const uint8_t* bs = V.B + bs_off;
  const uint32_t n_chunks = (uint32_t)min((uint64_t)0xffffffffu, (V.comp_bytes - bs_off) / 16);
  for (uint32_t jb = 0; jb < V.K; jb += 32) {
    const uint32_t j = jb + lane;
    SubBlock sb{0, 0, 0, 0, 0, 0};
    if (j < V.K) {
      const uint8_t* e = V.B + 192 + 12 * j;
      sb = SubBlock{A.sb_bit[j], ld_u32_nc(e), S.sb_out[j], ld_u32_nc(e + 4), A.sb_seq[j], ld_u32_nc(e + 8)};
    }
    const uint32_t cnt = huffman_lane<kLLBits, kOffBits, true>(A.ll, A.off, A.coff, A.sorted_off, A.u.bits[lane], bs, n_chunks, j < V.K, sb,
                                      V.n_seq, V.window, V.max_match, rec + rec_start(sb.out, j), err);
    if (j < V.K) S.sb_cnt[j] = cnt;
  }
  if (err) set_status(status, err);
  if (__any_sync(FULL, err != 0)) return false;
  __syncwarp();  // the records are visible to the whole warp
  return true;
}

// ---------------------------------------------------------------------------
// Phase B.
struct Window {
  uint32_t g0;       // output position of the next byte
  uint32_t cur;      // its place in buf
  uint32_t base;     // output position of buf[0] (a multiple of 16): g0 - cur
  uint32_t flushed;  // output bytes stored (a multiple of kFlush)
};
struct Group {
  uint32_t total, lits, shift;
  int err;
  bool slow;  // a Byte group too large for the window or the literal staging
};

__device__ __forceinline__ void slide(TileSmemB& S, Window& w, uint32_t shift) {
  const uint32_t lane = lane_id();
  // ascending strips, each loaded whole before it is stored: a strip's
  // destination ends at or below every later strip's source
  const uint32_t n = w.cur - shift;
  for (uint32_t u = 0; u < n; u += 512u) {
    const uint32_t c = u + 16u * lane;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (c < n) v = *reinterpret_cast<const uint4*>(S.buf + shift + c);
    __syncwarp();
    if (c < n) *reinterpret_cast<uint4*>(S.buf + c) = v;
    __syncwarp();
  }
  w.cur -= shift;
  w.base += shift;
}

__device__ __forceinline__ void flush(const TileSmemB& S, Window& w, uint8_t* out_blk, bool vec_ok) {
  if (w.g0 - w.flushed < kFlush) return;
  const uint32_t lane = lane_id(), end = w.g0 & ~(kFlush - 1u);
  if (vec_ok) {
    for (uint32_t c = w.flushed + 16u * lane; c < end; c += kFlush)
      *reinterpret_cast<uint4*>(out_blk + c) = *reinterpret_cast<const uint4*>(S.buf + (c - w.base));
  } else {
    for (uint32_t c = w.flushed + lane; c < end; c += 32u) out_blk[c] = S.buf[c - w.base];
  }
  w.flushed = end;
  __syncwarp();
}

// A Byte group that does not fit the fast path: record after record, the
// whole warp copying each literal string and each match.
__device__ __noinline__ void slow_group(TileSmemB& S, Window& w, const uint8_t* recs, uint32_t t0, uint32_t t1,
                                        const uint8_t* lits, uint8_t* out_blk, bool vec_ok) {
  const uint32_t lane = lane_id();
  auto room = [&](uint32_t n) {
    if (w.cur + n > kBuf) slide(S, w, (w.cur - kHist) & ~15u);
  };
  for (uint32_t t = t0; t < t1; t++) {
    const uint32_t r = ld_u32_nc(recs + 4ull * t), m = (r >> 10) & 63u, dist = (r >> 16) + 1u;
    uint32_t left = r & 1023u;
    const uint32_t ml = m ? m + 2u : 0u;
    while (left) {
      const uint32_t n = min(left, kFlush);
      room(n);
      for (uint32_t i = lane; i < n; i += 32) S.buf[w.cur + i] = __ldg(lits + i);
      __syncwarp();
      w.cur += n;
      w.g0 += n;
      lits += n;
      left -= n;
      flush(S, w, out_blk, vec_ok);
    }
    if (ml) {
      room(ml);
      for (uint32_t i = lane; i < ml; i += 32) {
        // an overlapping copy repeats the dist bytes before it
        const uint32_t src = w.g0 - dist + (dist < ml ? i % dist : i);
        S.buf[w.cur + i] = src >= w.base ? S.buf[src - w.base] : (uint8_t)__ldcg(out_blk + src);
      }
      __syncwarp();
      w.cur += ml;
      w.g0 += ml;
      flush(S, w, out_blk, vec_ok);
    }
  }
}

template <bool BYTE>
__device__ __forceinline__ void lz_block(TileSmem& SS, const BlockView& V, int32_t* status, const uint2* rec,
                                         uint8_t* out_blk) {
  TileSmemB& S = SS.u.b;
  const uint32_t lane = lane_id(), lt = (1u << lane) - 1u, le = lt | (1u << lane);
  const bool vec_ok = (((uintptr_t)out_blk) & 15u) == 0;
  const uint8_t* recs = V.B + 16;           // Byte blocks: the stream's records
  const uint8_t* lits = V.B + V.lit_off;    // and literals
  const uint32_t buf_a = smem_addr(S.buf);

  // records of the next group: Huffman blocks {literals, distance | match
  // length << 16 | literal count << 24} of one sub-block, Byte blocks the
  // stream's word; zero past the end
  uint32_t i_grp = 0;
  uint32_t j = 0, i0 = 0, n_j = 0;  // sub-block, record within it, its records (Byte: the block's)
  const uint2* rec_j = rec;
  if (BYTE) {
    n_j = V.n_seq;
  } else {
    while (j < V.K && (n_j = SS.sb_cnt[j]) == 0) j++;
    if (j < V.K) rec_j = rec + rec_start(SS.sb_out[j], j);
    else n_j = 0;
  }
  auto load = [&]() -> uint2 {
    const uint32_t i = i0 + lane;
    if (i >= n_j) return make_uint2(0, 0);
    if (BYTE) return make_uint2(0, ld_u32_nc(recs + 4ull * i));
    return __ldcg(rec_j + i);
  };
  auto step = [&]() {  // to the next group
    i0 += 32;
    if (i0 < n_j || BYTE) return;
    i0 = 0;
    n_j = 0;
    while (++j < V.K && (n_j = SS.sb_cnt[j]) == 0) {}
    if (j < V.K) rec_j = rec + rec_start(SS.sb_out[j], j);
  };

  // Lays out the group of records r at window w (its state before the
  // group): segment starts and entries, far sources and Byte literals staged
  // by cp.async.
  auto prep = [&](uint2 r, const Window& w, uint32_t litpos, int stage) -> Group {
    Group G;
    G.err = 0;
    G.slow = false;
    G.shift = 0;
    uint32_t ll, ml, dist, dst;
    if (BYTE) {
      const uint32_t m = (r.y >> 10) & 63u;
      ll = r.y & 1023u;
      ml = m ? m + 2u : 0u;  // code 63 has no length; as 65 it fails the check below
      dist = (r.y >> 16) + 1u;
      const uint32_t packed = (ll << 16) | (ll + ml);  // a group's sums stay below 2^16
      const uint32_t inc = warp_incl_scan(packed), sum = __shfl_sync(FULL, inc, 31);
      G.total = sum & 0xffffu;
      G.lits = sum >> 16;
      dst = (inc & 0xffffu) - (ll + ml);
      const uint32_t mst = w.g0 + dst + ll;
      if (__any_sync(FULL, ml > V.max_match)) G.err = GMP_STATUS_CORRUPT_SYMBOL;
      else if (__any_sync(FULL, ml > 0 && (dist > V.window || dist > mst))) G.err = GMP_STATUS_BAD_OFFSET;
      else if ((uint64_t)w.g0 + G.total > V.out_bytes || (uint64_t)litpos + G.lits > V.n_lit)
        G.err = GMP_STATUS_OUTPUT_OVERRUN;
      if (G.err) return G;
      const uint32_t l0 = litpos & ~15u, l1 = (litpos + G.lits + 15u) & ~15u;
      if (G.total > kGroupMax || l1 - l0 > kLitStage) {
        G.slow = true;
        return G;
      }
      if (16u * lane < l1 - l0) cp_async16(S.lit[stage] + 16u * lane, lits + l0 + 16u * lane);
      // literal string's place in the staging
      r.x = (litpos & 15u) + (inc >> 16) - ll;
    } else {
      ll = r.y >> 24;
      ml = (r.y >> 16) & 255u;
      dist = r.y & 0xffffu;
      const uint32_t inc = warp_incl_scan(ll + ml);
      G.total = __shfl_sync(FULL, inc, 31);
      G.lits = 0;
      dst = inc - (ll + ml);
      *reinterpret_cast<uint32_t*>(S.lit[stage] + 4u * lane) = r.x;
      r.x = 4u * lane;
    }
    G.shift = w.cur + G.total > kBuf ? (w.cur - kHist) & ~15u : 0u;
    const uint32_t cur = w.cur - G.shift, base = w.base + G.shift;
    // segment starts
    uint32_t* mark = S.mark[stage];
    for (uint32_t x = lane; x < ((G.total + 127u) >> 7) * 4u; x += 32) mark[x] = 0;
    __syncwarp();
    const uint32_t mst = dst + ll, src = w.g0 + mst - dist;
    const uint32_t b_l = __ballot_sync(FULL, ll > 0), b_m = __ballot_sync(FULL, ml > 0);
    uint32_t k = __popc(b_l & lt) + __popc(b_m & lt);
    uint32_t* seg = S.seg[stage];
    if (ll) {
      atomicOr(mark + (dst >> 5), 1u << (dst & 31u));
      seg[k++] = smem_addr(S.lit[stage]) + r.x - dst;
    }
    const bool is_far = ml > 0 && src < base;
    if (ml) {
      atomicOr(mark + (mst >> 5), 1u << (mst & 31u));
      seg[k] = is_far ? smem_addr(S.far[stage][lane]) + (src & 15u) - mst : buf_a + cur - dist;
    }
    // sources older than the window: at least kHist - 64 bytes back, hence
    // flushed (at most a group and a flush row are not)
    uint8_t* slot = S.far[stage][lane];
    if (vec_ok) {
      const uint8_t* g = out_blk + (src & ~15u);
      const uint32_t nc = is_far ? ((src & 15u) + ml + 15u) >> 4 : 0u;
      if (nc > 0) cp_async16(slot, g);
      if (nc > 1) cp_async16(slot + 16, g + 16);
      if (__any_sync(FULL, nc > 2)) {
        if (nc > 2) cp_async16(slot + 32, g + 32);
        if (nc > 3) cp_async16(slot + 48, g + 48);
        if (nc > 4) cp_async16(slot + 64, g + 64);
      }
    } else if (is_far) {
      for (uint32_t i = 0; i < ml; i++) slot[(src & 15u) + i] = (uint8_t)__ldcg(out_blk + src + i);
    }
    return G;
  };

  // Writes the group's bytes at buf + cur, tile by tile.
  auto tiles = [&](const Group& G, uint32_t cur, int stage) {
    const uint32_t* mark = S.mark[stage];
    const uint32_t* seg = S.seg[stage];
    uint32_t tile_a = buf_a + cur;  // shared address of the tile's first byte
    uint32_t before = 0xffffffffu;  // segments started before the tile, less one
    for (uint32_t t = 0; t < G.total; t += 128, tile_a += 128) {
      const uint4 m = *reinterpret_cast<const uint4*>(mark + (t >> 5));
      const uint32_t c0 = before + __popc(m.x), c1 = c0 + __popc(m.y), c2 = c1 + __popc(m.z);
      const uint32_t o = t + lane;
      uint32_t a0 = seg[before + __popc(m.x & le)] + o, a1 = seg[c0 + __popc(m.y & le)] + o + 32u;
      uint32_t a2 = seg[c1 + __popc(m.z & le)] + o + 64u, a3 = seg[c2 + __popc(m.w & le)] + o + 96u;
      before = c2 + __popc(m.w);
      const uint32_t n = G.total - t;
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
    }
  };

  Window w{0, 0, 0, 0};
  uint32_t litpos = 0, t_cur = 0;  // Byte: the group's first literal and record
  uint2 r = load();
  Group G{0, 0, 0, 0, false};  // an empty group before the first
  for (bool more = true; more;) {
    if (BYTE && G.err) {
      cp_async_wait<0>();
      if (lane == 0) set_status(status, G.err);
      return;
    }
    if (BYTE && G.slow) {
      cp_async_wait<0>();
      slow_group(S, w, recs, t_cur, min(t_cur + 32u, V.n_seq), lits + litpos, out_blk, vec_ok);
      litpos += G.lits;
      G = Group{0, 0, 0, 0, false};
    }
    // the next group is laid out, and its copies started, before this
    // group's bytes are written
    more = i0 < n_j;
    const int stage = (int)((i_grp++) & 1u);
    Window after = w;
    after.g0 += G.total;
    after.base += G.shift;
    after.cur = after.g0 - after.base;
    const Group N = prep(r, after, litpos + G.lits, stage);
    t_cur = i0;
    step();
    r = load();
    cp_async_commit();
    cp_async_wait<1>();
    __syncwarp();
    if (G.shift) slide(S, w, G.shift);
    tiles(G, w.cur, stage ^ 1);
    w.g0 += G.total;
    w.cur += G.total;
    litpos += G.lits;
    flush(S, w, out_blk, vec_ok);
    G = N;
  }
  cp_async_wait<0>();
  __syncwarp();
  // what is not flushed yet
  {
    uint32_t c = w.flushed;
    if (vec_ok) {
      for (uint32_t x = c + 16u * lane; x + 16u <= w.g0; x += 512u)
        *reinterpret_cast<uint4*>(out_blk + x) = *reinterpret_cast<const uint4*>(S.buf + (x - w.base));
      c = w.g0 & ~15u;
    }
    for (c += lane; c < w.g0; c += 32u) out_blk[c] = S.buf[c - w.base];
  }
  if ((w.g0 != V.out_bytes || (BYTE && litpos != V.n_lit)) && lane == 0) set_status(status, GMP_STATUS_OUTPUT_OVERRUN);
}

__device__ __forceinline__ void tile_block(TileSmem& S, const KParams& P, const gmp_file_desc& F, uint64_t b,
                                           int32_t* status, uint8_t* slot) {
  BlockView V;
  int err = open_block(F, b, V);
  if (!err && !V.byte_fmt && (V.out_bytes > P.max_out || V.n_seq > P.max_seq)) err = GMP_STATUS_CAPACITY;
  if (err) {
    if (lane_id() == 0) set_status(status, err);
    return;
  }
  uint2* rec = reinterpret_cast<uint2*>(slot);
  uint8_t* out_blk = F.out + V.out_offset;
  if (V.byte_fmt) {
    lz_block<true>(S, V, status, rec, out_blk);
  } else if (huffman_block(S, V, status, rec)) {
    lz_block<false>(S, V, status, rec, out_blk);
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

// Persistent kernel: warps take blocks until none are left (the first one
// fixed and interleaved over the CTAs when P.spread, as in gmp_decode.cu).
template <bool PIPE>
__global__ void __launch_bounds__(512, 1) tile_kernel(const KParams P) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const uint32_t warp = threadIdx.x >> 5, lane = lane_id();
  TileSmem& S = reinterpret_cast<TileSmem*>(smem_raw)[warp];
  const uint64_t gw = (uint64_t)blockIdx.x * (blockDim.x >> 5) + warp;
  uint8_t* slot = P.scratch + gw * P.slot_bytes;
  const uint64_t total = P.files ? P.item_start[P.n_files] : P.single.n_blocks;
  const unsigned long long fixed = P.spread ? (unsigned long long)gridDim.x * (blockDim.x >> 5) : 0ull;
  unsigned long long item = 0;
  if (P.spread) {
    item = (unsigned long long)warp * gridDim.x + blockIdx.x;
  } else {
    if (lane == 0) item = atomicAdd(P.counter, 1ull);
    item = __shfl_sync(FULL, item, 0);
  }
  while (item < total) {
    uint32_t file = 0;
    uint64_t b = item;
    gmp_file_desc F = P.single;
    if (P.files) {
      file = find_file(P, item);
      b = item - P.item_start[file];
      F = P.files[file];
    }
    if (!PIPE || !P.in_ready || wait_input(P.in_ready + file, P.abort_wait, P.gen, P.wait_ns)) {
      tile_block(S, P, F, b, P.status + file, slot);
    } else if (lane == 0) {
      set_status(P.status + file, GMP_STATUS_INPUT_TIMEOUT);
    }
    __syncwarp();
    if (PIPE && P.out_ready) block_done(P.done + file, P.out_ready + file, P.gen, F.n_blocks);
    unsigned long long next = 0;
    if (lane == 0) next = fixed + atomicAdd(P.counter, 1ull);
    item = __shfl_sync(FULL, next, 0);
  }
  if (PIPE && P.out_ready)
    pipeline_exit(P.exited, P.out_ready, P.gen, P.files ? P.n_files : 1u, gridDim.x * (blockDim.x >> 5));
}

}  // namespace

uint64_t tile_slot_bytes(uint64_t max_out) {
  // rec_start of the last sub-block and its records
  return ((max_out / 3 + 5ull * MAX_SUB + 8) * sizeof(uint2) + 255) & ~255ull;
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
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, tile_kernel<false>, warps_per_cta * 32,
                                                       warps_per_cta * sizeof(TileSmem));
}

cudaError_t launch_tile(const KParams& P, int grid, int warps_per_cta, bool pipe, cudaStream_t stream) {
  cudaError_t e = configure_tile();
  if (e != cudaSuccess) return e;
  const size_t smem = warps_per_cta * sizeof(TileSmem);
  if (pipe) tile_kernel<true><<<grid, warps_per_cta * 32, smem, stream>>>(P);
  else tile_kernel<false><<<grid, warps_per_cta * 32, smem, stream>>>(P);
  return cudaGetLastError();
}

}  // namespace gmp
