// gmp_gpucompress.cu - compression with the LZ77 parse on the GPU.
//
// Sec. 3.1: the input is cut into blocks that are compressed independently,
// hence in parallel; Sec. 4.2 adds the dependency rule of DE streams.  Here
// every step runs on the GPU: the match search and the parse of every block
// (this file), then the entropy coding (Huffman trees and sub-blocks, or Byte
// records; gmp_gpuencode.cu), writing the same stream format as
// gmp_compress.  The host only lays out the blocks from their sizes and
// writes the 64-byte file header and the block offset table.
//
//  chain_kernel: a CTA per block walks it 512 positions at a time, one per
//  thread, and writes each position's link: the distance to the latest
//  position of an earlier step with the same hash of its 3-byte prefix (0 =
//  none).  Positions of one step do not see each other, so every chain runs
//  through at most one position of a step.
//  search_kernel: given the links, every position's search is independent.  A
//  CTA takes a run of positions of one block, with the window before them and
//  all their links in shared memory.  A lane follows its position's chain for
//  up to chain_depth candidates within the window, keeps the longest match (at
//  most max_match bytes, the nearest of equals) and stores its length and
//  distance; then it takes the next position of its warp's share, so that
//  lanes whose chains are short do not wait for the longest one.
//  parse_kernel: a CTA per block parses it from its start: a match of at
//  least 3 bytes is taken unless the next position has a longer one
//  (one-step lazy evaluation), otherwise the byte becomes a literal.  What
//  follows from the matches alone is worked out for every position at once,
//  so that one warp has one lookup to do per token.  For DE streams a
//  candidate is cut at the first source byte that an earlier back-reference
//  of the same 32-sequence group writes, as in gmp_compress; for Byte streams
//  literal strings are cut into runs of at most 1023 bytes, which count as
//  sequences of their group.
//  Every token's position in its block is written beside it for the
//  entropy coder.
//
// Positions of the same step do not see each other, and one hash bucket per
// prefix is shared by several prefixes, so the parse can differ from
// gmp_compress's; any parse the checks accept is a valid stream.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "gmp.h"
#include "gmp_internal.h"

namespace {

constexpr uint32_t kFull = 0xffffffffu;
constexpr uint32_t kByteMaxLit = 1023;
constexpr uint32_t kStep = 512;          // positions of one step do not see each other
constexpr int kHeadBits = 12;            // hash buckets of 3-byte prefixes
constexpr uint32_t kLook = 64;           // longest match
constexpr int kSearchThreads = 1024;
constexpr int kSearchSmemMax = 3 * (32768 + 32768) + 64 + 64;  // window and run of 32 Ki positions
constexpr uint32_t kShare = 128;         // positions that a warp takes at a time
constexpr uint32_t kCompareAt = 10;      // lanes with a promising candidate that make the warp compare
constexpr int kWalkSteps = 4;           // candidates between the warp's votes
constexpr uint32_t kRefillAt = 6;        // idle lanes that make the warp deal out positions

__device__ __forceinline__ uint32_t prefix_hash(uint32_t b012) {
  return (b012 * 0x9E3779B1u) >> (32 - kHeadBits);
}

// One CTA per block.  Bound by its two barriers a step: 70 us for a 256 KiB
// block, whatever the number of blocks up to four per SM.
__global__ void __launch_bounds__(kStep) chain_kernel(const uint8_t* in, uint64_t n, uint32_t block_size,
                                                      uint16_t* link) {
  __shared__ uint32_t head[1 << kHeadBits];  // latest position + 1 of an earlier step, 0 = none
  const uint32_t tid = threadIdx.x;
  const uint64_t base = blockIdx.x * (uint64_t)block_size;
  const uint32_t len = (uint32_t)min((uint64_t)block_size, n - base);
  for (uint32_t i = tid; i < (1u << kHeadBits); i += kStep) head[i] = 0;
  // the 3 bytes at p, from the aligned words they lie in (the input has 16
  // bytes of slack)
  auto prefix = [&](uint32_t p) -> uint32_t {
    if (p + 3 > len) return 0;
    const uint64_t x = base + p;
    const uint32_t* w = reinterpret_cast<const uint32_t*>(in) + (x >> 2);
    return __funnelshift_r(__ldg(w), __ldg(w + 1), (uint32_t)(x & 3u) * 8u) & 0xffffffu;
  };
  uint32_t next = prefix(tid);
  __syncthreads();
  for (uint32_t s = 0; s < len; s += kStep) {
    const uint32_t p = s + tid, h = prefix_hash(next);
    const bool has_prefix = p + 3 <= len;
    next = prefix(p + kStep);
    const uint32_t c = has_prefix ? head[h] : 0u;
    if (p < len) link[base + p] = (c && p + 1 - c <= 0xffffu) ? (uint16_t)(p + 1 - c) : (uint16_t)0;
    __syncthreads();  // the step's lookups are done
    if (has_prefix) atomicMax(head + h, p + 1);
    __syncthreads();
  }
}

// A run of `span` positions per CTA.  Shared memory: links of the window and
// the run, then their bytes and a longest match more.  Bound by the load/store
// unit: three scattered shared-memory reads per candidate.  Dealing positions
// out to lanes that are done and comparing only when several lanes have a
// promising candidate keeps most lanes at work (one thread per position and
// step, with a barrier per step, had 7.5 of 32): 64 MiB of text 17.3 -> 3.6 ms.
__global__ void __launch_bounds__(kSearchThreads) search_kernel(const uint8_t* in, uint64_t n, uint32_t block_size,
                                                                uint32_t window, uint32_t max_match,
                                                                uint32_t chain_depth, uint32_t span,
                                                                uint32_t spans_per_block, const uint16_t* link,
                                                                uint8_t* best_len, uint16_t* best_dist) {
  extern __shared__ __align__(16) unsigned char search_smem[];
  __shared__ uint32_t dealt;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, lt = (1u << lane) - 1u;
  const uint64_t base = blockIdx.x / spans_per_block * (uint64_t)block_size;
  const uint32_t len = (uint32_t)min((uint64_t)block_size, n - base);
  const uint32_t t0 = blockIdx.x % spans_per_block * span;
  if (t0 >= len) return;
  const uint32_t t1 = min(t0 + span, len);
  const uint32_t lo = t0 > window ? t0 - window : 0u;  // the run's positions reach back to here
  const uint32_t shift = (uint32_t)((base + lo) & 3u);  // bytes are kept as aligned as in the input
  uint16_t* lnk = reinterpret_cast<uint16_t*>(search_smem);  // position lo + i at i
  uint32_t* words = reinterpret_cast<uint32_t*>(search_smem + ((2u * (window + span) + 15u) & ~15u));
  if (tid == 0) dealt = 0;
  // no link: one beyond every window
  for (uint32_t i = tid; i < t1 - lo; i += kSearchThreads) {
    const uint16_t l = __ldg(link + base + lo + i);
    lnk[i] = l ? l : (uint16_t)0xffffu;
  }
  {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(in) + ((base + lo) >> 2);
    const uint64_t all = (n + 3) >> 2;  // words of the input
    const uint32_t need = (shift + t1 - lo + kLook + 11u) >> 2;
    for (uint32_t i = tid; i < need; i += kSearchThreads)
      words[i] = ((base + lo) >> 2) + i < all ? __ldg(src + i) : 0u;
  }
  __syncthreads();
  // bytes x .. x + 3 of the block, x counted from lo
  auto word = [&](uint32_t x) {
    const uint32_t y = x + shift, i = y >> 2;
    return __funnelshift_r(words[i], words[i + 1], y << 3);
  };
  const uint32_t first = t0 - lo, count = t1 - t0;
  // a lane's search: position p and candidate c (from lo), the lowest one
  // allowed, best match, and what is compared first: the last four bytes that
  // a longer match needs (three while there is none).  A lane walks its chain,
  // or waits with a promising candidate, or is done.
  bool walk = false, promising = false, has = false;
  int c = 0, c_min = 0;
  uint32_t p = 0, ml = 0, dist = 0, lim = 0, left = 0, off = 0, key = 0, mask = 0;
  uint32_t next = 0, end = 0;  // the warp's share
  auto move = [&]() {  // to the candidate before
    c -= lnk[c];
    left--;
    walk = c >= c_min && left != 0;
  };
  for (;;) {
    const uint32_t idle = __ballot_sync(kFull, !(walk || promising));
    if (__popc(idle) >= (int)kRefillAt) {
      if (!(walk || promising) && has) {
        best_len[base + lo + p] = (uint8_t)ml;
        best_dist[base + lo + p] = (uint16_t)dist;
        has = false;
      }
      if (next >= end && next < count) {
        uint32_t x = 0;
        if (lane == 0) x = atomicAdd(&dealt, kShare);
        next = __shfl_sync(kFull, x, 0);
        end = min(next + kShare, count);
      }
      const uint32_t mine = next + __popc(idle & lt);
      if (!(walk || promising) && mine < end) {
        p = first + mine;
        c = (int)p;
        c_min = max((int)p - (int)window, 0);
        ml = dist = off = 0;
        mask = 0xffffffu;
        lim = min(max_match, len - (lo + p));
        left = chain_depth + 1;
        has = true;
        key = word(p);
        if (lim >= 3u) move();
      }
      if (next < end) next = min(next + __popc(idle), end);
      if (next >= count && !__any_sync(kFull, walk || promising || has)) break;
    }
#pragma unroll
    for (int u = 0; u < kWalkSteps; u++) {
      if (walk) {
        if (((word(c + off) ^ key) & mask) == 0) {
          promising = true;
          walk = false;
        } else {
          move();
        }
      }
    }
    const uint32_t ready = __ballot_sync(kFull, promising);
    if (__popc(ready) >= (int)kCompareAt || (ready && !__any_sync(kFull, walk))) {
      if (promising) {
        promising = false;
        uint32_t k = 0, x;
        do {
          x = word(c + k) ^ word(p + k);
          k += 4;
        } while (!x && k < lim);
        if (x) k = k - 4u + ((uint32_t)(__ffs((int)x) - 1) >> 3);
        k = min(k, lim);
        if (k >= 3 && k > ml) {
          ml = k;
          dist = p - (uint32_t)c;
          off = k - 3u;
          mask = 0xffffffffu;
          key = word(p + off);
        }
        if (ml != lim) move();
      }
    }
  }
}

// DE rule (Sec. 4.2, as read in gmp_compress): a match's source bytes before
// its own position must avoid the bytes that earlier back-references of its
// 32-sequence group write; it is cut at the first such byte (to nothing if
// fewer than 3 bytes remain).  Lane g holds the g-th range of the group
// (empty: a literal run), so that a cut is one reduction over the warp; the
// other values are the same in every lane.
struct Group {
  uint32_t lo = 0, hi = 0;  // this lane's range
  uint32_t n = 0;           // ranges so far
  uint32_t lo_min = ~0u;    // start of the first back-reference
  __device__ void add(uint32_t from, uint32_t to) {
    const bool here = (threadIdx.x & 31u) == n;
    lo = here ? from : lo;
    hi = here ? to : hi;
    lo_min = from != to ? min(lo_min, from) : lo_min;  // ranges rise
    if (++n == 32) {
      n = lo = hi = 0;
      lo_min = ~0u;
    }
  }
  __device__ void grow(uint32_t a, uint32_t first) {  // a ranges, set by their lanes, from `first` on
    lo_min = min(lo_min, first);
    n += a;
    if (n == 32) {
      n = lo = hi = 0;
      lo_min = ~0u;
    }
  }
  // what a match of L >= 3 bytes at q, distance D, is cut to
  __device__ uint32_t cut(uint32_t q, uint32_t L, uint32_t D) const {
    const uint32_t src = q - D, end = min(src + L, q);
    if (end <= lo_min) return L;
    // (an empty range is 0, 0)
    L = __reduce_min_sync(kFull, lo < end && hi > src ? max(lo, src) - src : L);
    return L >= 3 ? L : 0u;
  }
  // the same of a match of each lane's (less than 3 if nothing is left)
  __device__ uint32_t cut_each(uint32_t q, uint32_t L, uint32_t D) const {
    const uint32_t src = q - D, end = min(src + L, q);
    for (uint32_t g = 0; g < n; g++) {
      const uint32_t a = __shfl_sync(kFull, lo, g), z = __shfl_sync(kFull, hi, g);
      L = a < end && z > src ? min(L, max(a, src) - src) : L;
    }
    return L;
  }
};

constexpr uint32_t kParseThreads = 256;
constexpr uint32_t kChunk = 2048;  // positions parsed at a time
constexpr uint32_t kOver = 128;
constexpr uint32_t kNoMatch = 0xffffffffu;

struct ParseSmem {
  // per position of the chunk: where the next match token from here starts
  // (low half) and ends (high half), or kNoMatch, and the highest source end
  // (position in the block) of the matches looked at to decide so
  uint2 jump[kChunk];
  uint16_t next[kChunk + kOver];  // that end; where no token follows the chunk's stop; itself from there on
  uint2 list[kChunk / 3 + 2];  // the chunk's tokens: start of their literals; match start << 8 | length
  // matches of the chunk, and of the one after it while this one is walked
  // (it starts at most a match and its lazy steps past the chunk's end)
  // (length | distance << 8)
  uint32_t match[2][kChunk + kOver];
  uint32_t match_rows[kChunk / 32];  // a bit per position with a match
  uint32_t p, n_list, first_token;
};

// One CTA per block.  A chunk's decisions are independent but for where the
// parse enters it (and, for DE, the group's earlier ranges: a match whose
// sources end below the group's first back-reference cannot be cut, which the
// walking warp sees from one number; the others it decides one by one).
// Bound by that warp's chain of one shared-memory read per token.  One
// thread deciding every position took 10.6 ms for 64 MiB of text (256
// blocks), 16.5 for 16 MiB of CSV rows with DE; now 1.4 and 1.7.
__global__ void __launch_bounds__(kParseThreads) parse_kernel(const uint8_t* best_len, const uint16_t* best_dist,
                                                              uint64_t n, uint32_t block_size, uint32_t max_match,
                                                              int de, int byte_mode, int lazy, gmp::ParseToken* tok,
                                                              uint32_t* tpos, uint64_t stride, uint32_t* count) {
  __shared__ ParseSmem S;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const uint64_t b = blockIdx.x, base = b * (uint64_t)block_size;
  const uint32_t len = (uint32_t)min((uint64_t)block_size, n - base);
  gmp::ParseToken* t = tok + b * stride;
  uint32_t* tp = tpos + b * stride;
  // warp 0's state: tokens so far, start of the pending literals, DE group
  uint32_t nt = 0, lit_start = 0;
  Group grp;
  auto put = [&](uint32_t ll, uint32_t match) {  // a token at once (not by way of the list)
    if (nt < stride && lane == 0) {
      t[nt] = gmp::ParseToken{ll, match};
      tp[nt] = lit_start;
    }
    nt++;
  };
  // loads the matches of [from, from + kChunk + kOver) into buffer k; threads
  // t of m
  auto fetch = [&](int k, uint32_t from, uint32_t t_, uint32_t m) {
#pragma unroll 4
    for (uint32_t i = t_; i < kChunk + kOver; i += m) {
      const bool in = from + i < len;
      const uint8_t l = in ? __ldg(best_len + base + from + i) : (uint8_t)0;
      const uint16_t d = in ? __ldg(best_dist + base + from + i) : (uint16_t)0;
      S.match[k][i] = l | ((uint32_t)d << 8);
    }
  };
  int buf = 0;
  uint32_t buf_at = 0;  // position of the buffer's first entry
  fetch(0, 0, tid, kParseThreads);
  __syncthreads();
  for (uint32_t c0 = 0; c0 < len; buf ^= 1) {
    const uint32_t* match = S.match[buf] + (c0 - buf_at);
    const uint32_t cn = min(kChunk, len - c0);
    // decisions are taken up to `stop`, so that the lazy look at the next
    // position stays in the chunk, and look up to `end`
    const uint32_t stop = c0 + cn == len ? cn : cn - 1;
    // positions with a match: the token that a decision there gives
    for (uint32_t row = warp; row < kChunk / 32; row += kParseThreads / 32) {
      const uint32_t i = 32 * row + lane;
      const uint32_t x = match[i];
      uint32_t L = x & 255u;
      const bool any = L >= 3 && i < stop;
      const uint32_t bits = __ballot_sync(kFull, any);
      if (lane == 0) S.match_rows[row] = bits;
      if (any) {
        uint32_t m = i, src_end = min(c0 + i - (x >> 8) + L, c0 + i);
        if (lazy) {
          while (m + 1 < cn && L < max_match) {
            const uint32_t x2 = match[m + 1], L2 = x2 & 255u;
            if (L2 >= 3) src_end = max(src_end, min(c0 + m + 1 - (x2 >> 8) + L2, c0 + m + 1));
            if (L2 < 3 || L2 <= L) break;
            m++;  // the byte at m stays a literal
            L = L2;
          }
        }
        S.jump[i] = make_uint2(m | ((m + L) << 16), src_end);
      }
    }
    __syncthreads();
    // positions without one: the next one's
    for (uint32_t row = warp; row < kChunk / 32; row += kParseThreads / 32) {
      const uint32_t i = 32 * row + lane, bits = S.match_rows[row];
      if (!((bits >> lane) & 1u)) {
        uint32_t r = row, m = bits & (0xfffffffeu << lane);
        while (!m && ++r < kChunk / 32) m = S.match_rows[r];
        S.jump[i] = m ? S.jump[32 * r + (uint32_t)__ffs((int)m) - 1u] : make_uint2(kNoMatch, 0);
      }
      const uint32_t j = S.jump[i].x;
      S.next[i] = (uint16_t)(i >= stop ? i : j == kNoMatch ? stop : j >> 16);
    }
    if (tid < kOver) S.next[kChunk + tid] = (uint16_t)(kChunk + tid);
    __syncthreads();
    if (tid >= 32) {
      fetch(buf ^ 1, c0 + stop, tid - 32, kParseThreads - 32);
    } else {
      // the warp walks: up to 32 tokens (DE: the rest of the group) by one
      // read each, every lane keeping where one of them was decided; then each
      // lane looks its token up, and the warp takes those before the first
      // that needs a closer look
      uint32_t p = 0, k = 0, first_token = nt;  // position in the chunk, tokens in the list
      auto list = [&](uint32_t at, uint32_t lits, uint32_t m, uint32_t e) {
        S.list[at] = make_uint2(lits, (m << 8) | (e - m));
      };
      while (p < stop) {
        const uint32_t n = de ? grp.n : 0u;
        uint32_t mine = kChunk, q = p;
        for (uint32_t x = n; x < 32u && q < stop; x += 8) {
#pragma unroll
          for (uint32_t y = 0; y < 8; y++) {
            mine = lane == x + y ? q : mine;
            q = S.next[q];
          }
        }
        bool valid = lane >= n && mine < stop;
        const uint2 j = valid ? S.jump[mine] : make_uint2(kNoMatch, 0);
        valid = valid && j.x != kNoMatch;
        const uint32_t m = j.x & 0xffffu, e = j.x >> 16, lits = lane == n ? lit_start : c0 + mine;
        const uint32_t all = __ballot_sync(kFull, valid);  // lanes from n on, without gaps
        const uint32_t m_n = __shfl_sync(kFull, m, n);
        const uint32_t lo_min = lane == n ? grp.lo_min : min(grp.lo_min, c0 + m_n);
        const bool look = valid && ((de && j.y > lo_min) || (byte_mode && c0 + m - lits > kByteMaxLit));
        const uint32_t looks = __ballot_sync(kFull, look);
        const uint32_t taken = looks ? all & ((looks & (0u - looks)) - 1u) : all;
        const uint32_t a = (uint32_t)__popc(taken);
        if ((taken >> lane) & 1u) {
          list(k + lane - n, lits, m, e);
          grp.lo = c0 + m;
          grp.hi = c0 + e;
        }
        if (a) {
          p = __shfl_sync(kFull, e, n + a - 1u);
          lit_start = c0 + p;
          k += a;
          nt += a;
          if (de) grp.grow(a, c0 + m_n);
        }
        if (!looks) {
          if (n + a < 32u && __shfl_sync(kFull, mine, n + a) < stop) p = stop;  // no further match
          continue;
        }
        // the decision at p: in a DE stream a source may lie in the group;
        // in a Byte stream the literals before the match may be too many
        uint32_t from = p;
        if (de) {
          auto match_at = [&](uint32_t y) -> uint32_t {
            const uint32_t x = match[y], L = x & 255u;
            return L < 3 ? 0u : grp.cut(c0 + y, L, x >> 8);
          };
          for (uint32_t x; !(x = __ballot_sync(kFull, (match[p + lane] & 255u) >= 3)) || !(x & 1u);)
            p += x ? (uint32_t)__ffs((int)x) - 1u : 32u;  // there is a match before the chunk's stop
          uint32_t L = match_at(p);
          if (!L) {
            // the next position whose match the group leaves something of, 32
            // at a time: in a run of one byte nearly every source lies in the
            // group (16 MiB of zeros in 256 KiB blocks: one position per walk
            // 121 ms, 3.4 so; one thread for the block 58)
            uint32_t left = 0;
            while (!left && ++p < stop) {
              const uint32_t x = match[p + lane], q = c0 + p + lane;
              const uint32_t l = grp.cut_each(q, x & 255u, x >> 8);  // (every lane: it shuffles)
              left = __ballot_sync(kFull, l >= 3 && p + lane < stop);
              p += left ? (uint32_t)__ffs((int)left) - 1u : 31u;
            }
            p = min(p, stop);
            if (!left) continue;
            L = match_at(p);
          }
          if (lazy) {
            while (p + 1 < cn && L < max_match) {
              const uint32_t L2 = match_at(p + 1);
              if (L2 <= L) break;
              p++;
              L = L2;
            }
          }
          from = p;
          p += L;
        } else {
          from = S.jump[p].x & 0xffffu;
          p = S.jump[p].x >> 16;
        }
        if (byte_mode && c0 + from - lit_start > kByteMaxLit) {
          // the list goes out first, then the literal runs
          __syncwarp();
          for (uint32_t i = lane; i < k; i += 32) {
            const uint32_t x = S.list[i].y, at = x >> 8, u = first_token + i;
            if (u < stride) {
              t[u] = gmp::ParseToken{c0 + at - S.list[i].x, (match[at] & ~255u) | (x & 255u)};
              tp[u] = S.list[i].x;
            }
          }
          __syncwarp();
          k = 0;
          while (c0 + from - lit_start > kByteMaxLit) {
            put(kByteMaxLit, 0);
            lit_start += kByteMaxLit;
            if (de) grp.add(0, 0);
          }
          first_token = nt;
        }
        list(k, lit_start, from, p);  // the same from every lane
        k++;
        nt++;
        lit_start = c0 + p;
        if (de) grp.add(c0 + from, c0 + p);
      }
      if (lane == 0) {
        S.p = p;
        S.n_list = k;
        S.first_token = first_token;
      }
    }
    __syncthreads();
    for (uint32_t i = tid; i < S.n_list; i += kParseThreads) {
      const uint32_t x = S.list[i].y, at = x >> 8, u = S.first_token + i;
      if (u < stride) {
        t[u] = gmp::ParseToken{c0 + at - S.list[i].x, (match[at] & ~255u) | (x & 255u)};
        tp[u] = S.list[i].x;
      }
    }
    buf_at = c0 + stop;
    c0 += S.p;
    __syncthreads();
  }
  if (tid < 32) {
    for (; byte_mode && len - lit_start > kByteMaxLit; lit_start += kByteMaxLit) put(kByteMaxLit, 0);
    if (lit_start < len) put(len - lit_start, 0);
    if (lane == 0) count[b] = nt;
  }
}

// Device times of the calling thread's last gmp_compress_gpu.
thread_local gmp_gpu_compress_times g_times = {0, 0, 0, 0};

// A call's device memory: one allocation for everything whose size is known
// from the input's, and one for the stream's blocks when they do not fit where
// the matches were.  Eleven buffers allocated and freed one by one took 0.5 ms
// more: 64 MiB of text 8.30 -> 7.79 ms, 16 MiB of records (Byte) 4.81 -> 4.35,
// 1 MiB of text 2.44 -> 2.17.
struct DeviceBuffers {
  void* p[2] = {};
  uint64_t bytes = 0;
  uint64_t place(uint64_t n) {  // its offset in the first allocation
    const uint64_t at = bytes;
    bytes += (n + 255u) & ~(uint64_t)255u;
    return at;
  }
  ~DeviceBuffers() {
    for (void* q : p)
      if (q) cudaFree(q);
  }
};

}  // namespace

extern "C" {

int gmp_compress_gpu(int device, const void* host_in, size_t n, const gmp_compress_opts* opts, void* host_out,
                     size_t cap, size_t* out_bytes) {
  if ((!host_in && n) || !opts || !host_out || !out_bytes) return GMP_ERR_INVALID_ARG;
  const gmp_compress_opts o = *opts;
  if (!gmp::compress_opts_ok(o)) return GMP_ERR_INVALID_ARG;
  const uint8_t* in = static_cast<const uint8_t*>(host_in);
  const uint64_t nb = (n + o.block_size - 1) / o.block_size;
  g_times = gmp_gpu_compress_times{0, 0, 0, 0};
  if (nb == 0) {
    uint64_t total = 0;
    gmp::stream_layout(nullptr, 0, nullptr, &total);
    if (total > cap) return GMP_ERR_CAPACITY;
    gmp::write_stream_header(o, 0, 0, nullptr, total, static_cast<uint8_t*>(host_out));
    *out_bytes = total;
    return GMP_OK;
  }
  int prev = -1;
  if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
  cudaError_t e = cudaSetDevice(device);
  if (e != cudaSuccess) return gmp::cuda_error(e, "cudaSetDevice");
  int rc = GMP_OK;
  {
    // tokens per block: at most one per 3 bytes plus the literal-only runs
    const uint64_t stride = o.block_size / 3 + o.block_size / kByteMaxLit + 4;
    DeviceBuffers D;
    cudaEvent_t ev[5] = {};
    auto check = [&](cudaError_t err, const char* what) {
      if (err != cudaSuccess && rc == GMP_OK) rc = gmp::cuda_error(err, what);
      return rc == GMP_OK;
    };
    for (auto& x : ev) check(cudaEventCreate(&x), "cudaEventCreate");
    int sms = 0;
    check(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device), "cudaDeviceGetAttribute");
    uint8_t* d_in = nullptr;
    uint8_t* d_len = nullptr;
    uint16_t* d_dist = nullptr;
    gmp::ParseToken* d_tok = nullptr;
    uint32_t* d_tpos = nullptr;
    uint32_t* d_count = nullptr;
    unsigned long long* d_counter = nullptr;
    gmp::EncBlockPlan* d_plan = nullptr;
    gmp::EncShare* d_share = nullptr;
    uint64_t* d_bytes = nullptr;
    gmp::EncLaunch L{};
    L.n = n;
    L.block_size = o.block_size;
    L.n_sub = o.byte_mode ? 0u : o.n_sub;
    L.cwl = o.cwl;
    L.window = o.window;
    L.max_match = o.max_match;
    L.byte_mode = o.byte_mode ? 1 : 0;
    L.n_blocks = nb;
    L.stride = stride;
    L.threads = gmp::encode_threads(L, (uint32_t)std::max(sms, 1));
    L.n_share = (uint32_t)std::min<uint64_t>(L.threads, stride);
    L.grid = (unsigned)std::min<uint64_t>(nb, (uint64_t)std::max(sms, 1) * 16);
    uint64_t* d_off = nullptr;
    const uint64_t at_in = D.place(n + 16), at_len = D.place(n), at_dist = D.place(2 * n), matches_end = D.bytes;
    const uint64_t at_tok = D.place(nb * stride * sizeof(gmp::ParseToken)), at_tpos = D.place(nb * stride * sizeof(uint32_t));
    const uint64_t at_count = D.place(nb * sizeof(uint32_t)), at_counter = D.place(2 * sizeof(unsigned long long));
    const uint64_t at_plan = D.place(nb * sizeof(gmp::EncBlockPlan)), at_bytes = D.place(nb * sizeof(uint64_t));
    const uint64_t at_share = D.place(nb * L.n_share * sizeof(gmp::EncShare)), at_off = D.place(nb * sizeof(uint64_t));
    if (check(cudaMalloc(&D.p[0], D.bytes), "cudaMalloc")) {
      uint8_t* m = static_cast<uint8_t*>(D.p[0]);
      d_in = m + at_in;
      d_len = m + at_len;
      d_dist = reinterpret_cast<uint16_t*>(m + at_dist);
      d_tok = reinterpret_cast<gmp::ParseToken*>(m + at_tok);
      d_tpos = reinterpret_cast<uint32_t*>(m + at_tpos);
      d_count = reinterpret_cast<uint32_t*>(m + at_count);
      d_counter = reinterpret_cast<unsigned long long*>(m + at_counter);
      d_plan = reinterpret_cast<gmp::EncBlockPlan*>(m + at_plan);
      d_bytes = reinterpret_cast<uint64_t*>(m + at_bytes);
      d_share = reinterpret_cast<gmp::EncShare*>(m + at_share);
      d_off = reinterpret_cast<uint64_t*>(m + at_off);
    }
    int* d_error = reinterpret_cast<int*>(d_counter + 1);
    if (rc == GMP_OK) {
      check(cudaMemcpy(d_in, in, n, cudaMemcpyHostToDevice), "cudaMemcpy");
      check(cudaMemset(d_counter, 0, 2 * sizeof(unsigned long long)), "cudaMemset");
    }
    if (rc == GMP_OK) {
      check(cudaEventRecord(ev[0]), "cudaEventRecord");
      // the links lie where the tokens go later
      uint16_t* d_link = reinterpret_cast<uint16_t*>(d_tok);
      chain_kernel<<<(unsigned)nb, kStep>>>(d_in, n, o.block_size, d_link);
      check(cudaGetLastError(), "chain_kernel");
      // runs of 32 Ki positions, whose window of as many more is loaded once
      // for all of them; of fewer while there are not two per SM
      uint32_t span = 32768;
      auto runs = [&](uint32_t v) { return ((uint64_t)o.block_size + v - 1) / v * nb; };
      while (span > 4096 && (runs(span) < 2ull * (uint64_t)std::max(sms, 1) || span >= 2ull * o.block_size)) span /= 2;
      const uint64_t per_block = ((uint64_t)o.block_size + span - 1) / span;
      const int smem = (int)(((2 * (o.window + span) + 15) & ~15u) + o.window + span + kLook + 32);
      check(cudaFuncSetAttribute(search_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSearchSmemMax),
            "cudaFuncSetAttribute");
      if (rc == GMP_OK) {
        search_kernel<<<(unsigned)(per_block * nb), kSearchThreads, smem>>>(
            d_in, n, o.block_size, o.window, o.max_match, std::min(o.chain_depth, 64u), span, (uint32_t)per_block,
            d_link, d_len, d_dist);
        check(cudaGetLastError(), "search_kernel");
      }
    }
    if (rc == GMP_OK) {
      check(cudaEventRecord(ev[1]), "cudaEventRecord");
      parse_kernel<<<(unsigned)nb, kParseThreads>>>(d_len, d_dist, n, o.block_size, o.max_match, o.de ? 1 : 0,
                                                    o.byte_mode ? 1 : 0, o.lazy ? 1 : 0, d_tok, d_tpos, stride,
                                                    d_count);
      check(cudaGetLastError(), "parse_kernel");
    }
    // entropy coding on the GPU: plan every block (sizes), lay the blocks out
    // on the host, write them
    L.in = d_in;
    L.tok = d_tok;
    L.tpos = d_tpos;
    L.count = d_count;
    L.plan = d_plan;
    L.share = d_share;
    L.block_bytes = d_bytes;
    L.error = d_error;
    if (rc == GMP_OK) {
      check(cudaEventRecord(ev[2]), "cudaEventRecord");
      check(gmp::launch_encode_plan(L), "plan_kernel");
    }
    std::vector<uint64_t> sizes(nb), offsets(nb);
    int h_error = 0;
    if (rc == GMP_OK) check(cudaMemcpy(sizes.data(), d_bytes, nb * sizeof(uint64_t), cudaMemcpyDeviceToHost),
                            "cudaMemcpy");
    if (rc == GMP_OK) check(cudaMemcpy(&h_error, d_error, sizeof(int), cudaMemcpyDeviceToHost), "cudaMemcpy");
    if (rc == GMP_OK && h_error) rc = GMP_ERR_INVALID_ARG;  // a parse that fails its checks (not expected)
    uint64_t total = 0, first = 0;
    if (rc == GMP_OK) {
      first = gmp::stream_layout(sizes.data(), nb, offsets.data(), &total);
      if (total > cap) rc = GMP_ERR_CAPACITY;
    }
    const uint64_t body = total - first - 16;  // the blocks, back to back
    // where the matches were, which the parse was the last to read
    uint8_t* d_body = d_len;
    if (rc == GMP_OK && body > matches_end - at_len && check(cudaMalloc(&D.p[1], body), "cudaMalloc"))
      d_body = static_cast<uint8_t*>(D.p[1]);
    if (rc == GMP_OK) {
      for (uint64_t b = 0; b < nb; b++) offsets[b] -= first;
      check(cudaMemcpy(d_off, offsets.data(), nb * sizeof(uint64_t), cudaMemcpyHostToDevice), "cudaMemcpy");
      if (rc == GMP_OK) check(gmp::launch_encode_write(L, d_off, d_body), "write_kernel");
      if (rc == GMP_OK) check(cudaEventRecord(ev[3]), "cudaEventRecord");
      uint8_t* out = static_cast<uint8_t*>(host_out);
      if (rc == GMP_OK) check(cudaMemcpy(out + first, d_body, body, cudaMemcpyDeviceToHost), "cudaMemcpy");
      if (rc == GMP_OK) {
        for (uint64_t b = 0; b < nb; b++) offsets[b] += first;
        gmp::write_stream_header(o, n, nb, offsets.data(), total, out);
        *out_bytes = total;
        float t = 0;
        if (cudaEventElapsedTime(&t, ev[0], ev[1]) == cudaSuccess) g_times.match_ms = t;
        if (cudaEventElapsedTime(&t, ev[1], ev[2]) == cudaSuccess) g_times.parse_ms = t;
        if (cudaEventElapsedTime(&t, ev[2], ev[3]) == cudaSuccess) g_times.encode_ms = t;
        g_times.compressed_bytes = total;
      }
    }
    for (auto& x : ev)
      if (x) cudaEventDestroy(x);
  }
  if (prev >= 0) cudaSetDevice(prev);
  return rc;
}

void gmp_compress_gpu_last_times(gmp_gpu_compress_times* t) {
  if (t) *t = g_times;
}

}  // extern "C"
