// gmp_decode_common.h - device code shared by the decode kernels
// (gmp_decode.cu, gmp_tile.cu): launch parameters, the host-to-host
// pipeline's flags, canonical codes, small warp primitives.
#ifndef GMP_DECODE_COMMON_H_
#define GMP_DECODE_COMMON_H_

#include <cuda_runtime.h>
#include <stdint.h>

#include "gmp.h"
#include "gmp_internal.h"

namespace gmp {

constexpr uint32_t FULL = 0xffffffffu;

constexpr int LUT_BITS = 12;  // the longest code (cwl <= 12)
constexpr int LUT_SIZE = 1 << LUT_BITS;
constexpr uint16_t LONG_CODE = 0xffff;
constexpr int N_LL = 319;
constexpr int N_OFF = 30;
constexpr int MAX_SUB = 64;

// Canonical arrays of one tree (Sec. 3.1): per code length its code count,
// its first index in the symbol list sorted by (length, symbol), and its
// first code.
struct Canon {
  uint32_t cnt[16], idx[16], first[16];
};

struct KParams {
  const gmp_file_desc* files;  // batch mode; nullptr in single-stream mode
  const uint64_t* item_start;  // batch mode: n_files + 1 prefix sums
  uint32_t n_files;
  gmp_file_desc single;  // single-stream mode
  int32_t* status;       // one per file
  unsigned long long* counter;
  uint8_t* scratch;
  uint64_t slot_bytes;
  uint64_t shadow_off;  // offset of the literal shadow inside a slot (256-byte aligned)
  uint32_t max_seq, max_out;
  unsigned long long* stats;  // [groups, rounds, de_fallback, blocks, max_rounds, cycles x3]
  int collect_stats;
  int resolve;  // 0: by the stream's DE flag, 1: MRR always, 2: sequential copying (SC)
  const uint32_t* route;  // null, or: of a pair of launches the one it names (a Route) runs
  int spread;   // 1: first items fixed and interleaved over the CTAs; 0: all from the counter
  // Host-to-host pipeline (all null otherwise): a file's input is complete
  // once in_ready[file] reaches gen (written by the copy stream after the
  // copy); out_ready[file] is set to gen once all its blocks are decoded
  // (done[file] counts them), and by the last warp to exit (exited counts
  // the warps) for every file.
  const uint32_t* in_ready;
  uint32_t* abort_wait;  // set once a wait has run out: later waits give up at once
  unsigned long long wait_ns;
  uint32_t* out_ready;
  uint32_t* done;
  uint32_t* exited;
  uint32_t gen;
};

cudaError_t launch_tile(const KParams& P, int grid, int warps_per_cta, bool pipe, cudaStream_t stream);
cudaError_t launch_coop(const KParams& P, int grid, int warps, bool pipe, cudaStream_t stream);

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31u; }

__device__ __forceinline__ void set_status(int32_t* st, int code) { atomicCAS(st, 0, code); }

// ---- host-to-host pipeline flags
// The wait for a file's input is bounded: the host's limit (10 s unless the
// context sets another) of the global timer, and at most 2^24 polls; past
// that the file gets GMP_STATUS_INPUT_TIMEOUT, its blocks are skipped and
// every later wait of the launch gives up at once, so the launch always ends.
constexpr uint32_t kInputWaitPolls = 1u << 24;

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ uint32_t ld_acquire_sys(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.sys.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_sys(uint32_t* p, uint32_t v) {
  asm volatile("st.release.sys.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Whole warp: true once *flag has reached gen (cyclic comparison, as the
// copy stream's flag values wrap), false if the wait ran out.  The warp polls
// and sleeps as one: with lane 0 polling and sleeping alone while the other
// lanes waited at a shuffle, the warps decoded their next blocks 2 to 2.7
// times slower (measured on text256m, (In) mode).
static __device__ __noinline__ bool wait_input(const uint32_t* flag, uint32_t* abort_wait, uint32_t gen,
                                        unsigned long long wait_ns) {
  const unsigned long long t0 = global_ns();
  bool ok = false;
  for (uint32_t i = 0; i < kInputWaitPolls; i++) {
    // lane 0 reads the flag, the abort word and the clock; every decision
    // below is taken on its values, so the lanes leave the loop together
    uint32_t v = 0, stop = 0;
    if ((threadIdx.x & 31u) == 0) {
      v = ld_acquire_sys(flag);
      stop = *reinterpret_cast<volatile uint32_t*>(abort_wait) != 0u || global_ns() - t0 > wait_ns;
    }
    v = __shfl_sync(0xffffffffu, v, 0);
    stop = __shfl_sync(0xffffffffu, stop, 0);
    if ((int32_t)(v - gen) >= 0) {
      ok = true;
      break;
    }
    if (stop) break;
    __nanosleep(i < 64 ? 64 : 1024);
  }
  if (!ok && (threadIdx.x & 31u) == 0) atomicExch(abort_wait, 1u);
  __syncwarp();
  return ok;
}

// Whole warp, after a block of `file` (n_blocks blocks) is decoded: every
// lane's output stores are made visible before the block is counted, and
// the count that completes the file publishes its out_ready flag.
static __device__ __noinline__ void block_done(uint32_t* done, uint32_t* out_ready, uint32_t gen, uint64_t n_blocks) {
  __threadfence();
  __syncwarp();
  if ((threadIdx.x & 31u) == 0) {
    const uint32_t d = atomicAdd(done, 1u) + 1u;
    if (d == (uint32_t)n_blocks) {
      __threadfence_system();
      st_release_sys(out_ready, gen);
    }
  }
  __syncwarp();
}

// Whole warp, on leaving the persistent loop: the last warp of the launch
// sets every file's out_ready flag, so that no copy stream waits on a flag
// that is never written.
static __device__ __noinline__ void pipeline_exit(uint32_t* exited, uint32_t* out_ready, uint32_t gen, uint32_t n_files,
                                           uint32_t n_warps) {
  __threadfence();
  uint32_t last = 0;
  if ((threadIdx.x & 31u) == 0) last = atomicAdd(exited, 1u) + 1u == n_warps;
  last = __shfl_sync(0xffffffffu, last, 0);
  if (last) {
    __threadfence_system();
    for (uint32_t f = threadIdx.x & 31u; f < n_files; f += 32) st_release_sys(out_ready + f, gen);
  }
}

__device__ __forceinline__ uint32_t ld_u32_nc(const uint8_t* p) { return __ldg(reinterpret_cast<const uint32_t*>(p)); }
__device__ __forceinline__ uint64_t ld_u64_nc(const uint8_t* p) {
  return __ldg(reinterpret_cast<const unsigned long long*>(p));
}

// inclusive warp scan of a 32-bit value
__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v) {
  const uint32_t lane = lane_id();
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    uint32_t y = __shfl_up_sync(FULL, v, d);
    if (lane >= (uint32_t)d) v += y;
  }
  return v;
}

// A code longer than the table's bits, by the canonical ranges: the 12-bit
// peek, most significant bit first, lies in length L's range [first_L,
// first_L + cnt_L) shifted left by 12 - L.  Returns (L << 9) | symbol.
template <int TB>
__device__ __forceinline__ uint32_t decode_long(const Canon& C, const uint16_t* sorted, uint32_t peek12) {
  const uint32_t v = __brev(peek12) >> (32 - LUT_BITS);
  for (int L = TB + 1; L <= LUT_BITS; L++) {
    const uint32_t code = v >> (LUT_BITS - L);
    if (code - C.first[L] < C.cnt[L]) return ((uint32_t)L << 9) | sorted[C.idx[L] + code - C.first[L]];
  }
  return 0;
}

// ---------------------------------------------------------------------------
// cp.async (16-byte, L2-only) global -> shared copies and their groups.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const uint32_t sa = (uint32_t)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_1() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }


// ---- block header (every field checked before it is used)
struct BlockView {
  const uint8_t* B;      // the block's first byte
  uint64_t comp_bytes;   // its size in the stream
  uint64_t out_offset;   // its output's place in the file's output
  uint64_t lit_off;      // Byte blocks: the literal section's offset in the block
  uint32_t n_seq, out_bytes, n_lit, flags, K, window, max_match;
  bool byte_fmt;  // Gompresso/Byte block: records and raw literals, no Huffman phase
};

// Reads and checks the stream header, the block reference and the block's
// sizes; the whole warp gets the same result (a gmp_status, 0 = good).
__device__ __forceinline__ int open_block(const gmp_file_desc& F, uint64_t b, BlockView& V) {
  const uint8_t* comp = F.comp;
  if (F.comp_bytes < 64 || (((uintptr_t)comp) & 15u)) return GMP_STATUS_BAD_HEADER;
  const uint32_t magic = ld_u32_nc(comp), w1 = ld_u32_nc(comp + 4), w3 = ld_u32_nc(comp + 12);
  const uint32_t w5 = ld_u32_nc(comp + 20), cwl = (w3 >> 16) & 0xffu;
  V.window = ld_u32_nc(comp + 16);
  V.flags = w1 >> 16;
  V.K = w3 & 0xffffu;
  V.max_match = (w5 >> 8) & 0xffu;
  V.byte_fmt = !(V.flags & 2u);
  if (magic != 0x31504d47u || (w1 & 0xffffu) != 1u || V.flags > 3u || V.window == 0 || V.window > 32768 ||
      (w5 & 0xffu) != 3u || V.max_match < 3 || V.max_match > 64)
    return GMP_STATUS_BAD_HEADER;
  if (V.byte_fmt ? (V.K != 0 || cwl != 0) : (V.K == 0 || V.K > MAX_SUB || cwl == 0 || cwl > 12))
    return GMP_STATUS_BAD_HEADER;
  const gmp_block_ref br = F.index[b];
  if ((br.comp_offset & 15) || br.comp_offset > F.comp_bytes || br.comp_bytes > F.comp_bytes - br.comp_offset ||
      br.out_offset > F.out_cap || br.out_bytes > F.out_cap - br.out_offset)
    return GMP_STATUS_OUTPUT_OVERRUN;
  if (br.comp_bytes < (V.byte_fmt ? 16ull : (192 + 12ull * V.K + 15) & ~15ull))  // through the bitstream start
    return GMP_STATUS_BAD_HEADER;
  V.B = comp + br.comp_offset;
  V.comp_bytes = br.comp_bytes;
  V.out_offset = br.out_offset;
  V.n_seq = ld_u32_nc(V.B);
  V.out_bytes = ld_u32_nc(V.B + 4);
  V.n_lit = 0;
  V.lit_off = 0;
  if (V.out_bytes != br.out_bytes) return GMP_STATUS_BAD_HEADER;
  if (V.byte_fmt) {
    // the records and the padded literal section lie inside the block (whole
    // 16-byte chunks, which the literal staging reads)
    V.n_lit = ld_u32_nc(V.B + 8);
    V.lit_off = (16ull + 4ull * V.n_seq + 15ull) & ~15ull;
    if (V.lit_off + ((V.n_lit + 15ull) & ~15ull) > br.comp_bytes) return GMP_STATUS_BAD_HEADER;
  }
  return 0;
}

}  // namespace gmp

#endif  // GMP_DECODE_COMMON_H_
