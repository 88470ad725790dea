// Relational operators of the unified AI query on the GPU.
//
//  * predicate mask (Table 1, WHERE row): a conjunction of `column op const`
//    terms evaluated over 2048-row tiles, 8 consecutive rows per thread with
//    16-byte vector loads; the result is a bitmask (1 bit per row) plus each
//    tile's survivor count.  A join probe (Section 4: reviews joined with
//    movies on movie id) runs in the same pass for rows that pass the terms.
//  * order-preserving stream compaction: tile counts -> exclusive scan ->
//    each tile re-reads only its 256-byte bitmask slice and writes the ids of
//    its set bits at its offset (reduce-then-scan; no inter-block waits).  Up to
//    kScanTilesMax tiles the block that finishes last scans the counts itself, or,
//    where no host waits for their sum, each compacting block adds them up;
//    up to kSmallRows rows one block does the whole filter.
//  * open-addressing hash table (int64 key -> build row), linear probing with
//    a bounded probe sequence.
//  * decision (Fig. 2: strict yes > no, or first argmax) and the masked
//    aggregates (Table 1, SELECT row): label counts, yes bitmask for the
//    yes-row ids, GROUP BY build row with warp-aggregated atomics.
#include <cstdio>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace aiq {
namespace {

constexpr int kThreads = 256;  // 256 threads x 8 rows = kRowsPerBlock
constexpr unsigned long long kEmptyKey = 0x8000000000000000ull;

// Raw 8 rows [r0, r0 + 8) of one term's column, as four 16-byte words for
// 4-byte columns (two used) or 64-bit words for int64 columns.
struct TermRows {
  int4 w[4];
};

__device__ __forceinline__ void load_term(const PredDev& p, int64_t r0, int64_t n, TermRows& t) {
  const bool full = r0 + 8 <= n;
  if (p.type == 1) {
    const int64_t* c = static_cast<const int64_t*>(p.col) + r0;
    if (full) {
      const int4* q = reinterpret_cast<const int4*>(c);
#pragma unroll
      for (int j = 0; j < 4; ++j) t.w[j] = q[j];
    } else {
      int64_t* v = reinterpret_cast<int64_t*>(t.w);
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = r0 + j < n ? c[j] : 0;
    }
  } else {
    const int32_t* c = static_cast<const int32_t*>(p.col) + r0;
    if (full) {
      const int4* q = reinterpret_cast<const int4*>(c);
      t.w[0] = q[0];
      t.w[1] = q[1];
    } else {
      int32_t* v = reinterpret_cast<int32_t*>(t.w);
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = r0 + j < n ? c[j] : 0;
    }
  }
}

// The term's 8 result bits for rows loaded by load_term.  The operator is
// resolved once per term (the switch is outside the loop over the 8 values).
template <typename T>
__device__ __forceinline__ uint32_t cmp8(const T* v, int op, T c) {
  uint32_t bits = 0;
  switch (op) {
    case 0:
#pragma unroll
      for (int j = 0; j < 8; ++j) bits |= static_cast<uint32_t>(v[j] < c) << j;
      break;
    case 1:
#pragma unroll
      for (int j = 0; j < 8; ++j) bits |= static_cast<uint32_t>(v[j] <= c) << j;
      break;
    case 2:
#pragma unroll
      for (int j = 0; j < 8; ++j) bits |= static_cast<uint32_t>(v[j] > c) << j;
      break;
    case 3:
#pragma unroll
      for (int j = 0; j < 8; ++j) bits |= static_cast<uint32_t>(v[j] >= c) << j;
      break;
    case 4:
#pragma unroll
      for (int j = 0; j < 8; ++j) bits |= static_cast<uint32_t>(v[j] == c) << j;
      break;
    default:
#pragma unroll
      for (int j = 0; j < 8; ++j) bits |= static_cast<uint32_t>(v[j] != c) << j;
      break;
  }
  return bits;
}

// A term on a 4-byte column.
__device__ __forceinline__ uint32_t eval_term4(const PredDev& p, const TermRows& t) {
  if (p.type == 2) return cmp8<float>(reinterpret_cast<const float*>(t.w), p.op, static_cast<float>(p.fvalue));
  // int32: a constant outside the int32 range decides every row alike (as the
  // SQL comparison in int64 would); inside it, compare in 32 bits
  const int32_t* v = reinterpret_cast<const int32_t*>(t.w);
  if (p.ivalue > INT32_MAX || p.ivalue < INT32_MIN) {
    const bool below = p.ivalue > INT32_MAX;  // every value is below the constant
    const bool r = p.op == 0 || p.op == 1 ? below : (p.op == 2 || p.op == 3 ? !below : p.op == 5);
    return r ? 0xFFu : 0u;
  }
  return cmp8<int32_t>(v, p.op, static_cast<int32_t>(p.ivalue));
}

__device__ __forceinline__ uint32_t eval_term(const PredDev& p, const TermRows& t) {
  if (p.type == 1) return cmp8<int64_t>(reinterpret_cast<const int64_t*>(t.w), p.op, p.ivalue);
  return eval_term4(p, t);
}

// Each thread holds one byte of row bits (rows 8*t .. 8*t+7 of the tile);
// assemble 32-bit words (4 lanes each), write them, and return the tile's
// popcount (valid in thread 0).
__device__ __forceinline__ int write_words_and_count(uint32_t byte, uint32_t* bits_tile, int* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t w = byte << (8 * (lane & 3));
  w |= __shfl_xor_sync(0xffffffffu, w, 1);
  w |= __shfl_xor_sync(0xffffffffu, w, 2);
  if ((lane & 3) == 0) bits_tile[threadIdx.x >> 2] = w;
  int c = __popc(byte);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if (lane == 0) red[warp] = c;
  __syncthreads();
  int total = 0;
  if (threadIdx.x == 0)
    for (int i = 0; i < kThreads / 32; ++i) total += red[i];
  return total;
}

// Any number of terms (also none, or more than four): one 2048-row tile per
// block, thread t on rows 8t .. 8t+7.  Thread 0 first asks the bulk-copy engine to
// pull every later term's column chunk of the tile (2048 x 4 or 8 bytes) into L2,
// so all columns stream from DRAM at once while each thread's own 16-byte
// loads of successive terms follow one after the other.
__global__ void __launch_bounds__(kThreads) k_predicate_mask(PredSet ps, int64_t n, uint32_t* bits,
                                                             int32_t* block_counts) {
  grid_launch_next();
  grid_wait();
  __shared__ int red[kThreads / 32];
  const int64_t tile = blockIdx.x;
  if (threadIdx.x == 0 && (tile + 1) * kRowsPerBlock <= n) {
    for (int i = 1; i < ps.n; ++i) {
      const int esz = ps.p[i].type == 1 ? 8 : 4;
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(static_cast<const uint8_t*>(ps.p[i].col) +
                                                                        tile * kRowsPerBlock * esz),
                   "r"(kRowsPerBlock * esz)
                   : "memory");
    }
  }
  const int64_t r0 = tile * kRowsPerBlock + threadIdx.x * 8;
  uint32_t byte = 0;
  if (r0 < n) {
    byte = r0 + 8 <= n ? 0xFFu : ((1u << (n - r0)) - 1u);
    for (int i = 0; i < ps.n; ++i) {
      TermRows t;
      load_term(ps.p[i], r0, n, t);
      byte &= eval_term(ps.p[i], t);
    }
  }
  const int total = write_words_and_count(byte, bits + tile * (kRowsPerBlock / 32), red);
  if (threadIdx.x == 0) block_counts[tile] = total;
}

// Block-wide exclusive scan of one int per thread (NT threads).
template <int NT>
__device__ __forceinline__ int block_excl_scan(int v, int* sh, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sh[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int s = lane < NT / 32 ? sh[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    if (lane < NT / 32) sh[lane] = s;
  }
  __syncthreads();
  const int before = warp ? sh[warp - 1] : 0;
  *total = sh[NT / 32 - 1];
  return before + x - v;
}

// Called by every thread of every block once its tile's count is written (by
// thread 0): the block that arrives last scans all counts into offsets, writes
// the total wherever it is wanted and leaves the arrival counter at zero for the
// next launch.  No block waits for another.
template <int NT>
__device__ __forceinline__ void scan_in_last_block(const TileScan& ts) {
  __shared__ int sh[NT / 32];
  __shared__ int last;
  if (threadIdx.x == 0) {
    __threadfence();  // the count before the arrival
    last = atomicAdd(ts.arrived, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();  // the arrivals before the other blocks' counts
  constexpr int kPer = 16;
  const int64_t n = gridDim.x;
  int64_t carry = 0;
  for (int64_t base = 0; base < n; base += NT * kPer) {
    const int64_t i0 = base + threadIdx.x * kPer;
    int v[kPer];
    int s = 0;
#pragma unroll
    for (int j = 0; j < kPer; j += 4) {
      if (i0 + j + 4 <= n) {
        *reinterpret_cast<int4*>(v + j) = __ldcg(reinterpret_cast<const int4*>(ts.counts + i0 + j));
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) v[j + k] = i0 + j + k < n ? __ldcg(ts.counts + i0 + j + k) : 0;
      }
    }
#pragma unroll
    for (int j = 0; j < kPer; ++j) s += v[j];
    int total;
    int64_t run = carry + block_excl_scan<NT>(s, sh, &total);
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      if (i0 + j < n) ts.offsets[i0 + j] = run;
      run += v[j];
    }
    carry += total;
    __syncthreads();  // sh is reused
  }
  if (threadIdx.x == 0) {
    ts.offsets[n] = carry;
    if (ts.total) *ts.total = carry;
    *ts.arrived = 0;
  }
}

// 1..4 terms and no join probe (every workload's filter): N8 terms on int64
// columns, then N4 on 4-byte ones.  Every term's loads are issued before the
// first compare, in a coalesced layout (lane l of warp w takes rows 4l..4l+3 and
// 128+4l..128+4l+3 of the warp's 256 rows, so one 16-byte load instruction covers
// 512 contiguous bytes), and eight lanes' nibbles form one bitmask word.  Same
// bitmask and tile counts as k_predicate_mask, whose terms load one after the
// other.  4,195,081 rows of an int32, an int64 and a float32 term (67 MB) take 18.7
// us from a cold cache with the counts' scan in the last block, against 15.5 us for
// k_predicate_mask plus 7.4 for a scan and a copy of the count in launches of their own.
// SCAN takes registers of its own and is left out where another kernel scans, and up to
// 8 bytes a row the bounds ask for the 32 that let eight blocks share an SM: 2^28 rows
// of one 4-byte term 202 -> 182 us, of two 317 -> 312; 2^24 rows of one, with the scan,
// 28.5 -> 25.3.
template <int N8, int N4, bool SCAN>
__global__ void __launch_bounds__(kThreads, 2 * N8 + N4 <= 2 ? 8 : 1) k_predicate_cols(PredSet ps, int64_t n, uint32_t* bits,
                                                             int32_t* block_counts, TileScan ts) {
  grid_launch_next();
  grid_wait();
  __shared__ int red[kThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t ra = static_cast<int64_t>(blockIdx.x) * kRowsPerBlock + warp * 256 + lane * 4;
  const int64_t rb = ra + 128;
  TermRows t[N8 + N4];
  const bool full = rb + 4 <= n;
#pragma unroll
  for (int i = 0; i < N8 + N4; ++i) {
    if (i < N8) {
      const int64_t* c = static_cast<const int64_t*>(ps.p[i].col);
      if (full) {
        t[i].w[0] = *reinterpret_cast<const int4*>(c + ra);
        t[i].w[1] = reinterpret_cast<const int4*>(c + ra)[1];
        t[i].w[2] = *reinterpret_cast<const int4*>(c + rb);
        t[i].w[3] = reinterpret_cast<const int4*>(c + rb)[1];
      } else {
        int64_t* v = reinterpret_cast<int64_t*>(t[i].w);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          v[j] = ra + j < n ? c[ra + j] : 0;
          v[4 + j] = rb + j < n ? c[rb + j] : 0;
        }
      }
    } else {
      const int32_t* c = static_cast<const int32_t*>(ps.p[i].col);
      if (full) {
        t[i].w[0] = *reinterpret_cast<const int4*>(c + ra);
        t[i].w[1] = *reinterpret_cast<const int4*>(c + rb);
      } else {
        int32_t* v = reinterpret_cast<int32_t*>(t[i].w);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          v[j] = ra + j < n ? c[ra + j] : 0;
          v[4 + j] = rb + j < n ? c[rb + j] : 0;
        }
      }
    }
  }
  uint32_t byte = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) byte |= (static_cast<uint32_t>(ra + j < n) << j) | (static_cast<uint32_t>(rb + j < n) << (4 + j));
  // value j < 4 of a term is row ra + j, value 4 + j is row rb + j
#pragma unroll
  for (int i = 0; i < N8 + N4; ++i)
    byte &= i < N8 ? cmp8<int64_t>(reinterpret_cast<const int64_t*>(t[i].w), ps.p[i].op, ps.p[i].ivalue)
                   : eval_term4(ps.p[i], t[i]);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t w = ((byte >> (4 * h)) & 0xFu) << (4 * (lane & 7));
    w |= __shfl_xor_sync(0xffffffffu, w, 1);
    w |= __shfl_xor_sync(0xffffffffu, w, 2);
    w |= __shfl_xor_sync(0xffffffffu, w, 4);
    if ((lane & 7) == 0) bits[blockIdx.x * int64_t(kRowsPerBlock / 32) + warp * 8 + h * 4 + (lane >> 3)] = w;
  }
  int c = __popc(byte);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if (lane == 0) red[warp] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int total = 0;
    for (int i = 0; i < kThreads / 32; ++i) total += red[i];
    block_counts[blockIdx.x] = total;
  }
  if constexpr (SCAN) scan_in_last_block<kThreads>(ts);
}

// A term's 4 result bits for rows r0 .. r0 + 3 (r0 a multiple of 4).
__device__ __forceinline__ uint32_t eval_rows4(const PredDev& p, int64_t r0, int64_t n) {
  TermRows t;
  const bool full = r0 + 4 <= n;
  if (p.type == 1) {
    const int64_t* c = static_cast<const int64_t*>(p.col) + r0;
    int64_t* v = reinterpret_cast<int64_t*>(t.w);
    if (full) {
      t.w[0] = *reinterpret_cast<const int4*>(c);
      t.w[1] = reinterpret_cast<const int4*>(c)[1];
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = r0 + j < n ? c[j] : 0;
    }
#pragma unroll
    for (int j = 4; j < 8; ++j) v[j] = 0;
    return cmp8<int64_t>(v, p.op, p.ivalue) & 0xFu;
  }
  const int32_t* c = static_cast<const int32_t*>(p.col) + r0;
  int32_t* v = reinterpret_cast<int32_t*>(t.w);
  if (full) {
    t.w[0] = *reinterpret_cast<const int4*>(c);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = r0 + j < n ? c[j] : 0;
  }
#pragma unroll
  for (int j = 4; j < 8; ++j) v[j] = 0;
  return eval_term4(p, t) & 0xFu;
}

constexpr int kProbeThreads = 512;  // x 4 rows = kRowsPerBlock

// The terms and the join probe of one 2048-row tile.  A thread's four keys are
// hashed together and their table slots read together (a probe is a chain of
// dependent reads: 500,000 rows took 14.7 us with eight in turn and 9.6 for the
// scan's three launches, 12.5 now with the scan); collisions walk on for the keys
// that are left.
__global__ void __launch_bounds__(kProbeThreads) k_probe_mask(PredSet ps, ProbeSpec probe, int64_t n, uint32_t* bits,
                                                              int32_t* block_counts, TileScan ts) {
  grid_launch_next();
  grid_wait();
  __shared__ int red[kProbeThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t r0 = static_cast<int64_t>(blockIdx.x) * kRowsPerBlock + threadIdx.x * 4;
  uint32_t nib = 0;
  if (r0 < n) {
    nib = r0 + 4 <= n ? 0xFu : ((1u << (n - r0)) - 1u);
    unsigned long long key[4];
    if (r0 + 4 <= n) {
      const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(probe.keys + r0);
      const ulonglong2 b = reinterpret_cast<const ulonglong2*>(probe.keys + r0)[1];
      key[0] = a.x, key[1] = a.y, key[2] = b.x, key[3] = b.y;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) key[j] = r0 + j < n ? static_cast<unsigned long long>(probe.keys[r0 + j]) : kEmptyKey;
    }
    for (int i = 0; i < ps.n; ++i) nib &= eval_rows4(ps.p[i], r0, n);
    const unsigned long long mask = static_cast<unsigned long long>(probe.capacity - 1);
    unsigned long long slot[4];
    uint32_t open = 0;  // keys still looked for
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      slot[j] = hash64(key[j]) & mask;
      open |= static_cast<uint32_t>(((nib >> j) & 1u) && key[j] != kEmptyKey) << j;
    }
    nib &= open;
    for (int64_t step = 0; open && step < probe.capacity; ++step) {
      unsigned long long k[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if ((open >> j) & 1u) k[j] = probe.table_keys[slot[j]];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (!((open >> j) & 1u)) continue;
        if (k[j] == key[j]) {
          open &= ~(1u << j);  // found; slot[j] is its slot
        } else if (k[j] == kEmptyKey) {
          open &= ~(1u << j);
          nib &= ~(1u << j);
        } else {
          slot[j] = (slot[j] + 1) & mask;
        }
      }
    }
    nib &= ~open;  // a table without an empty slot: every slot has been looked at
    int m[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) m[j] = (nib >> j) & 1u ? probe.table_vals[slot[j]] : -1;
    if (r0 + 4 <= n)
      *reinterpret_cast<int4*>(probe.match_out + r0) = make_int4(m[0], m[1], m[2], m[3]);
    else
      for (int j = 0; r0 + j < n; ++j) probe.match_out[r0 + j] = m[j];
  }
  uint32_t w = nib << (4 * (lane & 7));
  w |= __shfl_xor_sync(0xffffffffu, w, 1);
  w |= __shfl_xor_sync(0xffffffffu, w, 2);
  w |= __shfl_xor_sync(0xffffffffu, w, 4);
  if ((lane & 7) == 0) bits[blockIdx.x * int64_t(kRowsPerBlock / 32) + warp * 4 + (lane >> 3)] = w;
  int c = __popc(nib);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if (lane == 0) red[warp] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int total = 0;
    for (int i = 0; i < kProbeThreads / 32; ++i) total += red[i];
    block_counts[blockIdx.x] = total;
  }
  if (ts.arrived) scan_in_last_block<kProbeThreads>(ts);
}

constexpr int kSmallThreads = 1024;

// The whole filter of a small table in one block: each pass evaluates 8 rows a
// thread, scans the survivor counts and writes the ids.  At these sizes a launch
// costs more than the rows: a call on 10,007 rows takes 8.0 us in one launch,
// against 14.7 in four.
__global__ void __launch_bounds__(kSmallThreads) k_filter_small(PredSet ps, int64_t n, int32_t* ids, int64_t* count) {
  grid_launch_next();
  grid_wait();
  __shared__ int sh[kSmallThreads / 32];
  int base = 0;
  for (int64_t p0 = 0; p0 < n; p0 += kSmallThreads * 8) {
    const int64_t r0 = p0 + threadIdx.x * 8;
    uint32_t byte = 0;
    if (r0 < n) {
      byte = r0 + 8 <= n ? 0xFFu : ((1u << (n - r0)) - 1u);
      for (int i = 0; i < ps.n; ++i) {
        TermRows t;
        load_term(ps.p[i], r0, n, t);
        byte &= eval_term(ps.p[i], t);
      }
    }
    int total;
    int at = base + block_excl_scan<kSmallThreads>(__popc(byte), sh, &total);
    for (uint32_t b = byte; b; b &= b - 1) ids[at++] = static_cast<int32_t>(r0) + __ffs(b) - 1;
    base += total;
    __syncthreads();  // sh is reused
  }
  if (threadIdx.x == 0) *count = base;
}

constexpr unsigned kWideTilesMax = 488;          // k_compact_wide without a payload
constexpr unsigned kWidePayloadTilesMax = 2432;  // and with one: 16 blocks per SM
constexpr unsigned kTriggerBlocksMax = 4096;  // blocks of k_compact that let the next kernel start early
constexpr int kCompactWarps = 4;  // warps (= 2048-row tiles at a time) per compaction block

// Survivors before tile `end`, by all threads of a block (NT of them) together.
template <int NT>
__device__ __forceinline__ int sum_counts(const int32_t* counts, unsigned end, int* sh) {
  int s = 0;
  const unsigned quads = end / 4;
#pragma unroll 4
  for (unsigned i = threadIdx.x; i < quads; i += NT) {
    const int4 v = __ldcg(reinterpret_cast<const int4*>(counts) + i);
    s += (v.x + v.y) + (v.z + v.w);
  }
  if (threadIdx.x < end % 4) s += __ldcg(counts + quads * 4 + threadIdx.x);
  s = __reduce_add_sync(0xffffffffu, s);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  s = 0;
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) s += sh[w];
  return s;
}

// One warp per 2048-row tile: lane l owns bitmask words l and 32 + l of the
// tile (two coalesced loads).  In two passes (words 0..31, then 32..63) a warp
// shuffle scan gives every lane its output position and the lane writes the
// row offsets of its word's set bits, in order, into the warp's own 16-bit
// shared-memory slice; the slice is then written out as one coalesced run of
// ids.  No block-wide barrier is involved.  A payload (the join's build row
// per probe row) is gathered in that last loop (PAYLOAD): in the set-bit loop each
// gather stalled its lane (8.5 us for 500,000 probe rows).
//
// DIRECT: no scan has run, a block adds up the counts before its tiles itself (all
// of them come from L2, at 8192 tiles 32 KB for the last block), which takes the scan
// out of the filter: 4,195,081 rows of three terms (67 MB) 22.0 -> 18.6 us, 16,777,211 rows of
// one term 35.6 -> 26.0, against a scan by the predicate's last block.  For a caller
// whose host must know the count before the ids have a place, the scan stays.
template <bool PAYLOAD, bool DIRECT>
__global__ void __launch_bounds__(kCompactWarps * 32) k_compact(const uint32_t* bits, TileBase tb,
                                                                int64_t n, int32_t* ids, const int32_t* payload,
                                                                int32_t* payload_out) {
  // With many short blocks the trigger costs more than the overlap gives: 2^28 rows
  // (32,768 blocks) 38 us with it, 25 without.
  if (gridDim.x <= kTriggerBlocksMax) grid_launch_next();
  grid_wait();
  __shared__ uint16_t s_ids[kCompactWarps][kRowsPerBlock];  // row offsets within the tile
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n_tiles = (n + kRowsPerBlock - 1) / kRowsPerBlock;
  const int64_t tile = static_cast<int64_t>(blockIdx.x) * kCompactWarps + warp;
  int64_t before = 0;
  if (DIRECT) {
    __shared__ int sh[kCompactWarps];
    before = sum_counts<kCompactWarps * 32>(tb.counts, blockIdx.x * kCompactWarps, sh);
    for (int w = 0; w < warp; ++w)
      if (tile - warp + w < n_tiles) before += __ldcg(tb.counts + tile - warp + w);
    if (tile == n_tiles - 1 && lane == 0) *tb.total = before + __ldcg(tb.counts + tile);
  }
  if (tile < n_tiles) {
    const uint32_t* wt = bits + tile * (kRowsPerBlock / 32);
    const uint32_t wa = wt[lane], wb = wt[32 + lane];
    const int64_t out = DIRECT ? before : tb.offsets[tile];
    const int64_t tile0 = tile * kRowsPerBlock;
    int at0 = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t b = h ? wb : wa;
      const int c = __popc(b);
      int incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      int at = at0 + incl - c;
      const int base = (h * 32 + lane) * 32;
      while (b) {
        const int j = __ffs(b) - 1;
        b &= b - 1;
        s_ids[warp][at] = static_cast<uint16_t>(base + j);
        ++at;
      }
      at0 += __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncwarp();
    for (int i = lane; i < at0; i += 32) {
      const int64_t row = tile0 + s_ids[warp][i];
      ids[out + i] = static_cast<int32_t>(row);
      if (PAYLOAD) payload_out[out + i] = payload[row];
    }
  }
}

// The same for few tiles: a block per tile, 8 rows a thread, so that a tile's ids
// and payload gathers are all in flight together (a warp per tile leaves most of
// the GPU idle and walks them in turn: 500,000 rows with a payload 11.5 us, here
// 3.8).  Without a payload the two are even at 489 tiles (3.6 us) and a warp per
// tile is the faster above (2049 tiles: 4.4 us against 5.1).
template <bool PAYLOAD, bool DIRECT>
__global__ void __launch_bounds__(kThreads) k_compact_wide(const uint32_t* bits, TileBase tb, int32_t* ids,
                                                           const int32_t* payload, int32_t* payload_out) {
  grid_launch_next();
  grid_wait();
  __shared__ int sh[kThreads / 32];
  const int64_t tile = blockIdx.x;
  const uint32_t byte = reinterpret_cast<const uint8_t*>(bits + tile * (kRowsPerBlock / 32))[threadIdx.x];
  int64_t out;
  if (DIRECT) {
    __shared__ int sums[kThreads / 32];
    out = sum_counts<kThreads>(tb.counts, blockIdx.x, sums);
  } else {
    out = tb.offsets[tile];
  }
  const int64_t r0 = tile * kRowsPerBlock + threadIdx.x * 8;
  int m[8];
  if (PAYLOAD) {
#pragma unroll
    for (int j = 0; j < 8; ++j) m[j] = (byte >> j) & 1u ? payload[r0 + j] : 0;
  }
  int total;
  int64_t at = out + block_excl_scan<kThreads>(__popc(byte), sh, &total);
  if (DIRECT && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *tb.total = out + total;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    if ((byte >> j) & 1u) {
      ids[at] = static_cast<int32_t>(r0 + j);
      if (PAYLOAD) payload_out[at] = m[j];
      ++at;
    }
  }
}

// ---------------------------------------------------------------- scans ---
// Tile sums (2048 ints per block) -> single-block scan of the tile sums ->
// per-tile scan with the tile's offset.

__global__ void __launch_bounds__(kThreads) k_tile_sums(const int32_t* in, int64_t n, int64_t* sums) {
  grid_launch_next();
  grid_wait();
  __shared__ int64_t red[kThreads / 32];
  const int64_t base = static_cast<int64_t>(blockIdx.x) * kRowsPerBlock;
  int64_t s = 0;
  for (int i = threadIdx.x; i < kRowsPerBlock; i += kThreads)
    if (base + i < n) s += in[base + i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    int64_t t = 0;
    for (int i = 0; i < kThreads / 32; ++i) t += red[i];
    sums[blockIdx.x] = t;
  }
}

// Exclusive scan of n int64 (or int32) values into out[0..n], one block of 1024
// threads, each scanning a contiguous run sequentially.
template <typename T>
__global__ void __launch_bounds__(1024) k_scan_single(const T* in, int64_t n, int64_t* out) {
  grid_launch_next();
  grid_wait();
  __shared__ int64_t sh[1024];
  const int64_t per = (n + 1023) / 1024;
  const int64_t b = threadIdx.x * per;
  int64_t s = 0;
  for (int64_t i = b; i < b + per && i < n; ++i) s += in[i];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {
    int64_t y = threadIdx.x >= o ? sh[threadIdx.x - o] : 0;
    __syncthreads();
    sh[threadIdx.x] += y;
    __syncthreads();
  }
  int64_t run = sh[threadIdx.x] - s;
  for (int64_t i = b; i < b + per && i < n; ++i) {
    out[i] = run;
    run += in[i];
  }
  if (threadIdx.x == 1023) out[n] = sh[1023];
}

__global__ void __launch_bounds__(kThreads) k_tile_scan(const int32_t* in, int64_t n, const int64_t* tile_off,
                                                        int64_t* out) {
  grid_launch_next();
  grid_wait();
  __shared__ int sh[kThreads / 32];
  const int64_t base = static_cast<int64_t>(blockIdx.x) * kRowsPerBlock + threadIdx.x * 8;
  int v[8];
  int s = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    v[j] = base + j < n ? in[base + j] : 0;
    s += v[j];
  }
  int total;
  int pre = block_excl_scan<kThreads>(s, sh, &total);
  int64_t run = tile_off[blockIdx.x] + pre;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    if (base + j < n) out[base + j] = run;
    run += v[j];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[n] = tile_off[gridDim.x];
}

// ----------------------------------------------------------- hash build ---

__device__ __forceinline__ void hash_insert(unsigned long long key, int32_t row, unsigned long long* tk, int32_t* tv,
                                            int64_t cap, int* err) {
  if (key == kEmptyKey) {
    set_dev_error(err, DEVERR_SENTINEL_KEY);
    return;
  }
  const unsigned long long mask = static_cast<unsigned long long>(cap - 1);
  unsigned long long slot = hash64(key) & mask;
  for (int64_t step = 0; step < cap; ++step) {
    const unsigned long long prev = atomicCAS(tk + slot, kEmptyKey, key);
    if (prev == kEmptyKey) {
      tv[slot] = row;
      return;
    }
    if (prev == key) {
      set_dev_error(err, DEVERR_DUP_BUILD_KEY);
      return;
    }
    slot = (slot + 1) & mask;
  }
  set_dev_error(err, DEVERR_HASH_FULL);
}

// The build rows given by id.
__global__ void k_hash_build(const int64_t* keys, const int32_t* rows, int64_t n, unsigned long long* tk,
                             int32_t* tv, int64_t cap, int* err) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  hash_insert(static_cast<unsigned long long>(keys[rows[i]]), rows[i], tk, tv, cap, err);
}

// The build rows that satisfy the terms, straight from the columns: the table is
// sized for all rows, so that neither their ids nor their number is needed first.
__global__ void k_hash_build_where(const int64_t* keys, PredSet ps, int64_t n, unsigned long long* tk, int32_t* tv,
                                   int64_t cap, int* err) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const unsigned long long key = static_cast<unsigned long long>(keys[i]);
  uint32_t pass = 1;
  for (int t = 0; t < ps.n; ++t) {
    TermRows v{};
    if (ps.p[t].type == 1)
      reinterpret_cast<int64_t*>(v.w)[0] = static_cast<const int64_t*>(ps.p[t].col)[i];
    else
      v.w[0].x = static_cast<const int32_t*>(ps.p[t].col)[i];
    pass &= eval_term(ps.p[t], v);
  }
  if (pass & 1u) hash_insert(key, static_cast<int32_t>(i), tk, tv, cap, err);
}

__global__ void k_fill_u64(unsigned long long* p, int64_t n, unsigned long long v) {
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    p[i] = v;
}

// ------------------------------------------------------ decide/aggregate ---

__global__ void __launch_bounds__(kThreads) k_decide(const float* logits, int64_t S, int K, int32_t* decision,
                                                     uint32_t* yes_bits, int32_t* block_counts,
                                                     unsigned long long* label_counts) {
  grid_launch_next();
  grid_wait();
  __shared__ int red[kThreads / 32];
  __shared__ unsigned int hist[16];
  if (threadIdx.x < 16) hist[threadIdx.x] = 0;
  __syncthreads();
  const int64_t r0 = static_cast<int64_t>(blockIdx.x) * kRowsPerBlock + threadIdx.x * 8;
  uint32_t byte = 0;
  for (int j = 0; j < 8; ++j) {
    const int64_t r = r0 + j;
    if (r >= S) break;
    const float* z = logits + r * K;
    int d;
    if (K == 2) {
      d = z[0] > z[1] ? 1 : 0;  // strict: a tie is "no"
      byte |= static_cast<uint32_t>(d) << j;
      atomicAdd(&hist[d ? 0 : 1], 1u);
    } else {
      d = 0;
      float best = z[0];
      for (int k = 1; k < K; ++k)
        if (z[k] > best) {
          best = z[k];
          d = k;
        }
      atomicAdd(&hist[d], 1u);
    }
    decision[r] = d;
  }
  const int total = write_words_and_count(byte, yes_bits + static_cast<int64_t>(blockIdx.x) * (kRowsPerBlock / 32), red);
  if (threadIdx.x == 0) block_counts[blockIdx.x] = total;
  if (threadIdx.x < K && hist[threadIdx.x]) atomicAdd(label_counts + threadIdx.x, (unsigned long long)hist[threadIdx.x]);
}

__global__ void __launch_bounds__(kThreads) k_flag_mask(const int32_t* flags, int64_t n, uint32_t* bits,
                                                         int32_t* block_counts) {
  __shared__ int red[kThreads / 32];
  const int64_t r0 = static_cast<int64_t>(blockIdx.x) * kRowsPerBlock + threadIdx.x * 8;
  uint32_t byte = 0;
  for (int j = 0; j < 8 && r0 + j < n; ++j) byte |= static_cast<uint32_t>(flags[r0 + j] != 0) << j;
  const int total = write_words_and_count(byte, bits + static_cast<int64_t>(blockIdx.x) * (kRowsPerBlock / 32), red);
  if (threadIdx.x == 0) block_counts[blockIdx.x] = total;
}

// Fixed-order reductions (warp shuffle tree, then the warps in order) so that
// the float sum is the same on every run.
template <typename T>
__device__ __forceinline__ T block_sum_fixed(T v, T* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  T t = 0;
  if (threadIdx.x == 0)
    for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) t += sh[w];
  return t;
}

template <typename T, typename C>
__global__ void __launch_bounds__(kThreads) k_masked_sum(const int32_t* decision, const int32_t* ids, const C* col,
                                                         int64_t S, T* partial) {
  __shared__ T sh[kThreads / 32];
  const int64_t r0 = static_cast<int64_t>(blockIdx.x) * kRowsPerBlock + threadIdx.x * 8;
  T acc = 0;
  for (int j = 0; j < 8; ++j) {
    const int64_t i = r0 + j;
    if (i < S && decision[i] == 1) acc += static_cast<T>(col[ids[i]]);
  }
  const T t = block_sum_fixed<T>(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = t;
}

template <typename T>
__global__ void __launch_bounds__(1024) k_sum_final(const T* partial, int64_t n, T* out) {
  __shared__ T sh[32];
  T acc = 0;
  for (int64_t i = threadIdx.x; i < n; i += 1024) acc += partial[i];
  const T t = block_sum_fixed<T>(acc, sh);
  if (threadIdx.x == 0) *out = t;
}

__global__ void k_group_build(const int32_t* decision, const int32_t* build_rows, int64_t S,
                              unsigned long long* counts) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const bool yes = i < S && decision[i] == 1;
  const unsigned active = __ballot_sync(0xffffffffu, yes);
  if (!yes) return;
  const int key = build_rows[i];
  // lanes of the warp that hit the same group add once (skewed foreign keys)
  const unsigned same = __match_any_sync(active, key);
  if ((threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(counts + key, (unsigned long long)__popc(same));
}

__global__ void __launch_bounds__(kThreads) k_nonzero_mask(const unsigned long long* counts, int64_t n, uint32_t* bits,
                                                           int32_t* block_counts) {
  __shared__ int red[kThreads / 32];
  const int64_t r0 = static_cast<int64_t>(blockIdx.x) * kRowsPerBlock + threadIdx.x * 8;
  uint32_t byte = 0;
  for (int j = 0; j < 8; ++j)
    if (r0 + j < n && counts[r0 + j] != 0) byte |= 1u << j;
  const int total = write_words_and_count(byte, bits + static_cast<int64_t>(blockIdx.x) * (kRowsPerBlock / 32), red);
  if (threadIdx.x == 0) block_counts[blockIdx.x] = total;
}

__global__ void k_gather_groups(const int32_t* rows, int64_t g, const int64_t* keys, const unsigned long long* counts,
                                int64_t* keys_out, int64_t* counts_out) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= g) return;
  const int32_t r = rows[i];
  keys_out[i] = keys[r];
  counts_out[i] = static_cast<int64_t>(counts[r]);
}

inline unsigned blocks_for(int64_t n, int64_t per) { return static_cast<unsigned>((n + per - 1) / per); }

}  // namespace

namespace {

template <int N8, int N4>
void launch_terms(unsigned grid, const PredSet& ps, int64_t n, uint32_t* bits, int32_t* counts, const TileScan& ts,
                  cudaStream_t s) {
  const auto kernel = ts.arrived ? k_predicate_cols<N8, N4, true> : k_predicate_cols<N8, N4, false>;
  launch_chained(kernel, dim3(grid), kThreads, 0, s, 1, ps, n, bits, counts, ts);
}

template <int N8>
void launch_cols(int n4, unsigned grid, const PredSet& ps, int64_t n, uint32_t* bits, int32_t* counts,
                 const TileScan& ts, cudaStream_t s) {
  switch (n4) {
    case 0:
      if constexpr (N8 > 0) launch_terms<N8, 0>(grid, ps, n, bits, counts, ts, s);
      break;
    case 1:
      if constexpr (N8 < 4) launch_terms<N8, 1>(grid, ps, n, bits, counts, ts, s);
      break;
    case 2:
      if constexpr (N8 < 3) launch_terms<N8, 2>(grid, ps, n, bits, counts, ts, s);
      break;
    case 3:
      if constexpr (N8 < 2) launch_terms<N8, 3>(grid, ps, n, bits, counts, ts, s);
      break;
    default:
      if constexpr (N8 < 1) launch_terms<N8, 4>(grid, ps, n, bits, counts, ts, s);
      break;
  }
}

// The terms on int64 columns first (k_predicate_cols); a conjunction has no order.
PredSet wide_first(const PredSet& ps, int* n8) {
  PredSet o = ps;
  int at = 0;
  for (int wide = 1; wide >= 0; --wide)
    for (int i = 0; i < ps.n; ++i)
      if ((ps.p[i].type == 1) == (wide == 1)) o.p[at++] = ps.p[i];
  *n8 = 0;
  while (*n8 < ps.n && o.p[*n8].type == 1) ++*n8;
  return o;
}

}  // namespace

bool filter_is_small(int64_t n_rows) { return n_rows > 0 && n_rows <= kSmallRows; }

void launch_filter_small(const PredSet& ps, int64_t n_rows, int32_t* ids, int64_t* count, cudaStream_t s) {
  launch_chained(k_filter_small, dim3(1), kSmallThreads, 0, s, 1, ps, n_rows, ids, count);
}

int launch_predicate_scan(const PredSet& ps, const ProbeSpec& probe, int64_t n_rows, uint32_t* bits,
                          int32_t* block_counts, int64_t* offsets, unsigned int* arrived, int64_t* total,
                          cudaStream_t s) {
  if (n_rows <= 0) {
    if (!offsets) return 0;
    cudaMemsetAsync(offsets, 0, sizeof(int64_t), s);
    if (total) cudaMemcpyAsync(total, offsets, sizeof(int64_t), cudaMemcpyDefault, s);
    return 0;
  }
  const unsigned grid = blocks_for(n_rows, kRowsPerBlock);
  bool aligned = true;
  for (int i = 0; i < ps.n; ++i) aligned = aligned && (reinterpret_cast<uintptr_t>(ps.p[i].col) & 15) == 0;
  // One block scans 2048 counts a microsecond: past kScanTilesMax tiles the caller
  // runs the three-kernel scan, whose blocks share the counts.
  TileScan ts{block_counts, offsets, offsets && grid <= kScanTilesMax ? arrived : nullptr, total};
  bool fused = ts.arrived != nullptr;
  if (probe.keys) {
    launch_chained(k_probe_mask, dim3(grid), kProbeThreads, 0, s, 1, ps, probe, n_rows, bits, block_counts, ts);
  } else if (ps.n >= 1 && ps.n <= 4 && aligned) {
    int n8 = 0;
    const PredSet o = wide_first(ps, &n8);
    switch (n8) {
      case 0: launch_cols<0>(o.n, grid, o, n_rows, bits, block_counts, ts, s); break;
      case 1: launch_cols<1>(o.n - 1, grid, o, n_rows, bits, block_counts, ts, s); break;
      case 2: launch_cols<2>(o.n - 2, grid, o, n_rows, bits, block_counts, ts, s); break;
      case 3: launch_cols<3>(o.n - 3, grid, o, n_rows, bits, block_counts, ts, s); break;
      default: launch_cols<4>(0, grid, o, n_rows, bits, block_counts, ts, s); break;
    }
  } else {
    launch_chained(k_predicate_mask, dim3(grid), kThreads, 0, s, 1, ps, n_rows, bits, block_counts);
    fused = false;
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    char buf[160];
    snprintf(buf, sizeof(buf), "predicate mask launch (grid %u, terms %d)", grid, ps.n);
    set_launch_error(buf, e);
  }
  if (fused || !offsets) return 1;
  launch_scan_counts(block_counts, grid, offsets, s);
  if (total) cudaMemcpyAsync(total, offsets + grid, sizeof(int64_t), cudaMemcpyDefault, s);
  return 2;
}

void launch_scan_counts(const int32_t* counts, int64_t n, int64_t* offsets, cudaStream_t s) {
  launch_chained(k_scan_single<int32_t>, dim3(1), 1024, 0, s, 1, counts, n, offsets);
}

void launch_compact(const uint32_t* bits, const int64_t* block_offsets, int64_t n_rows, int32_t* ids_out,
                    const int32_t* payload, int32_t* payload_out, cudaStream_t s) {
  if (n_rows <= 0) return;
  const unsigned tiles = blocks_for(n_rows, kRowsPerBlock);
  const TileBase tb{block_offsets, nullptr, nullptr};
  if (tiles <= (payload_out ? kWidePayloadTilesMax : kWideTilesMax)) {
    const auto kernel = payload_out ? k_compact_wide<true, false> : k_compact_wide<false, false>;
    launch_chained(kernel, dim3(tiles), kThreads, 0, s, 1, bits, tb, ids_out, payload, payload_out);
    return;
  }
  const unsigned grid = (tiles + kCompactWarps - 1) / kCompactWarps;  // one tile per warp
  const auto kernel = payload_out ? k_compact<true, false> : k_compact<false, false>;
  launch_chained(kernel, dim3(grid), kCompactWarps * 32, 0, s, 1, bits, tb, n_rows, ids_out, payload, payload_out);
}

void launch_compact_counts(const uint32_t* bits, const int32_t* block_counts, int64_t n_rows, int32_t* ids_out,
                           int64_t* total, cudaStream_t s) {
  if (n_rows <= 0) {
    cudaMemsetAsync(total, 0, sizeof(int64_t), s);
    return;
  }
  const unsigned tiles = blocks_for(n_rows, kRowsPerBlock);
  const TileBase tb{nullptr, block_counts, total};
  if (tiles <= kWideTilesMax)
    launch_chained(k_compact_wide<false, true>, dim3(tiles), kThreads, 0, s, 1, bits, tb, ids_out, nullptr, nullptr);
  else
    launch_chained(k_compact<false, true>, dim3((tiles + kCompactWarps - 1) / kCompactWarps), kCompactWarps * 32, 0, s,
                   1, bits, tb, n_rows, ids_out, nullptr, nullptr);
}

void launch_hash_build(const int64_t* keys, const int32_t* rows, int64_t n, unsigned long long* table_keys,
                       int32_t* table_vals, int64_t capacity, int* err, cudaStream_t s) {
  if (n <= 0) return;
  k_hash_build<<<blocks_for(n, 256), 256, 0, s>>>(keys, rows, n, table_keys, table_vals, capacity, err);
}

void launch_hash_build_where(const int64_t* keys, const PredSet& ps, int64_t n, unsigned long long* table_keys,
                             int32_t* table_vals, int64_t capacity, int* err, cudaStream_t s) {
  if (n <= 0) return;
  k_hash_build_where<<<blocks_for(n, 256), 256, 0, s>>>(keys, ps, n, table_keys, table_vals, capacity, err);
}

void launch_fill_u64(unsigned long long* p, int64_t n, unsigned long long v, cudaStream_t s) {
  if (n <= 0) return;
  const unsigned g = blocks_for(n, 256) < 4096 ? blocks_for(n, 256) : 4096;
  k_fill_u64<<<g, 256, 0, s>>>(p, n, v);
}

void launch_scan_lengths(const int32_t* lens, int64_t S, int64_t* cu, int64_t* scratch_blocks, cudaStream_t s) {
  // scratch_blocks: >= 2 * (tiles + 1) int64
  const int64_t tiles = (S + kRowsPerBlock - 1) / kRowsPerBlock;
  if (tiles == 0) {
    cudaMemsetAsync(cu, 0, sizeof(int64_t), s);
    return;
  }
  int64_t* sums = scratch_blocks;
  int64_t* off = scratch_blocks + tiles + 1;
  launch_chained(k_tile_sums, dim3(static_cast<unsigned>(tiles)), kThreads, 0, s, 1, lens, S, sums);
  launch_chained(k_scan_single<int64_t>, dim3(1), 1024, 0, s, 1, sums, tiles, off);
  launch_chained(k_tile_scan, dim3(static_cast<unsigned>(tiles)), kThreads, 0, s, 1, lens, S, off, cu);
}

void launch_decide(const float* logits, int64_t S, int K, int32_t* decision, uint32_t* yes_bits,
                   int32_t* block_counts, unsigned long long* label_counts, cudaStream_t s) {
  if (S <= 0) return;
  launch_chained(k_decide, dim3(blocks_for(S, kRowsPerBlock)), kThreads, 0, s, 1, logits, S, K, decision, yes_bits, block_counts,
                                                             label_counts);
}

void launch_flag_mask(const int32_t* flags, int64_t n, uint32_t* bits, int32_t* block_counts, cudaStream_t s) {
  if (n <= 0) return;
  k_flag_mask<<<blocks_for(n, kRowsPerBlock), kThreads, 0, s>>>(flags, n, bits, block_counts);
}

void launch_masked_sum(const int32_t* decision, const int32_t* ids, const void* col, int type, int64_t S,
                       void* partial, void* out, cudaStream_t s) {
  const unsigned nb = S > 0 ? blocks_for(S, kRowsPerBlock) : 0;
  if (type == 2) {
    if (nb) k_masked_sum<double, float><<<nb, kThreads, 0, s>>>(decision, ids, static_cast<const float*>(col), S,
                                                                 static_cast<double*>(partial));
    k_sum_final<double><<<1, 1024, 0, s>>>(static_cast<const double*>(partial), nb, static_cast<double*>(out));
  } else {
    // integers sum modulo 2^64 (unsigned arithmetic: a wrap is defined), read back as int64
    unsigned long long* pp = static_cast<unsigned long long*>(partial);
    if (nb && type == 0)
      k_masked_sum<unsigned long long, int32_t><<<nb, kThreads, 0, s>>>(decision, ids,
                                                                         static_cast<const int32_t*>(col), S, pp);
    if (nb && type == 1)
      k_masked_sum<unsigned long long, long long><<<nb, kThreads, 0, s>>>(decision, ids,
                                                                           static_cast<const long long*>(col), S, pp);
    k_sum_final<unsigned long long><<<1, 1024, 0, s>>>(pp, nb, static_cast<unsigned long long*>(out));
  }
}

void launch_group_build(const int32_t* decision, const int32_t* cand_build_rows, int64_t S,
                        unsigned long long* group_counts, cudaStream_t s) {
  if (S <= 0) return;
  k_group_build<<<blocks_for(S, 256), 256, 0, s>>>(decision, cand_build_rows, S, group_counts);
}

void launch_nonzero_mask(const unsigned long long* counts, int64_t n, uint32_t* bits, int32_t* block_counts,
                         cudaStream_t s) {
  if (n <= 0) return;
  k_nonzero_mask<<<blocks_for(n, kRowsPerBlock), kThreads, 0, s>>>(counts, n, bits, block_counts);
}

void launch_gather_groups(const int32_t* rows, int64_t g, const int64_t* build_keys,
                          const unsigned long long* counts, int64_t* keys_out, int64_t* counts_out,
                          cudaStream_t s) {
  if (g <= 0) return;
  k_gather_groups<<<blocks_for(g, 256), 256, 0, s>>>(rows, g, build_keys, counts, keys_out, counts_out);
}

}  // namespace aiq
