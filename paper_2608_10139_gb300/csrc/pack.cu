// Token packing of the candidate rows into a variable-length batch.
//
// Every candidate row's prompt is the shared prefix followed by the row's
// tokens (Table 1, AI_IF row: the text column feeds the causal LM; the prompt
// prefix is the instruction shared by all rows); a Q4 pair's prompt is the
// prefix followed by both rows' tokens (Table 2 Q4: AI_IF([A.text, B.text])).
// The prefix is run through the decoder once per query and its keys/values
// are reused by every row
// (causal attention makes the prefix's states independent of what follows),
// so the packed batch holds only each row's own tokens, at positions
// P, P+1, ...  Rows are concatenated with no padding; cu (int64 [S+1]) holds
// each row's start.  The prefill runs over token-budget chunks of
// consecutive rows, the GPU counterpart of the paper's scan over
// micro-batches (Section 3.2): row i belongs to chunk floor(cu[i] / step), so
// a chunk never holds more than step + max_len tokens.
#include "common.cuh"
#include "kernels.h"

namespace aiq {
namespace {

// lens[i] = text length of row ids[i] (plus row ids2[i]'s for a pair prompt);
// pairs += len * P + len * (len + 1) / 2 (the causal query-key pairs its tokens
// attend, for the executed-FLOP count).
__global__ void k_row_lengths(const int64_t* offsets, const int32_t* ids, const int32_t* ids2, int64_t S, int32_t P,
                              int32_t* lens, unsigned long long* pairs) {
  grid_launch_next();
  grid_wait();
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  unsigned long long pr = 0;
  if (i < S) {
    const int32_t r = ids[i];
    int64_t len = offsets[r + 1] - offsets[r];
    if (ids2) len += offsets[ids2[i] + 1] - offsets[ids2[i]];
    lens[i] = static_cast<int32_t>(len);
    pr = static_cast<unsigned long long>(len * P + len * (len + 1) / 2);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) pr += __shfl_xor_sync(0xffffffffu, pr, o);
  if ((threadIdx.x & 31) == 0 && pr) atomicAdd(pairs, pr);
}

// Few rows: what k_row_lengths and the three kernels of the lengths' scan do, in one
// block, with the totals straight into host memory that the device maps.  The chain
// is launches and little else at these sizes: a query over 319 rows took 322 us, with
// this kernel and no launch for the bounds of a single chunk 293.
__global__ void __launch_bounds__(1024) k_plan_rows(const int64_t* offsets, const int32_t* ids, const int32_t* ids2,
                                                    int32_t S, int32_t P, int64_t* cu, int64_t* total,
                                                    int64_t* pairs) {
  grid_launch_next();
  grid_wait();
  constexpr int PER = 4;  // consecutive rows a thread
  __shared__ int64_t sh[2][32];  // alternate, so that one barrier a round is enough
  __shared__ unsigned long long shp[32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int64_t carry = 0;
  unsigned long long pr = 0;
  for (int32_t b = 0, k = 0; b < S; b += 1024 * PER, k ^= 1) {
    const int32_t i0 = b + threadIdx.x * PER;
    int32_t r[PER], r2[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      r[j] = i0 + j < S ? ids[i0 + j] : -1;
      r2[j] = ids2 && i0 + j < S ? ids2[i0 + j] : -1;
    }
    int64_t len[PER], sum = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      len[j] = r[j] >= 0 ? offsets[r[j] + 1] - offsets[r[j]] : 0;
      if (r2[j] >= 0) len[j] += offsets[r2[j] + 1] - offsets[r2[j]];
    }
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      pr += static_cast<unsigned long long>(len[j] * P + len[j] * (len[j] + 1) / 2);
      sum += len[j];
    }
    int64_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) sh[k][warp] = incl;
    __syncthreads();
    int64_t tot = sh[k][lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, tot, o);
      if (lane >= o) tot += y;
    }
    const int64_t before = __shfl_sync(0xffffffffu, tot, (warp - 1) & 31);
    int64_t at = carry + (warp ? before : 0) + incl - sum;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      if (i0 + j < S) cu[i0 + j] = at;
      at += len[j];
    }
    carry += __shfl_sync(0xffffffffu, tot, 31);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) pr += __shfl_xor_sync(0xffffffffu, pr, o);
  if (lane == 0) shp[warp] = pr;
  __syncthreads();
  if (warp == 0) {
    pr = shp[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) pr += __shfl_xor_sync(0xffffffffu, pr, o);
    if (lane == 0) {
      cu[S] = carry;
      *total = carry;
      *pairs = static_cast<int64_t>(pr);
    }
  }
}

// chunk_rows[2c] = first row i with before + cu[i] >= c * step (S if none), chunk_rows[2c+1] = cu[that row].
__global__ void k_chunk_bounds(const int64_t* cu, int64_t S, int64_t before, int64_t step, int64_t n_chunks,
                               int64_t* out) {
  grid_launch_next();
  grid_wait();
  const int64_t c = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (c > n_chunks) return;
  int64_t lo = 0, hi = S;  // lower bound in cu[0..S)
  if (c == n_chunks) {
    lo = S;
  } else {
    const int64_t target = c * step - before;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (cu[mid] < target) lo = mid + 1;
      else hi = mid;
    }
  }
  out[2 * c] = lo;
  out[2 * c + 1] = cu[lo];
}

// chunk_rows[2c] = min(c * rows_per_chunk, S), chunk_rows[2c+1] = cu[that row].
__global__ void k_chunk_bounds_rows(const int64_t* cu, int64_t S, int64_t rows_per_chunk, int64_t n_chunks,
                                    int64_t* out) {
  grid_launch_next();
  grid_wait();
  const int64_t c = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (c > n_chunks) return;
  const int64_t row = c * rows_per_chunk < S ? c * rows_per_chunk : S;
  out[2 * c] = row;
  out[2 * c + 1] = cu[row];
}

// One warp per row: the row's tokens at positions P + j (for a pair prompt the
// first row's text, then the second's); a row with no tokens of its own gets
// last_idx = -1 (its last position is the prefix's last).  tok0 tokens (the
// prefix, packed as a sequence before them) come first.
__global__ void k_pack_chunk(const int64_t* cu, const int32_t* ids, const int32_t* ids2, const int64_t* offsets,
                             const int32_t* text, int32_t P, int64_t r0, int64_t r1, int32_t* tok, int32_t* pos,
                             int32_t* seq_start, int32_t* last_idx, int64_t tok0) {
  grid_launch_next();
  grid_wait();
  const int64_t w = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int64_t i = r0 + w;
  if (i >= r1) return;
  const int64_t base = cu[r0];
  const int64_t dst = tok0 + cu[i] - base;
  const int64_t len = cu[i + 1] - cu[i];
  const int32_t r = ids[i];
  const int32_t* src = text + offsets[r];
  const int64_t len_a = ids2 ? offsets[r + 1] - offsets[r] : len;
  const int64_t off_b = ids2 ? offsets[ids2[i]] : 0;
  for (int64_t j = lane; j < len; j += 32) {
    tok[dst + j] = j < len_a ? src[j] : text[off_b + (j - len_a)];
    pos[dst + j] = static_cast<int32_t>(P + j);
  }
  if (lane == 0) {
    seq_start[w] = static_cast<int32_t>(dst);
    last_idx[w] = len > 0 ? static_cast<int32_t>(dst + len - 1) : -1;
    if (i == r1 - 1) seq_start[w + 1] = static_cast<int32_t>(tok0 + cu[r1] - base);
  }
}

// Attention work list: one entry per (sequence, block of `tq` query tokens), one
// block.  A launch is a chain of barriers, so each 1024 sequences take one: a
// shuffle scan within the warps, then every warp scans the 32 warp totals.
__global__ void __launch_bounds__(1024) k_attn_tiles(const int32_t* seq_start, int32_t n, int32_t tq,
                                                     int32_t* tile_seq, int32_t* tile_q0, int32_t* n_tiles) {
  grid_launch_next();
  grid_wait();
  __shared__ int32_t sh[2][32];  // alternate, so that one barrier a round is enough
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int32_t carry = 0;
  for (int32_t b = 0, k = 0; b < n; b += 1024, k ^= 1) {
    const int32_t i = b + threadIdx.x;
    const int32_t cnt = i < n ? (seq_start[i + 1] - seq_start[i] + tq - 1) / tq : 0;
    int32_t incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) sh[k][warp] = incl;
    __syncthreads();
    int32_t tot = sh[k][lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, tot, o);
      if (lane >= o) tot += y;
    }
    const int32_t before = warp ? __shfl_sync(0xffffffffu, tot, (warp - 1) & 31) : 0;
    const int32_t at = carry + before + incl - cnt;
    for (int32_t q = 0; q < cnt; ++q) {
      tile_seq[at + q] = i;
      tile_q0[at + q] = q * tq;
    }
    carry += __shfl_sync(0xffffffffu, tot, 31);
  }
  if (threadIdx.x == 0) *n_tiles = carry;
}

// The prefix as one sequence: tokens, positions 0..P-1, seq_start = {0, P},
// last_idx = {P - 1}.
__global__ void k_pack_prefix(const int32_t* prefix, int32_t P, int32_t* tok, int32_t* pos, int32_t* seq_start,
                              int32_t* last_idx) {
  grid_launch_next();
  grid_wait();
  for (int j = threadIdx.x; j < P; j += blockDim.x) {
    tok[j] = prefix[j];
    pos[j] = j;
  }
  if (threadIdx.x == 0) {
    seq_start[0] = 0;
    seq_start[1] = P;
    last_idx[0] = P - 1;
  }
}

}  // namespace

void launch_pack_prefix(const int32_t* prefix, int32_t P, int32_t* tok, int32_t* pos, int32_t* seq_start,
                        int32_t* last_idx, cudaStream_t s) {
  launch_chained(k_pack_prefix, dim3(1), 256, 0, s, 1, prefix, P, tok, pos, seq_start, last_idx);
}

void launch_row_lengths(const int64_t* offsets, const int32_t* ids, int64_t S, int32_t prefix_len, int32_t* lens,
                        unsigned long long* pairs, cudaStream_t s, const int32_t* ids2) {
  if (S <= 0) return;
  launch_chained(k_row_lengths, dim3(static_cast<unsigned>((S + 255) / 256)), 256, 0, s, 1, offsets, ids, ids2, S, prefix_len, lens, pairs);
}

bool plan_is_small(int64_t S) { return S > 0 && S <= kPlanRows; }

void launch_plan_rows(const int64_t* offsets, const int32_t* ids, const int32_t* ids2, int64_t S, int32_t prefix_len,
                      int64_t* cu, int64_t* total, int64_t* pairs, cudaStream_t s) {
  launch_chained(k_plan_rows, dim3(1), 1024, 0, s, 1, offsets, ids, ids2, static_cast<int32_t>(S), prefix_len, cu,
                 total, pairs);
}

void launch_chunk_bounds(const int64_t* cu, int64_t S, int64_t before, int64_t step, int64_t n_chunks,
                         int64_t* chunk_rows, cudaStream_t s) {
  launch_chained(k_chunk_bounds, dim3(static_cast<unsigned>((n_chunks + 1 + 127) / 128)), 128, 0, s, 1, cu, S, before,
                 step, n_chunks, chunk_rows);
}

void launch_chunk_bounds_rows(const int64_t* cu, int64_t S, int64_t rows_per_chunk, int64_t n_chunks,
                              int64_t* chunk_rows, cudaStream_t s) {
  launch_chained(k_chunk_bounds_rows, dim3(static_cast<unsigned>((n_chunks + 1 + 127) / 128)), 128, 0, s, 1, cu, S, rows_per_chunk, n_chunks,
                                                                                       chunk_rows);
}

void launch_pack_chunk(const int64_t* cu, const int32_t* ids, const int64_t* offsets, const int32_t* text,
                       int32_t prefix_len, int64_t r0, int64_t r1, int32_t* tok, int32_t* pos, int32_t* seq_start,
                       int32_t* last_idx, cudaStream_t s, const int32_t* ids2, int64_t tok0) {
  if (r1 <= r0) return;
  const int64_t threads = (r1 - r0) * 32;
  launch_chained(k_pack_chunk, dim3(static_cast<unsigned>((threads + 255) / 256)), 256, 0, s, 1, cu, ids, ids2, offsets,
                 text, prefix_len, r0, r1, tok, pos, seq_start, last_idx, tok0);
}

void launch_attn_tiles(const int32_t* seq_start, int32_t n_seqs, int32_t tile_tokens, int32_t* tile_seq,
                       int32_t* tile_q0, int32_t* n_tiles_dev, cudaStream_t s) {
  launch_chained(k_attn_tiles, dim3(1), 1024, 0, s, 1, seq_start, n_seqs, tile_tokens, tile_seq, tile_q0, n_tiles_dev);
}

}  // namespace aiq
