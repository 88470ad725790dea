// Memory-bound steps of the decoder prefill: weight conversion at load,
// rotary-embedding table, token-embedding gather, RMSNorm, and the label head
// that reads only the label rows of the LM head at each row's last token
// (Fig. 2 slices logits[:, -1, :] at the label ids; the full vocabulary row is
// never formed).
#include "common.cuh"
#include "kernels.h"

namespace aiq {
namespace {

__device__ __forceinline__ float bf16_bits_to_float(uint16_t b) {
  return __uint_as_float(static_cast<uint32_t>(b) << 16);
}

// dst row r of a [rows, cols] fp16 matrix from a bf16 source.  With an
// interleave block ib > 0, the source holds two stacked [half_rows, cols]
// matrices (gate then up) and dst rows alternate blocks of ib gate rows and
// ib up rows, so that one GEMM output tile holds matching gate/up columns.
__global__ void k_bf16_to_f16(const uint16_t* src, __half* dst, int64_t rows, int64_t cols, int ib, int64_t half_rows,
                              int64_t ldd, int* err) {
  const int64_t n = rows * cols;
  bool bad = false;
  for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < n;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t r = e / cols, c = e - r * cols;
    int64_t sr = r;
    if (ib > 0) {
      const int64_t b = r / (2 * ib), w = r % (2 * ib);
      sr = w < ib ? b * ib + w : half_rows + b * ib + (w - ib);
    }
    const float v = bf16_bits_to_float(src[sr * cols + c]);
    bad |= !(fabsf(v) <= 65504.f);
    dst[r * ldd + c] = __float2half_rn(v);
  }
  if (bad) set_dev_error(err, DEVERR_FP16_RANGE);
}

__global__ void k_rope_table(float* cos_t, float* sin_t, int max_pos, int hd, double theta) {
  const int half = hd / 2;
  const int64_t n = static_cast<int64_t>(max_pos) * half;
  for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < n;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int p = static_cast<int>(e / half), i = static_cast<int>(e % half);
    const double inv = pow(theta, -2.0 * i / hd);
    const double a = p * inv;
    cos_t[e] = static_cast<float>(cos(a));
    sin_t[e] = static_cast<float>(sin(a));
  }
}

// One warp per token; 8 bf16 (16 bytes) per lane per step.  With xh / ss the
// row is also written as fp16, times the first layer's attention-norm gain
// when `gain` is given (the fused RMSNorm's input), and its sums of squares
// per 128 columns (16 lanes x 8 values, of the unscaled row) are stored, in a
// fixed order.  Bound by the copy bandwidth as long as the SMs are full of warps:
// eight blocks each need the 32 registers asked for here (the system-scope error
// word alone took it to 38 and six blocks: 92,000 rows of 2048 362 -> 402 us).
__global__ void __launch_bounds__(256, 8)
    k_embed(const int32_t* tok, int64_t T, const uint16_t* emb, int d, float* resid, __half* xh, float* ss,
            const uint16_t* gain, int* err) {
  grid_launch_next();
  grid_wait();
  const int64_t t = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (t >= T) return;
  const uint4* src = reinterpret_cast<const uint4*>(emb + static_cast<int64_t>(tok[t]) * d);
  float4* dst = reinterpret_cast<float4*>(resid + t * d);
  bool bad = false;
  for (int c0 = 0; c0 < d / 8; c0 += 32) {
    const int c = c0 + lane;
    float f[8];
    float part = 0.f;
    if (c < d / 8) {
      const uint4 v = src[c];
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        f[2 * j] = __uint_as_float(w[j] << 16);
        f[2 * j + 1] = __uint_as_float(w[j] & 0xFFFF0000u);
      }
      dst[2 * c] = make_float4(f[0], f[1], f[2], f[3]);
      dst[2 * c + 1] = make_float4(f[4], f[5], f[6], f[7]);
      if (xh) {
        uint32_t pk[4];
        float gf[8] = {1.f, 1.f, 1.f, 1.f, 1.f, 1.f, 1.f, 1.f};
        if (gain) {
          const uint4 gv = reinterpret_cast<const uint4*>(gain)[c];
          const uint32_t gw[4] = {gv.x, gv.y, gv.z, gv.w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            gf[2 * j] = __uint_as_float(gw[j] << 16);
            gf[2 * j + 1] = __uint_as_float(gw[j] & 0xFFFF0000u);
          }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float a = f[2 * j] * gf[2 * j], b = f[2 * j + 1] * gf[2 * j + 1];
          bad |= !(fabsf(a) <= 65504.f) || !(fabsf(b) <= 65504.f);
          __half2 h = __floats2half2_rn(a, b);
          pk[j] = *reinterpret_cast<uint32_t*>(&h);
          part += f[2 * j] * f[2 * j] + f[2 * j + 1] * f[2 * j + 1];
        }
        reinterpret_cast<uint4*>(xh + t * d)[c] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
      }
    }
    if (ss) {
      // lanes 16k .. 16k+15 hold columns [128 * (c0 / 16 + k), +128): reduce within the half-warp
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
      const int slot = (c0 * 8 + (lane >> 4) * 128) / 128;
      if ((lane & 15) == 0 && c < d / 8) ss[t * (d / 128) + slot] = part;
    }
  }
  if (bad) set_dev_error(err, DEVERR_FP16_RANGE);
}

// Sum of four squares, in a fixed order: a row's statistics are the same bits
// whichever of the two kernels below forms them.  It is the order in which the
// expression x * x + y * y + z * z + w * w is contracted (y's square rounded, the
// others joining it by fused steps), which gave these rows before.
__device__ __forceinline__ float sq4(const float4& v) {
  return __fmaf_rn(v.w, v.w, __fmaf_rn(v.z, v.z, __fmaf_rn(v.x, v.x, __fmul_rn(v.y, v.y))));
}

// Four normalised values of a row (columns c .. c + 3), stored as fp16 and, with
// `split`, as the two terms of k_rmsnorm.
__device__ __forceinline__ bool norm_store4(const float4& v, float inv, const uint16_t* g, int c, __half* row, int d,
                                            int split) {
  float g0 = 1.f, g1 = 1.f, g2 = 1.f, g3 = 1.f;
  if (g) {
    const uint2 gg = *reinterpret_cast<const uint2*>(g + c);
    g0 = __uint_as_float(gg.x << 16);
    g1 = __uint_as_float(gg.x & 0xFFFF0000u);
    g2 = __uint_as_float(gg.y << 16);
    g3 = __uint_as_float(gg.y & 0xFFFF0000u);
  }
  const float a = v.x * inv * g0, b = v.y * inv * g1, cc = v.z * inv * g2, e = v.w * inv * g3;
  __half2 h0 = __floats2half2_rn(a, b), h1 = __floats2half2_rn(cc, e);
  *reinterpret_cast<uint2*>(row + c) = make_uint2(*reinterpret_cast<uint32_t*>(&h0), *reinterpret_cast<uint32_t*>(&h1));
  if (split) {
    const float2 f0 = __half22float2(h0), f1 = __half22float2(h1);
    __half2 l0 = __floats2half2_rn(a - f0.x, b - f0.y), l1 = __floats2half2_rn(cc - f1.x, e - f1.y);
    *reinterpret_cast<uint2*>(row + d + c) =
        make_uint2(*reinterpret_cast<uint32_t*>(&l0), *reinterpret_cast<uint32_t*>(&l1));
  }
  return !(fabsf(a) <= 65504.f) || !(fabsf(b) <= 65504.f) || !(fabsf(cc) <= 65504.f) || !(fabsf(e) <= 65504.f);
}

// One warp per row: fp32 statistics, fp16 output for the next GEMM.
// split: out rows are 2d wide, fp16(v) in [0, d) and fp16(v - fp16(v)) in
// [d, 2d), a two-term operand for a GEMM that runs over K = 2d against the
// weight stored twice along K.
template <int PER_LANE>  // d / 32 / 4 float4 per lane (compile-time for register residency)
__global__ void k_rmsnorm(const float* x, int64_t T, int d, const uint16_t* g, float eps, __half* out, int split,
                          int* err) {
  grid_launch_next();
  grid_wait();
  const int64_t t = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (t >= T) return;
  const float4* row = reinterpret_cast<const float4*>(x + t * d);
  float4 v[PER_LANE];
  float ss = 0.f;
#pragma unroll
  for (int j = 0; j < PER_LANE; ++j) {
    v[j] = row[lane + 32 * j];
    ss = __fadd_rn(ss, sq4(v[j]));
  }
  ss = warp_sum(ss);
  const float inv = rsqrtf(ss / d + eps);
  bool bad = false;
  __half* o = out + t * d * (split ? 2 : 1);
#pragma unroll
  for (int j = 0; j < PER_LANE; ++j) bad |= norm_store4(v[j], inv, g, (lane + 32 * j) * 4, o, d, split);
  if (bad) set_dev_error(err, DEVERR_FP16_RANGE);
}

// Few rows: a block of eight warps per row.  With a warp per row each lane walks
// 16 or 32 loads of its own and most of the GPU idles: 24 rows of 2048 took 11.6 us
// from a cold cache, 128 rows of 4096 16.0 (now 4.0 and 5.2).  Warp w holds the
// row's 128-column groups w, w + 8, ...; every warp then adds the groups' sums in
// the order of k_rmsnorm.
template <int PER_LANE>
__global__ void __launch_bounds__(256) k_rmsnorm_rows(const float* x, int d, const uint16_t* g, float eps, __half* out,
                                                      int split, int* err) {
  constexpr int PER = PER_LANE / 8;
  grid_launch_next();
  grid_wait();
  __shared__ float part[PER_LANE][32];
  const int64_t t = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float4* row = reinterpret_cast<const float4*>(x + t * d);
  float4 v[PER];
#pragma unroll
  for (int i = 0; i < PER; ++i) v[i] = row[lane + 32 * (warp + 8 * i)];
#pragma unroll
  for (int i = 0; i < PER; ++i) part[warp + 8 * i][lane] = sq4(v[i]);
  __syncthreads();
  float ss = 0.f;
#pragma unroll
  for (int j = 0; j < PER_LANE; ++j) ss = __fadd_rn(ss, part[j][lane]);
  ss = warp_sum(ss);
  const float inv = rsqrtf(ss / d + eps);
  bool bad = false;
  __half* o = out + t * d * (split ? 2 : 1);
#pragma unroll
  for (int i = 0; i < PER; ++i) bad |= norm_store4(v[i], inv, g, (lane + 32 * (warp + 8 * i)) * 4, o, d, split);
  if (bad) set_dev_error(err, DEVERR_FP16_RANGE);
}

// Sums of squares of 128-column groups for the fused attention norm, after a
// product whose tiles are narrower than a group.  A group's 64 terms (a column's
// square and that of the column 32 on) are added one after the other, as the
// thread that holds a whole row does it in the large tiles, so that a row's norm
// does not depend on how many rows its product had.  A warp forms the terms of
// eight groups (its 32 loads all in flight) and eight lanes walk them; what
// bounds it is that walk behind one trip to memory: 590 rows of 2048 take 4.2 us from a
// cold cache.
constexpr int kSsWarps = 8, kSsGroups = 8;  // warps per block, groups per warp
__global__ void __launch_bounds__(kSsWarps * 32) k_row_ss(const float* x, int64_t groups, float* ss) {
  grid_launch_next();
  grid_wait();
  __shared__ float term[kSsWarps][kSsGroups][65];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t g0 = (static_cast<int64_t>(blockIdx.x) * kSsWarps + warp) * kSsGroups;
  float v[kSsGroups][4];
#pragma unroll
  for (int i = 0; i < kSsGroups; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) v[i][j] = g0 + i < groups ? x[(g0 + i) * 128 + j * 32 + lane] : 0.f;
#pragma unroll
  for (int i = 0; i < kSsGroups; ++i) {
    term[warp][i][lane] = __fmaf_rn(v[i][0], v[i][0], __fmul_rn(v[i][1], v[i][1]));
    term[warp][i][32 + lane] = __fmaf_rn(v[i][2], v[i][2], __fmul_rn(v[i][3], v[i][3]));
  }
  __syncwarp();
  if (lane < kSsGroups && g0 + lane < groups) {
    float part = 0.f;
#pragma unroll
    for (int j = 0; j < 64; ++j) part = __fadd_rn(part, term[warp][lane][j]);
    ss[g0 + lane] = part;
  }
}

// Generic-width fallback (d not a multiple of 128 handled elsewhere; d % 4 == 0 here).
__global__ void k_rmsnorm_any(const float* x, int64_t T, int d, const uint16_t* g, float eps, __half* out, int split,
                              int* err) {
  grid_launch_next();
  grid_wait();
  const int64_t t = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (t >= T) return;
  const float* row = x + t * d;
  float ss = 0.f;
  for (int c = lane; c < d; c += 32) ss += row[c] * row[c];
  ss = warp_sum(ss);
  const float inv = rsqrtf(ss / d + eps);
  bool bad = false;
  for (int c = lane; c < d; c += 32) {
    const float v = row[c] * inv * (g ? bf16_bits_to_float(g[c]) : 1.f);
    bad |= !(fabsf(v) <= 65504.f);
    const __half h = __float2half_rn(v);
    out[t * d * (split ? 2 : 1) + c] = h;
    if (split) out[t * d * 2 + d + c] = __float2half_rn(v - __half2float(h));
  }
  if (bad) set_dev_error(err, DEVERR_FP16_RANGE);
}

// One warp per candidate row: final RMSNorm of the last token's hidden state,
// then K dot products with the label rows of the LM head plus its bias.  A lane
// takes columns lane, lane + 32, ... in turn, the order that its sums have always
// had, 32 of them and two labels' rows in flight: one column at a time each walk of
// the row was a chain of 64 loads (46 rows of 2048, 2 labels: 28 -> 8.8 us from a cold
// cache).  PER: columns in flight.
template <int PER>
__global__ void __launch_bounds__(256) k_label_head(const float* resid, const int32_t* last_idx,
                                                    const float* prefix_last, int64_t n, int d, const uint16_t* g,
                                                    float eps, const uint16_t* W, const uint16_t* bias,
                                                    const int32_t* labels, int K, float* logits) {
  grid_launch_next();
  grid_wait();
  const int64_t r = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (r >= n) return;
  const int32_t li = last_idx[r];
  const float* x = li >= 0 ? resid + static_cast<int64_t>(li) * d : prefix_last;
  float ss = 0.f;
  for (int c0 = lane; c0 < d; c0 += 32 * PER) {
    float v[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) v[i] = c0 + 32 * i < d ? x[c0 + 32 * i] : 0.f;
#pragma unroll
    for (int i = 0; i < PER; ++i) ss = __fmaf_rn(v[i], v[i], ss);
  }
  ss = warp_sum(ss);
  const float inv = rsqrtf(ss / d + eps);
  for (int k = 0; k < K; k += 2) {
    const int l0 = labels[k], l1 = labels[k + 1 < K ? k + 1 : k];
    const uint16_t *w0 = W + static_cast<int64_t>(l0) * d, *w1 = W + static_cast<int64_t>(l1) * d;
    float a0 = 0.f, a1 = 0.f;
    for (int c0 = lane; c0 < d; c0 += 32 * PER) {
      float v[PER];
      uint16_t gv[PER], u0[PER], u1[PER];
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        const int c = c0 + 32 * i;
        if (c < d) v[i] = x[c], gv[i] = g[c], u0[i] = w0[c], u1[i] = w1[c];
      }
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        if (c0 + 32 * i >= d) break;
        const float t = v[i] * inv * bf16_bits_to_float(gv[i]);
        a0 = __fmaf_rn(t, bf16_bits_to_float(u0[i]), a0);
        a1 = __fmaf_rn(t, bf16_bits_to_float(u1[i]), a1);
      }
    }
    a0 = warp_sum(a0);
    a1 = warp_sum(a1);
    if (lane == 0) {
      logits[r * K + k] = a0 + bf16_bits_to_float(bias[l0]);
      if (k + 1 < K) logits[r * K + k + 1] = a1 + bf16_bits_to_float(bias[l1]);
    }
  }
}

// One warp copies n 16-byte words, eight a lane in flight.
__device__ __forceinline__ void copy_row(const uint4* src, uint4* dst, int n, int lane) {
  for (int c0 = lane; c0 < n; c0 += 32 * 8) {
    uint4 v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (c0 + 32 * i < n) v[i] = src[c0 + 32 * i];
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (c0 + 32 * i < n) dst[c0 + 32 * i] = v[i];
  }
}

// Final layer, rows only: gather each row's last token (attention output and
// residual) into dense [n, .] buffers; last_compact[r] = r, or -1 for a row
// without tokens of its own (its logits come from the prefix's last state).
__global__ void k_gather_last(const __half* att, int ld_att, const float* resid, int d, const int32_t* last_idx,
                              int64_t n, __half* att_out, float* resid_out, int32_t* last_compact) {
  grid_launch_next();
  grid_wait();
  const int64_t r = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (r >= n) return;
  const int32_t li = last_idx[r];
  if (lane == 0) last_compact[r] = li >= 0 ? static_cast<int32_t>(r) : -1;
  const int64_t src = li >= 0 ? li : 0;
  copy_row(reinterpret_cast<const uint4*>(att + src * ld_att), reinterpret_cast<uint4*>(att_out + r * ld_att), ld_att / 8,
           lane);
  copy_row(reinterpret_cast<const uint4*>(resid + src * d), reinterpret_cast<uint4*>(resid_out + r * d), d / 4, lane);
}

constexpr int64_t kRowBlocksMax = 2432;  // rows that take a block each: two waves of eight blocks per SM

inline unsigned grid_for(int64_t threads) { return static_cast<unsigned>((threads + 255) / 256); }

}  // namespace

void launch_bf16_to_f16(const uint16_t* src, __half* dst, int64_t rows, int64_t cols, int interleave_block,
                        int64_t half_rows, int* err, cudaStream_t s, int64_t ldd) {
  const int64_t n = rows * cols;
  if (n <= 0) return;
  unsigned g = grid_for(n);
  if (g > 8192) g = 8192;
  k_bf16_to_f16<<<g, 256, 0, s>>>(src, dst, rows, cols, interleave_block, half_rows, ldd > 0 ? ldd : cols, err);
}

void launch_rope_table(float* cos_t, float* sin_t, int max_pos, int head_dim, float theta, cudaStream_t s) {
  const int64_t n = static_cast<int64_t>(max_pos) * (head_dim / 2);
  if (n <= 0) return;
  unsigned g = grid_for(n);
  if (g > 4096) g = 4096;
  k_rope_table<<<g, 256, 0, s>>>(cos_t, sin_t, max_pos, head_dim, static_cast<double>(theta));
}

void launch_embed(const int32_t* tok, int64_t T, const uint16_t* emb, int d, float* resid, __half* xh, float* ss,
                  const uint16_t* gain, int* err, cudaStream_t s) {
  if (T <= 0) return;
  launch_chained(k_embed, dim3(grid_for(T * 32)), 256, 0, s, 1, tok, T, emb, d, resid, xh, ss, gain, err);
}

void launch_rmsnorm(const float* x, int64_t T, int d, const uint16_t* g, float eps, __half* out, int* err,
                    cudaStream_t s, bool split) {
  if (T <= 0) return;
  const unsigned grid = grid_for(T * 32);
  const int sp = split ? 1 : 0;
  if (T <= kRowBlocksMax) {
    switch (d) {
      case 1024: launch_chained(k_rmsnorm_rows<8>, dim3(static_cast<unsigned>(T)), 256, 0, s, 1, x, d, g, eps, out, sp, err); return;
      case 2048: launch_chained(k_rmsnorm_rows<16>, dim3(static_cast<unsigned>(T)), 256, 0, s, 1, x, d, g, eps, out, sp, err); return;
      case 4096: launch_chained(k_rmsnorm_rows<32>, dim3(static_cast<unsigned>(T)), 256, 0, s, 1, x, d, g, eps, out, sp, err); return;
    }
  }
  switch (d) {
    case 128: launch_chained(k_rmsnorm<1>, dim3(grid), 256, 0, s, 1, x, T, d, g, eps, out, sp, err); break;
    case 256: launch_chained(k_rmsnorm<2>, dim3(grid), 256, 0, s, 1, x, T, d, g, eps, out, sp, err); break;
    case 512: launch_chained(k_rmsnorm<4>, dim3(grid), 256, 0, s, 1, x, T, d, g, eps, out, sp, err); break;
    case 1024: launch_chained(k_rmsnorm<8>, dim3(grid), 256, 0, s, 1, x, T, d, g, eps, out, sp, err); break;
    case 2048: launch_chained(k_rmsnorm<16>, dim3(grid), 256, 0, s, 1, x, T, d, g, eps, out, sp, err); break;
    case 4096: launch_chained(k_rmsnorm<32>, dim3(grid), 256, 0, s, 1, x, T, d, g, eps, out, sp, err); break;
    default: launch_chained(k_rmsnorm_any, dim3(grid), 256, 0, s, 1, x, T, d, g, eps, out, sp, err); break;
  }
}

void launch_row_ss(const float* x, int64_t T, int d, float* ss, cudaStream_t s) {
  if (T <= 0) return;
  const int64_t groups = T * (d / 128);
  constexpr int64_t per = kSsWarps * kSsGroups;
  launch_chained(k_row_ss, dim3(static_cast<unsigned>((groups + per - 1) / per)), kSsWarps * 32, 0, s, 1, x, groups, ss);
}

void launch_gather_last(const __half* att, int ld_att, const float* resid, int d, const int32_t* last_idx, int64_t n,
                        __half* att_out, float* resid_out, int32_t* last_compact, cudaStream_t s) {
  if (n <= 0) return;
  launch_chained(k_gather_last, dim3(grid_for(n * 32)), 256, 0, s, 1, att, ld_att, resid, d, last_idx, n, att_out,
                 resid_out, last_compact);
}

void launch_label_head(const float* resid, const int32_t* last_idx, const float* prefix_last, int64_t n_rows, int d,
                       const uint16_t* g, float eps, const uint16_t* lm_head, const uint16_t* lm_bias,
                       const int32_t* labels, int n_labels, float* logits_out, cudaStream_t s) {
  if (n_rows <= 0) return;
  const auto kernel = d >= 1024 ? k_label_head<32> : k_label_head<4>;
  launch_chained(kernel, dim3(grid_for(n_rows * 32)), 256, 0, s, 1, resid, last_idx, prefix_last, n_rows, d, g, eps,
                 lm_head, lm_bias, labels, n_labels, logits_out);
}

}  // namespace aiq
