// Prefill GEMM on the 5th-generation tensor cores (tcgen05 + TMEM + TMA).
//
// C = A[M,K] * B[N,K]^T: A is the packed activation (tokens x features, fp16),
// B a linear layer's weight in [out, in] layout (fp16 copy of the bf16 model),
// accumulation in fp32 TMEM.  These are the decoder's dense contractions
// (QKV, O, gate/up and down projections of each layer) run over every token
// of the packed variable-length batch.
//
// Structure (one CTA per SM, persistent over 128 x BN output tiles, tiles
// ordered in bands of output columns so running CTAs share one L2-resident
// slice of the weight matrix):
//   warp 0  : TMA producer, STAGES-deep ring of (A 128x64, B BNx64) tiles,
//             128-byte swizzle, one mbarrier per stage (full / empty).
//   warp 1  : allocates 2*BN TMEM columns (two accumulators) and issues
//             tcgen05.mma 128xBNx16 from one thread; tcgen05.commit frees a
//             smem stage and, per tile, signals the epilogue.
//   warps 2-5: epilogue; each thread owns one accumulator row (TMEM lane),
//             reads 32-column slices with tcgen05.ld and applies the fused
//             epilogue (RoPE, SwiGLU, fp32 residual add) while the MMA warp
//             already fills the other accumulator.
// Pairs of CTAs on 256 x 256 tiles, and narrow tiles for few rows, follow the
// same structure and say where they differ.
#include <cudaTypedefs.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace aiq {
namespace {

constexpr int BM = 128;
constexpr int BK = 64;      // 64 fp16 = 128 bytes = one swizzle row
constexpr int UMMA_K = 16;  // K of one kind::f16 MMA
constexpr int kThreads = 192;

template <int BN>
struct Cfg {
  static constexpr int STAGES = BN == 256 ? 4 : 6;
  static constexpr int A_BYTES = BM * BK * 2;
  static constexpr int B_BYTES = BN * BK * 2;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int TMEM_COLS = 2 * BN;  // double-buffered fp32 accumulator
  static constexpr int BAR_BYTES = 256;
  static constexpr int SMEM = 1024 /*align slack*/ + STAGES * STAGE_BYTES + BAR_BYTES;
};

struct KArgs {
  int M, N, K;
  GemmEpilogue ep;
};

// EPI_RESID_ADD stages the accumulator in shared memory for TMA reduce-add:
// per epilogue warp two 32 x 32 fp32 buffers (4 KB each, 128-byte swizzle),
// after the operand ring and the barriers, 1024-byte aligned.
template <int EPI>
constexpr int epi_stage_bytes() {
  return EPI == EPI_RESID_ADD ? 4 * 2 * 4096 : 0;
}
constexpr int round_up_1k(int x) { return (x + 1023) & ~1023; }

// Tile order: bands of at most kBandTiles output-tile columns, all row tiles
// of a band before the next band, columns fastest within a band.  Running
// CTAs then share one band of the weight matrix (<= 32 MB for 2048-deep K)
// that stays in L2 while the activation rows stream past, instead of sweeping
// the whole weight matrix once per row tile.
constexpr int kBandTiles = 32;

__device__ __forceinline__ void tile_coords(int tile, int num_m, int num_n, int& mt, int& nt) {
  const int bw = num_n < kBandTiles ? num_n : kBandTiles;
  const int full_bands = num_n / bw;
  const int per_band = num_m * bw;
  const int band = tile / per_band;
  if (band < full_bands) {
    const int r = tile - band * per_band;
    mt = r / bw;
    nt = band * bw + r % bw;
  } else {  // the narrower last band
    const int w = num_n - full_bands * bw;
    const int r = tile - full_bands * per_band;
    mt = r / w;
    nt = full_bands * bw + r % w;
  }
}

__device__ __forceinline__ float u2f(uint32_t u) { return __uint_as_float(u); }

__device__ __forceinline__ void store_f16x32(__half* dst, const float* v, bool& bad) {
  uint4 pk[4];
  uint32_t* w = reinterpret_cast<uint32_t*>(pk);
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const float a = v[2 * j], b = v[2 * j + 1];
    bad |= !(fabsf(a) <= 65504.f) || !(fabsf(b) <= 65504.f);
    __half2 h = __floats2half2_rn(a, b);
    w[j] = *reinterpret_cast<uint32_t*>(&h);
  }
  uint4* d = reinterpret_cast<uint4*>(dst);
#pragma unroll
  for (int j = 0; j < 4; ++j) d[j] = pk[j];
}

__device__ __forceinline__ void load32(uint32_t taddr, float* v) {
  uint32_t r[32];
  tmem_ld_32x32b_x32(taddr, r);
  tmem_ld_wait();
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = u2f(r[j]);
}

// Two 32-column slices with one wait (both loads in flight together).
__device__ __forceinline__ void load2x32(uint32_t ta, uint32_t tb, float* va, float* vb) {
  uint32_t ra[32], rb[32];
  tmem_ld_32x32b_x32(ta, ra);
  tmem_ld_32x32b_x32(tb, rb);
  tmem_ld_wait();
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    va[j] = u2f(ra[j]);
    vb[j] = u2f(rb[j]);
  }
}

__device__ __forceinline__ void load_f32x32(const float* src, float* v) {
  const float4* p = reinterpret_cast<const float4*>(src);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float4 x = __ldg(p + j);
    v[4 * j] = x.x;
    v[4 * j + 1] = x.y;
    v[4 * j + 2] = x.z;
    v[4 * j + 3] = x.w;
  }
}

// dst += v (fp32), and the new values are returned in out.
__device__ __forceinline__ void add_store_f32x32(float* dst, const float* v, float* out) {
  float4* p = reinterpret_cast<float4*>(dst);
  float4 x[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) x[j] = p[j];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    x[j].x += v[4 * j];
    x[j].y += v[4 * j + 1];
    x[j].z += v[4 * j + 2];
    x[j].w += v[4 * j + 3];
    p[j] = x[j];
    out[4 * j] = x[j].x;
    out[4 * j + 1] = x[j].y;
    out[4 * j + 2] = x[j].z;
    out[4 * j + 3] = x[j].w;
  }
}

// 1 / RMS of an accumulator row from its partial sums of squares (fixed
// summation order), or 1 when the GEMM's input is already normalised.
__device__ __forceinline__ float row_inv_rms(const GemmEpilogue& ep, int row, bool live) {
  if (!ep.row_ss || !live) return 1.f;
  const float* p = ep.row_ss + static_cast<int64_t>(row) * ep.ss_parts;
  float s = 0.f;
  if ((ep.ss_parts & 3) == 0) {
    const float4* p4 = reinterpret_cast<const float4*>(p);
    for (int i = 0; i < ep.ss_parts / 4; ++i) {
      const float4 v = p4[i];
      s += v.x;
      s += v.y;
      s += v.z;
      s += v.w;
    }
  } else {
    for (int i = 0; i < ep.ss_parts; ++i) s += p[i];
  }
  return rsqrtf(s / ep.d_norm + ep.eps);
}

__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Issued before the epilogue waits for its accumulator: pulls the bytes this
// thread's row will read into L2 while the tile's MMAs still run.
template <int BN, int EPI>
__device__ __forceinline__ void epilogue_prefetch(const KArgs& a, int row, int n0) {
  if (row >= a.M) return;
  const GemmEpilogue& ep = a.ep;
  if constexpr (EPI == EPI_RESID_F32) {
    prefetch_l2(static_cast<const float*>(ep.out) + static_cast<int64_t>(row) * ep.ldo + n0, BN * 4);
  } else if constexpr (EPI == EPI_ROPE_F16) {
    if (n0 < ep.rope_cols) {
      const int half = ep.head_dim >> 1;
      const int64_t off = static_cast<int64_t>(ep.positions[row]) * half;
      prefetch_l2(ep.rope_cos + off, half * 4);
      prefetch_l2(ep.rope_sin + off, half * 4);
    }
  }
}

// inv: the row's 1/RMS (fused RMSNorm), computed by the caller before it
// waits for the accumulator, so that its loads overlap the tile's MMAs.
template <int BN, int EPI>
__device__ __forceinline__ void epilogue_tile(const KArgs& a, uint32_t trow, int row, int n0, float inv) {
  const GemmEpilogue& ep = a.ep;
  const bool live = row < a.M;
  bool bad = false;
  if constexpr (EPI == EPI_RESID_F32) {
    float* o = static_cast<float*>(ep.out) + static_cast<int64_t>(row) * ep.ldo + n0;
    float part = 0.f;  // sum of squares of the new residual over 128 columns (k_row_ss keeps its order)
#pragma unroll 1
    for (int c = 0; c < BN; c += 64) {
      float v0[32], v1[32];
      load2x32(trow + c, trow + c + 32, v0, v1);
      if (live) {
        add_store_f32x32(o + c, v0, v0);
        add_store_f32x32(o + c + 32, v1, v1);
        if (ep.xh_out) {
          __half* xh = ep.xh_out + static_cast<int64_t>(row) * ep.ldo + n0 + c;
#pragma unroll
          for (int j = 0; j < 32; ++j) part = __fadd_rn(part, __fmaf_rn(v0[j], v0[j], __fmul_rn(v1[j], v1[j])));
          if (ep.xh_gain) {
            // the next attention norm's gain goes on the activation (the QKV
            // weights stay exact): one fp16 rounding of x * g per element
            const uint4* g4 = reinterpret_cast<const uint4*>(ep.xh_gain + n0 + c);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              const uint4 gv = __ldg(g4 + q);
              const uint32_t gw[4] = {gv.x, gv.y, gv.z, gv.w};
              float* v = q < 4 ? v0 + 8 * q : v1 + 8 * (q - 4);
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                v[2 * j] *= __uint_as_float(gw[j] << 16);
                v[2 * j + 1] *= __uint_as_float(gw[j] & 0xFFFF0000u);
              }
            }
          }
          store_f16x32(xh, v0, bad);
          store_f16x32(xh + 32, v1, bad);
          if ((c & 127) == 64) {
            ep.ss_out[static_cast<int64_t>(row) * ep.ss_parts + (n0 + c) / 128] = part;
            part = 0.f;
          }
        }
      }
    }
  } else if constexpr (EPI == EPI_ARGMAX) {
    // logits = acc + bias; strictly-greater keeps the first column of a tie
    float best = -INFINITY;
    int bcol = -1;
#pragma unroll 1
    for (int c = 0; c < BN; c += 64) {
      float v0[32], v1[32];
      load2x32(trow + c, trow + c + 32, v0, v1);
      if (live) {
        float b0[32], b1[32];
        load_f32x32(ep.bias + n0 + c, b0);
        load_f32x32(ep.bias + n0 + c + 32, b1);
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const float x = v0[j] + b0[j];
          if (x > best) {
            best = x;
            bcol = n0 + c + j;
          }
        }
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const float x = v1[j] + b1[j];
          if (x > best) {
            best = x;
            bcol = n0 + c + 32 + j;
          }
        }
      }
    }
    if (live && bcol >= 0) {
      const uint32_t u = __float_as_uint(best);
      const uint32_t ord = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
      atomicMax(ep.best + row,
                (static_cast<unsigned long long>(ord) << 32) | (0xFFFFFFFFu - static_cast<uint32_t>(bcol)));
    }
  } else if constexpr (EPI == EPI_SWIGLU_F16) {
    __half* o = static_cast<__half*>(ep.out) + static_cast<int64_t>(row) * ep.ldo + n0 / 2;
#pragma unroll 1
    for (int c = 0; c < BN / 2; c += 32) {
      float g[32], u[32];
      load2x32(trow + c, trow + BN / 2 + c, g, u);
      // rows past M hold zeros, and a division of zero leaves the fast path:
      // skipping them takes a 128-row tile with dead rows from 21 to 6 us
      if (live) {
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const float gj = g[j] * inv;
          g[j] = gj / (1.0f + expf(-gj)) * (u[j] * inv);
        }
        store_f16x32(o + c, g, bad);
        if (ep.lo_off > 0) {
#pragma unroll
          for (int j = 0; j < 32; ++j) u[j] = g[j] - __half2float(__float2half_rn(g[j]));
          store_f16x32(o + ep.lo_off + c, u, bad);
        }
      }
    }
  } else {
    __half* o = static_cast<__half*>(ep.out) + static_cast<int64_t>(row) * ep.ldo + n0;
    int rot_end = 0;  // columns [0, rot_end) of the tile hold rotated (q, k) heads
    if constexpr (EPI == EPI_ROPE_F16) {
      const int hd = ep.head_dim;
      const int half = hd >> 1;
      rot_end = ep.rope_cols - n0;
      rot_end = rot_end < 0 ? 0 : (rot_end > BN ? BN : rot_end);
      const int64_t toff = live ? static_cast<int64_t>(ep.positions[row]) * half : 0;
      if (half >= 32) {
        // cos/sin of this row's position, 32 frequencies at a time, reused by every head of the tile
#pragma unroll 1
        for (int i0 = 0; i0 < half; i0 += 32) {
          float cs[32], sn[32];
          load_f32x32(ep.rope_cos + toff + i0, cs);
          load_f32x32(ep.rope_sin + toff + i0, sn);
#pragma unroll 1
          for (int h = 0; h < rot_end; h += hd) {
            float x1[32], x2[32];
            load2x32(trow + h + i0, trow + h + half + i0, x1, x2);
            if (live) {
#pragma unroll
              for (int j = 0; j < 32; ++j) {
                const float a1 = x1[j] * inv, a2 = x2[j] * inv;
                x1[j] = a1 * cs[j] - a2 * sn[j];
                x2[j] = a2 * cs[j] + a1 * sn[j];
              }
              store_f16x32(o + h + i0, x1, bad);
              store_f16x32(o + h + half + i0, x2, bad);
            }
          }
        }
      } else {  // head_dim 32: both halves of a head in one 32-column slice
        float cs[16], sn[16];
        const float4* c4 = reinterpret_cast<const float4*>(ep.rope_cos + toff);
        const float4* s4 = reinterpret_cast<const float4*>(ep.rope_sin + toff);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 cv = __ldg(c4 + j), sv = __ldg(s4 + j);
          cs[4 * j] = cv.x; cs[4 * j + 1] = cv.y; cs[4 * j + 2] = cv.z; cs[4 * j + 3] = cv.w;
          sn[4 * j] = sv.x; sn[4 * j + 1] = sv.y; sn[4 * j + 2] = sv.z; sn[4 * j + 3] = sv.w;
        }
#pragma unroll 1
        for (int h = 0; h < rot_end; h += 32) {
          float x[32];
          load32(trow + h, x);
          if (live) {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const float a1 = x[j] * inv, a2 = x[j + 16] * inv;
              x[j] = a1 * cs[j] - a2 * sn[j];
              x[j + 16] = a2 * cs[j] + a1 * sn[j];
            }
            store_f16x32(o + h, x, bad);
          }
        }
      }
    }
    // plain fp16 columns (all of them for EPI_F16; the value heads for EPI_ROPE_F16)
    int c = rot_end;
#pragma unroll 1
    for (; c + 64 <= BN; c += 64) {
      float v0[32], v1[32];
      load2x32(trow + c, trow + c + 32, v0, v1);
      if (live) {
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          v0[j] *= inv;
          v1[j] *= inv;
        }
        store_f16x32(o + c, v0, bad);
        store_f16x32(o + c + 32, v1, bad);
      }
    }
    if (c < BN) {
      float v[32];
      load32(trow + c, v);
      if (live) {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] *= inv;
        store_f16x32(o + c, v, bad);
      }
    }
  }
  if (bad) set_dev_error(ep.err, DEVERR_FP16_RANGE);
}

__device__ __forceinline__ void st_shared_v4(uint32_t saddr, uint4 v) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(saddr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}

// out[rows m0q .. m0q + 31][n0 .. n0 + BN) += acc, one 32 x 32 tile at a time:
// each lane writes its row (TMEM lane) into a swizzled staging buffer, lane 0
// hands the tile to the TMA unit as a reduce-add (rows past M are clipped by
// the tensor map).  Two buffers alternate; a buffer is rewritten only after
// the reduce issued from it two tiles earlier has read it.
template <int BN>
__device__ __forceinline__ void epilogue_tma_add(const CUtensorMap* tma_c, uint32_t trow, int m0q, int n0,
                                                 uint8_t* stage, int lane, uint32_t& nbuf) {
#pragma unroll 1
  for (int c = 0; c < BN; c += 32) {
    float v[32];
    load32(trow + c, v);
    uint8_t* buf = stage + (nbuf & 1) * 4096;
    if (lane == 0) bulk_wait_group_read<1>();
    __syncwarp();
    const uint32_t row = smem_u32(buf) + lane * 128;
#pragma unroll
    for (int j = 0; j < 8; ++j)
      st_shared_v4(row + ((j ^ (lane & 7)) << 4), make_uint4(__float_as_uint(v[4 * j]), __float_as_uint(v[4 * j + 1]),
                                                             __float_as_uint(v[4 * j + 2]),
                                                             __float_as_uint(v[4 * j + 3])));
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) {
      tma_reduce_add_2d(tma_c, buf, n0 + c, m0q);
      bulk_commit_group();
    }
    ++nbuf;
  }
}

template <int BN, int EPI>
__global__ void __launch_bounds__(kThreads, 1)
    k_gemm_tcgen05(const __grid_constant__ CUtensorMap tma_a, const __grid_constant__ CUtensorMap tma_b,
                   const __grid_constant__ CUtensorMap tma_c, KArgs args) {
  using C = Cfg<BN>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + C::STAGES * C::A_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::STAGES * C::STAGE_BYTES);
  uint64_t* full = bars;
  uint64_t* empty = bars + C::STAGES;
  uint64_t* tfull = bars + 2 * C::STAGES;
  uint64_t* tempty = tfull + 2;
  uint64_t* mma_done = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  int* err = args.ep.err;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], 4);  // one arrival per epilogue warp
    }
    mbar_init(mma_done, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tma_a);
    tma_prefetch_desc(&tma_b);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, C::TMEM_COLS);
    tmem_relinquish();
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  grid_launch_next();
  grid_wait();

  const int num_n = args.N / BN;
  const int num_m = (args.M + BM - 1) / BM;
  const int num_tiles = num_m * num_n;
  const int kblocks = args.K / BK;

  if (warp == 0) {
    if (lane == 0) {
      // ---------------------------------------------------- TMA producer
      uint32_t issued = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
        int mt, nt;
        tile_coords(tile, num_m, num_n, mt, nt);
        const int m0 = mt * BM;
        const int n0 = nt * BN;
        for (int kb = 0; kb < kblocks; ++kb) {
          const int s = issued % C::STAGES;
          const uint32_t ph = (issued / C::STAGES) & 1;
          if (!mbar_wait_bounded(&empty[s], ph ^ 1, abort_flag, err)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&full[s], C::STAGE_BYTES);
          tma_load_2d(sA + s * C::A_BYTES, &tma_a, &full[s], kb * BK, m0);
          tma_load_2d(sB + s * C::B_BYTES, &tma_b, &full[s], kb * BK, n0);
          ++issued;
        }
      }
      if (!ok) {
        // drain this thread's copies still in flight before the CTA can exit
        const uint32_t first = issued > (uint32_t)C::STAGES ? issued - C::STAGES : 0;
        volatile int never = 0;
        for (uint32_t i = first; i < issued; ++i)
          mbar_wait_bounded(&full[i % C::STAGES], (i / C::STAGES) & 1, &never, nullptr, 200000000ull);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ------------------------------------------------------ MMA issuer
      constexpr uint32_t idesc = idesc_f16_f32(BM, BN);
      uint32_t consumed = 0;
      int acc = 0;
      uint32_t acc_ph = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
        if (!mbar_wait_bounded(&tempty[acc], acc_ph ^ 1, abort_flag, err)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * BN;
        for (int kb = 0; kb < kblocks; ++kb) {
          const int s = consumed % C::STAGES;
          const uint32_t ph = (consumed / C::STAGES) & 1;
          if (!mbar_wait_bounded(&full[s], ph, abort_flag, err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a0 = smem_u32(sA + s * C::A_BYTES);
          const uint32_t b0 = smem_u32(sB + s * C::B_BYTES);
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; ++k) {
            // advancing K inside the 128-byte swizzle row = +32 bytes on the start address
            umma_f16_ss(d_tmem, smem_desc_k_sw128(a0 + k * UMMA_K * 2), smem_desc_k_sw128(b0 + k * UMMA_K * 2),
                        idesc, (kb | k) != 0);
          }
          umma_commit(&empty[s]);
          ++consumed;
        }
        if (!ok) break;
        umma_commit(&tfull[acc]);
        acc ^= 1;
        if (acc == 0) acc_ph ^= 1;
      }
      // every MMA issued above has completed once this arrives
      umma_commit(mma_done);
      volatile int never = 0;
      mbar_wait_bounded(mma_done, 0, &never, err);
    }
  } else {
    // ------------------------------------------------------------ epilogue
    const int quarter = warp & 3;  // TMEM lanes this warp may access
    uint8_t* stage = smem + round_up_1k(C::STAGES * C::STAGE_BYTES + C::BAR_BYTES) + quarter * 8192;
    uint32_t nbuf = 0;
    int acc = 0;
    uint32_t acc_ph = 0;
    for (int tile = blockIdx.x; tile < num_tiles; tile += gridDim.x) {
      int mt, nt;
      tile_coords(tile, num_m, num_n, mt, nt);
      const int m0 = mt * BM;
      const int n0 = nt * BN;
      epilogue_prefetch<BN, EPI>(args, m0 + quarter * 32 + lane, n0);
      const float inv = (EPI == EPI_ROPE_F16 || EPI == EPI_SWIGLU_F16)
                            ? row_inv_rms(args.ep, m0 + quarter * 32 + lane, m0 + quarter * 32 + lane < args.M)
                            : 1.f;
      // warp-uniform: a lane that gives up makes the whole warp give up, so no
      // lane is left alone in the warp-synchronous TMEM loads of the epilogue
      if (!__all_sync(0xffffffffu, mbar_wait_bounded(&tfull[acc], acc_ph, abort_flag, err))) break;
      tc_fence_after();
      const uint32_t trow = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + acc * BN;
      if constexpr (EPI == EPI_RESID_ADD)
        epilogue_tma_add<BN>(&tma_c, trow, m0 + quarter * 32, n0, stage, lane, nbuf);
      else
        epilogue_tile<BN, EPI>(args, trow, m0 + quarter * 32 + lane, n0, inv);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[acc]);
      acc ^= 1;
      if (acc == 0) acc_ph ^= 1;
    }
    if constexpr (EPI == EPI_RESID_ADD) {
      if (lane == 0) bulk_wait_group_all();  // the reduces have completed before the CTA leaves
    }
  }

  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, C::TMEM_COLS);
  }
}


// ------------------------------------------------------------ CTA pairs ---
// 256 x 256 output tiles on a cluster of two CTAs (tcgen05.mma.cta_group::2).
// Each CTA stages its own 128 rows of A and 128 columns of B per 128-deep
// k-block (two 64-deep swizzled sub-blocks per operand, 64 KB, 3 stages), so
// every SM moves half the B bytes of the single-CTA 128 x 256 tile for the
// same MMA work, and each barrier wait, fence and commit of the MMA issuer
// covers eight MMAs instead of four (3-6 % faster than 64-deep stages on the
// QKV and gate/up shapes); its TMA completes on the leader's barrier, the
// leader alone issues the M = 256 MMA, and each CTA's epilogue drains its own
// 128 accumulator rows and reports back to the leader.  Needs K % 128 == 0
// (other K take the single-CTA kernel).
struct CfgPair {
  static constexpr int STAGES = 3;
  static constexpr int SUB = 2;                  // 64-deep sub-blocks per stage
  static constexpr int A_BYTES = SUB * 128 * BK * 2;
  static constexpr int B_BYTES = SUB * 128 * BK * 2;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int TMEM_COLS = 512;
  static constexpr int SMEM = 1024 + STAGES * STAGE_BYTES + 256;
};

template <int EPI>
__global__ void __launch_bounds__(kThreads, 1)
    k_gemm_tcgen05_pair(const __grid_constant__ CUtensorMap tma_a, const __grid_constant__ CUtensorMap tma_b,
                        const __grid_constant__ CUtensorMap tma_c, KArgs args) {
  using C = CfgPair;
  constexpr int BN = 256;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + C::STAGES * C::A_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::STAGES * C::STAGE_BYTES);
  uint64_t* full = bars;                 // used in the leader only
  uint64_t* empty = bars + C::STAGES;    // per CTA, multicast by the leader's commits
  uint64_t* tfull = bars + 2 * C::STAGES;
  uint64_t* tempty = tfull + 2;          // used in the leader only: 4 warps x 2 CTAs
  uint64_t* mma_done = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int pair = blockIdx.x >> 1;
  const int n_pairs = gridDim.x >> 1;
  int* err = args.ep.err;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], 8);
    }
    mbar_init(mma_done, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tma_a);
    tma_prefetch_desc(&tma_b);
  }
  if (warp == 1) {
    tmem_alloc_pair(tmem_slot, C::TMEM_COLS);
    tmem_relinquish_pair();
    tc_fence_before();
  }
  __syncthreads();
  cluster_sync();  // barriers of both CTAs initialised before any remote arrival
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  grid_launch_next();
  grid_wait();

  const int num_n = args.N / BN;
  const int num_m = (args.M + 2 * BM - 1) / (2 * BM);
  const int num_tiles = num_m * num_n;
  const int kblocks = args.K / (BK * C::SUB);

  if (warp == 0) {
    if (lane == 0) {
      // ---------------------------------------------------- TMA producer
      const uint32_t full_leader = map_to_cta(smem_u32(full), 0);
      uint32_t issued = 0;
      bool ok = true;
      for (int tile = pair; tile < num_tiles && ok; tile += n_pairs) {
        int mt, nt;
        tile_coords(tile, num_m, num_n, mt, nt);
        const int m0 = mt * 2 * BM;
        const int n0 = nt * BN;
        for (int kb = 0; kb < kblocks; ++kb) {
          const int s = issued % C::STAGES;
          const uint32_t ph = (issued / C::STAGES) & 1;
          if (!mbar_wait_bounded(&empty[s], ph ^ 1, abort_flag, err)) {
            ok = false;
            break;
          }
          if (leader) mbar_arrive_expect_tx(&full[s], 2 * C::STAGE_BYTES);
#pragma unroll
          for (int sb = 0; sb < C::SUB; ++sb) {
            tma_load_2d_pair(sA + s * C::A_BYTES + sb * (128 * BK * 2), &tma_a, full_leader + s * 8,
                             (kb * C::SUB + sb) * BK, m0 + rank * BM);
            tma_load_2d_pair(sB + s * C::B_BYTES + sb * (128 * BK * 2), &tma_b, full_leader + s * 8,
                             (kb * C::SUB + sb) * BK, n0 + rank * 128);
          }
          ++issued;
        }
      }
      if (!ok && leader) {
        // the leader's barrier completes only once both CTAs' bytes have landed
        const uint32_t first = issued > (uint32_t)C::STAGES ? issued - C::STAGES : 0;
        volatile int never = 0;
        for (uint32_t i = first; i < issued; ++i)
          mbar_wait_bounded(&full[i % C::STAGES], (i / C::STAGES) & 1, &never, nullptr, 200000000ull);
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && leader) {
      // ------------------------------------------------ MMA issuer (leader)
      constexpr uint32_t idesc = idesc_f16_f32(2 * BM, BN);
      uint32_t consumed = 0;
      int acc = 0;
      uint32_t acc_ph = 0;
      bool ok = true;
      for (int tile = pair; tile < num_tiles && ok; tile += n_pairs) {
        if (!mbar_wait_bounded(&tempty[acc], acc_ph ^ 1, abort_flag, err)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * BN;
        for (int kb = 0; kb < kblocks; ++kb) {
          const int s = consumed % C::STAGES;
          const uint32_t ph = (consumed / C::STAGES) & 1;
          if (!mbar_wait_bounded(&full[s], ph, abort_flag, err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a0 = smem_u32(sA + s * C::A_BYTES);
          const uint32_t b0 = smem_u32(sB + s * C::B_BYTES);
#pragma unroll
          for (int sb = 0; sb < C::SUB; ++sb)
#pragma unroll
            for (int k = 0; k < BK / UMMA_K; ++k)
              umma_f16_ss_pair(d_tmem, smem_desc_k_sw128(a0 + sb * (128 * BK * 2) + k * UMMA_K * 2),
                               smem_desc_k_sw128(b0 + sb * (128 * BK * 2) + k * UMMA_K * 2), idesc,
                               (kb | sb | k) != 0);
          umma_commit_pair_mc(&empty[s], 0x3);
          ++consumed;
        }
        if (!ok) break;
        umma_commit_pair_mc(&tfull[acc], 0x3);
        acc ^= 1;
        if (acc == 0) acc_ph ^= 1;
      }
      umma_commit_pair_mc(mma_done, 0x1);
      volatile int never = 0;
      mbar_wait_bounded(mma_done, 0, &never, err);
    }
  } else {
    // ------------------------------------------------ epilogue (both CTAs)
    const int quarter = warp & 3;
    const uint32_t tempty_leader = map_to_cta(smem_u32(tempty), 0);
    uint8_t* stage = smem + round_up_1k(C::STAGES * C::STAGE_BYTES + 256) + quarter * 8192;
    uint32_t nbuf = 0;
    int acc = 0;
    uint32_t acc_ph = 0;
    for (int tile = pair; tile < num_tiles; tile += n_pairs) {
      int mt, nt;
      tile_coords(tile, num_m, num_n, mt, nt);
      const int m0 = mt * 2 * BM + rank * BM;
      const int n0 = nt * BN;
      epilogue_prefetch<BN, EPI>(args, m0 + quarter * 32 + lane, n0);
      const float inv = (EPI == EPI_ROPE_F16 || EPI == EPI_SWIGLU_F16)
                            ? row_inv_rms(args.ep, m0 + quarter * 32 + lane, m0 + quarter * 32 + lane < args.M)
                            : 1.f;
      // warp-uniform: a lane that gives up makes the whole warp give up, so no
      // lane is left alone in the warp-synchronous TMEM loads of the epilogue
      if (!__all_sync(0xffffffffu, mbar_wait_bounded(&tfull[acc], acc_ph, abort_flag, err))) break;
      tc_fence_after();
      const uint32_t trow = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + acc * BN;
      if constexpr (EPI == EPI_RESID_ADD)
        epilogue_tma_add<BN>(&tma_c, trow, m0 + quarter * 32, n0, stage, lane, nbuf);
      else
        epilogue_tile<BN, EPI>(args, trow, m0 + quarter * 32 + lane, n0, inv);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(tempty_leader + acc * 8);
      acc ^= 1;
      if (acc == 0) acc_ph ^= 1;
    }
    if constexpr (EPI == EPI_RESID_ADD) {
      if (lane == 0) bulk_wait_group_all();  // the reduces have completed before the CTA leaves
    }
  }

  __syncthreads();
  cluster_sync();  // no CTA leaves while its peer may still signal it
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, C::TMEM_COLS);
  }
}

// ------------------------------------------------------------- few rows ---
// Products with few rows (a generation step, the shared prefix's own pass, a
// small chunk, the final layer's last tokens), in narrow tiles, so that even N =
// 2048 gives every SM a slice of the weights to stream: tiles of up to 64 rows and BN
// = 16 .. 128 weight columns, by one CTA (k_gemm_few) or, with more rows, by two that
// share 128 rows and 2 BN columns (k_gemm_few_pair).  Bound by the weights' read from DRAM; what each CTA moves per
// 64-deep k-block is (rows of A + BN) x 128 bytes, so A's box holds only the
// rows that exist (rounded up to 8; the MMA's other rows read whatever follows
// in shared memory and are never stored).  One TMA per operand fills a stage
// of `sub` 64-deep blocks: A as {64, rows, sub}, B as {64, BN / 2, 2, sub}
// whose two halves lie `half` weight rows apart.  The halves hold what the
// epilogue combines: the gate and up columns (half = bn / 2, the interleave
// the caller laid the weights out with), the two halves of a head (half =
// head_dim / 2), or the tile's own halves (half = BN / 2, contiguous).
// Every element's products are summed in the order of the large-tile kernels
// and every epilogue step is the same operation, so a row's results do not
// depend on which kernel computed it.
constexpr int kFewRows = 64;           // rows that one CTA stages
constexpr int kFewSmem = 200 * 1024;  // operand ring
constexpr int kFewStages = 16;
constexpr int kFewEpiWarps = 8;
constexpr int kFewThreads = 64 + 32 * kFewEpiWarps;
constexpr int kFewSlack = kFewRows * 128;  // an A tile's MMA reads kFewRows rows from its slot's start

struct FewArgs {
  int a_rows;  // rows of A's box
  int sub;     // 64-deep blocks per stage
  int stages;
  int half;    // weight rows between the two halves of a tile
};

__device__ __forceinline__ void store_f16x8(__half* dst, const float* v, bool& bad) {
  uint32_t w[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float a = v[2 * j], b = v[2 * j + 1];
    bad |= !(fabsf(a) <= 65504.f) || !(fabsf(b) <= 65504.f);
    __half2 h = __floats2half2_rn(a, b);
    w[j] = *reinterpret_cast<uint32_t*>(&h);
  }
  *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
}

// First weight row of tile nt's two halves: tiles walk the `half` rows of a
// block in steps of BN / 2, then go to the next block of 2 * half rows.
template <int BN>
__device__ __forceinline__ int few_n0(int nt, int half) {
  const int per = half / (BN / 2);
  return (nt / per) * 2 * half + (nt % per) * (BN / 2);
}

// The accumulator's columns are shared by the two warps of a TMEM quarter (`part`
// 0 and 1): 16-column steps in turn where the threads add to the residual, else a
// half each of the tile's column pairs (tiles of 16 columns go to part 0).
template <int BN, int EPI>
__device__ __forceinline__ void epilogue_few(const KArgs& a, uint32_t trow, int row, bool live, int n0, int half,
                                             float inv, int part) {
  const GemmEpilogue& ep = a.ep;
  bool bad = false;
  const int64_t r = row;
  if constexpr (EPI == EPI_RESID_F32) {
#pragma unroll 1
    for (int c = part * 16; c < BN; c += 32) {
      uint32_t rv[16];
      tmem_ld_32x32b_x8(trow + c, rv);
      tmem_ld_32x32b_x8(trow + c + 8, rv + 8);
      tmem_ld_wait();
      if (live) {
        float v[16];
        float4* o4 = reinterpret_cast<float4*>(static_cast<float*>(ep.out) + r * ep.ldo + n0 + c);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float4 t = o4[j];
          t.x += u2f(rv[4 * j]);
          t.y += u2f(rv[4 * j + 1]);
          t.z += u2f(rv[4 * j + 2]);
          t.w += u2f(rv[4 * j + 3]);
          o4[j] = t;
          v[4 * j] = t.x;
          v[4 * j + 1] = t.y;
          v[4 * j + 2] = t.z;
          v[4 * j + 3] = t.w;
        }
        if (ep.xh_out) {
          __half* xh = ep.xh_out + r * ep.ldo + n0 + c;
#pragma unroll
          for (int j = 0; j < 16; j += 8) {
            if (ep.xh_gain) {
              const uint4 gv = __ldg(reinterpret_cast<const uint4*>(ep.xh_gain + n0 + c + j));
              const uint32_t gw[4] = {gv.x, gv.y, gv.z, gv.w};
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                v[j + 2 * i] *= __uint_as_float(gw[i] << 16);
                v[j + 2 * i + 1] *= __uint_as_float(gw[i] & 0xFFFF0000u);
              }
            }
            store_f16x8(xh + j, v + j, bad);
          }
        }
      }
      __syncwarp();
    }
  } else {
    constexpr int HB = BN / 2;
    constexpr int PER = HB < 16 ? HB : HB / 2;  // columns of each half per warp
    constexpr int W = PER < 16 ? PER : 16;      // and per step
    const int c1 = HB < 16 && part ? 0 : (part + 1) * PER;
#pragma unroll 1
    for (int c = part * PER; c < c1; c += W) {
      uint32_t ru[W], rv[W];
#pragma unroll
      for (int j = 0; j < W; j += 8) {
        tmem_ld_32x32b_x8(trow + c + j, ru + j);
        tmem_ld_32x32b_x8(trow + HB + c + j, rv + j);
      }
      tmem_ld_wait();
      if (live) {
        float x[W], y[W];
#pragma unroll
        for (int j = 0; j < W; ++j) {
          x[j] = u2f(ru[j]) * inv;
          y[j] = u2f(rv[j]) * inv;
        }
        if constexpr (EPI == EPI_SWIGLU_F16) {
          __half* o = static_cast<__half*>(ep.out) + r * ep.ldo + (n0 / (2 * half)) * half + n0 % (2 * half) + c;
#pragma unroll
          for (int j = 0; j < W; ++j) x[j] = x[j] / (1.0f + expf(-x[j])) * y[j];
#pragma unroll
          for (int j = 0; j < W; j += 8) store_f16x8(o + j, x + j, bad);
          if (ep.lo_off > 0) {
#pragma unroll
            for (int j = 0; j < W; ++j) y[j] = x[j] - __half2float(__float2half_rn(x[j]));
#pragma unroll
            for (int j = 0; j < W; j += 8) store_f16x8(o + ep.lo_off + j, y + j, bad);
          }
        } else {
          __half* o = static_cast<__half*>(ep.out) + r * ep.ldo + n0 + c;
          if (n0 < ep.rope_cols) {
            // column n0 + c + j of the head's first half and its partner `half` columns on
            const int64_t toff = static_cast<int64_t>(ep.positions[row]) * half + n0 % (2 * half) + c;
#pragma unroll
            for (int j = 0; j < W; j += 4) {
              const float4 cs4 = __ldg(reinterpret_cast<const float4*>(ep.rope_cos + toff + j));
              const float4 sn4 = __ldg(reinterpret_cast<const float4*>(ep.rope_sin + toff + j));
              const float cs[4] = {cs4.x, cs4.y, cs4.z, cs4.w}, sn[4] = {sn4.x, sn4.y, sn4.z, sn4.w};
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const float a1 = x[j + i], a2 = y[j + i];
                x[j + i] = a1 * cs[i] - a2 * sn[i];
                y[j + i] = a2 * cs[i] + a1 * sn[i];
              }
            }
          }
#pragma unroll
          for (int j = 0; j < W; j += 8) {
            store_f16x8(o + j, x + j, bad);
            store_f16x8(o + half + j, y + j, bad);
          }
        }
      }
      __syncwarp();
    }
  }
  if (bad) set_dev_error(ep.err, DEVERR_FP16_RANGE);
}

// One stage's MMAs: SUB 64-deep blocks of A (a_blk bytes apart) and B.
template <int SUB, int BN, bool PAIR = false>
__device__ __forceinline__ void few_issue(uint32_t d, uint64_t da, uint64_t db, uint32_t a_blk, uint32_t idesc,
                                          bool first) {
#pragma unroll
  for (int sb = 0; sb < SUB; ++sb)
#pragma unroll
    for (int k = 0; k < BK / UMMA_K; ++k) {
      // descriptors count 16-byte units; UMMA_K fp16 = 32 bytes
      const uint64_t a = da + sb * (a_blk >> 4) + 2 * k, b = db + sb * (BN * 128 >> 4) + 2 * k;
      if constexpr (PAIR) {
        if (sb == 0 && k == 0)
          umma_f16_ss_pair(d, a, b, idesc, !first);
        else
          umma_f16_ss_pair_acc(d, a, b, idesc);
      } else {
        if (sb == 0 && k == 0)
          umma_f16_ss(d, a, b, idesc, !first);
        else
          umma_f16_ss_acc(d, a, b, idesc);
      }
    }
}

template <int BN, int EPI>
__global__ void __launch_bounds__(kFewThreads, 1)
    k_gemm_few(const __grid_constant__ CUtensorMap tma_a, const __grid_constant__ CUtensorMap tma_b, KArgs args,
               FewArgs fa) {
  constexpr int TMEM_COLS = 2 * BN < 32 ? 32 : 2 * BN;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint64_t full[kFewStages], empty[kFewStages], tfull[2], tempty[2], mma_done;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_word;
  volatile int* abort_flag = &abort_word;

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  int* err = args.ep.err;
  const uint32_t stages = fa.stages, sub = fa.sub;
  const uint32_t a_blk = fa.a_rows * 128, a_bytes = sub * a_blk;  // one 64-deep block / one stage of A
  constexpr uint32_t b_blk = BN * 128;
  const uint32_t b_bytes = sub * b_blk;
  uint8_t* sA = smem;
  uint8_t* sB = smem + stages * a_bytes;

  if (threadIdx.x == 0) {
    for (uint32_t s = 0; s < stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], kFewEpiWarps);
    }
    mbar_init(&mma_done, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tma_a);
    tma_prefetch_desc(&tma_b);
  }
  if (warp == 1) {
    tmem_alloc(&tmem_slot, TMEM_COLS);
    tmem_relinquish();
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  grid_launch_next();
  grid_wait();

  const int num_m = (args.M + kFewRows - 1) / kFewRows;
  const int num_tiles = num_m * (args.N / BN);
  const int kblocks = args.K / (BK * sub);

  if (warp == 0) {
    if (lane == 0) {
      // ---------------------------------------------------- TMA producer
      uint32_t issued = 0, s = 0, ph = 1;
      bool ok = true;
      for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
        const int m0 = (tile % num_m) * kFewRows;
        const int n0 = few_n0<BN>(tile / num_m, fa.half);
        for (int kb = 0; kb < kblocks; ++kb) {
          if (!mbar_wait_bounded(&empty[s], ph, abort_flag, err)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&full[s], a_bytes + b_bytes);
          tma_load_4d(sB + s * b_bytes, &tma_b, &full[s], 0, n0, 0, kb * sub);
          tma_load_3d(sA + s * a_bytes, &tma_a, &full[s], 0, m0, kb * sub);
          ++issued;
          if (++s == stages) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      if (!ok) {
        // drain this thread's copies still in flight before the CTA can exit
        volatile int never = 0;
        for (uint32_t i = issued > stages ? issued - stages : 0; i < issued; ++i)
          mbar_wait_bounded(&full[i % stages], (i / stages) & 1, &never, nullptr, 200000000ull);
      }
    }
  } else if (warp == 1) {
    // -------------------------------------------------------- MMA issuer
    // The whole warp walks the stages and one elected lane issues: the
    // descriptors then stay in uniform registers.  Issue is what a short MMA
    // waits for: 90 clocks each when formed per MMA in one lane, against the
    // tensor core's own 23 (64 x 16 x 16).
    constexpr uint32_t idesc = idesc_f16_f32(kFewRows, BN);
    const uint64_t da0 = smem_desc_k_sw128(smem_u32(sA)), db0 = smem_desc_k_sw128(smem_u32(sB));
    const uint32_t tb = __shfl_sync(0xffffffffu, tmem_base, 0);
    uint32_t s = 0, ph = 0;
    int acc = 0;
    uint32_t acc_ph = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
      if (!__all_sync(0xffffffffu, mbar_wait_bounded(&tempty[acc], acc_ph ^ 1, abort_flag, err))) break;
      tc_fence_after();
      const uint32_t d_tmem = tb + acc * BN;
      for (int kb = 0; kb < kblocks; ++kb) {
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(&full[s], ph, abort_flag, err))) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint64_t da = da0 + s * (a_bytes >> 4), db = db0 + s * (b_bytes >> 4);
        if (elect_one()) {
          if (sub == 8)
            few_issue<8, BN>(d_tmem, da, db, a_blk, idesc, kb == 0);
          else if (sub == 4)
            few_issue<4, BN>(d_tmem, da, db, a_blk, idesc, kb == 0);
          else if (sub == 2)
            few_issue<2, BN>(d_tmem, da, db, a_blk, idesc, kb == 0);
          else
            few_issue<1, BN>(d_tmem, da, db, a_blk, idesc, kb == 0);
          umma_commit(&empty[s]);
        }
        __syncwarp();
        if (++s == stages) {
          s = 0;
          ph ^= 1;
        }
      }
      if (!ok) break;
      if (elect_one()) umma_commit(&tfull[acc]);
      __syncwarp();
      acc ^= 1;
      if (acc == 0) acc_ph ^= 1;
    }
    // every MMA issued above has completed once this arrives
    if (elect_one()) umma_commit(&mma_done);
    __syncwarp();
    volatile int never = 0;
    mbar_wait_bounded(&mma_done, 0, &never, err);
  } else {
    // ------------------------------------------------------------ epilogue
    const int quarter = warp & 3;  // TMEM lanes this warp may access
    const int part = (warp - 2) >> 2;
    int acc = 0;
    uint32_t acc_ph = 0;
    for (int tile = blockIdx.x; tile < num_tiles; tile += gridDim.x) {
      const int m0 = (tile % num_m) * kFewRows + quarter * 16;
      const int n0 = few_n0<BN>(tile / num_m, fa.half);
      // a 64-row accumulator takes the first 16 TMEM lanes of each quarter
      const int row = m0 + lane;
      const bool live = lane < 16 && row < args.M;
      if (EPI == EPI_RESID_F32) {
        if (live && part == 0)
          prefetch_l2(static_cast<const float*>(args.ep.out) + static_cast<int64_t>(row) * args.ep.ldo + n0, BN * 4);
      }
      const float inv = EPI == EPI_ROPE_F16 || EPI == EPI_SWIGLU_F16 ? row_inv_rms(args.ep, row, live) : 1.f;
      if (!__all_sync(0xffffffffu, mbar_wait_bounded(&tfull[acc], acc_ph, abort_flag, err))) break;
      tc_fence_after();
      if (m0 < args.M)  // warp-uniform: this warp holds at least one live row
        epilogue_few<BN, EPI>(args, tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + acc * BN, row, live,
                              n0, fa.half, inv, part);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[acc]);
      acc ^= 1;
      if (acc == 0) acc_ph ^= 1;
    }
  }

  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

// Two CTAs per tile of 128 rows x 2 BN columns (tcgen05.mma.cta_group::2, M =
// 128): each stages 64 of the rows and the BN weight columns of one of two
// neighbouring tiles of k_gemm_few, so that per product an SM takes in (64 + BN)
// bytes where a CTA by itself takes (128 + BN); the arrival of the operands is what
// bounds these products at more than 64 rows (60 to 68 bytes a clock per SM).  Each CTA's TMEM holds
// its 64 rows: the first tile's columns on lanes 0-63, the second's on lanes
// 64-127.  Barriers as in k_gemm_tcgen05_pair.  128 rows, 4096 x 14336: 47 -> 35 us
// (17 at the weights' read); the four products of a 128-row block of that size
// together 150 -> 130, one CTA taking 128 rows before.
template <int BN, int EPI>
__global__ void __launch_bounds__(kFewThreads, 1)
    k_gemm_few_pair(const __grid_constant__ CUtensorMap tma_a, const __grid_constant__ CUtensorMap tma_b, KArgs args,
                    FewArgs fa) {
  constexpr int TMEM_COLS = 2 * BN < 32 ? 32 : 2 * BN;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint64_t full[kFewStages], empty[kFewStages], tfull[2], tempty[2], mma_done;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_word;
  volatile int* abort_flag = &abort_word;

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int pair = blockIdx.x >> 1;
  const int n_pairs = gridDim.x >> 1;
  int* err = args.ep.err;
  const uint32_t stages = fa.stages, sub = fa.sub;
  constexpr uint32_t a_blk = 64 * 128, b_blk = BN * 128;
  const uint32_t a_bytes = sub * a_blk, b_bytes = sub * b_blk;  // a stage of this CTA
  uint8_t* sA = smem;
  uint8_t* sB = smem + stages * a_bytes;

  if (threadIdx.x == 0) {
    for (uint32_t s = 0; s < stages; ++s) {
      mbar_init(&full[s], 1);   // used in the leader only
      mbar_init(&empty[s], 1);  // per CTA, multicast by the leader's commits
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], 2 * kFewEpiWarps);  // used in the leader only
    }
    mbar_init(&mma_done, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tma_a);
    tma_prefetch_desc(&tma_b);
  }
  if (warp == 1) {
    tmem_alloc_pair(&tmem_slot, TMEM_COLS);
    tmem_relinquish_pair();
    tc_fence_before();
  }
  __syncthreads();
  cluster_sync();  // barriers of both CTAs initialised before any remote arrival
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  grid_launch_next();
  grid_wait();

  const int num_m = (args.M + 127) / 128;
  // row tiles fastest: the CTAs that share a weight slice run together
  const int num_tiles = num_m * (args.N / (2 * BN));
  const int kblocks = args.K / (BK * sub);

  if (warp == 0) {
    if (lane == 0) {
      // ---------------------------------------------------- TMA producer
      const uint32_t full_leader = map_to_cta(smem_u32(full), 0);
      uint32_t issued = 0, s = 0, ph = 1;
      bool ok = true;
      for (int tile = pair; tile < num_tiles && ok; tile += n_pairs) {
        const int m0 = (tile % num_m) * 128 + rank * 64;
        const int n0 = few_n0<BN>(2 * (tile / num_m) + rank, fa.half);
        for (int kb = 0; kb < kblocks; ++kb) {
          if (!mbar_wait_bounded(&empty[s], ph, abort_flag, err)) {
            ok = false;
            break;
          }
          if (leader) mbar_arrive_expect_tx(&full[s], 2 * (a_bytes + b_bytes));
          tma_load_4d_pair(sB + s * b_bytes, &tma_b, full_leader + s * 8, 0, n0, 0, kb * sub);
          tma_load_3d_pair(sA + s * a_bytes, &tma_a, full_leader + s * 8, 0, m0, kb * sub);
          ++issued;
          if (++s == stages) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      if (!ok && leader) {
        // the leader's barrier completes only once both CTAs' bytes have landed
        volatile int never = 0;
        for (uint32_t i = issued > stages ? issued - stages : 0; i < issued; ++i)
          mbar_wait_bounded(&full[i % stages], (i / stages) & 1, &never, nullptr, 200000000ull);
      }
    }
  } else if (warp == 1) {
    if (leader) {
      // ------------------------------------------------ MMA issuer (leader)
      constexpr uint32_t idesc = idesc_f16_f32(128, 2 * BN);
      const uint64_t da0 = smem_desc_k_sw128(smem_u32(sA)), db0 = smem_desc_k_sw128(smem_u32(sB));
      const uint32_t tb = __shfl_sync(0xffffffffu, tmem_base, 0);
      uint32_t s = 0, ph = 0;
      int acc = 0;
      uint32_t acc_ph = 0;
      bool ok = true;
      for (int tile = pair; tile < num_tiles && ok; tile += n_pairs) {
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(&tempty[acc], acc_ph ^ 1, abort_flag, err))) break;
        tc_fence_after();
        const uint32_t d_tmem = tb + acc * BN;
        for (int kb = 0; kb < kblocks; ++kb) {
          if (!__all_sync(0xffffffffu, mbar_wait_bounded(&full[s], ph, abort_flag, err))) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t da = da0 + s * (a_bytes >> 4), db = db0 + s * (b_bytes >> 4);
          if (elect_one()) {
            if (sub == 4)  // four stages of eight such blocks exceed the ring
              few_issue<4, BN, true>(d_tmem, da, db, a_blk, idesc, kb == 0);
            else if (sub == 2)
              few_issue<2, BN, true>(d_tmem, da, db, a_blk, idesc, kb == 0);
            else
              few_issue<1, BN, true>(d_tmem, da, db, a_blk, idesc, kb == 0);
            umma_commit_pair_mc(&empty[s], 0x3);
          }
          __syncwarp();
          if (++s == stages) {
            s = 0;
            ph ^= 1;
          }
        }
        if (!ok) break;
        if (elect_one()) umma_commit_pair_mc(&tfull[acc], 0x3);
        __syncwarp();
        acc ^= 1;
        if (acc == 0) acc_ph ^= 1;
      }
      // every MMA issued above has completed once this arrives
      if (elect_one()) umma_commit_pair_mc(&mma_done, 0x1);
      __syncwarp();
      volatile int never = 0;
      mbar_wait_bounded(&mma_done, 0, &never, err);
    }
  } else {
    // ------------------------------------------------ epilogue (both CTAs)
    const int quarter = warp & 3;  // TMEM lanes this warp may access
    const int part = (warp - 2) >> 2;
    const uint32_t tempty_leader = map_to_cta(smem_u32(tempty), 0);
    int acc = 0;
    uint32_t acc_ph = 0;
    for (int tile = pair; tile < num_tiles; tile += n_pairs) {
      const int m0 = (tile % num_m) * 128 + rank * 64 + (quarter & 1) * 32;
      const int n0 = few_n0<BN>(2 * (tile / num_m) + (quarter >> 1), fa.half);
      const int row = m0 + lane;
      const bool live = row < args.M;
      if (EPI == EPI_RESID_F32) {
        if (live && part == 0)
          prefetch_l2(static_cast<const float*>(args.ep.out) + static_cast<int64_t>(row) * args.ep.ldo + n0, BN * 4);
      }
      const float inv = EPI == EPI_ROPE_F16 || EPI == EPI_SWIGLU_F16 ? row_inv_rms(args.ep, row, live) : 1.f;
      if (!__all_sync(0xffffffffu, mbar_wait_bounded(&tfull[acc], acc_ph, abort_flag, err))) break;
      tc_fence_after();
      if (m0 < args.M)  // warp-uniform: this warp holds at least one live row
        epilogue_few<BN, EPI>(args, tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + acc * BN, row, live,
                              n0, fa.half, inv, part);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(tempty_leader + acc * 8);
      acc ^= 1;
      if (acc == 0) acc_ph ^= 1;
    }
  }

  __syncthreads();
  cluster_sync();  // no CTA leaves while its peer may still signal it
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, TMEM_COLS);
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    cudaDriverEntryPointQueryResult q;
    void* p = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// 2-D fp16 tensor [rows, cols] (cols contiguous, row pitch ld elements), box 64 x box_rows, 128B swizzle.
bool make_map(CUtensorMap* m, const __half* base, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
  cuuint64_t strides[1] = {static_cast<cuuint64_t>(ld * 2)};
  cuuint32_t box[2] = {static_cast<cuuint32_t>(BK), static_cast<cuuint32_t>(box_rows)};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// 2-D fp32 tensor [rows, cols] (row pitch ld elements), box 32 x 32, 128B swizzle:
// the target of EPI_RESID_ADD's reduce-add tiles.
bool make_map_out_f32(CUtensorMap* m, float* base, int64_t rows, int64_t cols, int64_t ld) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
  cuuint64_t strides[1] = {static_cast<cuuint64_t>(ld * 4)};
  cuuint32_t box[2] = {32, 32};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

template <int BN, int EPI>
constexpr int smem_single() {
  using C = Cfg<BN>;
  return EPI == EPI_RESID_ADD ? 1024 + round_up_1k(C::STAGES * C::STAGE_BYTES + C::BAR_BYTES) + epi_stage_bytes<EPI>()
                              : C::SMEM;
}
template <int EPI>
constexpr int smem_pair() {
  using C = CfgPair;
  return EPI == EPI_RESID_ADD ? 1024 + round_up_1k(C::STAGES * C::STAGE_BYTES + 256) + epi_stage_bytes<EPI>()
                              : C::SMEM;
}
static_assert(smem_single<256, EPI_RESID_ADD>() <= 232448 && smem_single<128, EPI_RESID_ADD>() <= 232448 &&
                  smem_pair<EPI_RESID_ADD>() <= 232448,
              "shared memory per block");

template <int BN, int EPI>
int launch(const CUtensorMap& ma, const CUtensorMap& mb, const CUtensorMap& mc, const KArgs& a, int num_sms,
           cudaStream_t stream) {
  constexpr int SM = smem_single<BN, EPI>();
  cudaError_t e = cudaFuncSetAttribute(k_gemm_tcgen05<BN, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, SM);
  if (e != cudaSuccess) return e;
  const int tiles = ((a.M + BM - 1) / BM) * (a.N / BN);
  const int grid = tiles < num_sms ? tiles : num_sms;
  return launch_chained(k_gemm_tcgen05<BN, EPI>, dim3(grid), kThreads, SM, stream, 1, ma, mb, mc, a);
}

template <int EPI>
int launch_pair(const CUtensorMap& ma, const CUtensorMap& mb, const CUtensorMap& mc, const KArgs& a, int num_sms,
                cudaStream_t stream) {
  constexpr int SM = smem_pair<EPI>();
  cudaError_t e = cudaFuncSetAttribute(k_gemm_tcgen05_pair<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, SM);
  if (e != cudaSuccess) return e;
  const int tiles = ((a.M + 2 * BM - 1) / (2 * BM)) * (a.N / 256);
  const int pairs = tiles < num_sms / 2 ? tiles : num_sms / 2;
  return launch_chained(k_gemm_tcgen05_pair<EPI>, dim3(2 * pairs), kThreads, SM, stream, 2, ma, mb, mc, a);
}

int dispatch_pair(const CUtensorMap& ma, const CUtensorMap& mb, const CUtensorMap& mc, const KArgs& a, int num_sms,
                  cudaStream_t s) {
  switch (a.ep.kind) {
    case EPI_F16: return launch_pair<EPI_F16>(ma, mb, mc, a, num_sms, s);
    case EPI_ROPE_F16: return launch_pair<EPI_ROPE_F16>(ma, mb, mc, a, num_sms, s);
    case EPI_RESID_F32: return launch_pair<EPI_RESID_F32>(ma, mb, mc, a, num_sms, s);
    case EPI_SWIGLU_F16: return launch_pair<EPI_SWIGLU_F16>(ma, mb, mc, a, num_sms, s);
    case EPI_ARGMAX: return launch_pair<EPI_ARGMAX>(ma, mb, mc, a, num_sms, s);
    case EPI_RESID_ADD: return launch_pair<EPI_RESID_ADD>(ma, mb, mc, a, num_sms, s);
  }
  return cudaErrorInvalidValue;
}

template <int BN>
int dispatch_epi(const CUtensorMap& ma, const CUtensorMap& mb, const CUtensorMap& mc, const KArgs& a, int num_sms,
                 cudaStream_t s) {
  switch (a.ep.kind) {
    case EPI_F16: return launch<BN, EPI_F16>(ma, mb, mc, a, num_sms, s);
    case EPI_ROPE_F16: return launch<BN, EPI_ROPE_F16>(ma, mb, mc, a, num_sms, s);
    case EPI_RESID_F32: return launch<BN, EPI_RESID_F32>(ma, mb, mc, a, num_sms, s);
    case EPI_SWIGLU_F16: return launch<BN, EPI_SWIGLU_F16>(ma, mb, mc, a, num_sms, s);
    case EPI_ARGMAX: return launch<BN, EPI_ARGMAX>(ma, mb, mc, a, num_sms, s);
    case EPI_RESID_ADD: return launch<BN, EPI_RESID_ADD>(ma, mb, mc, a, num_sms, s);
  }
  return cudaErrorInvalidValue;
}

// A of k_gemm_few, [rows, K] as {64, rows, K / 64}: box 64 x box_rows x sub.
bool make_map_few_a(CUtensorMap* m, const __half* base, int64_t rows, int64_t K, int64_t ld, int box_rows, int sub) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {BK, static_cast<cuuint64_t>(rows), static_cast<cuuint64_t>(K / BK)};
  cuuint64_t strides[2] = {static_cast<cuuint64_t>(ld * 2), BK * 2};
  cuuint32_t box[3] = {BK, static_cast<cuuint32_t>(box_rows), static_cast<cuuint32_t>(sub)};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<__half*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// B of k_gemm_few, [N, K] as {64, row, half, K / 64}: box 64 x BN / 2 x 2 x sub,
// the second half `half` rows after the first.
bool make_map_few_b(CUtensorMap* m, const __half* base, int64_t N, int64_t K, int64_t ld, int bn, int half, int sub) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[4] = {BK, static_cast<cuuint64_t>(N - half), 2, static_cast<cuuint64_t>(K / BK)};
  cuuint64_t strides[3] = {static_cast<cuuint64_t>(ld * 2), static_cast<cuuint64_t>(half * ld * 2), BK * 2};
  cuuint32_t box[4] = {BK, static_cast<cuuint32_t>(bn / 2), 2, static_cast<cuuint32_t>(sub)};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<__half*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Weight rows between the two halves of a tile (see k_gemm_few).
int few_half(int tile, int bn, const GemmEpilogue& ep) {
  if (ep.kind == EPI_SWIGLU_F16) return bn / 2;
  if (ep.kind == EPI_ROPE_F16) return ep.head_dim / 2;
  return tile / 2;
}

template <bool PAIR, int BN, int EPI>
int launch_few(const __half* A, int64_t lda, const __half* B, int64_t ldb, const KArgs& a, int bn, int num_sms,
               cudaStream_t stream) {
  FewArgs fa;
  fa.a_rows = a.M < kFewRows ? (a.M + 7) / 8 * 8 : kFewRows;
  fa.half = few_half(BN, bn, a.ep);
  // the deepest stage (one TMA per operand) that leaves four of them in the ring
  const int block = (fa.a_rows + BN) * 128;
  fa.sub = 1;
  for (int s = 8; s > 1; s /= 2)
    if (a.K % (BK * s) == 0 && 4 * s * block <= kFewSmem) {
      fa.sub = s;
      break;
    }
  fa.stages = kFewSmem / (fa.sub * block);
  if (fa.stages > kFewStages) fa.stages = kFewStages;
  CUtensorMap ma, mb;
  if (!make_map_few_a(&ma, A, a.M, a.K, lda, fa.a_rows, fa.sub) ||
      !make_map_few_b(&mb, B, a.N, a.K, ldb, BN, fa.half, fa.sub))
    return cudaErrorInvalidValue;
  constexpr int SM = 1024 + kFewSmem + kFewSlack;
  static_assert(SM + 1024 <= 232448, "shared memory per block");
  void (*kernel)(const CUtensorMap, const CUtensorMap, KArgs, FewArgs);
  int grid;
  if constexpr (PAIR) {
    kernel = k_gemm_few_pair<BN, EPI>;
    grid = 2 * std::min((a.M + 127) / 128 * (a.N / (2 * BN)), num_sms / 2);
  } else {
    kernel = k_gemm_few<BN, EPI>;
    grid = std::min((a.M + kFewRows - 1) / kFewRows * (a.N / BN), num_sms);
  }
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SM);
  if (e != cudaSuccess) return e;
  return launch_chained(kernel, dim3(grid), kFewThreads, SM, stream, PAIR ? 2 : 1, ma, mb, a, fa);
}

template <int BN, int EPI>
int launch_few_rows(const __half* A, int64_t lda, const __half* B, int64_t ldb, const KArgs& a, int bn, bool two,
                    int num_sms, cudaStream_t s) {
  return two ? launch_few<true, BN, EPI>(A, lda, B, ldb, a, bn, num_sms, s)
             : launch_few<false, BN, EPI>(A, lda, B, ldb, a, bn, num_sms, s);
}

template <int BN>
int dispatch_few(const __half* A, int64_t lda, const __half* B, int64_t ldb, const KArgs& a, int bn, bool two,
                 int num_sms, cudaStream_t s) {
  switch (a.ep.kind) {
    case EPI_ROPE_F16: return launch_few_rows<BN, EPI_ROPE_F16>(A, lda, B, ldb, a, bn, two, num_sms, s);
    case EPI_SWIGLU_F16: return launch_few_rows<BN, EPI_SWIGLU_F16>(A, lda, B, ldb, a, bn, two, num_sms, s);
    case EPI_RESID_F32:
    case EPI_RESID_ADD:  // the same sum, added by the epilogue threads
      return launch_few_rows<BN, EPI_RESID_F32>(A, lda, B, ldb, a, bn, two, num_sms, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

// The kernels' times are estimated from what bounds them, in SM clocks, and the
// smallest wins.  Per 64-deep k-block a CTA of the few-rows kernels takes the larger
// of its MMAs (45 clocks each, where issue bounds them) and of its operands' arrival
// (60 bytes per clock); the large tiles measure 720
// (128 x 256), 540 (128 x 128) and 660 (CTA pair).  An epilogue column costs 100
// clocks where the threads add to the residual, 50 for SwiGLU, 40 for RoPE and 22 for the
// TMA add with four epilogue warps, 70, 25 and 25 with the few-rows kernels' eight, and
// each epilogue 1200 more for its hand-offs (1800 in a pair, whose launch takes 1400
// longer: products of 64 to 3000 rows and N, K <= 512 take 10.5 us in pairs and 8.8
// without); a tile's epilogue runs beside the next tile's main loop.  A product that
// feeds a norm costs 4000 more in narrow tiles, the launch of k_row_ss behind it (a tiny
// decoder's query over 319 rows 300 us without this term, 288 with).  Measured
// (us, weights from DRAM; with about 7 us of launch and event overhead; from 128 rows
// on by pairs, and in brackets what one CTA per 128 rows took):
//   M     N      K      large   16          32          64          128
//   24    2048   8192   55.6    18.5        21.3        23.0        32.1
//   128   4096   14336  96.4    41.4 (82.7) 35.0 (47.1) 39.8 (49.6) 55.2 (71.5)
//   300   2048   8192   59.4    34.8 (72.9) 30.4 (52.4) 26.3 (33.4) 36.4 (46.5)
//   1000  2048   8192   54.0    69.6 (157)  50.7 (95.4) 42.4 (56.5) 36.8 (48.3)
//   24    28672  4096   53.3    67.1        48.5        44.7        48.9
//   500   28672  4096   98.8    216 (518)   140 (266)   106 (148)   87.2 (115)
// Eight epilogue warps against four: 16384 x 2048 SwiGLU, 500 rows 37.8 -> 35.6, 1000
// rows 57.2 -> 52.1; 1024 x 128, 10184 rows 33.1 -> 25.2.
FewTile gemm_few_tile(int M, int N, int K, int bn, bool pair, const GemmEpilogue& ep, int num_sms) {
  if (M > kFewRowsMax) return {};
  int epi = 0, epi_large = 0;  // clocks per column
  switch (ep.kind) {
    case EPI_ROPE_F16: epi = 25, epi_large = 40; break;
    case EPI_SWIGLU_F16: epi = 25, epi_large = 50; break;
    case EPI_RESID_F32: epi = 70, epi_large = 100; break;
    case EPI_RESID_ADD: epi = 70, epi_large = 22; break;
    default: return {};  // the plain and argmax epilogues
  }
  const int64_t kblocks = K / BK;
  auto cost = [&](int64_t tiles, int64_t units, int64_t per_kblock, int64_t epilogue, int64_t hand_off = 1200) {
    const int64_t waves = (tiles + units - 1) / units, main = kblocks * per_kblock;
    epilogue += hand_off;
    return main + (waves - 1) * std::max(main, epilogue) + epilogue;
  };
  const int64_t m128 = (M + 127) / 128;
  int64_t best = pair && K % (BK * CfgPair::SUB) == 0
                     ? cost((M + 255) / 256 * (N / 256), num_sms / 2, 660, 256 * epi_large)
                     : cost(m128 * (N / bn), num_sms, bn == 256 ? 720 : 540, bn * epi_large);
  FewTile tile;
  const int64_t sums = ep.ss_out ? 4000 : 0;
  const int rows = M < kFewRows ? (M + 7) / 8 * 8 : kFewRows;
  const int64_t m64 = (M + 63) / 64;
  for (int t = 16; t <= 128; t *= 2) {
    if (t / 2 > few_half(t, bn, ep)) break;  // a tile's halves lie within a gate / up block or a head
    const int64_t load = (rows + t) * 128 / 60;
    int64_t c = sums + cost(m64 * (N / t), num_sms, std::max<int64_t>({180, 2 * t, load}), t * epi);
    if (c < best) best = c, tile = {t, false};
    if (M <= kFewRows || N % (2 * t) != 0) continue;
    c = sums + 1400 + cost(m128 * (N / (2 * t)), num_sms / 2, std::max<int64_t>(180, load), t * epi, 1800);
    if (c < best) best = c, tile = {t, true};
  }
  return tile;
}

int gemm_f16_tcgen05(const __half* A, int64_t lda, const __half* B, int64_t ldb, int M, int N, int K, int bn,
                     bool pair, const GemmEpilogue& ep, int num_sms, cudaStream_t stream) {
  if (M == 0) return 0;
  if (M < 0 || N <= 0 || K <= 0 || K % BK != 0 || (bn != 128 && bn != 256) || N % bn != 0) return cudaErrorInvalidValue;
  if (pair && bn != 256) return cudaErrorInvalidValue;
  if (K % (BK * CfgPair::SUB) != 0) pair = false;  // CTA-pair stages hold 128-deep k-blocks
  if ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15) return cudaErrorMisalignedAddress;
  if ((lda * 2) % 16 != 0 || (ldb * 2) % 16 != 0) return cudaErrorInvalidValue;
  KArgs a{M, N, K, ep};
  if (ep.kind == EPI_ROPE_F16) {
    const int hd = ep.head_dim;
    if (!(hd == 32 || hd == 64 || hd == 128) || bn % hd != 0 || !ep.positions || !ep.rope_cos || !ep.rope_sin)
      return cudaErrorInvalidValue;
    // a head that starts below rope_cols is rotated whole: past this point the
    // kernels see multiples of a head only
    const int cols = std::min(std::max(ep.rope_cols, 0), N);
    a.ep.rope_cols = (cols + hd - 1) / hd * hd;
  }
  if (ep.kind == EPI_ARGMAX && (!ep.bias || !ep.best)) return cudaErrorInvalidValue;
  if (ep.kind == EPI_RESID_ADD &&
      (!ep.out || (reinterpret_cast<uintptr_t>(ep.out) & 15) || (ep.ldo * 4) % 16 != 0 || ep.xh_out))
    return cudaErrorInvalidValue;
  const FewTile few = gemm_few_tile(M, N, K, bn, pair, ep, num_sms);
  switch (few.bn) {
    case 16: return dispatch_few<16>(A, lda, B, ldb, a, bn, few.two_ctas, num_sms, stream);
    case 32: return dispatch_few<32>(A, lda, B, ldb, a, bn, few.two_ctas, num_sms, stream);
    case 64: return dispatch_few<64>(A, lda, B, ldb, a, bn, few.two_ctas, num_sms, stream);
    case 128: return dispatch_few<128>(A, lda, B, ldb, a, bn, few.two_ctas, num_sms, stream);
  }
  CUtensorMap ma, mb, mc;
  if (!make_map(&ma, A, M, K, lda, BM) || !make_map(&mb, B, N, K, ldb, pair ? 128 : bn)) return cudaErrorInvalidValue;
  if (ep.kind == EPI_RESID_ADD) {
    if (!make_map_out_f32(&mc, static_cast<float*>(ep.out), M, N, ep.ldo)) return cudaErrorInvalidValue;
  } else {
    mc = ma;  // unused by the other epilogues
  }
  if (pair) return dispatch_pair(ma, mb, mc, a, num_sms, stream);
  return bn == 256 ? dispatch_epi<256>(ma, mb, mc, a, num_sms, stream)
                   : dispatch_epi<128>(ma, mb, mc, a, num_sms, stream);
}

}  // namespace aiq
