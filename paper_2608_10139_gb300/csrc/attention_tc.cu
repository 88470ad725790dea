// Causal grouped-query attention on the 5th-generation tensor cores.
//
// One work item = (32 consecutive tokens of one sequence) x (the 4 query heads
// sharing one key/value head): its 128 query rows fill the M = 128 rows of a
// tcgen05 MMA, so every key/value block is fetched once per head group.  The
// keys of the shared prompt prefix (computed once per query, in prefix_kv)
// come first, then the sequence's own keys up to the tile's last token.
//
//   warp 0    TMA: the Q tile (3-D box hd x heads x tokens), then K and V blocks
//             of 64 keys into two rings (128-byte swizzle).  A K slot is free
//             once the S MMA that read it has completed, a V slot once the PV MMA
//             that read it has.  The same thread publishes each item's bounds in a
//             four-slot shared ring, an item ahead of its loads, so that no role
//             waits on global loads between items.
//   warp 1    tcgen05.mma: S = Q K^T into a 64-column TMEM score buffer, and
//             O += P V into the output accumulator, with P read from TMEM (it
//             overwrites its own scores) and V read as an MN-major operand
//             straight from its TMA tile.
//   warps 2-5 one query row per thread: read its 64 scores with tcgen05.ld, 32
//             at a time, apply the causal / prefix / length mask, and write
//             exp2(s - max) as fp16 pairs back over the first 32 columns of the
//             same score buffer with tcgen05.st.  The running max is raised
//             (and the output rescaled) only when it grows by more than 2^8, so
//             P never exceeds 256: the exponents are formed with the old max
//             while the new one is found, and formed again in the rare block
//             that raises it.  An item's output is divided by the row sum and
//             stored by its threads in 32-byte pieces, live rows only.
//
// Latency bounds it: a block costs a softmax warp some 500 issue clocks, and the
// way from its P to its next scores (two barriers, PV and S) takes as long.  So
// several CTAs share an SM, each SM sub-partition switching between their softmax
// warps, and every wait that can be taken before P arrives is: the MMA warp has
// the next block's K, V and Q in hand when P comes, and issues PV(g) and S(g+1)
// together.
//
// Ordering: tcgen05 MMAs of one thread run in issue order.  With one score
// buffer S(g+1) is issued after PV(g), which reads P(g) from that buffer; a
// softmax thread that has seen S(g) complete therefore knows that PV(g-1) has,
// too.  With two buffers S(g+1) is issued before PV(g) inside an item, S(g+2)
// after it, and seeing S(g) implies PV(g-2); the thread waits for PV(g-1) before
// it rescales the output.  Either way its parity waits on the two PV barriers
// can never be a full phase behind.  P is signalled on one barrier per score
// buffer: a warp cannot signal P(g + NS) before PV(g) has been issued.
// Work items are persistent per CTA; every wait is bounded.
#include <cudaTypedefs.h>

#include "common.cuh"
#include "kernels.h"

namespace aiq {
namespace {

constexpr int kThreadsTC = 192;
constexpr int kKeys = 64;  // keys per block

// Three CTAs per SM at head_dim 64, two at 128 (TMEM holds 512 columns).  The launch
// measures, for 970 rows of the select workload's text (128,867 tokens, 64 prefix
// keys, 32/8 heads, head_dim 64), 360 us, and 418 for two CTAs of 192 threads that
// double the score buffers and accumulators and store through shared memory; at
// head_dim 128 (150 rows, 34,972 tokens, 128 prefix keys) 202 us, and 326 for one such
// CTA per SM.  A whole call adds some 15 to 25 us.  What else was measured, each
// against the kernel it changed and with what the timing added: four CTAs with one Q
// slot and two K slots 399, two with four K and V slots 455, a CTA of two tiles that
// share K and V 427 and 346, its one MMA warp serving both tiles' hand-offs in turn,
// outputs staged in shared memory for TMA 418 and 242, 16-byte row stores 395 and 236,
// MMAs issued by one lane's control flow instead of a whole warp's 437 and 252, all
// against 387 and 222; outputs staged by each warp on its own 395 and 226 against 376
// and 217.
template <int HD>
struct ACfg {
  static constexpr int NC = HD / 64;             // 64-column sub-tiles of one head
  static constexpr int CTAS = HD == 64 ? 3 : 2;  // per SM
  static constexpr int NQ = HD == 64 ? 2 : 1;    // Q slots
  static constexpr int NK = HD == 64 ? 3 : 2;    // slots of the K ring
  static constexpr int NV = 2;                   // slots of the V ring
  static constexpr int NS = HD == 64 ? 1 : 2;    // score buffers
  static constexpr int Q_BYTES = 128 * HD * 2;   // 128 rows
  static constexpr int SUB = 64 * 128;           // one [64 x 64] fp16 sub-tile
  static constexpr int K_BYTES = NC * SUB;
  static constexpr int OFF_Q = 0;
  static constexpr int OFF_K = OFF_Q + NQ * Q_BYTES;
  static constexpr int OFF_V = OFF_K + NK * K_BYTES;
  static constexpr int OFF_INFO = OFF_V + NV * K_BYTES;  // item bounds ring, 4 x int4
  static constexpr int OFF_BAR = OFF_INFO + 4 * 16;
  static constexpr int N_BARS = 2 * NQ + 2 * NK + 2 * NV + 2 + 2 + 2 + 1 + 1 + 8;
  static constexpr int SMEM = OFF_BAR + N_BARS * 8 + 16;
  // the score buffers, then the output accumulator
  static constexpr int TMEM_COLS = HD == 64 ? 128 : 256;
  static constexpr int O_COL = NS * kKeys;
  static_assert(O_COL + HD <= TMEM_COLS && CTAS * TMEM_COLS <= 512, "TMEM columns");
  // each CTA also keeps 1 KB of the SM's shared memory
  static_assert(CTAS * (SMEM + 1024) <= 233472, "shared memory per SM");
};

struct AttnArgs {
  const int32_t* seq_start;
  const int32_t* tile_seq;
  const int32_t* tile_q0;
  const int32_t* n_tiles;
  int Hq, Hkv, G, TQ, P;
  bool prefix_is_seq0;  // the first sequence is the prefix: its items have no prefix keys
  float scale_log2;
  __half* out;
  int* err;
};

// 2^x with the SFU's approximation (relative error ~2^-22, flushes
// subnormals): plenty for probabilities that are rounded to fp16 next.
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Packed fp32 pairs (Blackwell f32x2): two IEEE fma / add per instruction,
// each lane's result identical to the scalar operation.
__device__ __forceinline__ unsigned long long f2_bits(float2 v) {
  return (static_cast<unsigned long long>(__float_as_uint(v.y)) << 32) | __float_as_uint(v.x);
}
__device__ __forceinline__ float2 bits_f2(unsigned long long b) {
  return make_float2(__uint_as_float(static_cast<uint32_t>(b)), __uint_as_float(static_cast<uint32_t>(b >> 32)));
}
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)), "l"(f2_bits(c)));
  return bits_f2(r);
}
__device__ __forceinline__ float2 fadd2(float2 a, float2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
  return bits_f2(r);
}

// 32 bytes to global memory in one instruction (32-byte aligned).
__device__ __forceinline__ void st_global_v8(void* p, const uint32_t* r) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(r[0]), "r"(r[1]), "r"(r[2]),
               "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}

// MN-major operand (N contiguous) in the 128-byte swizzle: rows of 64 N
// elements, 8-row groups 1024 B apart along K, 64-column atoms 8 KB apart along N.
__device__ __forceinline__ uint64_t smem_desc_mn_sw128(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>(lbo >> 4) << 16;
  d |= static_cast<uint64_t>(sbo >> 4) << 32;
  d |= static_cast<uint64_t>(1u) << 46;
  d |= static_cast<uint64_t>(2u) << 61;
  return d;
}

// D (TMEM) (+)= A (TMEM: lane = row, two fp16 per 32-bit column along K) * B (smem).
__device__ __forceinline__ void umma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// 32 scores of this thread's row from TMEM, those of keys >= lim masked.
__device__ __forceinline__ void load_scores(uint32_t taddr, float* v, bool mask, int lim) {
  uint32_t r[32];
  tmem_ld_32x32b_x32(taddr, r);
  tmem_ld_wait();
#pragma unroll
  for (int c = 0; c < 32; ++c) v[c] = __uint_as_float(r[c]);
  if (mask) {
    const uint32_t visible = lim >= 32 ? ~0u : (lim <= 0 ? 0u : (1u << lim) - 1u);
#pragma unroll
    for (int c = 0; c < 32; ++c) v[c] = (visible >> c) & 1u ? v[c] : -INFINITY;
  }
}

// Eight independent partial maxima keep the chain short.
__device__ __forceinline__ float max32(const float* v) {
  float pm[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) pm[c] = v[c];
#pragma unroll
  for (int c = 8; c < 32; ++c) pm[c & 7] = fmaxf(pm[c & 7], v[c]);
  return fmaxf(fmaxf(fmaxf(pm[0], pm[1]), fmaxf(pm[2], pm[3])), fmaxf(fmaxf(pm[4], pm[5]), fmaxf(pm[6], pm[7])));
}

// P of 32 scores: exp2(scale v - m) as fp16 pairs, added (in fp32) to ps.
__device__ __forceinline__ void exp32(const float* v, float scale_log2, float m, uint32_t* pk, float2* ps) {
  const float2 sc2 = make_float2(scale_log2, scale_log2), nm2 = make_float2(-m, -m);
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float2 x = ffma2(make_float2(v[2 * i], v[2 * i + 1]), sc2, nm2);
    const float2 p = make_float2(ex2_approx(x.x), ex2_approx(x.y));
    ps[i & 3] = fadd2(ps[i & 3], p);
    __half2 h = __floats2half2_rn(p.x, p.y);
    pk[i] = *reinterpret_cast<uint32_t*>(&h);
  }
}

template <int HD>
__global__ void __launch_bounds__(kThreadsTC, ACfg<HD>::CTAS)
    k_attention_tc(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_kv,
                   const __grid_constant__ CUtensorMap tm_pre, AttnArgs a) {
  using C = ACfg<HD>;
  constexpr int NQ = C::NQ, NK = C::NK, NV = C::NV, NS = C::NS;
  extern __shared__ __align__(1024) uint8_t smem[];  // swizzled tiles want 1024-byte alignment
  uint64_t* q_full = reinterpret_cast<uint64_t*>(smem + C::OFF_BAR);  // [NQ]
  uint64_t* q_empty = q_full + C::NQ;      // [NQ]: the item's S MMAs have completed
  uint64_t* k_full = q_empty + C::NQ;      // [NK]
  uint64_t* k_empty = k_full + NK;         // [NK]: the S MMA of the block has completed
  uint64_t* v_full = k_empty + NK;         // [NV]
  uint64_t* v_empty = v_full + NV;         // [NV]: the PV MMA of the block has completed
  uint64_t* s_full = v_empty + NV;         // [NS]: block g's scores, g % NS
  uint64_t* p_full = s_full + 2;           // [NS]: P of block g written over its scores
  uint64_t* o_done = p_full + 2;           // [2]: PV of block g commits o_done[g & 1]
  uint64_t* o_free = o_done + 2;           // the item's output has been read out
  uint64_t* mma_done = o_free + 1;
  uint64_t* info_full = mma_done + 1;      // [4]: item bounds published by the TMA thread
  uint64_t* info_empty = info_full + 4;    // [4]: read by the MMA warp and the four softmax warps
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(info_empty + 4);
  int4* info = reinterpret_cast<int4*>(smem + C::OFF_INFO);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  auto sQ = [&](int b) { return smem + C::OFF_Q + b * C::Q_BYTES; };
  auto sK = [&](int b) { return smem + C::OFF_K + b * C::K_BYTES; };
  auto sV = [&](int b) { return smem + C::OFF_V + b * C::K_BYTES; };
  if (smem_u32(smem) & 1023) {  // no tile is touched then
    grid_wait();  // not done before the kernel ahead is
    if (threadIdx.x == 0) set_dev_error(a.err, DEVERR_BOUNDS);
    return;
  }

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int* err = a.err;
  if (threadIdx.x == 0) {
    for (int b = 0; b < NQ; ++b) {
      mbar_init(&q_full[b], 1);
      mbar_init(&q_empty[b], 1);
    }
    for (int b = 0; b < NK; ++b) {
      mbar_init(&k_full[b], 1);
      mbar_init(&k_empty[b], 1);
    }
    for (int b = 0; b < NV; ++b) {
      mbar_init(&v_full[b], 1);
      mbar_init(&v_empty[b], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&s_full[b], 1);
      mbar_init(&p_full[b], 4);
      mbar_init(&o_done[b], 1);
    }
    mbar_init(o_free, 4);
    mbar_init(mma_done, 1);
    for (int b = 0; b < 4; ++b) {
      mbar_init(&info_full[b], 1);
      mbar_init(&info_empty[b], 5);
    }
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tm_q);
    tma_prefetch_desc(&tm_kv);
    tma_prefetch_desc(&tm_pre);
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

  const int n_work = *a.n_tiles * a.Hkv;
  // An item's bounds {start, length, first token, key/value head}; kNoPrefix is
  // added to the head of an item without prefix keys.
  constexpr int kNoPrefix = 1 << 24;
  const int n_prefix = (a.P + kKeys - 1) / kKeys;
  auto prefix_blocks = [&](const int4& inf) -> int { return inf.w < kNoPrefix ? n_prefix : 0; };
  // key blocks of an item: the shared prefix's, then the row's own up to the tile's last token
  auto blocks_of = [&](const int4& inf) -> int {
    return prefix_blocks(inf) + (min(inf.z + a.TQ, inf.y) + kKeys - 1) / kKeys;
  };
  // Every wait of the MMA and softmax warps is taken warp-uniformly: a lane that
  // gives up (timeout or abort) makes the whole warp give up, so no lane is left
  // alone in the warp-synchronous instructions that follow.
  auto wait_all = [&](uint64_t* bar, uint32_t parity) -> bool {
    return __all_sync(0xffffffffu, mbar_wait_bounded(bar, parity, abort_flag, err));
  };

  if (warp == 0) {
    if (lane == 0) {
      // ------------------------------------------------------------ TMA
      uint32_t g = 0;   // key blocks whose K load was issued (ring position)
      uint32_t gv = 0;  // key blocks whose V load was issued
      int it = 0;       // Q loads issued
      bool ok = true;
      // an item's bounds hang on two dependent loads: the work list is read three
      // items ahead, the sequence's bounds two ahead, and published one ahead
      auto list = [&](int w) -> int2 {
        if (w >= n_work) return make_int2(0, 0);
        const int i = w / a.Hkv;
        return make_int2(a.tile_seq[i], a.tile_q0[i]);
      };
      auto bounds = [&](int2 l, int w) -> int4 {
        const int st = a.seq_start[l.x];
        return make_int4(st, a.seq_start[l.x + 1] - st, l.y,
                         w % a.Hkv + (a.prefix_is_seq0 && l.x == 0 ? kNoPrefix : 0));
      };
      auto publish = [&](int item, const int4& inf) -> bool {
        const int is = item & 3;
        if (!mbar_wait_bounded(&info_empty[is], ((item >> 2) & 1) ^ 1, abort_flag, err)) return false;
        info[is] = inf;
        mbar_arrive(&info_full[is]);
        return true;
      };
      // the V load of the block whose K load came last
      const CUtensorMap* v_map = nullptr;
      int v_col = 0, v_row = 0;
      auto load_v = [&]() -> bool {
        const int vb = gv % NV;
        if (!mbar_wait_bounded(&v_empty[vb], ((gv / NV) & 1) ^ 1, abort_flag, err)) return false;
        mbar_arrive_expect_tx(&v_full[vb], C::K_BYTES);
        for (int c = 0; c < C::NC; ++c) tma_load_2d(sV(vb) + c * C::SUB, v_map, &v_full[vb], v_col + c * 64, v_row);
        ++gv;
        return true;
      };
      const int step = gridDim.x;
      int w = blockIdx.x;
      int4 cur = bounds(list(w), w), nxt = bounds(list(w + step), w + step);
      int2 ahead = list(w + 2 * step);
      if (w < n_work) ok = publish(0, cur);
      for (; w < n_work && ok; w += step) {
        const int4 after = bounds(ahead, w + 2 * step);
        ahead = list(w + 3 * step);
        const int st = cur.x, kvh = cur.w % kNoPrefix, n_pre = prefix_blocks(cur);
        const int n_kv = blocks_of(cur);
        const int qb = it % NQ;
        if (!mbar_wait_bounded(&q_empty[qb], ((it / NQ) & 1) ^ 1, abort_flag, err)) break;
        mbar_arrive_expect_tx(&q_full[qb], C::Q_BYTES);
        ++it;
        for (int c = 0; c < C::NC; ++c)
          tma_load_3d(sQ(qb) + c * (128 * 128), &tm_q, &q_full[qb], c * 64, kvh * a.G, st + cur.z);
        if (w + step < n_work && !publish(it, nxt)) break;
        for (int j = 0; j < n_kv; ++j, ++g) {
          const bool pre = j < n_pre;
          const CUtensorMap* map = pre ? &tm_pre : &tm_kv;
          const int kcol = pre ? kvh * HD : (a.Hq + kvh) * HD;
          const int row = pre ? j * kKeys : st + (j - n_pre) * kKeys;
          const int kb = g % NK;
          if (!mbar_wait_bounded(&k_empty[kb], ((g / NK) & 1) ^ 1, abort_flag, err)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&k_full[kb], C::K_BYTES);
          for (int c = 0; c < C::NC; ++c) tma_load_2d(sK(kb) + c * C::SUB, map, &k_full[kb], kcol + c * 64, row);
          // V a block behind K: its slot frees with the PV two blocks back, and the
          // next item's Q and first K must not wait for that
          if (g > 0 && !load_v()) {
            ok = false;
            ++g;  // this block's K load is in flight
            break;
          }
          v_map = map;
          v_col = pre ? (a.Hkv + kvh) * HD : (a.Hq + a.Hkv + kvh) * HD;
          v_row = row;
        }
        cur = nxt;
        nxt = after;
      }
      if (ok && g > gv && !load_v()) ok = false;
      if (!ok || *abort_flag) {
        // let this thread's copies still in flight land before the CTA can exit
        // (the last use of each slot is the only one that can be outstanding)
        volatile int never = 0;
        for (uint32_t i = g > NK ? g - NK : 0; i < g; ++i)
          mbar_wait_bounded(&k_full[i % NK], (i / NK) & 1, &never, nullptr, 200000000ull);
        for (uint32_t i = gv > NV ? gv - NV : 0; i < gv; ++i)
          mbar_wait_bounded(&v_full[i % NV], (i / NV) & 1, &never, nullptr, 200000000ull);
        for (int i = it > NQ ? it - NQ : 0; i < it; ++i)
          mbar_wait_bounded(&q_full[i % NQ], (i / NQ) & 1, &never, nullptr, 200000000ull);
      }
    }
  } else if (warp == 1) {
    // -------------------------------------------------------------- MMA
    // the whole warp walks the blocks and one elected lane issues, so that the
    // descriptors stay in uniform registers
    constexpr uint32_t idesc_s = idesc_f16_f32(128, kKeys);
    constexpr uint32_t idesc_o = idesc_f16_f32(128, HD) | (1u << 16);  // B (= V) MN-major
    const uint32_t tb = __shfl_sync(0xffffffffu, tmem_base, 0);
    const uint64_t dq0 = smem_desc_k_sw128(smem_u32(sQ(0))), dk0 = smem_desc_k_sw128(smem_u32(sK(0)));
    const uint64_t dv0 = smem_desc_mn_sw128(smem_u32(sV(0)), HD == 64 ? 1024u : 8192u, 1024u);
    // (one lane) S of block gg, its K and Q landed; `last`: its item's last block,
    // after which Q's slot is free
    auto issue_s = [&](uint32_t gg, int qb, bool last) {
      const uint32_t kb = gg % NK;
      const uint32_t d = tb + (gg % NS) * kKeys;
      const uint64_t dq = dq0 + qb * (C::Q_BYTES >> 4), dk = dk0 + kb * (C::K_BYTES >> 4);
#pragma unroll
      for (int c = 0; c < C::NC; ++c)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint64_t qa = dq + c * (128 * 128 >> 4) + 2 * k, ka = dk + c * (C::SUB >> 4) + 2 * k;
          if (c == 0 && k == 0)
            umma_f16_ss(d, qa, ka, idesc_s, 0);
          else
            umma_f16_ss_acc(d, qa, ka, idesc_s);
        }
      umma_commit(&s_full[gg % NS]);
      umma_commit(&k_empty[kb]);
      if (last) umma_commit(&q_empty[qb]);
    };
    // the blocks of item `item` (ring slot item & 3), once its Q and first K have landed
    auto take_item = [&](int item, uint32_t gg, int* n) -> bool {
      const int is = item & 3;
      if (!wait_all(&info_full[is], (item >> 2) & 1)) return false;
      *n = blocks_of(info[is]);
      __syncwarp();
      if (lane == 0) mbar_arrive(&info_empty[is]);
      return wait_all(&q_full[item % NQ], (item / NQ) & 1) && wait_all(&k_full[gg % NK], (gg / NK) & 1);
    };
    uint32_t g = 0;
    int it = 0, n_kv = 0;
    bool ok = true;
    int w = blockIdx.x;
    if (w < n_work) {
      // The blocks of all this CTA's items form one stream: the scores of the
      // next block, also the first block of the next item, are issued as soon
      // as their buffer allows, so an item boundary costs no extra hand-off.
      ok = take_item(0, 0, &n_kv);
      if (ok) {
        tc_fence_after();
        if (elect_one()) issue_s(0, 0, n_kv == 1);
        __syncwarp();
      }
      while (ok) {
        const bool more = w + static_cast<int>(gridDim.x) < n_work;
        int n_next = 0;
        for (int j = 0; j < n_kv; ++j, ++g) {
          const bool inside = j + 1 < n_kv;
          // With two score buffers the next scores of this item come before this
          // block's PV; the next item's come after it, as its Q may have to wait
          // for this item's last S.
          const bool early = NS == 2 && inside;
          if (inside) {
            if (!wait_all(&k_full[(g + 1) % NK], ((g + 1) / NK) & 1)) {
              ok = false;
              break;
            }
            if (early) {
              tc_fence_after();
              if (elect_one()) issue_s(g + 1, it % NQ, j + 2 == n_kv);
              __syncwarp();
            }
          } else if (more && NQ > 1 && !take_item(it + 1, g + 1, &n_next)) {
            ok = false;
            break;
          }
          // the first PV overwrites the accumulator: the softmax warps must have
          // read out the previous item's output
          const uint32_t vb = g % NV;
          if (!wait_all(&v_full[vb], (g / NV) & 1) || (j == 0 && !wait_all(o_free, (it & 1) ^ 1)) ||
              !wait_all(&p_full[g % NS], (g / NS) & 1)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t dv = dv0 + vb * (C::K_BYTES >> 4);
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
              umma_f16_ts(tb + C::O_COL, tb + (g % NS) * kKeys + k * 8, dv + k * (2048 >> 4), idesc_o, (j | k) != 0);
            umma_commit(&o_done[g & 1]);
            umma_commit(&v_empty[vb]);
            if (!early && inside) issue_s(g + 1, it % NQ, j + 2 == n_kv);
            if (!inside && more && NQ > 1) issue_s(g + 1, (it + 1) % NQ, n_next == 1);
          }
          __syncwarp();
          if (!inside && more && NQ == 1) {
            if (!take_item(it + 1, g + 1, &n_next)) {
              ok = false;
              break;
            }
            tc_fence_after();
            if (elect_one()) issue_s(g + 1, (it + 1) % NQ, n_next == 1);
            __syncwarp();
          }
        }
        if (!ok || !more) break;
        w += gridDim.x;
        n_kv = n_next;
        ++it;
      }
    }
    if (elect_one()) umma_commit(mma_done);
    __syncwarp();
    volatile int never = 0;
    mbar_wait_bounded(mma_done, 0, &never, err);
  } else {
    // ------------------------------------------------- softmax / epilogue
    const int quarter = warp & 3;
    const int r = quarter * 32 + lane;  // TMEM lane = query row of the tile
    const int t = r / a.G, gq = r % a.G;
    const uint32_t trow = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
    const uint32_t ocol = trow + C::O_COL;
    const bool wide = (reinterpret_cast<uintptr_t>(a.out) & 31) == 0;  // 32-byte stores
    uint32_t g = 0;
    int it = 0;
    bool ok = true;
    // PV of block gg done (see the ordering note above: the parity is exact)
    auto wait_pv = [&](uint32_t gg) -> bool { return wait_all(&o_done[gg & 1], (gg >> 1) & 1); };
    auto take_info = [&](int item, int4* inf) -> bool {
      const int is = item & 3;
      if (!wait_all(&info_full[is], (item >> 2) & 1)) return false;
      *inf = info[is];
      __syncwarp();
      if (lane == 0) mbar_arrive(&info_empty[is]);
      return true;
    };
    int4 inf = make_int4(0, 0, 0, 0), inf_next = inf;
    if (static_cast<int>(blockIdx.x) < n_work) ok = take_info(0, &inf_next);
    for (int w = blockIdx.x; w < n_work && ok; w += gridDim.x, ++it) {
      inf = inf_next;
      const int st = inf.x, len = inf.y, q0 = inf.z, kvh = inf.w % kNoPrefix;
      const int n_pre = prefix_blocks(inf), n_kv = blocks_of(inf);
      const int qpos = q0 + t;
      float m_used = 0.f, l = 0.f;
      for (int j = 0; j < n_kv; ++j, ++g) {
        const uint32_t sb = g % NS;
        if (!wait_all(&s_full[sb], (g / NS) & 1)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t scol = trow + sb * kKeys;
        const bool pre = j < n_pre;
        const int key0 = (pre ? j : j - n_pre) * kKeys;
        // warp-uniform: only the prefix's last block and the causal diagonal /
        // sequence end need a mask; then key c is visible iff c < lim
        const bool mask = pre ? (key0 + kKeys > a.P) : (key0 + kKeys - 1 > q0 || key0 + kKeys > len);
        const int lim = pre ? a.P - key0 : min(qpos + 1, len) - key0;
        float v[32];
        if (j == 0) {
          // running max on the raw scores; the softmax scale (with log2 e) is
          // folded into one FMA inside the exponent
          load_scores(scol, v, mask, lim);
          float mr = max32(v);
          load_scores(scol + 32, v, mask, lim - 32);
          mr = fmaxf(mr, max32(v));
          m_used = mr == -INFINITY ? 0.f : mr * a.scale_log2;
        }
        uint32_t pk[32];
        float2 ps[4];
        for (;;) {
#pragma unroll
          for (int i = 0; i < 4; ++i) ps[i] = make_float2(0.f, 0.f);
          load_scores(scol, v, mask, lim);
          float mr = max32(v);
          exp32(v, a.scale_log2, m_used, pk, ps);
          load_scores(scol + 32, v, mask, lim - 32);
          mr = fmaxf(mr, max32(v));
          exp32(v, a.scale_log2, m_used, pk + 16, ps);
          const float mx = mr * a.scale_log2;
          const bool grow = j > 0 && mx > m_used + 8.f;
          if (!__any_sync(0xffffffffu, grow)) break;
          // rescale this warp's output rows once the previous block's PV is done,
          // and form this block's P again from its scores, still in place
          if (NS == 2) {
            if (!wait_pv(g - 1)) {
              ok = false;
              break;
            }
            tc_fence_after();
          }
          const float f = grow ? ex2_approx(m_used - mx) : 1.f;
          if (grow) {
            l *= f;
            m_used = mx;
          }
#pragma unroll 1
          for (int c = 0; c < HD; c += 32) {
            uint32_t o[32];
            tmem_ld_32x32b_x32(ocol + c, o);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * f);
            tmem_st_32x32b_x32(ocol + c, o);
          }
          tmem_st_wait();
        }
        if (!ok) break;
        l += ((ps[0].x + ps[0].y) + (ps[1].x + ps[1].y)) + ((ps[2].x + ps[2].y) + (ps[3].x + ps[3].y));
        // P (fp16 pairs) over the first 32 columns of this block's score buffer
        tmem_st_32x32b_x32(scol, pk);
        tmem_st_wait();
        tc_fence_before();  // this block's score reads and P writes are complete
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_full[sb]);
      }
      if (!ok) break;
      // the next item's bounds while this item's last PV runs
      if (w + static_cast<int>(gridDim.x) < n_work && !take_info(it + 1, &inf_next)) break;
      // O / l of the tile's real tokens, once the item's last PV is done
      if (!wait_pv(g - 1)) break;
      tc_fence_after();
      const float inv = l > 0.f ? 1.f / l : 0.f;
      __half* dst = a.out + static_cast<int64_t>(st + qpos) * (a.Hq * HD) + (kvh * a.G + gq) * HD;
#pragma unroll 1
      for (int c = 0; c < HD; c += 32) {
        uint32_t o[32], pk[16];
        tmem_ld_32x32b_x32(ocol + c, o);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          __half2 h = __floats2half2_rn(__uint_as_float(o[2 * i]) * inv, __uint_as_float(o[2 * i + 1]) * inv);
          pk[i] = *reinterpret_cast<uint32_t*>(&h);
        }
        if (qpos < len) {
          if (wide) {
            st_global_v8(dst + c, pk);
            st_global_v8(dst + c + 16, pk + 8);
          } else {
#pragma unroll
            for (int q4 = 0; q4 < 4; ++q4)
              reinterpret_cast<uint4*>(dst + c)[q4] = make_uint4(pk[4 * q4], pk[4 * q4 + 1], pk[4 * q4 + 2], pk[4 * q4 + 3]);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(o_free);
    }
  }

  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, C::TMEM_COLS);
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn_attn() {
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

bool map2d(CUtensorMap* m, const __half* base, int64_t rows, int64_t cols, int64_t ld) {
  auto fn = encode_fn_attn();
  if (!fn) return false;
  cuuint64_t dims[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
  cuuint64_t strides[1] = {static_cast<cuuint64_t>(ld * 2)};
  cuuint32_t box[2] = {64, 64};
  cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// qkv viewed as [T][heads][hd]; box = 64 columns x G heads x TQ tokens.
bool map3d_q(CUtensorMap* m, const __half* base, int64_t T, int heads, int hd, int G, int TQ) {
  auto fn = encode_fn_attn();
  if (!fn) return false;
  cuuint64_t dims[3] = {static_cast<cuuint64_t>(hd), static_cast<cuuint64_t>(heads), static_cast<cuuint64_t>(T)};
  cuuint64_t strides[2] = {static_cast<cuuint64_t>(hd * 2), static_cast<cuuint64_t>(int64_t(heads) * hd * 2)};
  cuuint32_t box[3] = {64, static_cast<cuuint32_t>(G), static_cast<cuuint32_t>(TQ)};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<__half*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int HD>
int launch_tc(const CUtensorMap& mq, const CUtensorMap& mkv, const CUtensorMap& mpre, const AttnArgs& a,
              int n_work_max, int num_sms, cudaStream_t s) {
  using C = ACfg<HD>;
  cudaError_t e = cudaFuncSetAttribute(k_attention_tc<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e != cudaSuccess) return e;
  const int grid = n_work_max < num_sms * C::CTAS ? n_work_max : num_sms * C::CTAS;
  if (grid <= 0) return 0;
  return launch_chained(k_attention_tc<HD>, dim3(grid), kThreadsTC, C::SMEM, s, 1, mq, mkv, mpre, a);
}

}  // namespace

bool attention_tc_supported(int hd, int Hq, int Hkv) {
  if (hd != 64 && hd != 128) return false;
  const int G = Hq / Hkv;
  return Hq % Hkv == 0 && G >= 1 && G <= 128 && 128 % G == 0;
}

int attention_tc_tile_tokens(int Hq, int Hkv) { return 128 / (Hq / Hkv); }

int launch_attention_tc(const __half* qkv, int64_t T, const int32_t* seq_start, const int32_t* tile_seq,
                        const int32_t* tile_q0, int n_tiles_max, const int32_t* n_tiles_dev, int Hq, int Hkv, int hd,
                        const PrefixKV& prefix, __half* out, int* err, int num_sms, cudaStream_t s) {
  if (n_tiles_max <= 0 || T <= 0) return 0;
  const int G = Hq / Hkv, TQ = 128 / G;
  const int heads = Hq + 2 * Hkv;
  CUtensorMap mq, mkv, mpre;
  if (!map3d_q(&mq, qkv, T, heads, hd, G, TQ) || !map2d(&mkv, qkv, T, int64_t(heads) * hd, int64_t(heads) * hd))
    return cudaErrorInvalidValue;
  // the output's rows are written in 16- or 32-byte pieces
  if (reinterpret_cast<uintptr_t>(out) & 15) return cudaErrorInvalidValue;
  int P = prefix.P;
  if (prefix.kv && P > 0) {
    if (!map2d(&mpre, prefix.kv, P, int64_t(2) * Hkv * hd, prefix.ld)) return cudaErrorInvalidValue;
  } else {
    mpre = mkv;
    P = 0;
  }
  AttnArgs a{seq_start, tile_seq, tile_q0, n_tiles_dev, Hq, Hkv, G, TQ, P, prefix.is_seq0,
             1.4426950408889634f / sqrtf(static_cast<float>(hd)), out, err};
  const int n_work_max = n_tiles_max * Hkv;
  return hd == 64 ? launch_tc<64>(mq, mkv, mpre, a, n_work_max, num_sms, s)
                  : launch_tc<128>(mq, mkv, mpre, a, n_work_max, num_sms, s);
}

}  // namespace aiq
