// Causal attention of a run of queries (the decoder prefill) on the tcgen05
// tensor cores, for head width 128 (fp16 / bf16 storage, fp32 arithmetic).
//
// Per head h, query t (position pos0 + t) attends to cache positions
// 0 .. pos0 + t:  out[t] = sum_j softmax_j(q_t . k_j / sqrt(128)) v_j.  Both
// contractions are dense and run on the tensor cores; the softmax is exact,
// computed online over key tiles in fp32.
//
// One CTA owns 128 queries of one head.  For each tile of 128 keys:
//   S = Q K^T   tcgen05.mma kind::f16, M 128 (queries) x N 128 (keys) x K 128
//               (head dims); Q and the key tile by TMA (128-byte swizzle,
//               K-major); S in one of two TMEM buffers, so the next tile's S
//               is computed during this tile's softmax
//   P           warps 2..9, two threads per query row (64 keys each): the
//               scores from TMEM into registers, causal mask (only in tiles
//               that the diagonal or the end of the run crosses), running max
//               m (the halves exchange theirs through shared memory) and
//               denominator l, p = e^(s - m) written to shared memory as two
//               bf16/fp16 parts p_hi + p_lo (p_lo = round(p - p_hi)), so the
//               product with V keeps about 16 significant bits of p, not 8;
//               runs of fewer than 64 queries keep all 24 (SHORT)
//   O_t = P V   tcgen05.mma, M 128 x N 128 x K 16 steps for each part; V
//               is the value tile as loaded by TMA (two 64-dim boxes),
//               [keys][dims] with the dims contiguous, i.e. the B operand in
//               MN-major layout
//   O           each softmax thread keeps 64 of its row's outputs in
//               registers: O = O * e^(m_old - m_new) + O_t, added while the
//               next tile's scores are already there
// and at the end writes O / l.  Warp 0 issues the TMA loads (key and value
// tiles double-buffered), warp 1 owns TMEM and issues the MMAs.  What bounds
// it is the softmax's instruction stream, about 9 per score on eight warps;
// 512 queries of 32 heads 24.0 us with one thread per query, the scores read
// twice and every phase waiting for the one before, 14.5 us now; 79 queries
// on a cache of 100, 8 heads, 14.2 -> 9.3 us (both alone, launch included).
// Few queries on a long cache leave most SMs idle and the key tiles one
// after the other: then a cluster of 3 to 8 CTAs shares a (query tile,
// head)'s key tiles (SPLIT; tile kt to CTA kt mod parts, parts known once the
// position is), and the CTAs' (m, l, O) are combined in CTA order through
// distributed shared memory, M = max m, O = sum O e^(m - M) / sum l e^(m - M).
// On 900 earlier keys: 64 queries of 8 heads 18.9 -> 9.7 us, 512 of 8 heads
// 27.1 -> 15.2, 128 of 32 heads 21.9 -> 16.2; a nearly empty cache of 1500
// keys pays 0.4-0.8 us for the possibility.
// Every wait is bounded: on timeout the kernel records kDevErrTimeout, drains
// the loads and MMAs it started, frees TMEM and returns.
#include <cooperative_groups.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "device.cuh"
#include "internal.h"
#include "kernels.h"

namespace swapnet {

namespace {

constexpr int kAQ = 128;        // queries per CTA (MMA M)
constexpr int kAK = 128;        // keys per tile
constexpr int kAD = 128;        // head width
constexpr int kASoft = 256;      // softmax threads: two per query
constexpr int kAThreads = 64 + kASoft;  // warp 0 TMA, warp 1 MMA, warps 2..9 softmax
constexpr int kHalf = 128 * 64 * 2;  // one 128-row x 64-column swizzled half tile (16 KB)
constexpr int kTile = 2 * kHalf;     // 128 x 128 elements
// shared memory: Q | K stage 0, 1 | V stage 0, 1 | P (its parts) | exchange | barriers
constexpr int kOffQ = 0;
constexpr int kOffK = kOffQ + kTile;
constexpr int kOffV = kOffK + 2 * kTile;
constexpr int kOffP = kOffV + 2 * kTile;
constexpr int kOffX = kOffP + 2 * kTile;  // [half][query] floats
constexpr int kOffBar = kOffX + 2 * kAQ * 4;
constexpr int kASmem = kOffBar + 128 + 1024;  // + barriers, TMEM slot, flags; + alignment slack
static_assert(kASmem <= 232448, "attention tile set exceeds the shared memory of a CTA");
// SHORT: runs of fewer than 64 queries use half of the MMA's rows, so the room
// of two parts of P holds three of 64 rows (the MMA's other rows read whatever
// lies behind them, results nobody uses): p = p_hi + p_mid + p_lo, all of its
// 24 bits, as the split-key kernel has them for fewer (query, head) pairs.
// Outputs that are not the rounded float64 result, 63 queries of 8 heads on 900
// keys, bf16: 2.1e-4 there, 2.2e-3 with two parts, 4.5e-4 so (the rest is the
// sums of the tensor cores).  The third part costs 0.2-0.6 us per key tile of
// a CTA (63 x 8 on 900 keys 9.6 -> 9.7 us, 17 x 16 on 3000 14.1 -> 15.9).
// fp16 parts carry p * 2^15, so that their exponent range takes the small ones.
constexpr int kShortRows = 64;
template <bool SHORT> struct PCfg {
  static constexpr int kParts = SHORT ? 3 : 2;
  static constexpr int kHalfBytes = SHORT ? kHalf / 2 : kHalf;  // 64 columns of a part
  static constexpr int kPartBytes = 2 * kHalfBytes;
  static constexpr int kWriters = SHORT ? kASoft / 2 : kASoft;  // threads that own a row
  static_assert((kParts - 1) * kPartBytes + kHalfBytes + kHalf <= 2 * kTile, "the parts and the rows behind them");
};
constexpr int kAMaxSplit = 8;   // portable cluster size
constexpr int kORow = kAD + 4;  // floats of an output row handed to the cluster (over the key and value tiles)
static_assert(kAQ * kORow * 4 <= 4 * kTile, "the output rows overlay the key and value tiles");

constexpr uint32_t kTmemCols = 512;  // S: [0, 128) and [128, 256), O_t: [256, 384)

// Shared-memory descriptor of a B operand stored MN-major with the 128-byte
// swizzle (the layout TMA gives a [K rows][64 N] box): 8-row K groups are
// 1024 bytes apart (stride byte offset); the two 64-column N blocks of the
// value tile (the two TMA boxes) are kHalf bytes apart (leading byte
// offset), so one N = 128 MMA covers all head dims.
__device__ __forceinline__ uint64_t smem_desc_sw128_mn(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(kHalf >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Sharing a query tile's keys out costs about 2 us (the cluster's barriers,
// the outputs through distributed shared memory), a key tile 1.6 us.
__host__ __device__ inline bool split_pays(int tiles, int split) { return tiles - (tiles + split - 1) / split >= 3; }

struct AttnArgs {
  void* out;
  const int* pos_ptr;
  int tokens, heads, width, max_seq;
  float scale_log2;  // log2(e) / sqrt(head width)
  int split;         // CTAs of a cluster that may share a (query tile, head)'s keys
  int* err;
};

template <typename T> __device__ __forceinline__ uint32_t pack2(float lo, float hi);
template <> __device__ __forceinline__ uint32_t pack2<__half>(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
template <> __device__ __forceinline__ uint32_t pack2<__nv_bfloat16>(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
template <typename T> __device__ __forceinline__ float2 unpack2(uint32_t u);
template <> __device__ __forceinline__ float2 unpack2<__half>(uint32_t u) {
  return make_float2(__half2float(__ushort_as_half((unsigned short)(u & 0xffffu))),
                     __half2float(__ushort_as_half((unsigned short)(u >> 16))));
}
template <> __device__ __forceinline__ float2 unpack2<__nv_bfloat16>(uint32_t u) {
  return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
}

template <typename T, bool SPLIT, bool SHORT>
__global__ void __launch_bounds__(kAThreads, 1)
    attention_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                        const __grid_constant__ CUtensorMap tmV, const AttnArgs p) {
  using P = PCfg<SHORT>;
  constexpr float kPScale = SHORT && std::is_same<T, __half>::value ? 32768.0f : 1.0f;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kOffBar);
  const uint32_t q_full = smem_u32(bars + 0);
  auto kv_full = [&](int s) { return smem_u32(bars + 1 + s); };
  auto kv_empty = [&](int s) { return smem_u32(bars + 3 + s); };
  auto s_full = [&](int b) { return smem_u32(bars + 5 + b); };
  const uint32_t p_full = smem_u32(bars + 7);
  const uint32_t o_full = smem_u32(bars + 8);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 9);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + 10);
  const uint32_t done_bar = smem_u32(bars + 11);

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int t0 = blockIdx.x * kAQ, h = blockIdx.y;
  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(kv_full(s), 1);
      mbar_init(kv_empty(s), 1);
    }
    mbar_init(s_full(0), 1);
    mbar_init(s_full(1), 1);
    mbar_init(p_full, P::kWriters);
    mbar_init(o_full, 1);
    mbar_init(done_bar, 1);
    *abort_flag = 0;
    fence_barrier_init();
    prefetch_tmap(&tmQ);
    prefetch_tmap(&tmK);
    prefetch_tmap(&tmV);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t tO = tmem + 256;
  // The launch before rotates q and appends the run's own cache rows; it let
  // this one start only after every launch before it had completed, so the
  // position and the key and value tiles of earlier runs are read already.
  const int pos0 = min(*p.pos_ptr, p.max_seq);  // (a position outside the cache is reported by the rotation)
  const int last_q = min(t0 + kAQ, p.tokens) - 1;
  const int n_keys = max(0, min(pos0 + last_q + 1, p.max_seq));
  const int nkt = (n_keys + kAK - 1) / kAK;
  const int col0 = h * kAD;
  // this CTA's key tiles: z, z + parts, ...
  const int z = SPLIT ? blockIdx.z : 0;
  const int parts = SPLIT && split_pays(nkt, p.split) ? min(p.split, nkt) : 1;
  const int nloc = z < parts ? (nkt - z + parts - 1) / parts : 0;
  auto load_kv = [&](int i) {
    const int s = i & 1, k0 = (z + i * parts) * kAK;
    mbar_arrive_expect_tx(kv_full(s), 2 * kTile);
    const uint32_t ks = smem_u32(smem + kOffK + s * kTile), vs = smem_u32(smem + kOffV + s * kTile);
    tma_load_2d(ks, &tmK, kv_full(s), col0, k0);
    tma_load_2d(ks + kHalf, &tmK, kv_full(s), col0 + 64, k0);
    tma_load_2d(vs, &tmV, kv_full(s), col0, k0);
    tma_load_2d(vs + kHalf, &tmV, kv_full(s), col0 + 64, k0);
  };
  // whole tiles of older rows, one per buffer
  const int early = min(min(2, nloc), (max(pos0, 0) / kAK + parts - 1 - z) / parts);
  if (warp == 0 && elect_one())
    for (int i = 0; i < early; ++i) load_kv(i);
  pdl_wait();
  pdl_launch_dependents();

  if (warp == 0) {
    if (nloc > 0 && elect_one()) {
      // ---------------- TMA producer
      mbar_arrive_expect_tx(q_full, kTile);
      tma_load_2d(smem_u32(smem + kOffQ), &tmQ, q_full, col0, t0);
      tma_load_2d(smem_u32(smem + kOffQ + kHalf), &tmQ, q_full, col0 + 64, t0);
      int i = early;
      for (; i < nloc; ++i) {
        if (i >= 2 && !mbar_wait_bounded(kv_empty(i & 1), ((i >> 1) - 1) & 1, abort_flag, p.err)) break;
        load_kv(i);
      }
      // let every load issued land before the CTA can exit
      volatile int no_abort = 0;
      mbar_wait_bounded(q_full, 0, &no_abort, nullptr);
      for (int j = (i > 2 ? i - 2 : 0); j < i; ++j)
        mbar_wait_bounded(kv_full(j & 1), (j >> 1) & 1, &no_abort, nullptr);
    }
  } else if (warp == 1) {
    if (nloc > 0 && elect_one()) {
      // ---------------- MMA issuer
      constexpr int bf = std::is_same<T, __nv_bfloat16>::value ? 1 : 0;
      constexpr uint32_t idesc_s = idesc_f16(bf, kAQ, kAK);
      constexpr uint32_t idesc_pv = idesc_f16(bf, kAQ, kAD) | (1u << 16);  // B (values) MN-major, N = 128
      const uint64_t qd = smem_desc_sw128(smem_u32(smem + kOffQ)), kd = smem_desc_sw128(smem_u32(smem + kOffK));
      const uint64_t pd = smem_desc_sw128(smem_u32(smem + kOffP));
      const uint64_t vd = smem_desc_sw128_mn(smem_u32(smem + kOffV));
      // scores of the CTA's tile kt into TMEM buffer kt % 2 (read by the
      // softmax of tile kt - 2, which has handed its P over by now)
      auto scores = [&](int kt) -> bool {
        const uint32_t b = (uint32_t)(kt & 1);
        if (!mbar_wait_bounded(kv_full(b), (kt >> 1) & 1, abort_flag, p.err)) return false;
        tc_fence_after();
        const uint64_t kb_d = kd + b * (uint32_t)(kTile >> 4);  // the descriptors' address field counts 16 bytes
#pragma unroll
        for (int kb = 0; kb < 2; ++kb)
#pragma unroll
          for (int k = 0; k < 4; ++k)
            tc_mma_f16(tmem + b * 128u, qd + (uint64_t)(kb * (kHalf >> 4) + 2 * k), kb_d + (uint64_t)(kb * (kHalf >> 4) + 2 * k),
                       idesc_s, (kb | k) != 0);
        tc_commit(s_full(b));
        return true;
      };
      bool ok = mbar_wait_bounded(q_full, 0, abort_flag, p.err) && scores(0);
      for (int kt = 0; ok && kt < nloc; ++kt) {
        if (kt + 1 < nloc && !scores(kt + 1)) break;
        if (!mbar_wait_bounded(p_full, kt & 1, abort_flag, p.err)) break;
        tc_fence_after();
        const uint64_t vt = vd + (uint32_t)(kt & 1) * (uint32_t)(kTile >> 4);
#pragma unroll
        for (int part = 0; part < P::kParts; ++part) {
#pragma unroll
          for (int ks = 0; ks < 8; ++ks)  // 16 keys per step, all 128 head dims (both 64-wide halves)
            tc_mma_f16(tO, pd + (uint64_t)((part * P::kPartBytes + (ks >> 2) * P::kHalfBytes) / 16 + 2 * (ks & 3)),
                       vt + (uint64_t)(ks * (2048 >> 4)), idesc_pv, (part | ks) != 0);
        }
        tc_commit(o_full);
        tc_commit(kv_empty(kt & 1));
      }
      // every MMA issued must have finished before TMEM is freed (on the
      // normal path the softmax warps have already waited for the last one)
      tc_commit(done_bar);
      volatile int no_abort = 0;
      mbar_wait_bounded(done_bar, 0, &no_abort, nullptr);
    }
  } else if (!SHORT || (warp & 3) < kShortRows / 32) {
    // ---------------- softmax and output: warps 2..9, half a query row per thread
    const int q4 = warp & 3, half = (warp - 2) >> 2;
    const int row = q4 * 32 + lane;
    const int tq = t0 + row;
    // last visible key: padding rows reuse the last query's horizon; never
    // past the cache (a position beyond it is reported by the RoPE kernel)
    const int qpos = min(pos0 + min(tq, p.tokens - 1), p.max_seq - 1);
    // horizon of the warp's first row: keys up to it are visible to all 32
    const int qpos_min = min(pos0 + min(t0 + q4 * 32, p.tokens - 1), p.max_seq - 1);
    const uint32_t lane_off = (uint32_t)(q4 * 32) << 16;
    const uint32_t prow = (uint32_t)half * P::kHalfBytes + (uint32_t)((row >> 3) * 1024 + (row & 7) * 128);
    const uint32_t psw = (uint32_t)(row & 7);
    float* xch = reinterpret_cast<float*>(smem + kOffX);
    // the two warps of a row quarter meet here; both take part in every
    // tile's exchange, also after a timeout
    auto pair_sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(1 + q4) : "memory"); };
    float m = -INFINITY, l = 0.f, alpha = 0.f;
    float o[64];
#pragma unroll
    for (int d = 0; d < 64; ++d) o[d] = 0.f;
    bool ok = true;
    // O = O * alpha + O_t of tile kt (alpha: that tile's rescaling)
    auto add_tile = [&](int kt) {
      ok = ok && mbar_wait_bounded(o_full, kt & 1, abort_flag, p.err);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) return;
      tc_fence_after();
#pragma unroll
      for (int c0 = 0; c0 < 64; c0 += 16) {
        uint32_t r[16];
        tmem_ld_32x32b_x16(tO + lane_off + (uint32_t)(half * 64 + c0), r);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 16; ++i) o[c0 + i] = fmaf(o[c0 + i], alpha, __uint_as_float(r[i]));
      }
    };
    for (int kt = 0; kt < nloc; ++kt) {
      const int b = kt & 1, k0 = (z + kt * parts) * kAK + half * 64;  // this thread's first key
      ok = ok && mbar_wait_bounded(s_full(b), (kt >> 1) & 1, abort_flag, p.err);
      ok = __all_sync(0xffffffffu, ok);
      tc_fence_after();
      uint32_t s[64];
      float mx = -INFINITY;
      if (ok) {
#pragma unroll
        for (int c0 = 0; c0 < 64; c0 += 32) {
          uint32_t (&r)[32] = *reinterpret_cast<uint32_t (*)[32]>(s + c0);
          tmem_ld_32x32b_x32(tmem + (uint32_t)b * 128u + lane_off + (uint32_t)(half * 64 + c0), r);
        }
        tmem_ld_wait();
        if (k0 + 63 > qpos_min) {  // the diagonal or the run's end crosses these keys
#pragma unroll
          for (int i = 0; i < 64; ++i)
            if (k0 + i > qpos) s[i] = 0xff800000u;  // -inf
        }
#pragma unroll
        for (int i = 0; i < 64; ++i) mx = fmaxf(mx, __uint_as_float(s[i]));
      }
      xch[half * kAQ + row] = mx;
      pair_sync();
      // (key 0 is visible to every query; a row may see none of another CTA's tiles)
      mx = fmaxf(m, fmaxf(mx, xch[(half ^ 1) * kAQ + row]));
      const float base = SPLIT && mx == -INFINITY ? 0.f : mx;
      pair_sync();  // read by both before either writes again
      if (kt > 0) add_tile(kt - 1);  // and P may be written again
      alpha = exp2f((m - base) * p.scale_log2);  // 0 on the first tile (m = -inf)
      m = mx;
      if (ok) {
        float lt = 0.f;
#pragma unroll
        for (int c = 0; c < 8; ++c) {  // 8 keys: one 16-byte chunk of each part
          uint32_t part[P::kParts][4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float p0 = exp2f((__uint_as_float(s[8 * c + 2 * i]) - base) * p.scale_log2);
            const float p1 = exp2f((__uint_as_float(s[8 * c + 2 * i + 1]) - base) * p.scale_log2);
            lt += p0;
            lt += p1;
            float2 rest = make_float2(p0 * kPScale, p1 * kPScale);
#pragma unroll
            for (int j = 0; j < P::kParts; ++j) {
              part[j][i] = pack2<T>(rest.x, rest.y);
              const float2 h = unpack2<T>(part[j][i]);
              rest = make_float2(rest.x - h.x, rest.y - h.y);
            }
          }
          const uint32_t off = prow + (((uint32_t)c ^ psw) << 4);
#pragma unroll
          for (int j = 0; j < P::kParts; ++j)
            asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(smem_u32(smem + kOffP + j * P::kPartBytes) + off), "r"(part[j][0]),
                         "r"(part[j][1]), "r"(part[j][2]), "r"(part[j][3])
                         : "memory");
        }
        l = l * alpha + lt;
        fence_proxy_async_smem();  // P is read by the tensor cores (async proxy)
        tc_fence_before();
        mbar_arrive(p_full);
      }
    }
    if (nloc > 0) {
      add_tile(nloc - 1);
      xch[half * kAQ + row] = l;
      pair_sync();
      const float other = xch[(half ^ 1) * kAQ + row];
      if (SPLIT && parts > 1) {
        pair_sync();  // both have read
        if (half == 0) {
          xch[row] = m;
          xch[kAQ + row] = l + other;
        }
        float4* mine = reinterpret_cast<float4*>(smem + kOffK) + row * (kORow / 4) + half * 16;
#pragma unroll
        for (int c = 0; c < 16; ++c) mine[c] = make_float4(o[4 * c], o[4 * c + 1], o[4 * c + 2], o[4 * c + 3]);
      } else if (ok && tq < p.tokens) {
        const float inv = 1.0f / (kPScale * (half ? other + l : l + other));
        uint4* dst = reinterpret_cast<uint4*>(static_cast<T*>(p.out) + (int64_t)tq * p.width + col0 + half * 64);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          uint4 v;
          v.x = pack2<T>(o[8 * c] * inv, o[8 * c + 1] * inv);
          v.y = pack2<T>(o[8 * c + 2] * inv, o[8 * c + 3] * inv);
          v.z = pack2<T>(o[8 * c + 4] * inv, o[8 * c + 5] * inv);
          v.w = pack2<T>(o[8 * c + 6] * inv, o[8 * c + 7] * inv);
          dst[c] = v;
        }
      }
    }
    tc_fence_before();
  }
  tc_fence_before();
  __syncthreads();
  if (SPLIT && parts > 1) {
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    cluster.sync();
    // a warp per row, four columns per lane: rows shared out over the CTAs
    // (several rows at a time take registers that the tile loop needs)
    const int rows = min(kAQ, p.tokens - t0);
    if (z < parts && warp >= 2) {
      float* x = reinterpret_cast<float*>(smem + kOffX);
      float4* ov = reinterpret_cast<float4*>(smem + kOffK);
      for (int row = (warp - 2) * parts + z; row < rows; row += parts * (kASoft / 32)) {
        float mr[kAMaxSplit], lr[kAMaxSplit], M = -INFINITY;
        float4 v[kAMaxSplit];
#pragma unroll
        for (int c = 0; c < kAMaxSplit; ++c) {
          if (c < parts) {
            const float* rx = cluster.map_shared_rank(x, c);
            mr[c] = rx[row];
            lr[c] = rx[kAQ + row];
            v[c] = cluster.map_shared_rank(ov, c)[row * (kORow / 4) + lane];
          }
        }
#pragma unroll
        for (int c = 0; c < kAMaxSplit; ++c)
          if (c < parts) M = fmaxf(M, mr[c]);
        float L = 0.f;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int c = 0; c < kAMaxSplit; ++c) {
          if (c < parts) {
            const float w = exp2f((mr[c] - M) * p.scale_log2);  // 0 where no key of the CTA is visible
            L = fmaf(lr[c], w, L);
            a.x = fmaf(v[c].x, w, a.x);
            a.y = fmaf(v[c].y, w, a.y);
            a.z = fmaf(v[c].z, w, a.z);
            a.w = fmaf(v[c].w, w, a.w);
          }
        }
        const float inv = 1.0f / (kPScale * L);
        *reinterpret_cast<uint2*>(static_cast<T*>(p.out) + (int64_t)(t0 + row) * p.width + col0 + lane * 4) =
            make_uint2(pack2<T>(a.x * inv, a.y * inv), pack2<T>(a.z * inv, a.w * inv));
      }
    }
    cluster.sync();  // every row has been read before any CTA exits
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

int done(cudaError_t e, const char* what) {
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) SN_FAIL(SWAPNET_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
  return SWAPNET_OK;
}

// Clusters of c CTAs of this kernel that the device runs at once (cached per size and device).
template <typename T> int active_clusters(int c) {
  static std::atomic<int> cached[64][kAMaxSplit + 1];  // the count + 1, 0 until known
  const int dev = device_index();
  if (dev >= 0) {
    const int v = cached[dev][c].load(std::memory_order_relaxed);
    if (v > 0) return v - 1;
  }
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(1, 1, c);
  cfg.blockDim = dim3(kAThreads);
  cfg.dynamicSmemBytes = kASmem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = c;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, attention_tc_kernel<T, true, false>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
  if (dev >= 0) cached[dev][c].store(n + 1, std::memory_order_relaxed);
  return n;
}

template <typename T>
int launch_t(const void* q, const void* kc, const void* vc, const int* pos_ptr, int tokens, int heads, int width,
             int max_seq, void* out, int* err, cudaStream_t s) {
  static std::atomic<uint64_t> attr_done{0};
  if (attr_needed(attr_done)) {
    for (auto kern : {attention_tc_kernel<T, false, false>, attention_tc_kernel<T, true, false>,
                      attention_tc_kernel<T, false, true>, attention_tc_kernel<T, true, true>})
      if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kASmem) != cudaSuccess)
        return done(cudaGetLastError(), "attention shared memory");
    attr_set(attr_done);
  }
  const int dt = std::is_same<T, __nv_bfloat16>::value ? SWAPNET_BF16 : SWAPNET_F16;
  CUtensorMap tq, tk, tv;
  int rc = make_tmap_2d(&tq, dt, q, (uint64_t)width, (uint64_t)tokens, (uint64_t)width * 2, 64, kAQ);
  if (!rc) rc = make_tmap_2d(&tk, dt, kc, (uint64_t)width, (uint64_t)max_seq, (uint64_t)width * 2, 64, kAK);
  if (!rc) rc = make_tmap_2d(&tv, dt, vc, (uint64_t)width, (uint64_t)max_seq, (uint64_t)width * 2, 64, kAK);
  if (rc) return rc;
  AttnArgs a;
  std::memset(&a, 0, sizeof(a));
  a.out = out;
  a.pos_ptr = pos_ptr;
  a.tokens = tokens;
  a.heads = heads;
  a.width = width;
  a.max_seq = max_seq;
  a.scale_log2 = 1.4426950408889634f / sqrtf((float)kAD);
  a.err = err;
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  // the widest split of a cache's key tiles whose clusters all run at once;
  // not two: 64 clusters of two cost 2 us more on a short prefix (32 heads,
  // 256 tokens on 200 keys of a 1500-key cache 13.8 us unsplit, 15.9) and
  // save 3.8 on 900 keys
  const int tiles = (max_seq + kAK - 1) / kAK, ctas = (tokens + kAQ - 1) / kAQ * heads;
  a.split = std::min(tiles, kAMaxSplit);
  while (a.split > 1 && ctas > active_clusters<T>(a.split)) --a.split;
  if (a.split < 3 || !split_pays(tiles, a.split)) a.split = 1;
  cfg.gridDim = dim3((tokens + kAQ - 1) / kAQ, heads, a.split);
  cfg.blockDim = dim3(kAThreads);
  cfg.dynamicSmemBytes = kASmem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 1;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = a.split;
  cfg.attrs = attr;
  cfg.numAttrs = a.split > 1 ? 2 : 1;
  const auto kern = tokens < kShortRows
                        ? (a.split > 1 ? attention_tc_kernel<T, true, true> : attention_tc_kernel<T, false, true>)
                        : (a.split > 1 ? attention_tc_kernel<T, true, false> : attention_tc_kernel<T, false, false>);
  return done(cudaLaunchKernelEx(&cfg, kern, tq, tk, tv, a), "tensor-core attention launch");
}

}  // namespace

// Where this kernel takes over from the split-key one (a cluster of CTAs per
// query and head), whose time grows with queries x heads x keys while this
// one's is about 6.6 us and 2 us per 128 keys of the cache's filled part
// (which only the device knows) on one CTA.  Measured, split-key against this,
// RoPE included: 128 (query, head) pairs in a cache of 160 7.1-7.6 against
// 6.5-8.9 us, of 340 10.6-11.5 against 6.5-11.4, of 1030 13.3-22.9 against
// 6.8-11.8; caches of at most 128 keys 4.9-8.0 against 6.9 us at 256 pairs,
// 10.9-11.4 against 6.8 at 384.  (64 pairs on more than 1000 keys, 12.6
// against 8.5-11, would pay 2 us in a cache that is still nearly empty.)
bool attention_tc_supported(int dtype, int tokens, int heads, int width, int max_seq) {
  return (dtype == SWAPNET_F16 || dtype == SWAPNET_BF16) && heads > 0 && width == heads * kAD &&
         (int64_t)tokens * heads >= (max_seq > kAK ? 128 : 384);
}

int launch_attention_tc(int dtype, const void* q, const void* kc, const void* vc, const int* pos_ptr, int tokens,
                        int heads, int width, int max_seq, void* out, int* err, cudaStream_t s) {
  if ((dtype != SWAPNET_F16 && dtype != SWAPNET_BF16) || heads < 1 || width != heads * kAD)
    SN_FAIL(SWAPNET_ERR_UNSUPPORTED, "tensor-core attention: fp16/bf16, head width 128");
  if (((uintptr_t)q | (uintptr_t)kc | (uintptr_t)vc | (uintptr_t)out) & 15)
    SN_FAIL(SWAPNET_ERR_MISALIGNED, "tensor-core attention: operands must be 16-byte aligned");
  if (dtype == SWAPNET_BF16)
    return launch_t<__nv_bfloat16>(q, kc, vc, pos_ptr, tokens, heads, width, max_seq, out, err, s);
  return launch_t<__half>(q, kc, vc, pos_ptr, tokens, heads, width, max_seq, out, err, s);
}

}  // namespace swapnet
