// tcgen05 tensor-core GEMM and implicit-GEMM convolution for sm_103a.
//
//   C[m, n] = sum_k A[m, k] * B[n, k],  fp16/bf16 operands, fp32 accumulate
//   in TMEM, fused epilogue (bias, residual, activation) on the way out.
//
// B is a weight matrix [N][K] (K contiguous) that lives in the arena slot of
// the block being executed; it is staged by TMA (128-byte swizzle).  A is
// either a row-major activation matrix (linear layers, 1x1 stride-1 convs),
// also staged by TMA, or the implicit im2col of an NHWC input for general
// convolutions, gathered by four warps with cp.async (zero fill for padding)
// into the same swizzled layout.  One CTA computes one 128 x BN tile (BN 64
// or 128; 256 for linear layers of at most kFewRows rows):
//   warp 0      TMA producer (one elected lane)
//   warp 1      TMEM allocation and MMA issue (one elected lane)
//   warps 2..5  im2col gather (conv)
//   warps 2..9  epilogue: TMEM -> registers -> shared memory -> global, warp w
//               reading TMEM lanes 32*(w % 4) .. +31 of one half of the columns.
// Every wait is bounded; on timeout the kernel records kDevErrTimeout in
// the error word, drains what it started, frees TMEM and returns.
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "device.cuh"
#include "internal.h"
#include "kernels.h"
#include "tc_epi.cuh"

namespace swapnet {

__device__ int g_tc_err;

namespace {

constexpr int kBM = 128;
constexpr int kBK = 64;  // 64 x 2 bytes = one 128-byte swizzle row
constexpr int kEpiThreads = 256;
constexpr int kThreads = 64 + kEpiThreads;
constexpr int kABytes = kBM * kBK * 2;

// A operand: kA2d (2-D TMA of a row-major matrix: linear layers, 1x1
// stride-1 convs), kAGather (cp.async im2col gather by warps 2..5), kATap
// (convs whose taps are whole 64-channel k-blocks: one 4-D TMA per k-block
// of the tap's 64 channels over a wt x ht patch of output pixels, zero fill
// for the padding; the CTA's 128 rows are that patch, rows >= wt * ht unused),
// kAFew (2-D TMA of at most kFewRows rows, whose work is streaming the weight
// matrix: only those rows are loaded and the other MMA rows read whatever
// lies behind them, results nobody uses, so a stage is 2 KB of A and the
// weight tile and the stages hold 128-170 KB of weights in flight; an N tile
// of 256 exists for it alone; the splits' partials are shared out by column).
// Measured inside chains of such layers, weights from HBM, 16 rows, with
// 16 KB of A per stage and 4-6 stages before: 1024 -> 1024 4.2 to 3.4 us, 1024 <-> 2752 5.8
// to 3.9, 2048 <-> 8192 12.9 to 8.4, 4096 -> 4096 9.4 to 8.7, 8192 -> 8192
// 26.2 to 24.3 (5.5 TB/s); 25088 -> 4096 alone 37.9 to 33.2.
// Siblings share a launch of it: twelve layers 2048 -> 11008 of 8 rows 131.0
// us one by one, 102.6 three to a launch.
constexpr int kA2d = 0, kAGather = 1, kATap = 2, kAFew = 3;
constexpr int kFewRows = 16;

template <int BN, int AMODE> struct Cfg {
  static constexpr bool kFew = AMODE == kAFew;
  static constexpr int kStages = kFew ? (BN == 64 ? 16 : (BN == 128 ? 10 : 5)) : (BN == 64 ? 6 : 4);
  static constexpr int kLag = kStages - 2;  // gather: cp.async groups in flight per thread
  static constexpr int kAStage = kFew ? kFewRows * kBK * 2 : kABytes;
  static constexpr int kARegion = kStages * kAStage + kABytes - kAStage;  // the last stage's MMA reads 128 rows too
  static constexpr int kBBytes = BN * kBK * 2;
  static constexpr int kStageBytes = kARegion + kStages * kBBytes;
  // cluster split-K receive buffer.  Row owners: up to kTcMaxSplit splits x
  // ceil(128/splits) rows.  Few rows (column owners): splits x kFewRows rows x
  // (columns per owner, a multiple of 8, + 4): 2 to 8 splits of up to BN + 76 floats.
  static constexpr int kRecvBytes = kFew ? kFewRows * (BN + 76) * 4 : (kBM + kTcMaxSplit - 1) * (BN + 4) * 4;
  static constexpr int kBiasBytes = BN * 4;
  static constexpr int kSmem = kStageBytes + kRecvBytes + kBiasBytes + 512 + 1024;
  static_assert(kSmem <= 232448, "dynamic shared memory above the 227 KB per-CTA limit");
};

// NS: layers that a launch may hold (1, or kTcMaxSeg siblings)
template <typename T, int BN, int AMODE, int NS>
__global__ void __launch_bounds__(kThreads, 1)
    tc_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ TcSegs<NS> sg, const TcArgs p) {
  constexpr bool GATHER = AMODE == kAGather;
  constexpr bool TAP = AMODE == kATap;
  constexpr bool FEW = AMODE == kAFew;
  using C = Cfg<BN, AMODE>;
  constexpr int kStages = C::kStages;
  constexpr int kLag = C::kLag;
  constexpr int kAStage = C::kAStage;
  constexpr int kBBytes = C::kBBytes;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + C::kARegion;
  float* recv = reinterpret_cast<float*>(smem + C::kStageBytes);
  float* sbias = reinterpret_cast<float*>(smem + C::kStageBytes + C::kRecvBytes);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::kStageBytes + C::kRecvBytes + C::kBiasBytes);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + kStages);
  const uint32_t accum_bar = smem_u32(bars + 2 * kStages);
  auto full_bar = [&](int s) { return full0 + 8u * s; };
  auto empty_bar = [&](int s) { return empty0 + 8u * s; };

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int m0 = TAP ? 0 : blockIdx.x * kBM;
  int seg = 0, n0 = (int)blockIdx.y * BN;
  if constexpr (NS > 1) {
    const int nt = (p.N + BN - 1) / BN;
    seg = (int)blockIdx.y / nt;
    n0 -= seg * nt * BN;
  }
  const CUtensorMap* tmB = &sg.m[seg];
  // tap mode: this CTA's patch (image, patch row th, patch column tw)
  int pimg = 0, pth = 0, ptw = 0;
  if (TAP) {
    const int patches = p.tiles_w * p.tiles_h;
    pimg = blockIdx.x / patches;
    const int rem = blockIdx.x - pimg * patches;
    pth = rem / p.tiles_w;
    ptw = rem - pth * p.tiles_w;
  }
  const uint32_t a_bytes = TAP ? (uint32_t)(p.wt * p.ht * 128) : (GATHER ? 0u : (uint32_t)kAStage);
  // output row of tile row r (-1: no output)
  auto row_m = [&](int r) -> int {
    if (TAP) {
      if (r >= p.wt * p.ht) return -1;
      const int oy = pth * p.ht + r / p.wt, ox = ptw * p.wt + r % p.wt;
      return (oy < p.Ho && ox < p.Wo) ? (pimg * p.Ho + oy) * p.Wo + ox : -1;
    }
    return m0 + r < p.M ? m0 + r : -1;
  };
  const int KB = (p.K + kBK - 1) / kBK;
  const int kb0 = blockIdx.z * p.kb_per_split;
  const int nk = min(KB, kb0 + p.kb_per_split) - kb0;  // >= 1 by construction
  const int splits = gridDim.z;
  const bool csplit = splits > 1;  // the splits of a tile are a cluster

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full_bar(s), GATHER ? 1 + 128 : 1);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(accum_bar, 1);
    *abort_flag = 0;
    fence_barrier_init();
    fence_proxy_async_smem();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), BN);
    tmem_relinquish();
  }
  if (threadIdx.x == 0) {
    prefetch_tmap(tmB);
    if (!GATHER) prefetch_tmap(&tmA);
  }
  // bias of this tile to shared memory (weights: ready before the kernel)
  if (threadIdx.x >= 64) {
    const T* bias = seg_bias<T>(p, sg, seg);
    for (int j = threadIdx.x - 64; j < BN; j += kEpiThreads) sbias[j] = (bias && n0 + j < p.N) ? to_f<T>(bias[n0 + j]) : 0.f;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_launch_dependents();
  if (csplit) asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");  // peers started (waited before DSMEM use)

  const bool vec = epi_vec_ok(p, seg_y<T>(p, sg, seg));
  const int rmode = res_mode(p.e);
  // cluster split-K: what epilogue thread t sums after the exchange, and its
  // residual, requested while the MMAs run.  row owners: 8 columns of up to
  // kRedN rows of this CTA's share of the rows; few rows: 8 columns of one row
  // of this CTA's share of the columns
  constexpr int kColGroups = BN / 8, kRedRows = kEpiThreads / kColGroups, kRedN = FEW ? 1 : 64 / kRedRows;
  const int t = (int)threadIdx.x - 64;
  int red_m[kRedN];
  uint4 red_res[kRedN];

  if (warp == 0) {
    if (elect_one()) {
      // ---------------- TMA producer: weight tiles of the first stages go
      // out before waiting for the previous kernel (they do not depend on it)
      // The loop runs on one thread, whose every dependent instruction takes
      // 4-5 cycles: with the stage and filter tap found by divisions an
      // iteration took 300 cycles and set the pace of the whole kernel (a
      // k-block's MMAs take 192), so everything advances by increments.
      const int early = min(nk, kStages);
      const uint32_t a0 = smem_u32(sA), b0 = smem_u32(sB);
      const uint32_t tx = kBBytes + a_bytes;
      for (int i = 0; i < early; ++i) {
        mbar_arrive_expect_tx(full_bar(i), tx);
        tma_load_2d(b0 + i * kBBytes, tmB, full_bar(i), (kb0 + i) * kBK, n0);
      }
      // the next A k-block: channel c0 of filter tap (rx, ry), whose patch
      // starts at pixel (px + rx, py + ry)
      int c0 = 0, rx = 0, ry = 0, px = 0, py = 0;
      if (TAP) {
        const int k0 = kb0 * kBK, tap = k0 / p.C;
        c0 = k0 - tap * p.C;
        ry = tap / p.kw;
        rx = tap - ry * p.kw;
        px = ptw * p.wt * p.stride - p.pad;
        py = pth * p.ht * p.stride - p.pad;
      }
      auto load_a = [&](int s, int i) {
        if (TAP) {
          tma_load_4d(a0 + s * kAStage, &tmA, full_bar(s), c0, px + rx, py + ry, pimg);
          c0 += kBK;
          if (c0 == p.C) {
            c0 = 0;
            if (++rx == p.kw) { rx = 0; ++ry; }
          }
        } else {
          tma_load_2d(a0 + s * kAStage, &tmA, full_bar(s), (kb0 + i) * kBK, m0);
        }
      };
      pdl_wait();
      if (!GATHER)
        for (int i = 0; i < early; ++i) load_a(i, i);
      int i = early, s = 0;
      uint32_t par = 0;
      for (; i < nk; ++i) {
        if (!mbar_wait_bounded(empty_bar(s), par, abort_flag, p.err)) break;
        mbar_arrive_expect_tx(full_bar(s), tx);
        tma_load_2d(b0 + s * kBBytes, tmB, full_bar(s), (kb0 + i) * kBK, n0);
        if (!GATHER) load_a(s, i);
        if (++s == kStages) {
          s = 0;
          par ^= 1;
        }
      }
      if (i < nk) {
        // aborted: let the loads already issued land before the CTA exits
        volatile int no_abort = 0;
        for (int j = (i > kStages ? i - kStages : 0); j < i; ++j)
          mbar_wait_bounded(full_bar(j % kStages), (j / kStages) & 1, &no_abort, nullptr);
      }
    } else {
      pdl_wait();
    }
  } else if (warp == 1) {
    pdl_wait();
    if (elect_one()) {
      // ---------------- MMA issuer
      constexpr uint32_t idesc = idesc_f16(std::is_same<T, __nv_bfloat16>::value ? 1 : 0, kBM, BN);
      const uint64_t ad0 = smem_desc_sw128(smem_u32(sA)), bd0 = smem_desc_sw128(smem_u32(sB));
      uint32_t s = 0, par = 0;
      for (int i = 0; i < nk; ++i) {
        if (!mbar_wait_bounded(full_bar(s), par, abort_flag, p.err)) break;
        tc_fence_after();
        // the descriptors' address field counts 16 bytes
        const uint64_t ad = ad0 + s * (uint32_t)(kAStage >> 4), bd = bd0 + s * (uint32_t)(kBBytes >> 4);
#pragma unroll
        for (int k = 0; k < kBK / 16; ++k) tc_mma_f16(tmem, ad + 2ull * k, bd + 2ull * k, idesc, (i | k) != 0);
        tc_commit(empty_bar(s));
        if (++s == kStages) {
          s = 0;
          par ^= 1;
        }
      }
      tc_commit(accum_bar);  // fires once every MMA issued above has completed
    }
  } else {
    pdl_wait();
    if (GATHER && t < 128) {
      // ---------------- implicit im2col gather of A (row t of the tile)
      const int m = m0 + t;
      const bool mvalid = m < p.M;
      int img = 0, oy = 0, ox = 0;
      if (mvalid) {
        const int hw = p.Ho * p.Wo;
        img = m / hw;
        const int rem = m - img * hw;
        oy = rem / p.Wo;
        ox = rem - oy * p.Wo;
      }
      const int iy0 = oy * p.stride - p.pad, ix0 = ox * p.stride - p.pad;
      const T* xb = static_cast<const T*>(p.x) + (int64_t)img * p.H * p.Wd * p.C;
      const uint32_t row_off = (uint32_t)((t >> 3) * 1024 + (t & 7) * 128);
      const uint32_t sw = (uint32_t)(t & 7);
      // position of the first K element of this split: tap (ry, rx), channel c
      int k = kb0 * kBK;
      int tap = k / p.C;
      int c = k - tap * p.C;
      int ry = tap / p.kw, rx = tap - (tap / p.kw) * p.kw;
      const bool whole_tap = (p.C % kBK) == 0;  // a 64-wide K block never straddles taps
      int i = 0;
      for (; i < nk; ++i) {
        const int s = i % kStages, r = i / kStages;
        if (!mbar_wait_bounded(empty_bar(s), (r & 1) ^ 1, abort_flag, p.err)) break;
        const uint32_t dst_row = smem_u32(sA + s * kAStage) + row_off;
        if (whole_tap) {
          const int iy = iy0 + ry, ix = ix0 + rx;
          const bool valid = mvalid && k < p.K && (unsigned)iy < (unsigned)p.H && (unsigned)ix < (unsigned)p.Wd;
          const T* src = valid ? xb + ((int64_t)iy * p.Wd + ix) * p.C + c : static_cast<const T*>(p.x);
#pragma unroll
          for (int j = 0; j < 8; ++j) cp_async_16(dst_row + (((uint32_t)j ^ sw) << 4), src + (valid ? 8 * j : 0), valid);
          k += kBK;
          c += kBK;
          if (c == p.C) {
            c = 0;
            if (++rx == p.kw) { rx = 0; ++ry; }
          }
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int iy = iy0 + ry, ix = ix0 + rx;
            const bool valid =
                mvalid && k < p.K && (unsigned)iy < (unsigned)p.H && (unsigned)ix < (unsigned)p.Wd;
            const T* src = valid ? xb + ((int64_t)iy * p.Wd + ix) * p.C + c : static_cast<const T*>(p.x);
            cp_async_16(dst_row + (((uint32_t)j ^ sw) << 4), src, valid);
            k += 8;
            c += 8;
            if (c == p.C) {
              c = 0;
              if (++rx == p.kw) { rx = 0; ++ry; }
            }
          }
        }
        cp_async_commit();
        if (i >= kLag) {
          cp_async_wait<kLag>();
          fence_proxy_async_smem();
          mbar_arrive(full_bar((i - kLag) % kStages));
        }
      }
      cp_async_wait<0>();
      fence_proxy_async_smem();
      for (int j = (i > kLag ? i - kLag : 0); j < i; ++j) mbar_arrive(full_bar(j % kStages));
    }
    // ---------------- epilogue
    const int q = warp & 3;
    const int row = q * 32 + lane;
    const int m = row_m(row);  // -1: this row has no output
    const bool any_row = __any_sync(0xffffffffu, m >= 0);
    const int c_lo = (warp - 2) / 4 * (BN / 2), c_hi = c_lo + BN / 2;  // this warp's columns
    const uint32_t lanes = tmem + ((uint32_t)(q * 32) << 16);
    uint4 rnext[4];
    if (splits == 1) {
      epi_res_load<T>(rnext, p, m, n0 + c_lo, vec);
    } else if (csplit && FEW) {
      const int cpo = (((BN + splits - 1) / splits) + 7) & ~7;
      const int w8 = (min(BN, ((int)blockIdx.z + 1) * cpo) - (int)blockIdx.z * cpo) / 8;
      const int rr = w8 > 0 ? t / w8 : kFewRows;
      red_m[0] = rr < kFewRows ? row_m(rr) : -1;
      if (red_m[0] >= 0) red_res[0] = res8<T>(p, red_m[0], n0 + (int)blockIdx.z * cpo + 8 * (t - rr * w8), vec);
    } else if (csplit) {
      const int rpo = (kBM + splits - 1) / splits;
#pragma unroll
      for (int j = 0; j < kRedN; ++j) {
        const int rr = j * kRedRows + t / kColGroups;
        red_m[j] = rr < rpo && (int)blockIdx.z * rpo + rr < kBM ? row_m((int)blockIdx.z * rpo + rr) : -1;
        red_res[j] = res8<T>(p, red_m[j], n0 + 8 * (t % kColGroups), vec);
      }
    }
    const bool ok = mbar_wait_bounded(accum_bar, 0, abort_flag, p.err);
    tc_fence_after();
    const bool all_ok = __all_sync(0xffffffffu, ok);  // tcgen05.ld is warp-collective
    if (splits == 1) {
      // the stage ring is idle now (every load was consumed by an MMA that
      // has completed): its first 16 KB stage the warps' pieces
      const uint32_t stage = smem_u32(sA) + (uint32_t)((warp - 2) * kEpiStage);
      if (all_ok && any_row) {
#pragma unroll 1
        for (int c0 = c_lo; c0 < c_hi && n0 + c0 < p.N; c0 += 32) {
          uint4 rcur[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) rcur[i] = rnext[i];
          if (c0 + 32 < c_hi) epi_res_load<T>(rnext, p, m, n0 + c0 + 32, vec);
          epi_piece<T>(lanes + (uint32_t)c0, sbias + c0, stage, p, seg_y<T>(p, sg, seg), m, n0 + c0, vec, rmode,
                       rcur);
        }
      }
    } else {
      asm volatile("barrier.cluster.wait;" ::: "memory");  // every peer is running
      // push this split's partial rows to their owners, slot = this split's index
      const bool mine = FEW ? m >= 0 && row < kFewRows : m >= 0;
      if (all_ok && __any_sync(0xffffffffu, mine)) {
        // owner of row w = w / rows_per_owner; few rows: columns [o * cpo, (o + 1) * cpo) belong to CTA o
        const int rpo = (kBM + splits - 1) / splits;
        const int cpo = (((BN + splits - 1) / splits) + 7) & ~7;
        const uint32_t owner = (uint32_t)(row / rpo);
        uint32_t base = 0;
        if (!FEW) {
          const uint32_t la = smem_u32(recv) + (uint32_t)((((int)blockIdx.z * rpo + row - (int)owner * rpo) * (BN + 4)) * 4);
          asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(base) : "r"(la), "r"(owner));
        }
#pragma unroll 1
        for (int c0 = c_lo; c0 < c_hi; c0 += 16) {
          uint32_t r[16];
          tmem_ld_32x32b_x16(lanes + (uint32_t)c0, r);
          tmem_ld_wait();
          if (mine) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int c = c0 + 4 * j;
              uint32_t ra = base + (uint32_t)c * 4;
              if (FEW) {
                const uint32_t o = (uint32_t)(c / cpo);
                const uint32_t la =
                    smem_u32(recv) + (uint32_t)((((int)blockIdx.z * kFewRows + row) * (cpo + 4) + c - (int)o * cpo) * 4);
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(la), "r"(o));
              }
              asm volatile("st.shared::cluster.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(ra), "f"(__uint_as_float(r[4 * j])),
                           "f"(__uint_as_float(r[4 * j + 1])), "f"(__uint_as_float(r[4 * j + 2])),
                           "f"(__uint_as_float(r[4 * j + 3]))
                           : "memory");
            }
          }
          __syncwarp();
        }
      }
    }
  }
  if (csplit) {
    if (threadIdx.x < 64) asm volatile("barrier.cluster.wait;" ::: "memory");  // pairs the early arrive
    // all pushes are visible after this barrier; each CTA reduces its share
    // from its own receive buffer, in split order 0..S-1
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    if (t >= 0) {
      const int rpo = (kBM + splits - 1) / splits;
      const int cpo = (((BN + splits - 1) / splits) + 7) & ~7;
      const int c_own = FEW ? (int)blockIdx.z * cpo : 0;  // this CTA's first column
      const int w8 = FEW ? max(1, (min(BN, c_own + cpo) - c_own) / 8) : kColGroups;
      const int rs = FEW ? cpo + 4 : BN + 4;                      // floats per receive row
      const int zs = (FEW ? kFewRows : rpo) * rs;                 // floats per split
      const int c8 = t % w8 * 8;
#pragma unroll
      for (int j = 0; j < kRedN; ++j) {
        const int rr = j * kRedRows + t / w8, n = n0 + c_own + c8;
        if (red_m[j] < 0 || n >= p.N) continue;
        const float* src = recv + rr * rs + c8;
        float4 a0 = *reinterpret_cast<const float4*>(src), a1 = *reinterpret_cast<const float4*>(src + 4);
#pragma unroll 4
        for (int z = 1; z < splits; ++z) {
          const float4 f = *reinterpret_cast<const float4*>(src + z * zs);
          const float4 g = *reinterpret_cast<const float4*>(src + z * zs + 4);
          a0.x += f.x; a0.y += f.y; a0.z += f.z; a0.w += f.w;
          a1.x += g.x; a1.y += g.y; a1.z += g.z; a1.w += g.w;
        }
        const float v[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
        finish8<T>(v, sbias + c_own + c8, p, seg_y<T>(p, sg, seg), red_m[j], n, vec, rmode, red_res[j]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, BN);
  }
}

// ------------------------------------------------------------ host side
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
  });
  return fn;
}

// A tiled map of 16-bit elements with zero fill.  The CUDA driver's call needs a
// current context, which a thread whose first CUDA call leads here does not
// have yet (the runtime binds one at its own calls): bind that of the thread's
// device and ask again.
CUresult encode_tiled(CUtensorMap* m, int dtype, int rank, const void* base, const cuuint64_t* dims, const cuuint64_t* strides,
                      const cuuint32_t* box, const cuuint32_t* estr, CUtensorMapSwizzle swizzle) {
  auto fn = encode_fn();
  if (!fn) return CUDA_ERROR_NOT_FOUND;
  auto encode = [&] {
    return fn(m, dtype == SWAPNET_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, (cuuint32_t)rank,
              const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  };
  CUresult r = encode();
  int dev = 0;
  if (r == CUDA_ERROR_INVALID_CONTEXT && cudaGetDevice(&dev) == cudaSuccess && cudaSetDevice(dev) == cudaSuccess) r = encode();
  return r;
}

int make_tmap(CUtensorMap* m, int dtype, const void* base, uint64_t inner, uint64_t rows, uint64_t row_stride_bytes,
              uint32_t box_rows) {
  if (((uintptr_t)base & 15) || (row_stride_bytes & 15))
    SN_FAIL(SWAPNET_ERR_MISALIGNED, "TMA operand must be 16-byte aligned with a 16-byte multiple row stride");
  const cuuint64_t dims[2] = {inner, rows};
  const cuuint64_t strides[1] = {row_stride_bytes};
  const cuuint32_t box[2] = {(cuuint32_t)kBK, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = encode_tiled(m, dtype, 2, base, dims, strides, box, estr, CU_TENSOR_MAP_SWIZZLE_128B);
  if (r != CUDA_SUCCESS) SN_FAIL(SWAPNET_ERR_CUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
  return SWAPNET_OK;
}

// 4-D map of an NHWC activation tensor for per-tap im2col loads: box of 64
// channels x wt columns x ht rows of one image, every s-th column and row
// (the conv stride), zero fill outside the image (the conv padding).
int make_tmap_conv4d(CUtensorMap* m, int dtype, const void* base, int n, int h, int w, int c, int wt, int ht,
                     int stride) {
  if (((uintptr_t)base & 15) || (c * 2) % 16)
    SN_FAIL(SWAPNET_ERR_MISALIGNED, "TMA conv operand must be 16-byte aligned");
  const cuuint64_t dims[4] = {(cuuint64_t)c, (cuuint64_t)w, (cuuint64_t)h, (cuuint64_t)n};
  const cuuint64_t strides[3] = {(cuuint64_t)c * 2, (cuuint64_t)w * c * 2, (cuuint64_t)h * w * c * 2};
  const cuuint32_t box[4] = {(cuuint32_t)(c == kTap2C ? kTap2C : kBK), (cuuint32_t)(wt * stride), (cuuint32_t)(ht * stride), 1};
  const cuuint32_t estr[4] = {1, (cuuint32_t)stride, (cuuint32_t)stride, 1};
  const CUresult r = encode_tiled(m, dtype, 4, base, dims, strides, box, estr,
                                  c == kTap2C ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B);
  if (r != CUDA_SUCCESS)
    SN_FAIL(SWAPNET_ERR_CUDA, "cuTensorMapEncodeTiled (conv) failed (" + std::to_string((int)r) + ")");
  return SWAPNET_OK;
}

// Output patch (wt x ht pixels, wt * ht <= 128) for per-tap TMA loads that
// wastes the fewest of the 128 MMA rows; returns the used fraction.
double conv_patch(int ho, int wo, int stride, int* wt, int* ht) {
  double best = 0.0;
  *wt = *ht = 0;
  for (int cand : {wo, 128, 64, 32, 16, 8, 4}) {
    if (cand < 1 || cand > 128 || cand * stride > 256) continue;
    const int w_ = cand, h_ = std::min(128 / w_, ho);
    if (h_ < 1 || h_ * stride > 256) continue;
    const double tiles = (double)((wo + w_ - 1) / w_) * ((ho + h_ - 1) / h_);
    const double util = (double)ho * wo / (tiles * kBM);
    if (util > best + 1e-9) {
      best = util;
      *wt = w_;
      *ht = h_;
    }
  }
  return best;
}

template <typename T, int BN, int AMODE, int NS = 1>
int launch_inst(const TcGemm& g, const TcPlan& pl, int* err, cudaStream_t s) {
  static std::atomic<uint64_t> attr_done{0};  // per instantiation, one bit per device
  auto kern = tc_gemm_kernel<T, BN, AMODE, NS>;
  if (attr_needed(attr_done)) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (Cfg<BN, AMODE>::kSmem)) != cudaSuccess)
      SN_FAIL(SWAPNET_ERR_CUDA, "cudaFuncSetAttribute failed");
    attr_set(attr_done);
  }
  TcArgs a;
  std::memset(&a, 0, sizeof(a));
  a.M = g.M; a.N = g.N; a.K = g.K;
  a.x = g.A;
  a.H = g.H; a.Wd = g.Wd; a.C = g.C; a.Ho = g.Ho; a.Wo = g.Wo;
  a.kh = g.kh; a.kw = g.kw; a.stride = g.stride; a.pad = g.pad;
  a.e = g.e; a.y = g.y; a.ldy = g.ldy; a.err = err;
  a.kb_per_split = pl.kb_per_split;
  a.wt = pl.wt; a.ht = pl.ht; a.tiles_w = pl.tiles_w; a.tiles_h = pl.tiles_h;
  const int64_t mtiles = AMODE == kATap ? (int64_t)g.M / ((int64_t)g.Ho * g.Wo) * pl.tiles_w * pl.tiles_h
                                        : (g.M + kBM - 1) / kBM;
  const dim3 grid((unsigned)mtiles, (g.N + BN - 1) / BN * std::max(1, g.nseg), pl.splits);
  const bool csplit = pl.splits > 1;
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = (Cfg<BN, AMODE>::kSmem);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int na = 0;
  if (!g.no_pdl) {
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
  }
  if (csplit) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = 1;
    attr[na].val.clusterDim.y = 1;
    attr[na].val.clusterDim.z = pl.splits;
    ++na;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  const cudaError_t le = cudaLaunchKernelEx(&cfg, kern, pl.tmA, make_segs<NS>(g, pl), a);
  if (le != cudaSuccess) SN_FAIL(SWAPNET_ERR_CUDA, std::string("tcgen05 GEMM launch: ") + cudaGetErrorString(le));
  return SWAPNET_OK;
}

template <typename T, int NS> int launch_few(const TcGemm& g, const TcPlan& pl, int* err, cudaStream_t s) {
  if (pl.bn == 64) return launch_inst<T, 64, kAFew, NS>(g, pl, err, s);
  if (pl.bn == 128) return launch_inst<T, 128, kAFew, NS>(g, pl, err, s);
  return launch_inst<T, 256, kAFew, NS>(g, pl, err, s);
}

// Clusters of c CTAs (2 to kTcMaxSplit, along the split dimension) of this kernel
// instance that the device runs at once (cudaOccupancyMaxActiveClusters;
// cached per instance, size and device).
template <typename T, int BN, int AMODE>
int active_clusters_inst(int c) {
  static std::atomic<int> cached[64][kTcMaxSplit + 1];  // the count + 1, 0 until known
  if (c < 2 || c > kTcMaxSplit) return 0;
  const int dev = device_index();
  if (dev >= 0) {
    const int v = cached[dev][c].load(std::memory_order_relaxed);
    if (v > 0) return v - 1;
  }
  auto kern = tc_gemm_kernel<T, BN, AMODE, 1>;
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (Cfg<BN, AMODE>::kSmem));
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(1, 1, c);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = (Cfg<BN, AMODE>::kSmem);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = c;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
  if (dev >= 0) cached[dev][c].store(n + 1, std::memory_order_relaxed);
  return n;
}

template <typename T>
int active_clusters_t(int bn, bool gather, bool few, int c) {
  if (few)
    return bn == 256 ? active_clusters_inst<T, 256, kAFew>(c)
                     : (bn == 64 ? active_clusters_inst<T, 64, kAFew>(c) : active_clusters_inst<T, 128, kAFew>(c));
  if (bn == 64) return gather ? active_clusters_inst<T, 64, kAGather>(c) : active_clusters_inst<T, 64, kA2d>(c);
  return gather ? active_clusters_inst<T, 128, kAGather>(c) : active_clusters_inst<T, 128, kA2d>(c);
}

int active_clusters(int dtype, int bn, bool gather, bool few, int c) {
  return dtype == SWAPNET_BF16 ? active_clusters_t<__nv_bfloat16>(bn, gather, few, c)
                               : active_clusters_t<__half>(bn, gather, few, c);
}

// ---- which kernel, N tile and split of K: the least of the times below, in
// us per launch inside a chain of dependent launches.  The constants are fits
// to sweeps on the GB300 over every N tile, sub-tile count and split of linear
// layers of 40 to 100000 rows and of 1x1 to 7x7 convolutions at batch 1 to 32
// (3 to 25 choices each; mean error 8 %).  What counts is the ranking: of 137
// layers 130 got the fastest choice or one within 2 %.  The others lost 0.1-0.5 us,
// but for two odd widths, whose 2-byte stores are not in the fits: 3x3 64 -> 71
// at 48 x 48, batch 8, 8.4 us, 7.3 on pairs; 3x3 128 -> 255 at 52 x 52, batch 16,
// 27.1 on pairs, 25.8 on single SMs.
// (The fits before, of deep layers alone, took pairs of SMs with N tiles of 64
// for wide layers of short K, 20000 x 256 x 256 11.4 us against 7.8 on single SMs,
// and no split of a gathered operand, see tile_us.)

// Per-tile kernel: `base` from the previous kernel's end to the last store
// without a k-block, the k-blocks of one CTA (a split below five hides
// nothing of the fill), and the exchange of a split.  More tiles than SMs
// repeat everything but the launch.  A gathered operand costs several times a
// TMA one, more as more CTAs gather (3x3 96 -> 96 at 9 x 9, 14 k-blocks: 9.4 us
// unsplit, 4.9 seven ways).  Ragged rows (K odd in units of 16 values, so that
// a row starts in the middle of a 32-byte sector) load at about half the rate
// (512 x 2752 x 2040 13.9 us, x 2048 8.5).  thin: a convolution of so few
// features that all CTAs fetch the same few weight rows at once (3x3 256 -> 12 at
// 182 x 182: 32.8 us on single SMs, 16.7 on pairs, half of which fetch none).  Filter
// taps on N tiles of 128 slow down as more CTAs load them (3x3, 36 k-blocks: 8.4 us
// on 24 CTAs, 9.4 on 112).
double tile_us(int bn, int64_t tiles, int splits, int KB, bool tap, bool gather, bool ragged, bool thin, int sms) {
  const int kb = (KB + splits - 1) / splits;
  const int64_t ctas = tiles * splits, waves = (ctas + sms - 1) / sms;
  const double split = splits > 1 ? (bn == 64 ? 1.5 : 2.8) + 0.02 * splits : 0.0;
  // (long K: the weights come from HBM at the pace the stages allow)
  const double per_kb = gather ? (bn == 64 ? 0.5 : 0.6) + 0.002 * std::min<int64_t>(ctas, sms)
                        : ragged ? (bn == 64 ? 0.235 : 0.345)
                               : (bn == 64 ? (tap ? 0.14 : 0.125) + 0.0002 * kb
                                : tap    ? 0.155 + 0.0003 * std::min<int64_t>(ctas, sms)
                                         : 0.16 + 0.0008 * kb) +
                                     (thin ? 0.0011 * std::min<int64_t>(ctas, sms) : 0.0);
  return (bn == 64 ? 2.1 : 2.9) + split + waves * std::max(per_kb * kb, splits > 1 && !gather ? (bn == 64 ? (tap ? 0.7 : 0.63) : 0.82) : 0.0) +
         (waves - 1) * (bn == 64 ? 2.2 : 2.9);
}

// The per-tile kernel on at most kFewRows rows: streaming the weights is the
// work.  A k-block slows down as more CTAs share the L2 (from 64 of them on),
// and the whole matrix may have to come from HBM, at a rate that needs a CTA
// on most SMs.  More CTAs than SMs cost a
// whole CTA's fill again.
double few_us(int bn, int64_t tiles, int splits, int KB, int64_t N, int sms) {
  const int kb = (KB + splits - 1) / splits;
  const double alone = bn == 64 ? 0.118 : (bn == 128 ? 0.133 : 0.27);
  const double shared = bn == 64 ? 0.082 : (bn == 128 ? 0.057 : 0.04);
  const double base = bn == 64 ? 1.95 : (bn == 128 ? 2.5 : 3.6);
  const int64_t ctas = tiles * splits, waves = (ctas + sms - 1) / sms;
  const double busy = std::min(1.0, std::max(0.0, (ctas - 64) / 88.0));
  const double hbm = 6.9e6 * (0.6 + 0.4 * std::min(1.0, ctas / 128.0));  // bytes per us
  const double split = splits > 1 ? 1.0 + 0.08 * splits : 0.0;
  return base + split + std::max(waves * (alone + shared * busy) * kb, (double)N * KB * kBK * 2.0 / hbm) +
         (waves - 1) * 2.5;
}

// Persistent kernel, one CTA per tile of msub x 128 rows: the fill, then per
// tile the longer of its epilogue (which the next tile's MMAs overlap, not
// wholly while they are short) and its k-blocks, at the pace of the loads (A: a
// matrix by TMA, or one of ragged rows; 4-D TMA per filter tap; two taps per
// k-block; gathered).
enum class AFrom { kMatrix, kRagged, kTap, kTapPair, kGather };
double persist_us(int bn, int msub, int64_t tiles, int KB, AFrom a, bool thin, int sms) {
  const int64_t rounds = (tiles + sms - 1) / sms;
  if (a == AFrom::kGather)
    return (bn == 64 ? 2.3 : (bn == 128 ? 3.0 : 4.8)) +
           rounds * KB * ((bn == 256 ? 0.6 : 0.5) + 0.002 * std::min<int64_t>(tiles, sms));
  double fill, tile, tap;
  if (bn == 64 && msub == 1) {
    fill = 1.4 + std::min(0.1 * KB, 1.3);
    tile = std::max({1.05, 0.75 + 0.075 * KB, 0.125 * KB});
    tap = std::max(0.9 + 0.13 * KB, 0.173 * KB);
  } else if (bn == 64) {
    fill = 1.7 + std::min(0.06 * KB, 0.6);
    tile = std::max(1.7, 0.95 + 0.22 * KB);
    tap = std::max(0.95 + 0.25 * KB, 0.287 * KB);
  } else if (bn == 128) {
    fill = 1.7 + std::min(0.14 * KB, 1.2);
    tile = std::max({1.8, 1.0 + 0.135 * KB, 0.25 + 0.18 * KB});
    // (all SMs at once; without the last term 256 -> 512 at 26 x 26, batch 4, came
    // here at 10.2 us, 9.4 per tile, and 64 -> 71 at 217 x 217, batch 16, at 210 us,
    // 160 on pairs)
    tap = std::max(0.9 + 0.155 * KB, 0.178 * KB) + 0.03 * KB * std::min<int64_t>(tiles, sms) / sms;
  } else {
    fill = 2.15 + std::min(0.12 * KB, 1.7);
    tile = std::max({3.15, 2.5 + 0.16 * KB, 0.295 * KB});
    tap = 1.0 + 0.275 * KB;
  }
  if (a == AFrom::kTap) tile = std::max(tile, tap + (thin ? (msub > 1 ? 0.002 : 0.0009) * std::min<int64_t>(tiles, sms) * KB : 0.0));
  if (a == AFrom::kTapPair) tile = std::max(tile, (msub > 1 ? 0.42 : 0.257) * KB);
  if (a == AFrom::kRagged) tile = std::max(tile, (msub > 1 ? 0.5 : 0.17 + 0.0015 * bn) * KB);
  return fill + rounds * tile;
}

// Persistent kernel on pairs of SMs, tiles of 256 x bn: the same, a tile's
// hand-over between the two SMs costs more than on one.
double pair_us(int bn, int64_t tiles, int KB, bool tap, bool ragged, int sms) {
  const int64_t slots = sms / 2, rounds = (tiles + slots - 1) / slots;
  const double fill = 1.6 + 0.0042 * bn + std::min(KB, 16) * (0.03 + 0.0005 * bn);
  const double loads = std::max((ragged ? 0.17 : 0.06) + 0.00085 * bn, 0.14);
  return fill + rounds * std::max({1.1 + 0.01 * bn + (KB - 1) * (0.055 + 0.00005 * bn), 0.2 + KB * loads,
                                   tap ? 1.0 + 0.15 * KB : 0.0});
}

// N tile of the paired kernel with the least pair_us (ties: the widest) for
// mt 128-row blocks and nseg segments of N columns.
int pair_tile(int64_t mt, int64_t N, int nseg, int KB, bool tap, bool ragged, int sms, double* us) {
  int best_bn = 0;
  for (int bn = 256; bn >= 64; bn -= 32) {
    const double t = pair_us(bn, (mt + 1) / 2 * ((N + bn - 1) / bn) * nseg, KB, tap, ragged, sms);
    if (!best_bn || t < *us) {
      best_bn = bn;
      *us = t;
    }
  }
  return best_bn;
}

}  // namespace

int tc_prepare(const TcGemm& g, TcPlan* p) {
  std::memset(p, 0, sizeof(*p));
  if (g.dtype != SWAPNET_F16 && g.dtype != SWAPNET_BF16) SN_FAIL(SWAPNET_ERR_UNSUPPORTED, "tcgen05 path: fp16/bf16 only");
  if (g.K % 8) SN_FAIL(SWAPNET_ERR_UNSUPPORTED, "tcgen05 path: K must be a multiple of 8");
  if (g.conv && g.C % 8) SN_FAIL(SWAPNET_ERR_UNSUPPORTED, "tcgen05 conv: channels must be a multiple of 8");
  if ((uintptr_t)g.y % 2) SN_FAIL(SWAPNET_ERR_MISALIGNED, "unaligned output");
  const int sms = g.num_sms > 0 ? g.num_sms : 148;
  const int Nd = g.N_layer > 0 ? g.N_layer : g.N;  // decisions follow the whole layer
  const int64_t mt = (g.M + kBM - 1) / kBM;
  const int KB = (g.K + kBK - 1) / kBK;
  // Convolutions whose taps are whole 64-channel k-blocks load A by one 4-D
  // TMA per tap over a pixel patch instead of the cp.async gather: in the
  // persistent kernels when the patches fill the 128 rows to 75 %, per tile
  // also when they need no more CTAs than 128-row tiles would (such layers
  // are latency-bound: unused MMA rows cost nothing, the gather's address
  // work does).
  int wt = 0, ht = 0;
  int64_t patches = 0;
  bool tap = false, tap_persist = false;
  const bool pair_taps = g.conv && g.C == kTap2C && Nd <= 128;  // two taps per k-block
  if (g.conv && (g.C % kBK == 0 || pair_taps)) {
    const double util = conv_patch(g.Ho, g.Wo, g.stride, &wt, &ht);
    if (wt > 0)
      patches = (int64_t)g.M / ((int64_t)g.Ho * g.Wo) * ((g.Wo + wt - 1) / wt) * ((g.Ho + ht - 1) / ht);
    tap_persist = wt > 0 && util >= 0.75;
    tap = !pair_taps && (tap_persist || (wt > 0 && patches <= mt));
  }
  const bool gather = g.conv && !tap;
  const int nseg = std::max(1, g.nseg);
  if (nseg > kTcMaxSeg || (nseg > 1 && (g.conv || g.e.res))) SN_FAIL(SWAPNET_ERR_UNSUPPORTED, "segments: linear layers without residual");
  const int64_t mt_tile = tap ? patches : mt, mt_pers = tap_persist ? patches : mt;
  double best = 0.0;
  // ---- per tile, K split over clusters
  const int cap = std::max(1, std::min(std::min(kTcMaxSplit, g.cluster_max), KB));
  auto consider = [&](int bn, int splits, double us) {
    if (best > 0.0 && us >= best) return;
    best = us;
    p->bn = bn;
    p->splits = splits;
  };
  const bool few = !g.conv && g.M <= kFewRows, ragged = !g.conv && g.K % 16, thin = tap && Nd <= 24;
  for (int bn : {64, 128, 256}) {
    if ((bn == 128 && Nd <= 64) || (bn == 256 && (!few || KB < 16))) continue;
    const int64_t tiles = mt_tile * ((Nd + bn - 1) / bn) * nseg;
    // segments: an unsplit sum, as each layer's own launch makes it
    for (int c = 1; c <= (nseg > 1 ? 1 : cap); ++c) {
      const int per = (KB + c - 1) / c, used = (KB + per - 1) / per;  // splits that get a k-block
      if (used != c) continue;
      // every cluster at once: a second wave of them costs more than a split saves
      if (c > 1 && tiles > active_clusters(g.dtype, bn, gather, few, c)) continue;
      consider(bn, c, few ? few_us(bn, tiles, c, KB, (int64_t)Nd * nseg, sms) : tile_us(bn, tiles, c, KB, tap, gather, ragged, thin, sms));
    }
  }
  // ---- persistent, no split
  if (g.allow_persist && !few) {
    // N tiles of 64, 128 or 256 as the width needs, and 128 where 256 leaves SMs
    // idle.  N tiles of 64 with A by TMA: two 128-row sub-tiles per tile share
    // each weight stage where that still leaves a tile per SM.  (Four: their
    // epilogue is twice as long and the stages shallower; 3x3 64 -> 64 at batch
    // 8, 112x112 16.5 us with four, 12.1 so; batch 16, 224x224: 84.3, 69.7.)
    const AFrom a = !g.conv ? (ragged ? AFrom::kRagged : AFrom::kMatrix)
                            : (!tap_persist ? AFrom::kGather : (pair_taps ? AFrom::kTapPair : AFrom::kTap));
    auto persist = [&](int bn, int ms) {
      const double us = persist_us(bn, ms, (mt_pers + ms - 1) / ms * ((Nd + bn - 1) / bn), KB, a, thin, sms);
      if (us >= best) return;
      best = us;
      p->persist = 1;
      p->bn = bn;
      p->msub = ms;
    };
    if (nseg == 1) {
      if (Nd > 128) persist(256, 1);
      if (Nd > 64) persist(128, 1);
      else persist(64, 1);
      if (Nd <= 64 && a != AFrom::kGather && (mt_pers + 1) / 2 >= sms) persist(64, 2);
    }
    if (mt_pers > 1 && (!g.conv || (tap_persist && !pair_taps))) {
      double two = 0.0;
      const int bn2 = pair_tile(mt_pers, Nd, nseg, KB, tap_persist, ragged, sms, &two);
      if (two < best) {
        p->persist = p->pair = 1;
        p->bn = bn2;
        p->msub = 1;
      }
    }
  }
  if (p->persist) p->splits = 1;
  p->few = few && !p->persist;
  p->kb_per_split = (KB + p->splits - 1) / p->splits;
  p->tma_conv = p->persist ? tap_persist : tap;
  const int64_t mt_used = p->persist ? mt_pers : mt_tile;
  const int mtile = p->pair ? 2 : (p->persist ? p->msub : 1);
  p->tiles = (mt_used + mtile - 1) / mtile * ((g.N + p->bn - 1) / p->bn) * nseg;
  int rc = SWAPNET_OK;
  for (int i = 0; i < nseg && !rc; ++i)
    rc = make_tmap(&p->tmB[i], g.dtype, i ? g.Wx[i - 1] : g.W, (uint64_t)g.K, (uint64_t)g.N, (uint64_t)g.K * 2,
                   (uint32_t)(p->pair ? p->bn / 2 : p->bn));
  if (rc) return rc;
  if (!g.conv && g.A) {
    rc = make_tmap(&p->tmA, g.dtype, g.A, (uint64_t)g.K, (uint64_t)g.M, (uint64_t)g.lda * 2,
                   (uint32_t)(p->few ? kFewRows : kBM));
    if (rc) return rc;
  }
  if (p->tma_conv) {
    p->wt = wt;
    p->ht = ht;
    p->tiles_w = (g.Wo + wt - 1) / wt;
    p->tiles_h = (g.Ho + ht - 1) / ht;
    if (g.A) {
      const int n_img = (int)((int64_t)g.M / ((int64_t)g.Ho * g.Wo));
      rc = make_tmap_conv4d(&p->tmA, g.dtype, g.A, n_img, g.H, g.Wd, g.C, wt, ht, g.stride);
      if (rc) return rc;
    }
  }
  p->ready = 1;
  return SWAPNET_OK;
}

int launch_tc_gemm(const TcGemm& g, const TcPlan& pl, int* err, cudaStream_t s) {
  if (!pl.ready) SN_FAIL(SWAPNET_ERR_INVALID_ARG, "tcgen05 GEMM not prepared");
  if (pl.pair) return launch_tc_pair(g, pl, err, s);
  if (pl.persist) return launch_tc_persist(g, pl, err, s);
  const bool bf = g.dtype == SWAPNET_BF16;
  if (pl.few)
    return g.nseg > 1 ? (bf ? launch_few<__nv_bfloat16, kTcMaxSeg>(g, pl, err, s) : launch_few<__half, kTcMaxSeg>(g, pl, err, s))
                      : (bf ? launch_few<__nv_bfloat16, 1>(g, pl, err, s) : launch_few<__half, 1>(g, pl, err, s));
  if (g.nseg > 1) {
    if (pl.bn == 64)
      return bf ? launch_inst<__nv_bfloat16, 64, kA2d, kTcMaxSeg>(g, pl, err, s) : launch_inst<__half, 64, kA2d, kTcMaxSeg>(g, pl, err, s);
    return bf ? launch_inst<__nv_bfloat16, 128, kA2d, kTcMaxSeg>(g, pl, err, s) : launch_inst<__half, 128, kA2d, kTcMaxSeg>(g, pl, err, s);
  }
  if (g.conv && pl.tma_conv) {
    if (pl.bn == 64) return bf ? launch_inst<__nv_bfloat16, 64, kATap>(g, pl, err, s) : launch_inst<__half, 64, kATap>(g, pl, err, s);
    return bf ? launch_inst<__nv_bfloat16, 128, kATap>(g, pl, err, s) : launch_inst<__half, 128, kATap>(g, pl, err, s);
  }
  if (g.conv) {
    if (pl.bn == 64) return bf ? launch_inst<__nv_bfloat16, 64, kAGather>(g, pl, err, s) : launch_inst<__half, 64, kAGather>(g, pl, err, s);
    return bf ? launch_inst<__nv_bfloat16, 128, kAGather>(g, pl, err, s) : launch_inst<__half, 128, kAGather>(g, pl, err, s);
  }
  if (pl.bn == 64) return bf ? launch_inst<__nv_bfloat16, 64, kA2d>(g, pl, err, s) : launch_inst<__half, 64, kA2d>(g, pl, err, s);
  return bf ? launch_inst<__nv_bfloat16, 128, kA2d>(g, pl, err, s) : launch_inst<__half, 128, kA2d>(g, pl, err, s);
}

// ------------------------------------------------------------ allocation-free GEMM
namespace {
struct NoAllocDevice {
  int* err = nullptr;  // device address of g_tc_err
  int sms = 0;
};
std::mutex g_noalloc_mu;
NoAllocDevice g_noalloc_dev[64];

// The entry point's limit on a problem: the fp32 partial sums of a K split
// over as many SMs as its 128 x 64 (or, with a tile per SM, 128 x 128) output
// tiles leave idle, plus 64 KiB, fit SWAPNET_NOALLOC_SCRATCH_BYTES.  Returns
// the bytes (0: nothing to split).
uint64_t noalloc_bytes(int64_t M, int64_t N, int64_t K, int sms) {
  const int64_t mt = (M + kBM - 1) / kBM, KB = (K + kBK - 1) / kBK;
  const int64_t bn = N > 64 && mt * ((N + 127) / 128) >= sms ? 128 : 64;
  const int64_t tiles = mt * ((N + bn - 1) / bn);
  if (tiles >= sms) return 0;
  const int64_t want = std::max<int64_t>(1, std::min<int64_t>(32, std::min<int64_t>(sms / tiles, std::max<int64_t>(1, KB / 2))));
  const int64_t per = (KB + want - 1) / want, splits = (KB + per - 1) / per;
  return splits > 1 ? (uint64_t)(splits * M * N) * sizeof(float) + 64 * 1024 : 0;
}
}  // namespace

int make_tmap_2d(CUtensorMap* m, int dtype, const void* base, uint64_t inner, uint64_t rows, uint64_t row_stride_bytes,
                 uint32_t box_inner, uint32_t box_rows) {
  if (((uintptr_t)base & 15) || (row_stride_bytes & 15) || (box_inner * 2) % 16)
    SN_FAIL(SWAPNET_ERR_MISALIGNED, "TMA operand must be 16-byte aligned with a 16-byte multiple row stride");
  const cuuint64_t dims[2] = {inner, rows};
  const cuuint64_t strides[1] = {row_stride_bytes};
  const cuuint32_t box[2] = {box_inner, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = encode_tiled(m, dtype, 2, base, dims, strides, box, estr, CU_TENSOR_MAP_SWIZZLE_128B);
  if (r != CUDA_SUCCESS) SN_FAIL(SWAPNET_ERR_CUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
  return SWAPNET_OK;
}

int tc_error_word(int** ptr) {
  void* p = nullptr;
  if (cudaGetSymbolAddress(&p, g_tc_err) != cudaSuccess) SN_FAIL(SWAPNET_ERR_CUDA, "cudaGetSymbolAddress failed");
  *ptr = static_cast<int*>(p);
  return SWAPNET_OK;
}

}  // namespace swapnet

extern "C" int swapnet_gemm_noalloc(int32_t dtype, const void* A, const void* W, const void* bias, void* Y,
                                    int32_t M, int32_t N, int32_t K, int32_t act, swapnet_stream stream) {
  return swapnet::guard_abi([&]() -> int {
    using namespace swapnet;
    if (dtype != SWAPNET_F16 && dtype != SWAPNET_BF16) SN_FAIL(SWAPNET_ERR_UNSUPPORTED, "fp16 or bf16 only");
    if (!A || !W || !bias || !Y || M < 1 || N < 1 || K < 1) SN_FAIL(SWAPNET_ERR_INVALID_ARG, "null pointer or empty shape");
    if (act < SWAPNET_ACT_NONE || act > SWAPNET_ACT_LEAKY) SN_FAIL(SWAPNET_ERR_INVALID_ARG, "bad activation");
    if (K % 8) SN_FAIL(SWAPNET_ERR_UNSUPPORTED, "K must be a multiple of 8");
    if (((uintptr_t)A | (uintptr_t)W | (uintptr_t)bias | (uintptr_t)Y) & 15)
      SN_FAIL(SWAPNET_ERR_MISALIGNED, "pointers must be 16-byte aligned");
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
      cudaGetLastError();
      SN_FAIL(SWAPNET_ERR_CUDA, "no current CUDA device");
    }
    NoAllocDevice d;
    {
      std::lock_guard<std::mutex> lk(g_noalloc_mu);
      NoAllocDevice& c = g_noalloc_dev[dev];
      if (!c.err) {  // once per device, with that device current
        void* e = nullptr;
        cudaError_t r = cudaGetSymbolAddress(&e, g_tc_err);
        if (r != cudaSuccess || !e) {
          cudaGetLastError();
          SN_FAIL(SWAPNET_ERR_CUDA, std::string("cudaGetSymbolAddress(error word): ") + cudaGetErrorString(r));
        }
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
          cudaGetLastError();
          SN_FAIL(SWAPNET_ERR_CUDA, "device attribute query failed");
        }
        c.err = static_cast<int*>(e);
        c.sms = sms;
      }
      d = c;
    }
    const uint64_t need = noalloc_bytes(M, N, K, d.sms);
    if (need > SWAPNET_NOALLOC_SCRATCH_BYTES)
      SN_FAIL(SWAPNET_ERR_INVALID_ARG, "problem counts for " + std::to_string(need) + " bytes of split-K scratch; the limit is " +
                                           std::to_string(SWAPNET_NOALLOC_SCRATCH_BYTES));
    TcGemm g;
    std::memset(&g, 0, sizeof(g));
    g.dtype = dtype;
    g.M = M; g.N = N; g.K = K;
    g.W = W;
    g.A = A; g.lda = K; g.conv = 0;
    g.e.bias = bias; g.e.res = nullptr; g.e.ldr = N; g.e.act = act; g.e.res_post = 0;
    g.y = Y; g.ldy = N;
    g.num_sms = d.sms;
    g.cluster_max = kTcMaxSplit;
    g.allow_persist = 1;
    // W and bias are caller memory that the previous work on the stream (an
    // earlier call, say) may have written: no early start before it completes
    g.no_pdl = 1;
    TcPlan pl;
    int rc = tc_prepare(g, &pl);
    if (rc) return rc;
    return launch_tc_gemm(g, pl, d.err, reinterpret_cast<cudaStream_t>(stream));
  });
}
