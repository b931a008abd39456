// Persistent tcgen05 GEMM / implicit-GEMM convolution on pairs of SMs
// (cta_group::2), for problems with enough output to give every pair a tile:
//
//   C[m, n] = sum_k A[m, k] * B[n, k],  fp16/bf16 in, fp32 accumulate in TMEM
//
// The two CTAs of a cluster own one 256 x BN output tile at a time: CTA r
// loads rows 128 r .. + 127 of A (a row block, or a pixel patch of a
// convolution) and rows r BN/2 .. + BN/2 - 1 of the weight tile, and holds
// the accumulator of its own 128 rows in its TMEM; one thread of CTA 0
// issues the MMAs for both.
//
// Why pairs: with one CTA per 128 x BN tile the loads bound the kernel, not
// the tensor pipe.  All SMs together read L2 at about 85 bytes per clock and
// SM, so a 64-deep k-block of a 128 x 128 tile (32 KB) takes 380 cycles
// against 256 of MMA, of a 128 x 256 tile (48 KB) 780 against 512.  A pair
// needs half of B per CTA: 24 KB and 282 cycles for 256 x 128, 32 KB and 512
// (the MMA's own time) for 256 x 256.
//
// BN is any multiple of 32 up to 256, chosen by the host (pair_tile) so that
// the tiles fill whole waves of the pairs.  Measured against the one-CTA
// kernel, per launch: 512 x 11008 x 4096 bf16 about 49 -> 31.2 us (128 x 256
// tiles left a second wave 13 % full; 256 x 160 tiles fill 1.8 of 2), 512 x
// 4096 x 11008 38 -> 34.4 us, 512 x 4096 x 4096 about 15.5 -> 14.1 us (1214
// TFLOP/s), a 3x3 convolution 256 -> 256 at 56 x 56, batch 16, 39 -> 35.9 us
// (1650 TFLOP/s).  What bounds it now: the MMA rate where BN is 256, the L2
// reads below.  Warp roles in both CTAs:
//   warp 0      TMA producer (its own operands; they are counted on CTA 0's
//               full barriers)
//   warp 1      TMEM owner; in CTA 0 also the MMA issuer
//   warps 2..9  epilogue of the CTA's own 128 rows, as in the one-CTA kernel
// Barriers: full (CTA 0: both CTAs' bytes), empty and tfull (both CTAs, by
// multicast commits), tempty (CTA 0: the epilogue warps of both).  Every wait
// is bounded; on timeout the error is recorded, every role leaves its loop,
// copies and MMAs in flight are given time to finish, TMEM is freed, and the
// CTAs leave together.
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "device.cuh"
#include "internal.h"
#include "kernels.h"
#include "tc_epi.cuh"

namespace swapnet {

namespace {

constexpr int kQBM = 128;  // rows per CTA
constexpr int kQBK = 64;   // one 128-byte swizzle row of 16-bit elements
constexpr int kQA = kQBM * kQBK * 2;
constexpr int kQEpiWarps = 8;
constexpr int kQThreads = 64 + 32 * kQEpiWarps;
constexpr int kQStaging = kQEpiWarps * kEpiStage;
constexpr int kQBias = kQEpiWarps * 128 * 4;
constexpr int kQMaxStages = 8;
constexpr int kQSmem = 232448;
constexpr int kQRing = kQSmem - 1024 - 256 - kQStaging - kQBias;  // bytes of the stage ring
constexpr uint32_t kQTmemCols = 512;                              // two accumulators of up to 256 columns
static_assert(2 * (kQA + 256 / 2 * 128) <= kQRing, "two stages of the widest tile");

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// Tiled loads into this CTA's shared memory, counted on a barrier of either
// CTA of the pair (bar: shared::cluster address).
__device__ __forceinline__ void tma2_load_2d(uint32_t dst, const void* tmap, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(
          dst),
      "l"(tmap), "r"(bar), "r"(x), "r"(y)
      : "memory");
}
__device__ __forceinline__ void tma2_load_4d(uint32_t dst, const void* tmap, uint32_t bar, int x, int y, int z, int w) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(
          dst),
      "l"(tmap), "r"(bar), "r"(x), "r"(y), "r"(z), "r"(w)
      : "memory");
}
__device__ __forceinline__ void tc2_mma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive once on the barrier at this offset in the CTAs of `mask` when all prior MMAs of this thread complete.
__device__ __forceinline__ void tc2_commit(uint32_t bar, uint16_t mask) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"(mask)
      : "memory");
}

// AMODE: 0 (row-major A) or 1 (convolution, A by filter tap); NS: layers that a
// launch may hold (1, or kTcMaxSeg siblings)
template <typename T, int AMODE, int NS>
__global__ void __launch_bounds__(kQThreads, 1)
    tc_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ TcSegs<NS> sg, const TcArgs p,
                   const int bn, const int stages) {
  constexpr bool TAP = AMODE == 1;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int b_bytes = bn / 2 * 128, stage_bytes = kQA + b_bytes;  // B: this CTA's half of the weight tile
  uint8_t* staging = smem + kQRing;
  float* sbias = reinterpret_cast<float*>(staging + kQStaging);
  uint64_t* bars = reinterpret_cast<uint64_t*>(staging + kQStaging + kQBias);
  // bars: full[8], empty[8], tfull[2], tempty[2], drain
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kQMaxStages + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + kQMaxStages);
  const uint32_t tfull0 = smem_u32(bars + 2 * kQMaxStages), tempty0 = smem_u32(bars + 2 * kQMaxStages + 2);
  const uint32_t drain_bar = smem_u32(bars + 2 * kQMaxStages + 4);

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int rank = (int)cluster_rank();  // 0: leader
  const int pair = (int)blockIdx.x >> 1, pairs = (int)gridDim.x >> 1;
  const int patches = p.tiles_w * p.tiles_h;
  // 128-row blocks of the output matrix, or pixel patches
  const int mt = TAP ? (p.M / (p.Ho * p.Wo)) * patches : (p.M + kQBM - 1) / kQBM;
  const int nt = (p.N + bn - 1) / bn;  // n-tiles per segment
  const int mtp = (mt + 1) / 2;
  int nseg = 1;
  if constexpr (NS > 1) nseg = sg.nseg;
  const int tiles = mtp * nt * nseg;
  const int KB = (p.K + kQBK - 1) / kQBK;
  const int my_tiles = pair < tiles ? (tiles - 1 - pair) / pairs + 1 : 0;
  const int work = my_tiles * KB;
  const uint32_t a_bytes = TAP ? (uint32_t)(p.wt * p.ht * 128) : (uint32_t)kQA;
  auto tile_of = [&](int lt) { return pair + lt * pairs; };

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(full0 + 8u * s, 1);
      mbar_init(empty0 + 8u * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull0 + 8u * b, 1);
      mbar_init(tempty0 + 8u * b, 2 * kQEpiWarps);
    }
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    fence_barrier_init();
    fence_proxy_async_smem();
    for (int i = 0; i < nseg; ++i) prefetch_tmap(&sg.m[i]);
    prefetch_tmap(&tmA);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(kQTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  // both CTAs' barriers are initialised before either counts on the other's
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_launch_dependents();

  if (warp == 0) {
    if (elect_one()) {
      // ---------------- TMA producer.  The weight tiles of the first stages
      // go out before waiting for the previous kernel (they do not depend on it).
      const uint32_t lfull0 = map_rank(full0, 0);
      const uint32_t tx = 2 * (a_bytes + (uint32_t)b_bytes);  // both CTAs' bytes of a stage
      int n0 = 0, ay = 0, az = 0, aw = 0;
      const CUtensorMap* tmB = &sg.m[0];
      auto start_tile = [&](int lt) {
        const int tile = tile_of(lt);
        const int ntile = tile / mtp, seg = NS > 1 ? ntile / nt : 0;
        tmB = &sg.m[seg];
        n0 = (ntile - seg * nt) * bn + rank * (bn / 2);
        const int idx = (tile % mtp) * 2 + rank;  // past the last one: only out-of-range coordinates (zero fill)
        if (TAP) {
          const int img = idx / patches, rem = idx - img * patches;
          const int th = rem / p.tiles_w, tw = rem - th * p.tiles_w;
          ay = tw * p.wt * p.stride - p.pad;
          az = th * p.ht * p.stride - p.pad;
          aw = img;
        } else {
          ay = idx * kQBM;
        }
      };
      // position of k-block kb of the current tile
      int kb = 0, lt = 0, c0 = 0, rx = 0, ry = 0;
      auto advance = [&]() {
        if (++kb == KB) {
          kb = c0 = rx = ry = 0;
          if (++lt < my_tiles) start_tile(lt);
        } else if (TAP) {
          c0 += kQBK;
          if (c0 == p.C) {
            c0 = 0;
            if (++rx == p.kw) { rx = 0; ++ry; }
          }
        }
      };
      auto load_b = [&](int s) {
        if (rank == 0) mbar_arrive_expect_tx(full0 + 8u * s, tx);
        tma2_load_2d(smem_u32(smem) + (uint32_t)(s * stage_bytes + kQA), tmB, lfull0 + 8u * s, kb * kQBK, n0);
      };
      auto load_a = [&](int s) {
        const uint32_t dst = smem_u32(smem) + (uint32_t)(s * stage_bytes);
        if (TAP) tma2_load_4d(dst, &tmA, lfull0 + 8u * s, c0, ay + rx, az + ry, aw);
        else tma2_load_2d(dst, &tmA, lfull0 + 8u * s, kb * kQBK, ay);
      };
      const int early = min(work, stages);
      if (work > 0) start_tile(0);
      for (int g = 0; g < early; ++g, advance()) load_b(g);
      pdl_wait();
      kb = lt = c0 = rx = ry = 0;
      if (work > 0) start_tile(0);
      for (int g = 0; g < early; ++g, advance()) load_a(g);
      int g = early, s = early == stages ? 0 : early;
      uint32_t par = 0;  // parity of the next release of a stage
      for (; g < work; ++g, advance()) {
        if (!mbar_wait_bounded(empty0 + 8u * s, par, abort_flag, p.err)) break;
        load_b(s);
        load_a(s);
        if (++s == stages) { s = 0; par ^= 1; }
      }
      if (g == work) {
        // the last releases of the stages have arrived before this CTA can leave
        if (work < stages) s = 0;
        for (int i = 0; i < early; ++i) {
          if (!mbar_wait_bounded(empty0 + 8u * s, par, abort_flag, p.err)) break;
          if (++s == stages) { s = 0; par ^= 1; }
        }
      } else {
        // aborted: the copies in flight (a few microseconds) land before the
        // CTAs leave.  They are counted on CTA 0's barriers, whose phases
        // are unknown here, so this waits for a time far above theirs
        const uint64_t t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 5000000ull) {
        }
      }
    } else {
      pdl_wait();
    }
  } else if (warp == 1) {
    pdl_wait();
    if (rank == 0) {
      if (elect_one()) {
        // ---------------- MMA issuer (for both CTAs)
        const uint32_t idesc = idesc_f16(std::is_same<T, __nv_bfloat16>::value ? 1 : 0, 2 * kQBM, bn);
        const uint64_t ad0 = smem_desc_sw128(smem_u32(smem)), bd0 = smem_desc_sw128(smem_u32(smem) + kQA);
        const uint32_t dstep = (uint32_t)stage_bytes >> 4;  // the descriptors' address field counts 16 bytes
        uint32_t s = 0, par = 0;
        bool ok = true;
        for (int lt = 0; lt < my_tiles && ok; ++lt) {
          const int buf = lt & 1, use = lt >> 1;
          if (!mbar_wait_bounded(tempty0 + 8u * buf, (use & 1) ^ 1, abort_flag, p.err)) break;
          tc_fence_after();
          const uint32_t d = tmem + (uint32_t)(buf * 256);
          for (int kb = 0; kb < KB; ++kb) {
            if (!mbar_wait_bounded(full0 + 8u * s, par, abort_flag, p.err)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint64_t ad = ad0 + s * dstep, bd = bd0 + s * dstep;
#pragma unroll
            for (int k = 0; k < kQBK / 16; ++k) tc2_mma_f16(d, ad + 2ull * k, bd + 2ull * k, idesc, (kb | k) != 0);
            tc2_commit(empty0 + 8u * s, 3);
            if (++s == (uint32_t)stages) {
              s = 0;
              par ^= 1;
            }
          }
          if (ok) tc2_commit(tfull0 + 8u * buf, 3);
        }
        // every MMA issued above has completed once this arrives
        tc2_commit(drain_bar, 1);
        volatile int no_abort = 0;
        mbar_wait_bounded(drain_bar, 0, &no_abort, p.err);
      }
    }
  } else {
    // ---------------- epilogue of this CTA's 128 rows
    pdl_wait();
    const int q = warp & 3;
    const int row = q * 32 + lane;
    const int half = (warp - 2) / 4, h0 = (bn / 32 + 1) / 2 * 32;
    const int c_lo = half * h0, cols = half ? bn - h0 : h0;  // this warp's columns, a multiple of 32 (may be none)
    float* sb = sbias + (warp - 2) * 128;                    // its own copy of their bias: no cross-warp barrier
    const uint32_t stage = smem_u32(staging) + (uint32_t)((warp - 2) * kEpiStage);
    const uint32_t ltempty0 = map_rank(tempty0, 0);
    const int rmode = res_mode(p.e);
    for (int lt = 0; lt < my_tiles; ++lt) {
      const int buf = lt & 1, use = lt >> 1;
      const int tile = tile_of(lt);
      const int ntile = tile / mtp, seg = NS > 1 ? ntile / nt : 0;
      const int n0 = (ntile - seg * nt) * bn + c_lo;
      T* const y = seg_y<T>(p, sg, seg);
      const bool vec = epi_vec_ok(p, y);
      const T* bias = seg_bias<T>(p, sg, seg);
      for (int j = lane; j < cols; j += 32) sb[j] = (bias && n0 + j < p.N) ? to_f<T>(bias[n0 + j]) : 0.f;
      __syncwarp();
      const int idx = (tile % mtp) * 2 + rank;
      int m = -1;  // output row of this thread's TMEM lane
      if (idx < mt) {
        if (TAP) {
          const int img = idx / patches, rem = idx - img * patches;
          const int th = rem / p.tiles_w, tw = rem - th * p.tiles_w;
          if (row < p.wt * p.ht) {
            const int oy = th * p.ht + row / p.wt, ox = tw * p.wt + row % p.wt;
            if (oy < p.Ho && ox < p.Wo) m = (img * p.Ho + oy) * p.Wo + ox;
          }
        } else {
          m = idx * kQBM + row;
          if (m >= p.M) m = -1;
        }
      }
      uint4 rnext[4];
      epi_res_load<T>(rnext, p, m, n0, vec && cols > 0);
      const bool got = mbar_wait_bounded(tfull0 + 8u * buf, use & 1, abort_flag, p.err);
      if (!__all_sync(0xffffffffu, got)) break;  // tcgen05.ld is warp-collective
      tc_fence_after();
#pragma unroll 1
      for (int c = 0; c < cols && n0 + c < p.N; c += 32) {
        uint4 rcur[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) rcur[i] = rnext[i];
        if (c + 32 < cols) epi_res_load<T>(rnext, p, m, n0 + c + 32, vec);
        epi_piece<T>(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * 256 + c_lo + c), sb + c, stage, p, y, m, n0 + c,
                     vec, rmode, rcur);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(ltempty0 + 8u * buf);
    }
  }
  tc_fence_before();
  __syncthreads();
  // neither CTA leaves while the other may still read its operands or signal its barriers
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kQTmemCols) : "memory");
  }
}

template <typename T, int AMODE, int NS = 1>
int launch_pair_inst(const TcGemm& g, const TcPlan& pl, int* err, cudaStream_t s) {
  static std::atomic<uint64_t> attr_done{0};  // per instantiation, one bit per device
  auto kern = tc_pair_kernel<T, AMODE, NS>;
  if (attr_needed(attr_done)) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kQSmem) != cudaSuccess)
      SN_FAIL(SWAPNET_ERR_CUDA, "cudaFuncSetAttribute failed");
    attr_set(attr_done);
  }
  TcArgs a;
  std::memset(&a, 0, sizeof(a));
  a.M = g.M; a.N = g.N; a.K = g.K;
  a.Ho = g.Ho; a.Wo = g.Wo; a.C = g.C;
  a.kh = g.kh; a.kw = g.kw; a.stride = g.stride; a.pad = g.pad;
  a.e = g.e; a.y = g.y; a.ldy = g.ldy; a.err = err;
  a.wt = pl.wt; a.ht = pl.ht; a.tiles_w = pl.tiles_w; a.tiles_h = pl.tiles_h;
  const int sms = g.num_sms > 0 ? g.num_sms : 148;
  const int stages = std::min(kQMaxStages, kQRing / (kQA + pl.bn / 2 * 128));
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(2 * (unsigned)std::min<int64_t>(pl.tiles, sms / 2));
  cfg.blockDim = dim3(kQThreads);
  cfg.dynamicSmemBytes = kQSmem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = g.no_pdl ? 1 : 2;
  const cudaError_t le = cudaLaunchKernelEx(&cfg, kern, pl.tmA, make_segs<NS>(g, pl), a, (int)pl.bn, stages);
  if (le != cudaSuccess) SN_FAIL(SWAPNET_ERR_CUDA, std::string("paired GEMM launch: ") + cudaGetErrorString(le));
  return SWAPNET_OK;
}

}  // namespace

int launch_tc_pair(const TcGemm& g, const TcPlan& pl, int* err, cudaStream_t s) {
  if (pl.bn < 32 || pl.bn > 256 || pl.bn % 32 || (g.conv && !pl.tma_conv))
    SN_FAIL(SWAPNET_ERR_INVALID_ARG, "paired GEMM: bad tile");
  if (g.nseg > 1)
    return g.dtype == SWAPNET_BF16 ? launch_pair_inst<__nv_bfloat16, 0, kTcMaxSeg>(g, pl, err, s)
                                   : launch_pair_inst<__half, 0, kTcMaxSeg>(g, pl, err, s);
  if (g.dtype == SWAPNET_BF16)
    return g.conv ? launch_pair_inst<__nv_bfloat16, 1>(g, pl, err, s) : launch_pair_inst<__nv_bfloat16, 0>(g, pl, err, s);
  return g.conv ? launch_pair_inst<__half, 1>(g, pl, err, s) : launch_pair_inst<__half, 0>(g, pl, err, s);
}

}  // namespace swapnet
