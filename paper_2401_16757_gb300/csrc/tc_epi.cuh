// Shared pieces of the tcgen05 GEMM kernels: launch arguments and the fused
// epilogue (bias, residual, activation, conversion).
#pragma once
#include "device.cuh"
#include "kernels.h"

namespace swapnet {
namespace {

// Weight maps of a launch and, for siblings sharing it (NS > 1: same input, K
// and N), each layer's output and bias.  A launch of one layer has its output
// and bias in TcArgs: with the arrays in every launch, YOLOv3's 75 layers
// took 424 us, without 416.
template <int NS> struct TcSegs {
  CUtensorMap m[NS];
  void* y[NS];
  const void* bias[NS];
  int nseg;
};
template <> struct TcSegs<1> {
  CUtensorMap m[1];
};

struct TcArgs {
  int M, N, K;
  const void* x;  // conv input (gather)
  int H, Wd, C, Ho, Wo, kh, kw, stride, pad;
  Epi e;
  void* y;
  int64_t ldy;
  int* err;
  int kb_per_split;  // k-blocks per split; gridDim.z splits
  // TMA im2col (persistent kernel): output tiles are wt x ht pixel patches of
  // one image, tiles_w x tiles_h of them per image; rows >= wt * ht are unused
  int wt, ht, tiles_w, tiles_h;
};

// A launch's weight maps, outputs and biases (host side).
template <int NS>
inline TcSegs<NS> make_segs(const TcGemm& g, const TcPlan& pl) {
  TcSegs<NS> r;
  for (int i = 0; i < NS; ++i) r.m[i] = pl.tmB[i < g.nseg ? i : 0];
  if constexpr (NS > 1) {
    r.nseg = g.nseg;
    for (int i = 0; i < NS; ++i) {
      r.y[i] = i && i < g.nseg ? g.yx[i - 1] : g.y;
      r.bias[i] = i && i < g.nseg ? g.bx[i - 1] : g.e.bias;
    }
  }
  return r;
}
// Output and bias of segment seg.
template <typename T, int NS>
__device__ __forceinline__ T* seg_y(const TcArgs& p, const TcSegs<NS>& sg, int seg) {
  if constexpr (NS > 1) return static_cast<T*>(sg.y[seg]);
  else return static_cast<T*>(p.y);
}
template <typename T, int NS>
__device__ __forceinline__ const T* seg_bias(const TcArgs& p, const TcSegs<NS>& sg, int seg) {
  if constexpr (NS > 1) return static_cast<const T*>(sg.bias[seg]);
  else return static_cast<const T*>(p.e.bias);
}

// ---- epilogue helpers
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
template <typename T> __device__ __forceinline__ float lo_f(uint32_t u);
template <typename T> __device__ __forceinline__ float hi_f(uint32_t u);
template <> __device__ __forceinline__ float lo_f<__half>(uint32_t u) {
  return __half2float(__ushort_as_half((unsigned short)(u & 0xffffu)));
}
template <> __device__ __forceinline__ float hi_f<__half>(uint32_t u) {
  return __half2float(__ushort_as_half((unsigned short)(u >> 16)));
}
template <> __device__ __forceinline__ float lo_f<__nv_bfloat16>(uint32_t u) { return __uint_as_float(u << 16); }
template <> __device__ __forceinline__ float hi_f<__nv_bfloat16>(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }

// How an epilogue uses the residual: not at all, before the activation,
// after it, or as the gate of a SwiGLU layer.  Chosen once per tile, so that
// the per-element code has no branch on it.
constexpr int kResNone = 0, kResPre = 1, kResPost = 2, kResGate = 3;

__device__ __forceinline__ int res_mode(const Epi& e) {
  if (e.act == SWAPNET_ACT_SWIGLU) return kResGate;
  return !e.res ? kResNone : (e.res_post ? kResPost : kResPre);
}

// r / d for d = 1 + e^-r >= 1: an approximate quotient and one correction by
// its exact remainder (P. Markstein, "Computation of elementary functions on
// the IBM RISC System/6000 processor", 1990), without the test and branch per
// element of the general division, which kept the elements of a thread from
// overlapping (a 32 x 32 SwiGLU piece took 5.8 us of a warp, and a 79 x 2752 x
// 1024 SwiGLU layer 9.9 us, 5.0 with this; 4.0 without an activation).
// The correctly rounded quotient for every 16-bit r and for 2^26 fp32 values of
// r in [-110, 110]: near the end of fp32's range too, where the reciprocal is
// subnormal and a few bits short, which the correction bears.  Where r or d is
// infinite the remainder is not a number and the first quotient is exact.
__device__ __forceinline__ float gate_quotient(float r, float d) {
  float rc;
  asm("rcp.approx.f32 %0, %1;" : "=f"(rc) : "f"(d));
  const float q = r * rc;
  const float c = fmaf(-fmaf(q, d, -r), rc, q);  // (this sign of the remainder keeps that of a zero r)
  return c == c ? c : q;
}

// One output element; the arithmetic of epilogue() in device.cuh.
template <int RES>
__device__ __forceinline__ float epi1(float acc, float bias, float r, int act) {
  if (RES == kResGate) return gate_quotient(r, 1.0f + expf(-r)) * (acc + bias);
  float v = acc + bias;
  if (RES == kResPre) v += r;
  const float neg = act == SWAPNET_ACT_RELU ? 0.f : (act == SWAPNET_ACT_LEAKY ? 0.1f * v : v);
  v = v > 0.f ? v : neg;
  if (RES == kResPost) v += r;
  return v;
}

// 8 consecutive outputs: fp32 sums a, 8 bias values at sb (shared memory),
// 8 residual values r as stored -> 8 packed outputs.
template <typename T, int RES>
__device__ __forceinline__ uint4 epi8(const float (&a)[8], const float* sb, const uint4& r, int act) {
  const float4 b0 = *reinterpret_cast<const float4*>(sb);
  const float4 b1 = *reinterpret_cast<const float4*>(sb + 4);
  const float bf[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
  const uint32_t rw[4] = {r.x, r.y, r.z, r.w};
  uint32_t o[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float r0 = RES ? lo_f<T>(rw[i]) : 0.f, r1 = RES ? hi_f<T>(rw[i]) : 0.f;
    o[i] = pack2<T>(epi1<RES>(a[2 * i], bf[2 * i], r0, act), epi1<RES>(a[2 * i + 1], bf[2 * i + 1], r1, act));
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}

template <typename T>
__device__ __forceinline__ uint4 epi8_any(const float (&a)[8], const float* sb, const uint4& r, int act, int res) {
  switch (res) {
    case kResNone: return epi8<T, kResNone>(a, sb, r, act);
    case kResPre: return epi8<T, kResPre>(a, sb, r, act);
    case kResPost: return epi8<T, kResPost>(a, sb, r, act);
    default: return epi8<T, kResGate>(a, sb, r, act);
  }
}

// ---- tile epilogue of one warp: its 32 rows (TMEM lanes) x 32 columns at a
// time.  In TMEM a thread has a row; written like that to global memory,
// every store (and every residual load) of a warp would touch 32 rows, 16
// bytes each.  So a warp passes each 32 x 32 piece through 2 KB of shared
// memory of its own (rows of 64 bytes, 16-byte chunks swizzled by row, no
// bank conflicts in either direction) and reads and writes global memory
// eight whole 64-byte row pieces per instruction.  What bounds it at batch 1
// is latency and instruction fetch, not bandwidth: the code is kept short
// (16 columns per step, one variant per residual mode), and the residual is
// requested before the accumulator is waited for.  A 1x1 layer's 64-column
// tile: 2.4 us from the accumulator to the last store with one thread per
// row, four warps and the activation chosen per element.
constexpr int kEpiStage = 32 * 64;  // bytes of shared memory per warp

// Rows can be moved in 16-byte pieces: N, the strides and the bases allow it.
__device__ __forceinline__ bool epi_vec_ok(const TcArgs& p, const void* y) {
  return ((p.N | p.ldy) % 8 == 0) && ((uintptr_t)y & 15) == 0 &&
         (!p.e.res || (p.e.ldr % 8 == 0 && ((uintptr_t)p.e.res & 15) == 0));
}

__device__ __forceinline__ uint32_t epi_stage_addr(uint32_t stage, int row, int chunk) {
  return stage + (uint32_t)(row * 64 + ((chunk ^ ((row >> 1) & 3)) << 4));
}

// Residual of columns [n, n + 32) of the warp's rows, four 16-byte pieces
// per lane in the layout of the coalesced pass (m: this lane's output row,
// -1 for none).  Zeros without a residual or where the 16-byte path does
// not apply.
template <typename T>
__device__ __forceinline__ void epi_res_load(uint4 (&r)[4], const TcArgs& p, int m, int n, bool vec) {
  const int lane = threadIdx.x & 31;
  const T* res = static_cast<const T*>(p.e.res);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int mr = __shfl_sync(0xffffffffu, m, i * 8 + (lane >> 2)), c = n + (lane & 3) * 8;
    r[i] = make_uint4(0u, 0u, 0u, 0u);
    if (vec && res && mr >= 0 && c < p.N) r[i] = *reinterpret_cast<const uint4*>(res + (int64_t)mr * p.e.ldr + c);
  }
}

template <typename T, int RES>
__device__ __forceinline__ void epi_rows(uint32_t taddr, const float* sb, uint32_t stage, int act) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    uint32_t v[16];
    tmem_ld_32x32b_x16(taddr + 16u * h, v);
    tmem_ld_wait();
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const uint32_t addr = epi_stage_addr(stage, lane, 2 * h + c);
      uint4 r = make_uint4(0u, 0u, 0u, 0u);
      if (RES) asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "r"(addr));
      float a[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) a[j] = __uint_as_float(v[8 * c + j]);
      r = epi8<T, RES>(a, sb + 16 * h + 8 * c, r, act);
      asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(r.x), "r"(r.y), "r"(r.z), "r"(r.w) : "memory");
    }
  }
}

// Columns [n, n + 32) of the warp's rows of output y: accumulator at taddr
// (the warp's TMEM lanes, first column), bias at sb, residual r from
// epi_res_load.  All lanes call it together.
template <typename T>
__device__ __forceinline__ void epi_piece(uint32_t taddr, const float* sb, uint32_t stage, const TcArgs& p, T* y, int m,
                                          int n, bool vec, int res, const uint4 (&r)[4]) {
  const int lane = threadIdx.x & 31;
  if (res != kResNone) {
    if (vec) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(epi_stage_addr(stage, i * 8 + (lane >> 2), lane & 3)),
                     "r"(r[i].x), "r"(r[i].y), "r"(r[i].z), "r"(r[i].w)
                     : "memory");
    } else {
      const uint16_t* rs = static_cast<const uint16_t*>(p.e.res);
#pragma unroll 4
      for (int row = 0; row < 32; ++row) {
        const int mr = __shfl_sync(0xffffffffu, m, row);
        const uint16_t e = rs && mr >= 0 && n + lane < p.N ? rs[(int64_t)mr * p.e.ldr + n + lane] : (uint16_t)0;
        asm volatile("st.shared.u16 [%0], %1;" ::"r"(epi_stage_addr(stage, row, lane >> 3) + (lane & 7) * 2), "h"(e)
                     : "memory");
      }
    }
    __syncwarp();
  }
  switch (res) {
    case kResNone: epi_rows<T, kResNone>(taddr, sb, stage, p.e.act); break;
    case kResPre: epi_rows<T, kResPre>(taddr, sb, stage, p.e.act); break;
    case kResPost: epi_rows<T, kResPost>(taddr, sb, stage, p.e.act); break;
    default: epi_rows<T, kResGate>(taddr, sb, stage, p.e.act); break;
  }
  __syncwarp();
  if (vec) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int row = i * 8 + (lane >> 2), c = n + (lane & 3) * 8;
      const int mr = __shfl_sync(0xffffffffu, m, row);
      uint4 v;
      asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                   : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                   : "r"(epi_stage_addr(stage, row, lane & 3)));
      if (mr >= 0 && c < p.N) *reinterpret_cast<uint4*>(y + (int64_t)mr * p.ldy + c) = v;
    }
  } else {
#pragma unroll 4
    for (int row = 0; row < 32; ++row) {
      const int mr = __shfl_sync(0xffffffffu, m, row);
      uint16_t e;
      asm volatile("ld.shared.u16 %0, [%1];"
                   : "=h"(e)
                   : "r"(epi_stage_addr(stage, row, lane >> 3) + (lane & 7) * 2));
      if (mr >= 0 && n + lane < p.N) reinterpret_cast<uint16_t*>(y)[(int64_t)mr * p.ldy + n + lane] = e;
    }
  }
  __syncwarp();  // the staging rows may be written again
}

// 8 outputs [n, n + 8) of row m from fp32 sums (split-K reductions); r: the
// residual already loaded by res8 on the 16-byte path.
template <typename T>
__device__ __forceinline__ uint4 res8(const TcArgs& p, int m, int n, bool vec) {
  if (!vec || !p.e.res || m < 0 || n >= p.N) return make_uint4(0u, 0u, 0u, 0u);
  return *reinterpret_cast<const uint4*>(static_cast<const T*>(p.e.res) + (int64_t)m * p.e.ldr + n);
}
template <typename T>
__device__ __forceinline__ void finish8(const float (&a)[8], const float* sb, const TcArgs& p, T* y0, int m, int n,
                                        bool vec, int res, const uint4& r) {
  T* y = y0 + (int64_t)m * p.ldy + n;
  if (vec) {
    *reinterpret_cast<uint4*>(y) = epi8_any<T>(a, sb, r, p.e.act, res);
  } else {
    const T* rr = p.e.res ? static_cast<const T*>(p.e.res) + (int64_t)m * p.e.ldr + n : nullptr;
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (n + j < p.N)
        y[j] = from_f<T>(epilogue(a[j], sb[j], rr ? to_f<T>(rr[j]) : 0.f, rr != nullptr, p.e.act, p.e.res_post));
  }
}

}  // namespace
}  // namespace swapnet
