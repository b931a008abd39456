// SIMT layer kernels: skinny linear (M <= 16: the HBM-bound GEMV and the
// few-row fp32 kernel), tiled fp32 linear,
// direct convolution for channel counts the tensor-core path cannot tile,
// pooling, upsampling and channel concatenation.  NHWC everywhere.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstring>

#include "device.cuh"
#include "internal.h"
#include "kernels.h"

namespace swapnet {

namespace {

template <typename T> struct Vec16 { static constexpr int N = 16 / sizeof(T); };

// Launch with programmatic stream serialization: the kernel may start while
// the previous kernel on the stream drains; it waits (pdl_wait) before
// reading that kernel's output.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

__device__ __forceinline__ uint4 ld_stream16(const void* p) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}

// 16 bytes of the launch before's output: a plain load, kept behind the wait
// (both are volatile) but free to pass this kernel's own stores, none of which
// writes there.
__device__ __forceinline__ uint4 ld_input16(const void* p) {
  uint4 r;
  asm volatile("ld.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
  return r;
}

template <typename T> __device__ __forceinline__ void unpack16(const uint4& v, float* f) {
  const T* e = reinterpret_cast<const T*>(&v);
#pragma unroll
  for (int i = 0; i < Vec16<T>::N; ++i) f[i] = to_f<T>(e[i]);
}

template <typename T> __device__ __forceinline__ uint4 pack16(const float* f) {
  uint4 v;
  T* e = reinterpret_cast<T*>(&v);
#pragma unroll
  for (int i = 0; i < Vec16<T>::N; ++i) e[i] = from_f<T>(f[i]);
  return v;
}

// ------------------------------------------------------------ GEMV
// Linear layers of 1 to 4 rows of 16-bit values, or one row of fp32: the time
// is streaming the weights.  Persistent CTAs (as many as are resident: two per
// SM, one with sums for 3 or 4 rows) take groups of eight weight rows; K is walked in passes, of which a lane takes one 16-byte chunk
// of every row (chunk 32 w + l of the pass for lane l of warp w), so a loaded
// chunk of x meets eight rows.  The loads of two passes are in flight ahead of
// the one being summed, across groups, so that a group's reductions and
// stores never leave HBM idle; the first two passes' weights are requested
// before the programmatic wait (they do not depend on the kernel before).  A
// lane's sums are halved across the lanes, the warps' added in warp order
// through shared memory: a fixed order for every output.
//
// One launch may serve several layers that read the same input (SkJob
// segments, e.g. the q, k, v projections): the groups are dealt to the
// segments in order.  In pair mode (a gate and the layer whose epilogue takes
// the gate's output as its residual, e.g. SwiGLU) a group is four features of
// both: the gate's rounded output is stored and that same rounded value is
// the second layer's residual.  Every output is summed as in a one-layer
// launch, so the results are bit-identical to launching the layers one by
// one.
// Bound by HBM: against one warp per feature with eight loads in flight and
// none while it sums, whose last wave of CTAs leaves the chip part empty:
// 11008 x 4096 bf16 19.0 -> 13.7 us (6.6 TB/s, launch included), 4096 x 11008
// 19.1 -> 15.0, 4096 x 4096 (from L2) 6.1 -> 4.4, 32000 x 4096 40.2 -> 36.7.
// Four rows of 4096 x 4096 14.5 -> 9.0 (FMAs and conversions; 9.6 with twice the
// CTAs that fit).
constexpr int kGvWarps = 8;
constexpr int kGvRows = 8;  // weight rows per group
// CTAs of an instance on an SM: 118-124 registers a thread with sums for one
// or two rows of x, 206 with four.
constexpr int gv_ctas(int mt) { return mt <= 2 ? 2 : 1; }

// Short rows (TEAMS): a row that needs only wk = 1, 2 or 4 of the warps leaves
// the CTA room for kGvWarps / wk teams of wk warps, each on groups of its own:
// the same chunks on the same lanes and the same order of sums (an idle warp
// added zeros), with all warps loading.  1 row of 512 bf16 by 32000 features
// 16.7 us with one team, 6.2 with four.
template <typename T, int MT, bool TEAMS>
__global__ void __launch_bounds__(kGvWarps * 32, gv_ctas(MT)) gemv_kernel(const SkJob j, const int groups, const int team_warps) {
  constexpr int V = Vec16<T>::N;
  constexpr int NV = MT * kGvRows;
  __shared__ float red[2][kGvWarps][NV];
  const int wk = TEAMS ? team_warps : kGvWarps;  // warps that share a group
  const int kPass = wk * 32 * V;                 // k per pass
  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int team = TEAMS ? warp / wk : 0, warp0 = team * wk;
  const int K = j.K, k0 = ((warp - warp0) * 32 + lane) * V;
  const int passes = TEAMS ? 1 : (K + kPass - 1) / kPass;
  const int teams = TEAMS ? kGvWarps / wk : 1;
  const int G = (int)gridDim.x * teams, g0 = (int)blockIdx.x * teams + team;
  const int items = g0 < groups ? (groups - 1 - g0) / G + 1 : 0;
  const T* x = static_cast<const T*>(j.x);
  const int per = j.pair ? kGvRows / 2 : kGvRows;  // features per group
  // segment and first feature of a group
  auto locate = [&](int g, int* o) {
    int si = 0;
    if (!j.pair)
      while (si + 1 < j.nseg) {
        const int n = (j.seg[si].N + per - 1) / per;
        if (g < n) break;
        g -= n;
        ++si;
      }
    *o = g * per;
    return si;
  };
  // load cursor: rows 0..3 of its group start at pa, rows 4..7 at pb; of each
  // four, va and vb exist
  int lg = g0, lp = 0, va = 0, vb = 0;
  const T *pa = nullptr, *pb = nullptr;
  auto open_group = [&]() {
    if (lg >= groups) {
      va = vb = 0;
      return;
    }
    int o;
    const int si = locate(lg, &o);
    const T* W = static_cast<const T*>(j.seg[0].W);
    int N = j.seg[0].N;
#pragma unroll
    for (int i = 1; i < kSkMaxSeg; ++i)
      if (i == si) {
        W = static_cast<const T*>(j.seg[i].W);
        N = j.seg[i].N;
      }
    pa = W + (int64_t)o * K + k0;
    va = min(4, N - o);
    if (j.pair) {
      pb = static_cast<const T*>(j.seg[1].W) + (int64_t)o * K + k0;
      vb = va;
    } else {
      pb = pa + (int64_t)4 * K;
      vb = max(0, min(4, N - o - 4));
    }
  };
  struct Buf {
    uint4 w[kGvRows];
    uint4 x[MT];
  };
  auto load_w = [&](Buf& b) {
    const bool in = k0 + lp * kPass < K;
#pragma unroll
    for (int f = 0; f < kGvRows; ++f) {
      b.w[f] = make_uint4(0u, 0u, 0u, 0u);
      const bool ok = in && (f < 4 ? f < va : f - 4 < vb);
      if (ok) b.w[f] = ld_stream16((f < 4 ? pa : pb) + (int64_t)(f & 3) * K + (int64_t)lp * kPass);
    }
  };
  auto load_x = [&](Buf& b, int p) {
    const int k = k0 + p * kPass;
#pragma unroll
    for (int m = 0; m < MT; ++m)
      b.x[m] = m < j.M && k < K ? ld_input16(x + (int64_t)m * K + k) : make_uint4(0u, 0u, 0u, 0u);
  };
  auto next_load = [&]() {
    if (++lp == passes) {
      lp = 0;
      lg += G;
      open_group();
    }
  };
  Buf A, B;
  open_group();
  load_w(A);
  const int pA = lp;
  next_load();
  load_w(B);
  const int pB = lp;
  next_load();
  pdl_wait();
  pdl_launch_dependents();
  load_x(A, pA);
  load_x(B, pB);
  float acc[NV];  // [row of x][weight row]
#pragma unroll
  for (int i = 0; i < NV; ++i) acc[i] = 0.f;
  auto sum = [&](const Buf& b) {
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      float xf[V];
      unpack16<T>(b.x[m], xf);
#pragma unroll
      for (int f = 0; f < kGvRows; ++f) {
        float wf[V];
        unpack16<T>(b.w[f], wf);
#pragma unroll
        for (int i = 0; i < V; ++i) acc[m * kGvRows + f] = fmaf(wf[i], xf[i], acc[m * kGvRows + f]);
      }
    }
  };
  // a group's sums across lanes and warps, its outputs
  auto finish = [&](int g, int par) {
    // halve the sums a lane holds while there are several, then add across
    // the lanes that hold the same one; the highest lane bits say which
#pragma unroll
    for (int off = 16, n = NV / 2; off > 0; off >>= 1, n >>= 1) {
      if (n > 0) {
#pragma unroll
        for (int i = 0; i < n; ++i) {
          const bool up = lane & off;
          const float send = up ? acc[i] : acc[i + n], keep = up ? acc[i + n] : acc[i];
          acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
      } else {
        acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], off);
      }
    }
    if (NV >= 32) {
#pragma unroll
      for (int i = 0; i < (NV + 31) / 32; ++i) red[par][warp][lane * (NV / 32) + i] = acc[i];
    } else if (lane % (32 / (NV < 32 ? NV : 32)) == 0) {
      red[par][warp][lane / (32 / (NV < 32 ? NV : 32))] = acc[0];
    }
#pragma unroll
    for (int i = 0; i < NV; ++i) acc[i] = 0.f;
    if (TEAMS) asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(wk * 32) : "memory");
    else __syncthreads();
    const int tid = TEAMS ? (warp - warp0) * 32 + lane : (int)threadIdx.x;
    const int f = tid % per, m = tid / per;
    if (m >= j.M) return;
    int o;
    const int si = locate(g, &o);
    o += f;
    SkSeg S = j.seg[0];
#pragma unroll
    for (int i = 1; i < kSkMaxSeg; ++i)
      if (i == si) S = j.seg[i];
    if (o >= S.N) return;
    auto total = [&](int i) {
      float t = red[par][warp0][i];
      if constexpr (TEAMS) {
        for (int h = 1; h < wk; ++h) t += red[par][warp0 + h][i];
      } else {
#pragma unroll
        for (int h = 1; h < kGvWarps; ++h) t += red[par][h][i];
      }
      return t;
    };
    auto emit = [&](const SkSeg& q, float t, float r, bool has_r) {
      const float bias = q.e.bias ? to_f<T>(static_cast<const T*>(q.e.bias)[o]) : 0.f;
      const T out = from_f<T>(epilogue(t, bias, r, has_r, q.e.act, q.e.res_post));
      static_cast<T*>(q.y)[(int64_t)m * q.ldy + o] = out;
      return to_f<T>(out);  // the stored value, as a paired layer reads it
    };
    const bool has_r = S.e.res != nullptr;
    const float r = has_r ? to_f<T>(static_cast<const T*>(S.e.res)[(int64_t)m * S.e.ldr + o]) : 0.f;
    const float gate = emit(S, total(m * kGvRows + f), r, has_r);
    if (j.pair) emit(j.seg[1], total(m * kGvRows + f + 4), gate, true);
  };
  int cp = 0, cg = g0, par = 0;  // pass and group being summed
  const int total = items * passes;
  auto step = [&](Buf& b, int it) {
    sum(b);
    if (it + 2 < total) {
      load_w(b);
      load_x(b, lp);
      next_load();
    }
    if (++cp == passes) {
      cp = 0;
      finish(cg, par);
      cg += G;
      par ^= 1;
    }
  };
  for (int it = 0; it < total; it += 2) {
    step(A, it);
    if (it + 1 < total) step(B, it + 1);
  }
}

// ------------------------------------------------------------ few-row fp32 linear
// fp32 layers of 2 to 16 rows: one CTA per FT output features, K walked
// in chunks of 1024, of which warp w takes the k 128 w .. + 127 and lane l four
// of them.  Weights and x come straight from global memory, 16 bytes per lane
// and row, every load of a chunk in flight at once (the first chunk's weights
// before the programmatic wait), and each loaded value of x meets FT weights
// in registers.  The MT x FT sums of a lane are reduced across the lanes by
// halving (62 shuffles for 64 sums), then across the warps in warp order
// through shared memory: a fixed order for every output, whatever the other
// features, and the same for weights in device and in mapped host memory.
// Bound by the chain of one launch: the load round trip, the sums and two
// reductions.  The one-warp-per-feature kernels read x from shared memory or
// L1 once per feature and warp: 8 x 1024 x 1024, weights in L2, 6.3 us
// in a chain of layers, 2.3 with this; 8 x 4096 x 4096 79 -> 13 us; 16 x 2048 x
// 2048 26 -> 7.8. One row alone is left to the GEMV (1024 x 1024 1.8 against 1.9).
// Six blocks of three siblings, a SwiGLU pair and a layer, width 256, 8 rows:
// 41.0 us with shared launches, 59.5 with one each (1024: 112.6, 122.8).
constexpr int kRwWarps = 8;

// One launch may serve several layers that read the same x, as the GEMV's: the
// CTAs are dealt to the segments in order, or (pair) a CTA takes FT / 2 features
// of the gate and of its paired layer.  NS: layers that a launch may hold (1 or
// kSkMaxSeg; a layer alone does not carry the parameters of three).
//
// TEAMS: rows of up to 512 values need only wk = 1, 2 or 4 of the warps; with
// more CTAs than are resident (two per SM) a CTA is kRwWarps / wk teams of wk
// warps, each with features of its own (same lanes, same order of sums): 2 rows of
// 64 by 3648 features 3.46 us without, 1.85 with; 8 of 512 by 8000 8.1 and 5.9.
// Longer rows, two of them, take 16 features per CTA there instead of 8: 1024 by
// 3648 4.06 -> 3.16 (1024 by 1024, one round of CTAs either way, 1.92 and 1.95).
template <int NS> struct RowsJob {
  const float* x;
  int M, K, nseg, pair, wk;
  SkSeg seg[NS];
};

template <int MT, int FT, int NS, bool TEAMS>
__global__ void __launch_bounds__(kRwWarps * 32, 2) linear_rows_kernel(const RowsJob<NS> j) {
  constexpr bool MULTI = NS > 1;
  constexpr int NV = MT * FT;  // sums per lane, a power of two of at least 32
  static_assert(NV >= 32 && (NV & (NV - 1)) == 0 && NV <= kRwWarps * 32, "halving reduction");
  __shared__ float red[kRwWarps][NV];
  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int M = j.M, K = j.K;
  const float* x = j.x;
  const bool pair = MULTI && j.pair;
  const int per = pair ? FT / 2 : FT;  // features of a layer per CTA
  const int wk = TEAMS ? j.wk : kRwWarps;
  const int warp0 = TEAMS ? warp / wk * wk : 0;  // the team's first warp
  int cta = TEAMS ? (int)blockIdx.x * (kRwWarps / wk) + warp / wk : (int)blockIdx.x, si = 0;
  if (MULTI && !pair)
    while (si + 1 < j.nseg && cta >= (j.seg[si].N + FT - 1) / FT) cta -= (j.seg[si++].N + FT - 1) / FT;
  SkSeg S = j.seg[0];
#pragma unroll
  for (int i = 1; i < NS; ++i)
    if (i == si) S = j.seg[i];
  const int o0 = cta * per;
  const int k0 = (warp - warp0) * 128 + lane * 4;
  float4 w[FT];
  auto load_w = [&](int k) {
#pragma unroll
    for (int f = 0; f < FT; ++f) {
      const bool up = pair && f >= FT / 2;  // the paired layer's half
      const int o = o0 + (up ? f - FT / 2 : f);
      w[f] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (o < S.N && k < K) {
        const uint4 u = ld_stream16(static_cast<const float*>(up ? j.seg[NS > 1].W : S.W) + (int64_t)o * K + k);
        w[f] = make_float4(__uint_as_float(u.x), __uint_as_float(u.y), __uint_as_float(u.z), __uint_as_float(u.w));
      }
    }
  };
  load_w(k0);
  pdl_wait();
  pdl_launch_dependents();
  float v[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) v[i] = 0.f;
  for (int k = k0; k - k0 < K; k += kRwWarps * 128) {  // (one round for teams)
    if (k != k0) load_w(k);
    float4 xv[MT];
#pragma unroll
    for (int m = 0; m < MT; ++m)
      xv[m] = m < M && k < K ? *reinterpret_cast<const float4*>(x + (int64_t)m * K + k) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int f = 0; f < FT; ++f) {
        float a = v[m * FT + f];
        a = fmaf(w[f].x, xv[m].x, a);
        a = fmaf(w[f].y, xv[m].y, a);
        a = fmaf(w[f].z, xv[m].z, a);
        v[m * FT + f] = fmaf(w[f].w, xv[m].w, a);
      }
  }
  // across the lanes: each step halves the sums a lane holds; lane bits pick
  // the half, from the highest bit down, so lane l ends with the sums of
  // indexes [l * NV / 32, (l + 1) * NV / 32)
#pragma unroll
  for (int off = 16, n = NV / 2; off > 0; off >>= 1, n >>= 1) {
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const bool up = lane & off;
      const float send = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
#pragma unroll
  for (int i = 0; i < NV / 32; ++i) red[warp][lane * (NV / 32) + i] = v[i];
  if (TEAMS) asm volatile("bar.sync %0, %1;" ::"r"(1 + warp / wk), "r"(wk * 32) : "memory");
  else __syncthreads();
  auto total = [&](int i) {
    float s = red[warp0][i];
    if constexpr (TEAMS) {
      for (int h = 1; h < wk; ++h) s += red[warp0 + h][i];
    } else {
#pragma unroll
      for (int h = 1; h < kRwWarps; ++h) s += red[h][i];
    }
    return s;
  };
  auto emit = [&](const SkSeg& q, int m, int o, float s, float r, bool has_r) {
    const float* bias = static_cast<const float*>(q.e.bias);
    const float out = epilogue(s, bias ? bias[o] : 0.f, r, has_r, q.e.act, q.e.res_post);
    static_cast<float*>(q.y)[(int64_t)m * q.ldy + o] = out;
    return out;
  };
  auto finish = [&](int i) {
    const int m = i / per, f = i % per, o = o0 + f;
    if (m >= M || o >= S.N) return;
    const float* res = static_cast<const float*>(S.e.res);
    const float gate = emit(S, m, o, total(m * FT + f), res ? res[(int64_t)m * S.e.ldr + o] : 0.f, res != nullptr);
    if (pair) emit(j.seg[NS > 1], m, o, total(m * FT + f + FT / 2), gate, true);
  };
  if constexpr (TEAMS) {
    for (int i = (warp - warp0) * 32 + lane; i < MT * per; i += wk * 32) finish(i);
  } else {
    finish((int)threadIdx.x);
  }
}

// CTAs that take all features of a launch, FT each.
inline int rows_ctas(const SkJob& j, int ft) {
  const int per = j.pair ? ft / 2 : ft;
  int n = (j.seg[0].N + per - 1) / per;
  for (int i = 1; i < j.nseg && !j.pair; ++i) n += (j.seg[i].N + per - 1) / per;
  return n;
}

template <int MT, int FT, int NS>
int rows_launch_ns(const SkJob& j, cudaStream_t s) {
  RowsJob<NS> r{static_cast<const float*>(j.x), j.M, j.K, j.nseg, j.pair, 1, {}};
  for (int i = 0; i < NS; ++i) r.seg[i] = j.seg[i];
  int ctas = rows_ctas(j, FT);
  while (r.wk < kRwWarps && r.wk * 128 < j.K) r.wk *= 2;
  const bool teams = r.wk < kRwWarps && ctas > 2 * j.num_sms;
  if (teams) ctas = (ctas + kRwWarps / r.wk - 1) / (kRwWarps / r.wk);
  const cudaError_t e = launch_pdl(teams ? linear_rows_kernel<MT, FT, NS, true> : linear_rows_kernel<MT, FT, NS, false>,
                                   dim3(ctas), dim3(kRwWarps * 32), 0, s, r);
  return e == cudaSuccess ? SWAPNET_OK : SWAPNET_ERR_CUDA;
}
template <int MT, int FT> int rows_launch(const SkJob& j, cudaStream_t s) {
  return j.nseg > 1 ? rows_launch_ns<MT, FT, kSkMaxSeg>(j, s) : rows_launch_ns<MT, FT, 1>(j, s);
}

template <typename T, int MT, bool TEAMS> int gemv_launch_as(const SkJob& j, int groups, int wk, cudaStream_t s) {
  const int teams = kGvWarps / wk;
  const int grid = std::max(1, std::min((groups + teams - 1) / teams, gv_ctas(MT) * std::max(1, j.num_sms)));
  const cudaError_t e = launch_pdl(gemv_kernel<T, MT, TEAMS>, dim3(grid), dim3(kGvWarps * 32), 0, s, j, groups, wk);
  return e == cudaSuccess ? SWAPNET_OK : SWAPNET_ERR_CUDA;
}
// Teams pay from more groups than SMs on, of fp32 from twice as many: 1 row of
// 512 bf16, 2432 features (304 groups) 2.11 us without, 1.86 with; 1024 (128
// groups) 1.70 and 1.84; 1 row of 308 fp32, 2093 features 1.75 and 1.95, of 256,
// 3648 features 2.19 and 1.96.
template <typename T, int MT> int gemv_launch(const SkJob& j, int groups, cudaStream_t s) {
  int wk = 1;  // warps that a row needs
  while (wk < kGvWarps && wk * 32 * Vec16<T>::N < j.K) wk *= 2;
  return wk < kGvWarps && groups > (sizeof(T) == 4 ? 2 : 1) * j.num_sms ? gemv_launch_as<T, MT, true>(j, groups, wk, s)
                                             : gemv_launch_as<T, MT, false>(j, groups, kGvWarps, s);
}

template <typename T> int skinny_dispatch(const SkJob& j, cudaStream_t s) {
  if constexpr (sizeof(T) == 4) {
    if (j.M == 2 && j.K > 512 && rows_ctas(j, 8) > 2 * j.num_sms) return rows_launch<2, 16>(j, s);
    if (j.M > 1) return j.M <= 4 ? rows_launch<4, 8>(j, s) : (j.M <= 8 ? rows_launch<8, 8>(j, s) : rows_launch<16, 4>(j, s));
  }
  const int per = j.pair ? kGvRows / 2 : kGvRows;
  int groups = (j.seg[0].N + per - 1) / per;
  if (!j.pair)
    for (int i = 1; i < j.nseg; ++i) groups += (j.seg[i].N + per - 1) / per;
  if (j.M <= 1) return gemv_launch<T, 1>(j, groups, s);
  if constexpr (sizeof(T) == 2) {  // (fp32 layers of more rows have been launched above)
    if (j.M <= 2) return gemv_launch<T, 2>(j, groups, s);
    if (j.M <= 4) return gemv_launch<T, 4>(j, groups, s);
  }
  // 16-bit layers of 5 rows and more run on the tensor cores
  SN_FAIL(SWAPNET_ERR_UNSUPPORTED, "skinny linear: more rows than the GEMV takes");
}

// ------------------------------------------------------------ tiled linear
// General fallback for any M, K, N and dtype (fp32 rows beyond the skinny
// kernel's 16, 16-bit layers whose K the other kernels do not take): one
// TM x TN output tile per CTA, fp32 FMAs.  K is walked in chunks of BK that
// cp.async brings into a ring of kTlStages stages (the weights' first stages
// before the programmatic wait), rows as they lie in memory, padded by four
// floats so that eight rows' 16-byte pieces fall on different banks.  A
// chunk's k are shared out to KG groups of threads; each thread keeps RM x RN
// outputs of its group's sum, two partial sums (even and odd k) per output in
// one packed fma.rn.f32x2.  At the end the groups' sums are added in group
// order through shared memory, so a result does not depend on scheduling.
//
// What bounds it: for the batches it serves (17 to a few hundred rows) the
// parallelism, hence two tiles: 32 x 32 with K split 8 ways inside the CTA
// for up to 127 tiles of 64 x 64, 64 x 64 (K split in two) from there on.
// 100 x 1000 x 1000 fp32: 91 us with 64 x 64 tiles of 16 k per step, loaded and
// waited for element by element; 12.4 us now (40.3 with the wide tiles).  By
// count, its reads of shared memory, 12 of 16 bytes per 64 packed FMAs of a
// thread, take about 6 of them.
constexpr int kTlStages = 4;
constexpr int kTlThreads = 256;
// 64 x 64 tiles from which they are taken: wide against narrow 39.0 and 29.7 us
// at 112 tiles (256 x 1024 x 1792), 38.9 and 38.5 at 128 (256 x 1024 x 2048),
// 20.7 and 21.1 (64 x 512 x 8192), 52.3 and 55.3 at 132 (700 x 1023 x 768), 12.8
// and 14.5 at 136 (512 x 260 x 1029).  (With a second round of wide tiles, from
// 153 on, the narrow ones are faster again at first: 53.6 and 39.5 at 160.)
constexpr int kTlWideTiles = 128;

template <int TM, int TN, int RM, int RN, int BK> struct TlCfg {
  static constexpr int kCols = TM / RM;                     // threads along M in a group
  static constexpr int kGroup = kCols * (TN / RN);          // threads per k group
  static constexpr int KG = kTlThreads / kGroup;
  static constexpr int kRow = BK + 4;                       // floats per staged row
  static constexpr int kStage = (TM + TN) * kRow;           // floats per stage
  static constexpr int kPartRow = TN + 4;
  static constexpr int kSmem = 4 * (kTlStages * kStage > KG * TM * kPartRow ? kTlStages * kStage : KG * TM * kPartRow);
  static_assert(BK % (4 * KG) == 0 && TM * (BK / 4) % kTlThreads == 0 && TN * (BK / 4) % kTlThreads == 0, "shares");
};

__device__ __forceinline__ void cp_async_4(uint32_t dst, const void* src, bool valid) {
  const int n = valid ? 4 : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}

// acc.xy += a.xy * b.xy, both halves rounded as a scalar FMA would.
__device__ __forceinline__ void fma2(uint64_t& acc, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

// Four consecutive k of row r (of `rows`) of a row-major matrix into shared
// memory; zeros past the matrix.  vec: rows are 16-byte aligned (fp32).
template <typename T>
__device__ __forceinline__ void tl_load4(uint32_t dst, const T* base, int r, int rows, int k, int K, bool vec) {
  const T* src = base + (int64_t)r * K + k;
  if constexpr (sizeof(T) == 4) {
    if (vec) {
      const bool ok = r < rows && k < K;
      cp_async_16(dst, ok ? src : base, ok);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const bool ok = r < rows && k + j < K;
        cp_async_4(dst + 4 * j, ok ? src + j : base, ok);
      }
    }
  } else {
    float f[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) f[j] = r < rows && k + j < K ? to_f<T>(src[j]) : 0.f;
    asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(dst), "f"(f[0]), "f"(f[1]), "f"(f[2]), "f"(f[3])
                 : "memory");
  }
}

template <typename T, int TM, int TN, int RM, int RN, int BK>
__global__ void __launch_bounds__(kTlThreads, 2) linear_tiled_kernel(const T* x, int M, int K,
                                                                     const T* __restrict__ W, int N, Epi e,
                                                                     T* __restrict__ y, int64_t ldy, int vec) {
  using C = TlCfg<TM, TN, RM, RN, BK>;
  extern __shared__ __align__(16) float tl_smem[];
  const int tid = threadIdx.x;
  const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
  const int chunks = (K + BK - 1) / BK;
  const uint32_t base = smem_u32(tl_smem);
  auto load_x = [&](int c) {
    const uint32_t st = base + (uint32_t)((c % kTlStages) * C::kStage * 4);
#pragma unroll
    for (int i = tid; i < TM * (BK / 4); i += kTlThreads) {
      const int r = i / (BK / 4), q = i % (BK / 4);
      tl_load4<T>(st + (uint32_t)(r * C::kRow + 4 * q) * 4, x, m0 + r, M, c * BK + 4 * q, K, vec);
    }
  };
  auto load_w = [&](int c) {
    const uint32_t st = base + (uint32_t)((c % kTlStages) * C::kStage * 4);
#pragma unroll
    for (int i = tid; i < TN * (BK / 4); i += kTlThreads) {
      const int r = i / (BK / 4), q = i % (BK / 4);
      tl_load4<T>(st + (uint32_t)((TM + r) * C::kRow + 4 * q) * 4, W, n0 + r, N, c * BK + 4 * q, K, vec);
    }
  };
  // the weights do not depend on the kernel before
  for (int c = 0; c < kTlStages - 1 && c < chunks; ++c) load_w(c);
  pdl_wait();
  pdl_launch_dependents();
  for (int c = 0; c < kTlStages - 1; ++c) {
    if (c < chunks) load_x(c);
    cp_async_commit();
  }
  const int g = tid / C::kGroup, tg = tid % C::kGroup;
  const int tm = tg % C::kCols, tn = tg / C::kCols;
  uint64_t acc[RM][RN];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) acc[i][j] = 0ull;
  for (int c = 0; c < chunks; ++c) {
    cp_async_wait<kTlStages - 2>();
    __syncthreads();  // chunk c has landed for every thread; the stage refilled below is no longer read
    const int cn = c + kTlStages - 1;
    if (cn < chunks) {
      load_w(cn);
      load_x(cn);
    }
    cp_async_commit();
    const float* st = tl_smem + (c % kTlStages) * C::kStage + g * (BK / C::KG);
#pragma unroll
    for (int kk = 0; kk < BK / C::KG; kk += 4) {
      ulonglong2 a[RM];
#pragma unroll
      for (int i = 0; i < RM; ++i)
        a[i] = *reinterpret_cast<const ulonglong2*>(st + (tm + i * C::kCols) * C::kRow + kk);
#pragma unroll
      for (int j = 0; j < RN; ++j) {
        const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(st + (TM + tn + j * (TN / RN)) * C::kRow + kk);
#pragma unroll
        for (int i = 0; i < RM; ++i) {
          fma2(acc[i][j], a[i].x, b.x);
          fma2(acc[i][j], a[i].y, b.y);
        }
      }
    }
  }
  cp_async_wait<0>();
  __syncthreads();
  // the groups' sums, added in group order
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j)
      tl_smem[(g * TM + tm + i * C::kCols) * C::kPartRow + tn + j * (TN / RN)] =
          __uint_as_float((uint32_t)acc[i][j]) + __uint_as_float((uint32_t)(acc[i][j] >> 32));
  __syncthreads();
  const T* bias = static_cast<const T*>(e.bias);
  const T* res = static_cast<const T*>(e.res);
#pragma unroll 1
  for (int i = tid; i < TM * (TN / 4); i += kTlThreads) {
    const int r = i / (TN / 4), q = i % (TN / 4);
    const int m = m0 + r, n = n0 + 4 * q;
    if (m >= M) continue;
    float4 s = *reinterpret_cast<const float4*>(tl_smem + r * C::kPartRow + 4 * q);
#pragma unroll
    for (int h = 1; h < C::KG; ++h) {
      const float4 v = *reinterpret_cast<const float4*>(tl_smem + (h * TM + r) * C::kPartRow + 4 * q);
      s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    const float v[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (n + j >= N) continue;
      const float rv = res ? to_f<T>(res[(int64_t)m * e.ldr + n + j]) : 0.f;
      y[(int64_t)m * ldy + n + j] =
          from_f<T>(epilogue(v[j], bias ? to_f<T>(bias[n + j]) : 0.f, rv, res != nullptr, e.act, e.res_post));
    }
  }
}

template <typename T, int TM, int TN, int RM, int RN, int BK>
int tiled_launch(const T* x, int M, int K, const T* W, int N, const Epi& e, T* y, int64_t ldy, int vec, cudaStream_t s) {
  using C = TlCfg<TM, TN, RM, RN, BK>;
  static std::atomic<uint64_t> attr_done{0};  // per instantiation, one bit per device
  auto kern = linear_tiled_kernel<T, TM, TN, RM, RN, BK>;
  if (attr_needed(attr_done)) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmem) != cudaSuccess)
      SN_FAIL(SWAPNET_ERR_CUDA, "cudaFuncSetAttribute failed");
    attr_set(attr_done);
  }
  launch_pdl(kern, dim3((N + TN - 1) / TN, (M + TM - 1) / TM), dim3(kTlThreads), (size_t)C::kSmem, s, x, M, K, W, N, e, y,
             ldy, vec);
  return SWAPNET_OK;
}

// ------------------------------------------------------------ direct conv
// Thread = one output pixel x 16 output channels.  The CTA's 16 filters are
// staged in shared memory as fp32, laid out [tap][cin][16] so each input
// value meets 16 weights read as four broadcast float4 loads.  Used for
// channel counts the tensor-core path cannot tile (e.g. a 3-channel image).
constexpr int kDcCo = 16;

template <typename T>
__global__ void __launch_bounds__(128) conv_direct_kernel(const T* x, int n, int h, int w, int cin,
                                                          const T* __restrict__ W, int cout, int kh, int kw,
                                                          int stride, int pad, int oh, int ow, Epi e,
                                                          T* __restrict__ y) {
  extern __shared__ float ws[];  // [kh*kw*cin][kDcCo]
  const int co0 = blockIdx.y * kDcCo;
  const int taps = kh * kw * cin;
  for (int i = threadIdx.x; i < taps * kDcCo; i += blockDim.x) {
    const int j = i % kDcCo, tc = i / kDcCo;  // tc = (r*kw + s)*cin + c
    const int co = co0 + j;
    ws[i] = co < cout ? to_f<T>(W[(int64_t)co * taps + tc]) : 0.f;
  }
  pdl_wait();  // the filters come from the arena; the input from the previous kernel
  pdl_launch_dependents();
  __syncthreads();
  const int64_t pix = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t npix = (int64_t)n * oh * ow;
  if (pix >= npix) return;
  const int img = (int)(pix / ((int64_t)oh * ow));
  const int rem = (int)(pix % ((int64_t)oh * ow));
  const int oy = rem / ow, ox = rem % ow;
  float acc[kDcCo];
#pragma unroll
  for (int j = 0; j < kDcCo; ++j) acc[j] = 0.f;
  for (int r = 0; r < kh; ++r) {
    const int iy = oy * stride + r - pad;
    if (iy < 0 || iy >= h) continue;
    for (int s = 0; s < kw; ++s) {
      const int ix = ox * stride + s - pad;
      if (ix < 0 || ix >= w) continue;
      const T* xp = x + (((int64_t)img * h + iy) * w + ix) * cin;
      const float4* wp = reinterpret_cast<const float4*>(ws + (int64_t)((r * kw + s) * cin) * kDcCo);
      for (int c = 0; c < cin; ++c) {
        const float xv = to_f<T>(xp[c]);
#pragma unroll
        for (int q = 0; q < kDcCo / 4; ++q) {
          const float4 wv = wp[c * (kDcCo / 4) + q];
          acc[4 * q + 0] = fmaf(xv, wv.x, acc[4 * q + 0]);
          acc[4 * q + 1] = fmaf(xv, wv.y, acc[4 * q + 1]);
          acc[4 * q + 2] = fmaf(xv, wv.z, acc[4 * q + 2]);
          acc[4 * q + 3] = fmaf(xv, wv.w, acc[4 * q + 3]);
        }
      }
    }
  }
  const T* bias = reinterpret_cast<const T*>(e.bias);
  const T* res = reinterpret_cast<const T*>(e.res);
#pragma unroll
  for (int j = 0; j < kDcCo; ++j) {
    const int co = co0 + j;
    if (co < cout) {
      const float rv = res ? to_f<T>(res[pix * e.ldr + co]) : 0.f;
      y[pix * cout + co] =
        from_f<T>(epilogue(acc[j], bias ? to_f<T>(bias[co]) : 0.f, rv, res != nullptr, e.act, e.res_post));
    }
  }
}

// ------------------------------------------------------------ pooling etc.
template <typename T>
__global__ void maxpool_kernel(const T* x, int n, int h, int w, int c, int kh, int kw, int stride,
                               int pad, int oh, int ow, T* __restrict__ y) {
  pdl_wait();
  pdl_launch_dependents();
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t total = (int64_t)n * oh * ow * c;
  if (idx >= total) return;
  const int ch = (int)(idx % c);
  const int64_t p = idx / c;
  const int ox = (int)(p % ow);
  const int oy = (int)((p / ow) % oh);
  const int img = (int)(p / ((int64_t)ow * oh));
  float m = -INFINITY;
  for (int r = 0; r < kh; ++r) {
    const int iy = oy * stride + r - pad;
    if (iy < 0 || iy >= h) continue;
    for (int s = 0; s < kw; ++s) {
      const int ix = ox * stride + s - pad;
      if (ix < 0 || ix >= w) continue;
      m = fmaxf(m, to_f<T>(x[(((int64_t)img * h + iy) * w + ix) * c + ch]));
    }
  }
  y[idx] = from_f<T>(m);
}

template <typename T>
__global__ void gap_kernel(const T* x, int n, int hw, int c, T* __restrict__ y) {
  pdl_wait();
  pdl_launch_dependents();
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)n * c) return;
  const int img = (int)(idx / c), ch = (int)(idx % c);
  const T* p = x + (int64_t)img * hw * c + ch;
  float s = 0.f;
  for (int i = 0; i < hw; ++i) s += to_f<T>(p[(int64_t)i * c]);
  y[idx] = from_f<T>(s / (float)hw);
}

template <typename T>
__global__ void upsample2x_kernel(const T* x, int n, int h, int w, int c, T* __restrict__ y) {
  pdl_wait();
  pdl_launch_dependents();
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t total = (int64_t)n * 2 * h * 2 * w * c;
  if (idx >= total) return;
  const int ch = (int)(idx % c);
  const int64_t p = idx / c;
  const int ox = (int)(p % (2 * w));
  const int oy = (int)((p / (2 * w)) % (2 * h));
  const int img = (int)(p / ((int64_t)4 * w * h));
  y[idx] = x[(((int64_t)img * h + oy / 2) * w + ox / 2) * c + ch];
}

template <typename T>
__global__ void concat_kernel(const T* a, int ca, const T* b, int cb, int64_t pixels,
                              T* __restrict__ y) {
  pdl_wait();
  pdl_launch_dependents();
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int c = ca + cb;
  if (idx >= pixels * c) return;
  const int64_t p = idx / c;
  const int ch = (int)(idx % c);
  y[idx] = ch < ca ? a[p * ca + ch] : b[p * cb + (ch - ca)];
}

// Vectorised variants: a thread handles 16 bytes of channels (channels a
// multiple of the vector width, rows 16-byte aligned).  Max is exact, so
// the result equals the scalar kernels'.
template <typename T>
__global__ void maxpool_vec_kernel(const uint4* x, int n, int h, int w, int cv, int kh, int kw,
                                   int stride, int pad, int oh, int ow, uint4* __restrict__ y) {
  constexpr int V = Vec16<T>::N;
  pdl_wait();
  pdl_launch_dependents();
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t total = (int64_t)n * oh * ow * cv;
  if (idx >= total) return;
  const int ch = (int)(idx % cv);
  const int64_t p = idx / cv;
  const int ox = (int)(p % ow);
  const int64_t q = p / ow;
  const int oy = (int)(q % oh);
  const int img = (int)(q / oh);
  float m[V];
#pragma unroll
  for (int i = 0; i < V; ++i) m[i] = -INFINITY;
  // four taps' loads in flight at a time
  const int taps = kh * kw;
  int r = 0, t = 0;
  for (int k = 0; k < taps; k += 4) {
    uint4 v[4];
    bool ok[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int iy = oy * stride + r - pad, ix = ox * stride + t - pad;
      ok[u] = k + u < taps && (unsigned)iy < (unsigned)h && (unsigned)ix < (unsigned)w;
      if (ok[u]) v[u] = x[(((int64_t)img * h + iy) * w + ix) * cv + ch];
      if (++t == kw) {
        t = 0;
        ++r;
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (!ok[u]) continue;
      float f[V];
      unpack16<T>(v[u], f);
#pragma unroll
      for (int i = 0; i < V; ++i) m[i] = fmaxf(m[i], f[i]);
    }
  }
  y[idx] = pack16<T>(m);
}

__global__ void upsample2x_vec_kernel(const uint4* x, int n, int h, int w, int cv,
                                      uint4* __restrict__ y) {
  pdl_wait();
  pdl_launch_dependents();
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t total = (int64_t)n * 2 * h * 2 * w * cv;
  if (idx >= total) return;
  const int ch = (int)(idx % cv);
  const int64_t p = idx / cv;
  const int ox = (int)(p % (2 * w));
  const int64_t q = p / (2 * w);
  const int oy = (int)(q % (2 * h));
  const int img = (int)(q / (2 * h));
  y[idx] = x[(((int64_t)img * h + oy / 2) * w + ox / 2) * cv + ch];
}

__global__ void concat_vec_kernel(const uint4* a, int ca, const uint4* b, int cb,
                                  int64_t pixels, uint4* __restrict__ y) {
  pdl_wait();
  pdl_launch_dependents();
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int c = ca + cb;
  if (idx >= pixels * c) return;
  const int64_t p = idx / c;
  const int ch = (int)(idx % c);
  y[idx] = ch < ca ? a[p * ca + ch] : b[p * cb + (ch - ca)];
}

inline int grid1d(int64_t total, int block) { return (int)((total + block - 1) / block); }



}  // namespace

#define SN_DISPATCH(dtype, T, ...)                    \
  switch (dtype) {                                    \
    case SWAPNET_F32: { using T = float; __VA_ARGS__; break; }          \
    case SWAPNET_F16: { using T = __half; __VA_ARGS__; break; }         \
    case SWAPNET_BF16: { using T = __nv_bfloat16; __VA_ARGS__; break; } \
    default: return SWAPNET_ERR_INVALID_ARG;          \
  }

static int last_launch() {
  const cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) {
    set_error(std::string("kernel launch: ") + cudaGetErrorString(err));
    return SWAPNET_ERR_CUDA;
  }
  return SWAPNET_OK;
}

int launch_linear_skinny_job(int dtype, const SkJob& j, cudaStream_t s) {
  const int es = dtype_size(dtype);
  if (j.M < 1 || j.M > 16 || j.K < 1 || j.nseg < 1 || j.nseg > kSkMaxSeg || (j.pair && j.nseg != 2))
    SN_FAIL(SWAPNET_ERR_UNSUPPORTED, "skinny linear: M must be in [1, 16], 1 to 3 layers");
  if ((j.K * es) % 16 || (uintptr_t)j.x % 16) SN_FAIL(SWAPNET_ERR_MISALIGNED, "skinny linear: rows must be 16-byte aligned");
  for (int i = 0; i < j.nseg; ++i) {
    if (j.seg[i].N < 1) SN_FAIL(SWAPNET_ERR_UNSUPPORTED, "skinny linear: no output features");
    if ((uintptr_t)j.seg[i].W % 16) SN_FAIL(SWAPNET_ERR_MISALIGNED, "skinny linear: rows must be 16-byte aligned");
  }
  if (j.pair && j.seg[0].N != j.seg[1].N) SN_FAIL(SWAPNET_ERR_UNSUPPORTED, "skinny linear: paired layers differ in width");
  SN_DISPATCH(dtype, T, return skinny_dispatch<T>(j, s));
  return SWAPNET_OK;
}

int launch_linear_skinny(int dtype, const void* x, int M, int K, const void* W, int N, const Epi& e, void* y,
                         int64_t ldy, int num_sms, cudaStream_t s) {
  SkJob j{};
  j.x = x;
  j.M = M;
  j.K = K;
  j.nseg = 1;
  j.seg[0] = SkSeg{W, N, e, y, ldy};
  j.num_sms = num_sms;
  return launch_linear_skinny_job(dtype, j, s);
}

int launch_linear_tiled(int dtype, const void* x, int M, int K, const void* W, int N, int N_layer, const Epi& e, void* y,
                        int64_t ldy, cudaStream_t s) {
  if (M < 1 || K < 1 || N < 1) SN_FAIL(SWAPNET_ERR_INVALID_ARG, "tiled linear: empty shape");
  // 16-byte copies need 16-byte aligned fp32 rows
  const int vec = dtype == SWAPNET_F32 && K % 4 == 0 && (((uintptr_t)x | (uintptr_t)W) & 15) == 0;
  // 64 x 64 tiles once they give most SMs one.  The two tiles share K out
  // differently, so the choice follows the whole layer's width: a column
  // piece of a layer sums each output as the whole layer would
  const int64_t tiles = (int64_t)((M + 63) / 64) * ((N_layer + 63) / 64);
  int rc = SWAPNET_OK;
  SN_DISPATCH(dtype, T, {
    const T* xt = static_cast<const T*>(x);
    const T* wt = static_cast<const T*>(W);
    if (tiles >= kTlWideTiles) rc = tiled_launch<T, 64, 64, 8, 4, 32>(xt, M, K, wt, N, e, static_cast<T*>(y), ldy, vec, s);
    else rc = tiled_launch<T, 32, 32, 4, 8, 64>(xt, M, K, wt, N, e, static_cast<T*>(y), ldy, vec, s);
  });
  if (rc) return rc;
  return last_launch();
}

int launch_conv_direct(int dtype, const void* x, int n, int h, int w, int cin, const void* W, int cout, int kh,
                       int kw, int stride, int pad, int oh, int ow, const Epi& e, void* y, cudaStream_t s) {
  const int64_t npix = (int64_t)n * oh * ow;
  const size_t smem = (size_t)kh * kw * cin * kDcCo * sizeof(float);
  if (smem > 200 * 1024) SN_FAIL(SWAPNET_ERR_UNSUPPORTED, "direct conv: filter too large for shared memory");
  const dim3 grid(grid1d(npix, 128), (cout + kDcCo - 1) / kDcCo);
  SN_DISPATCH(dtype, T, {
    auto kern = conv_direct_kernel<T>;
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
      SN_FAIL(SWAPNET_ERR_CUDA, "cudaFuncSetAttribute failed");
    launch_pdl(kern, grid, dim3(128), smem, s, static_cast<const T*>(x), n, h, w, cin, static_cast<const T*>(W), cout,
               kh, kw, stride, pad, oh, ow, e, static_cast<T*>(y));
  });
  return last_launch();
}

int launch_maxpool(int dtype, const void* x, int n, int h, int w, int c, int kh, int kw, int stride, int pad,
                   int oh, int ow, void* y, cudaStream_t s) {
  SN_DISPATCH(dtype, T, {
    constexpr int V = Vec16<T>::N;
    if (c % V == 0 && ((uintptr_t)x | (uintptr_t)y) % 16 == 0) {
      const int64_t tv = (int64_t)n * oh * ow * (c / V);
      launch_pdl(maxpool_vec_kernel<T>, dim3(grid1d(tv, 256)), dim3(256), 0, s, static_cast<const uint4*>(x), n, h,
                 w, c / V, kh, kw, stride, pad, oh, ow, static_cast<uint4*>(y));
      return last_launch();
    }
  });
  const int64_t total = (int64_t)n * oh * ow * c;
  SN_DISPATCH(dtype, T,
              launch_pdl(maxpool_kernel<T>, dim3(grid1d(total, 256)), dim3(256), 0, s, static_cast<const T*>(x), n, h,
                         w, c, kh, kw, stride, pad, oh, ow, static_cast<T*>(y)));
  return last_launch();
}

int launch_gap(int dtype, const void* x, int n, int h, int w, int c, void* y, cudaStream_t s) {
  SN_DISPATCH(dtype, T,
              launch_pdl(gap_kernel<T>, dim3(grid1d((int64_t)n * c, 256)), dim3(256), 0, s, static_cast<const T*>(x),
                         n, h * w, c, static_cast<T*>(y)));
  return last_launch();
}

int launch_upsample2x(int dtype, const void* x, int n, int h, int w, int c, void* y, cudaStream_t s) {
  {
    const int es = dtype == SWAPNET_F32 ? 4 : 2;
    if ((c * es) % 16 == 0 && ((uintptr_t)x | (uintptr_t)y) % 16 == 0) {
      const int cv = c * es / 16;
      launch_pdl(upsample2x_vec_kernel, dim3(grid1d((int64_t)n * 4 * h * w * cv, 256)), dim3(256), 0, s,
                 static_cast<const uint4*>(x), n, h, w, cv, static_cast<uint4*>(y));
      return last_launch();
    }
  }
  const int64_t total = (int64_t)n * 4 * h * w * c;
  SN_DISPATCH(dtype, T,
              launch_pdl(upsample2x_kernel<T>, dim3(grid1d(total, 256)), dim3(256), 0, s, static_cast<const T*>(x), n,
                         h, w, c, static_cast<T*>(y)));
  return last_launch();
}

int launch_concat(int dtype, const void* a, int ca, const void* b, int cb, int64_t pixels, void* y,
                  cudaStream_t s) {
  {
    const int es = dtype == SWAPNET_F32 ? 4 : 2;
    if ((ca * es) % 16 == 0 && (cb * es) % 16 == 0 && ((uintptr_t)a | (uintptr_t)b | (uintptr_t)y) % 16 == 0) {
      const int av = ca * es / 16, bv = cb * es / 16;
      launch_pdl(concat_vec_kernel, dim3(grid1d(pixels * (av + bv), 256)), dim3(256), 0, s,
                 static_cast<const uint4*>(a), av, static_cast<const uint4*>(b), bv, pixels,
                 static_cast<uint4*>(y));
      return last_launch();
    }
  }
  const int64_t total = pixels * (ca + cb);
  SN_DISPATCH(dtype, T,
              launch_pdl(concat_kernel<T>, dim3(grid1d(total, 256)), dim3(256), 0, s, static_cast<const T*>(a), ca,
                         static_cast<const T*>(b), cb, pixels, static_cast<T*>(y)));
  return last_launch();
}

}  // namespace swapnet
