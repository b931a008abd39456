// Decoder-layer kernels: embedding gather (zero-copy from the host-resident
// table), RMSNorm, RoPE + KV-cache append, causal attention for short query
// runs (the decode step: keys split over a thread-block cluster), row argmax,
// and the device-side advance of the cache position.
// bf16 / fp16 storage, fp32 arithmetic, fixed reduction orders.
#include <cooperative_groups.h>

#include <algorithm>
#include <cstring>

#include "device.cuh"
#include "internal.h"
#include "kernels.h"

namespace swapnet {

namespace cg = cooperative_groups;

namespace {

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

int done(cudaError_t e, const char* what) {
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) SN_FAIL(SWAPNET_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
  return SWAPNET_OK;
}

// ------------------------------------------------------------ embedding
// Row t of the output is row ids[t] of the table, read straight from the
// page-locked host table (device alias) with 16-byte loads.
template <typename T>
__global__ void __launch_bounds__(256) embed_kernel(const T* __restrict__ table, const int* ids,
                                                    int vocab, int d, T* __restrict__ out, int* err) {
  pdl_wait();
  pdl_launch_dependents();
  const int t = blockIdx.x;
  const int id = ids[t];
  const bool ok = id >= 0 && id < vocab;
  if (!ok && threadIdx.x == 0) atomicExch(err, kDevErrBounds);
  const uint4* src = reinterpret_cast<const uint4*>(table + (int64_t)(ok ? id : 0) * d);
  uint4* dst = reinterpret_cast<uint4*>(out + (int64_t)t * d);
  const int n16 = d * (int)sizeof(T) / 16;
  for (int i = threadIdx.x; i < n16; i += blockDim.x) dst[i] = ok ? src[i] : make_uint4(0, 0, 0, 0);
}

// ------------------------------------------------------------ RMSNorm
// One CTA per row; the sum of squares is reduced in a fixed order (each
// thread's elements in index order, warp butterfly, warps in index order).
// Rows of whole 16-byte chunks are read once into registers (up to
// kNormKeep chunks per thread, the rest read again for the scaling pass).
constexpr int kNormThreads = 256;
constexpr int kNormKeep = 4;

template <typename T> struct Chunk8 {
  static_assert(sizeof(T) == 2, "16-bit element types");
  __device__ static void unpack(const uint4& v, float* f) {
    const T* e = reinterpret_cast<const T*>(&v);
#pragma unroll
    for (int i = 0; i < 8; ++i) f[i] = to_f<T>(e[i]);
  }
  __device__ static uint4 pack(const float* f) {
    uint4 v;
    T* e = reinterpret_cast<T*>(&v);
#pragma unroll
    for (int i = 0; i < 8; ++i) e[i] = from_f<T>(f[i]);
    return v;
  }
};

template <typename T>
__global__ void __launch_bounds__(kNormThreads) rmsnorm_kernel(const T* x, const T* __restrict__ g,
                                                               int d, float eps, T* __restrict__ y, int vec) {
  __shared__ float wsum[kNormThreads / 32];
  pdl_wait();
  pdl_launch_dependents();
  const T* xr = x + (int64_t)blockIdx.x * d;
  T* yr = y + (int64_t)blockIdx.x * d;
  const int t = threadIdx.x;
  float s = 0.f;
  uint4 keep[kNormKeep];
  const int nc = d / 8;
  if (vec) {
    const uint4* xv = reinterpret_cast<const uint4*>(xr);
#pragma unroll
    for (int j = 0; j < kNormKeep; ++j) {
      const int c = t + j * kNormThreads;
      keep[j] = c < nc ? xv[c] : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int j = 0; j < kNormKeep; ++j) {
      float f[8];
      Chunk8<T>::unpack(keep[j], f);
#pragma unroll
      for (int i = 0; i < 8; ++i) s = fmaf(f[i], f[i], s);
    }
    for (int c = t + kNormKeep * kNormThreads; c < nc; c += kNormThreads) {
      float f[8];
      Chunk8<T>::unpack(xv[c], f);
#pragma unroll
      for (int i = 0; i < 8; ++i) s = fmaf(f[i], f[i], s);
    }
  } else {
    for (int i = t; i < d; i += kNormThreads) {
      const float v = to_f<T>(xr[i]);
      s = fmaf(v, v, s);
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if ((t & 31) == 0) wsum[t >> 5] = s;
  __syncthreads();
  float tot = 0.f;
#pragma unroll
  for (int w = 0; w < kNormThreads / 32; ++w) tot += wsum[w];
  const float r = 1.0f / sqrtf(tot / (float)d + eps);
  if (vec) {
    const uint4* xv = reinterpret_cast<const uint4*>(xr);
    const uint4* gv = reinterpret_cast<const uint4*>(g);
    uint4* yv = reinterpret_cast<uint4*>(yr);
    auto scale = [&](int c, const uint4& xc) {
      float f[8], gf[8], o[8];
      Chunk8<T>::unpack(xc, f);
      Chunk8<T>::unpack(gv[c], gf);
#pragma unroll
      for (int i = 0; i < 8; ++i) o[i] = f[i] * r * gf[i];
      yv[c] = Chunk8<T>::pack(o);
    };
#pragma unroll
    for (int j = 0; j < kNormKeep; ++j)
      if (t + j * kNormThreads < nc) scale(t + j * kNormThreads, keep[j]);
    for (int c = t + kNormKeep * kNormThreads; c < nc; c += kNormThreads) scale(c, xv[c]);
  } else {
    for (int i = t; i < d; i += kNormThreads) yr[i] = from_f<T>(to_f<T>(xr[i]) * r * to_f<T>(g[i]));
  }
}

// ------------------------------------------------------------ RoPE + cache
// Thread = NP adjacent pairs (2i, 2i+1) of HPT heads of one token: rotates q
// in place and k into the key cache at the state position, copies v into the
// value cache.  Angles: position * theta^(-2i/Dh), computed in fp32, once for
// the thread's heads.  A decode step takes one pair and head per thread (its
// time is one chain of loads, power and sine), long runs four pairs (16
// bytes) of four heads: 512 tokens of 32 heads 10.8 us with one pair and head
// per thread, 8.5 with four of four.
template <int NP> struct RopeVec;
template <> struct RopeVec<1> { using type = uint32_t; };
template <> struct RopeVec<4> { using type = uint4; };

template <typename T, int HPT, int NP>
__global__ void __launch_bounds__(128) rope_append_kernel(T* __restrict__ q, const T* k,
                                                          const T* v, T* __restrict__ kc,
                                                          T* __restrict__ vc, const int* pos_ptr,
                                                          int heads, int dh, float theta, int max_seq, int* err) {
  using Vec = typename RopeVec<NP>::type;
  const int t = blockIdx.y;
  const int chunks = dh / (2 * NP);  // chunks of NP pairs in a head
  const int id = blockIdx.x * blockDim.x + threadIdx.x;
  const int ch = id % chunks, h0 = id / chunks * HPT;
  float inv[NP];
#pragma unroll
  for (int u = 0; u < NP; ++u) inv[u] = powf(theta, -2.0f * (float)(ch * NP + u) / (float)dh);
  pdl_wait();
  // After the wait, in every CTA: both attention kernels (each launched right
  // behind this one) read the position and the cache rows of earlier runs
  // before their own wait, which only ends with this launch.
  pdl_launch_dependents();
  if (h0 >= heads) return;
  const int pos0 = *pos_ptr;
  if (pos0 < 0 || pos0 >= max_seq - t) {  // (no sum that could overflow)
    if (id == 0) atomicExch(err, kDevErrBounds);
    return;
  }
  const int pos = pos0 + t;
  const int width = heads * dh;
  Vec qv[HPT], kv[HPT], vv[HPT];
#pragma unroll
  for (int j = 0; j < HPT; ++j) {
    if (h0 + j < heads) {
      const int64_t col = (int64_t)t * width + (h0 + j) * dh + ch * 2 * NP;
      qv[j] = *reinterpret_cast<const Vec*>(q + col);
      kv[j] = *reinterpret_cast<const Vec*>(k + col);
      vv[j] = *reinterpret_cast<const Vec*>(v + col);
    }
  }
  float sn[NP], cs[NP];
#pragma unroll
  for (int u = 0; u < NP; ++u) sincosf((float)pos * inv[u], &sn[u], &cs[u]);
  auto rotate = [&](const Vec& x) {
    Vec y;
    const T* e = reinterpret_cast<const T*>(&x);
    T* r = reinterpret_cast<T*>(&y);
#pragma unroll
    for (int u = 0; u < NP; ++u) {
      const float a = to_f<T>(e[2 * u]), b = to_f<T>(e[2 * u + 1]);
      r[2 * u] = from_f<T>(a * cs[u] - b * sn[u]);
      r[2 * u + 1] = from_f<T>(a * sn[u] + b * cs[u]);
    }
    return y;
  };
#pragma unroll
  for (int j = 0; j < HPT; ++j) {
    if (h0 + j < heads) {
      const int64_t col = (h0 + j) * dh + ch * 2 * NP;
      *reinterpret_cast<Vec*>(q + (int64_t)t * width + col) = rotate(qv[j]);
      *reinterpret_cast<Vec*>(kc + (int64_t)pos * width + col) = rotate(kv[j]);
      *reinterpret_cast<Vec*>(vc + (int64_t)pos * width + col) = vv[j];
    }
  }
}

// ------------------------------------------------------------ attention
// Runs of many queries (the prefill) take the tcgen05 kernel (k_attn_tc.cu,
// attention_tc_supported).
//
// Short query runs (a decode step): the visible keys of one (query t,
// head h) are split into S consecutive chunks of `chunk` keys, one CTA per
// chunk, and the S CTAs of a (t, h) form a thread-block cluster.  Each CTA
// computes, over its chunk only (256 threads):
//   phase 1: scores s_j = q . k_j / sqrt(128): 16 threads per key, one
//            16-byte load each (8 head dims), summed over the 16 lanes in a
//            fixed butterfly order; 16 keys per pass, the loads of four
//            passes issued before their arithmetic;
//   phase 2: the chunk's max m_c, p_j = exp(s_j - m_c) and l_c = sum p_j
//            (block reductions in a fixed order);
//   phase 3: a_c[d] = sum_j p_j v_j[d]: thread (key group g, 8-dim slice)
//            over keys g, g + 16, ... with 16-byte loads (the first eight of
//            them issued before phase 1, so that they arrive during it),
//            then the two groups of each warp and the warps in index order.
// Every CTA leaves (m_c, l_c, a_c) in the shared memory of the cluster's
// first CTA, which after a cluster barrier combines them in chunk order:
// M = max m_c, L = sum l_c e^(m_c - M), out[d] = sum a_c[d] e^(m_c - M) / L
// (chunks past the visible keys hold l_c = 0 and are skipped).  The result is
// that of one exact softmax over all visible keys, with every sum in a fixed
// order.
// A decode step is bound by this chain of latencies (at 32 heads and 540
// keys its 8.9 MB would take 1.3 us).  The cache rows of earlier runs are
// requested while rope_append_kernel still runs: it lets this kernel start
// only after every launch before it has completed.  With the rotation, 32
// heads of 540 keys: 7.35 us with all loads after the wait and the results
// read by the first CTA one after the other, 6.7 with the results pushed,
// 5.75 with the early loads.  (The rotation within this launch: 6.9, and
// 4.5 us more inside a decode step, where its clusters can only be placed
// once the projections have left; the small rotation grid hides that.)
constexpr int kDh = 128;
constexpr int kSpThreads = 256;
constexpr int kSpMaxSplit = 8;      // portable cluster size
constexpr int kSpKeysPerPass = kSpThreads / 16;
constexpr int kSpVPre = 8;          // value rows per thread requested with the keys
constexpr int kRopeManyHeads = 4096;  // (token, head) pairs from which a RoPE thread takes four heads

struct SplitPlan {
  int split, chunk;
};

// Chunks of at least 64 keys (a multiple of 16), at most kSpMaxSplit of them.
inline SplitPlan split_plan(int max_seq) {
  int split = std::min(kSpMaxSplit, std::max(1, (max_seq + 63) / 64));
  int chunk = ((max_seq + split - 1) / split + 15) / 16 * 16;
  return SplitPlan{split, chunk};
}

__device__ __forceinline__ float sp_block_reduce(float v, float* red, bool is_max) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float o = __shfl_xor_sync(0xffffffffu, v, off);
    v = is_max ? fmaxf(v, o) : v + o;
  }
  __syncthreads();  // red is reused between calls
  if (lane == 0) red[warp] = v;
  __syncthreads();
  float r = red[0];
  for (int w = 1; w < kSpThreads / 32; ++w) r = is_max ? fmaxf(r, red[w]) : r + red[w];
  return r;
}

// Shared memory, in floats: one partial sum per warp, the cluster's a_c and
// (m_c, l_c) (used in the first CTA), the reductions' partials, the chunk's
// scores.
constexpr int kSpWarps = kSpThreads / 32;
constexpr int kSpPart = kSpWarps * kDh, kSpAcc = kSpMaxSplit * kDh;
constexpr int kSpFixed = kSpPart + kSpAcc + 2 * kSpMaxSplit + kSpWarps;

size_t attention_split_smem_bytes(int chunk) { return sizeof(float) * (kSpFixed + (size_t)chunk); }

template <typename T>
__global__ void __launch_bounds__(kSpThreads, 2)
    attention_split_kernel(const T* q, const T* kc, const T* vc, const int* pos_ptr, int width, int max_seq, int chunk,
                           T* out) {
  extern __shared__ __align__(16) float sp_smem[];
  float* part = sp_smem;
  float* acc = part + kSpPart;
  float* ml = acc + kSpAcc;
  float* red = ml + 2 * kSpMaxSplit;
  float* sc = red + kSpWarps;
  cg::cluster_group cluster = cg::this_cluster();
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");  // started: its shared memory may be written
  const int tid = threadIdx.x;
  const int c = (int)cluster.block_rank();
  const int split = (int)cluster.num_blocks();
  const int h = blockIdx.y, t = blockIdx.z;
  const int pos0 = min(*pos_ptr, max_seq);  // (a position outside the cache is reported by the rotation)
  const int n = min(pos0 + t + 1, max_seq);
  const int j0 = c * chunk, j1 = min(j0 + chunk, n);
  const int jo = min(j1, pos0);  // keys from pos0 on belong to this run
  const int64_t col = (int64_t)h * kDh;
  const int sl = tid & 15, kq = tid >> 4;
  const T* kcol = kc + col + sl * 8;
  const T* vcol = vc + col + sl * 8;
  const float scale = rsqrtf((float)kDh);
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  auto row = [&](const T* p, int j) { return *reinterpret_cast<const uint4*>(p + (int64_t)j * width); };
  // the first four passes of keys and the first kSpVPre value rows this
  // thread sums in phase 3 (keys kq, kq + 16, ... of the chunk both)
  uint4 ku[4], vpre[kSpVPre];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int j = j0 + kq + r * kSpKeysPerPass;
    ku[r] = j < jo ? row(kcol, j) : zero;
  }
#pragma unroll
  for (int r = 0; r < kSpVPre; ++r) {
    const int j = j0 + kq + r * 16;
    vpre[r] = j < jo ? row(vcol, j) : zero;
  }
  pdl_wait();
  pdl_launch_dependents();
  float m_c = -INFINITY, l_c = 0.f;
  if (j0 < j1) {
    // phase 1: lane group of 16 per key, 8 dims per thread
    float qv[8];
    {
      const uint4 u = *reinterpret_cast<const uint4*>(q + (int64_t)t * width + col + sl * 8);
      const T* e = reinterpret_cast<const T*>(&u);
#pragma unroll
      for (int i = 0; i < 8; ++i) qv[i] = to_f<T>(e[i]);
    }
    if (jo < j1) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int j = j0 + kq + r * kSpKeysPerPass;
        if (j >= jo && j < j1) ku[r] = row(kcol, j);
      }
#pragma unroll
      for (int r = 0; r < kSpVPre; ++r) {
        const int j = j0 + kq + r * 16;
        if (j >= jo && j < j1) vpre[r] = row(vcol, j);
      }
    }
    float mx = -INFINITY;
    for (int jb = j0; jb < j1; jb += 4 * kSpKeysPerPass) {
      if (jb > j0) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int j = jb + r * kSpKeysPerPass + kq;
          ku[r] = j < j1 ? row(kcol, j) : zero;
        }
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int j = jb + r * kSpKeysPerPass + kq;
        const T* e = reinterpret_cast<const T*>(&ku[r]);
        float sdot = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) sdot = fmaf(qv[i], to_f<T>(e[i]), sdot);
#pragma unroll
        for (int off = 8; off > 0; off >>= 1) sdot += __shfl_xor_sync(0xffffffffu, sdot, off);
        sdot *= scale;
        if (j < j1) {
          if (sl == 0) sc[j - j0] = sdot;
          mx = fmaxf(mx, sdot);
        }
      }
    }
    // phase 2
    m_c = sp_block_reduce(mx, red, true);
    float l = 0.f;
    for (int j = tid; j < j1 - j0; j += kSpThreads) {
      const float pj = expf(sc[j] - m_c);
      sc[j] = pj;
      l += pj;
    }
    l_c = sp_block_reduce(l, red, false);  // the barriers inside also publish sc[]
    // phase 3: key group kq, dims 8 * sl .. + 7
    float a[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) a[i] = 0.f;
    auto add = [&](const uint4& vv, int j) {
      if (j < j1) {
        const float pj = sc[j - j0];
        const T* e = reinterpret_cast<const T*>(&vv);
#pragma unroll
        for (int i = 0; i < 8; ++i) a[i] = fmaf(pj, to_f<T>(e[i]), a[i]);
      }
    };
#pragma unroll
    for (int r = 0; r < kSpVPre; ++r) add(vpre[r], j0 + kq + r * 16);
    for (int jb = j0 + kq + kSpVPre * 16; jb < j1; jb += 4 * 16) {
      uint4 vu[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) vu[r] = jb + r * 16 < j1 ? row(vcol, jb + r * 16) : zero;
#pragma unroll
      for (int r = 0; r < 4; ++r) add(vu[r], jb + r * 16);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) a[i] += __shfl_xor_sync(0xffffffffu, a[i], 16);
    if (tid % 32 < 16) {
      float4* pw = reinterpret_cast<float4*>(part + (tid >> 5) * kDh + sl * 8);
      pw[0] = make_float4(a[0], a[1], a[2], a[3]);
      pw[1] = make_float4(a[4], a[5], a[6], a[7]);
    }
    __syncthreads();
  }
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  if (j0 < j1 && tid < kDh) {
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < kSpWarps; ++w) sum += part[w * kDh + tid];
    cluster.map_shared_rank(acc, 0)[c * kDh + tid] = sum;
  }
  if (tid == 0) {
    float* rml = cluster.map_shared_rank(ml, 0) + 2 * c;
    rml[0] = m_c;
    rml[1] = l_c;
  }
  cluster.sync();  // every chunk's (m_c, l_c, a_c) is visible to the first CTA
  if (c != 0) return;
  if (tid < kDh) {
    float M = -INFINITY;
#pragma unroll
    for (int r = 0; r < kSpMaxSplit; ++r)
      if (r < split && ml[2 * r + 1] > 0.f) M = fmaxf(M, ml[2 * r]);
    float L = 0.f, o = 0.f;
#pragma unroll
    for (int r = 0; r < kSpMaxSplit; ++r) {
      if (r < split && ml[2 * r + 1] > 0.f) {
        const float w = expf(ml[2 * r] - M);
        L += ml[2 * r + 1] * w;
        o += acc[r * kDh + tid] * w;
      }
    }
    out[(int64_t)t * width + col + tid] = from_f<T>(o / L);
  }
}

// ------------------------------------------------------------ argmax
// One CTA per row.  Each thread scans its elements in index order keeping
// the first maximum; threads, then warps, are combined by (larger value,
// then smaller index), an order-independent rule, so ties go to the
// lowest index.  Rows of whole 16-byte chunks are read kArgBatch chunks
// per thread at a time.
constexpr int kArgThreads = 1024;
constexpr int kArgBatch = 4;

__device__ __forceinline__ void arg_take(float& best, int& bi, float ov, int oi) {
  if (ov > best || (ov == best && oi < bi)) {
    best = ov;
    bi = oi;
  }
}

template <typename T>
__global__ void __launch_bounds__(kArgThreads) argmax_kernel(const T* x, int n, int* __restrict__ out,
                                                             int vec) {
  __shared__ float sv[kArgThreads / 32];
  __shared__ int si[kArgThreads / 32];
  pdl_wait();
  pdl_launch_dependents();
  const T* row = x + (int64_t)blockIdx.x * n;
  const int t = threadIdx.x;
  float best = -INFINITY;
  int bi = 0x7fffffff;
  if (vec) {
    const uint4* rv = reinterpret_cast<const uint4*>(row);
    const int nc = n / 8;
    for (int c0 = t; c0 < nc; c0 += kArgBatch * kArgThreads) {
      uint4 v[kArgBatch];
#pragma unroll
      for (int u = 0; u < kArgBatch; ++u) {
        const int c = c0 + u * kArgThreads;
        v[u] = c < nc ? rv[c] : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int u = 0; u < kArgBatch; ++u) {
        const int c = c0 + u * kArgThreads;
        if (c < nc) {
          float f[8];
          Chunk8<T>::unpack(v[u], f);
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (f[i] > best) {  // strictly greater: the first index wins
              best = f[i];
              bi = c * 8 + i;
            }
        }
      }
    }
  } else {
    for (int j = t; j < n; j += kArgThreads) {
      const float v = to_f<T>(row[j]);
      if (v > best) {
        best = v;
        bi = j;
      }
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
    arg_take(best, bi, __shfl_xor_sync(0xffffffffu, best, off), __shfl_xor_sync(0xffffffffu, bi, off));
  if ((t & 31) == 0) {
    sv[t >> 5] = best;
    si[t >> 5] = bi;
  }
  __syncthreads();
  if (t < 32) {
    best = sv[t];
    bi = si[t];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
      arg_take(best, bi, __shfl_xor_sync(0xffffffffu, best, off), __shfl_xor_sync(0xffffffffu, bi, off));
    if (t == 0) out[blockIdx.x] = bi == 0x7fffffff ? 0 : bi;
  }
}

__global__ void advance_kernel(int* pos_ptr, int n) {
  pdl_wait();
  pdl_launch_dependents();
  *pos_ptr += n;
}

}  // namespace

#define SN_DISPATCH16(dtype, T, ...)                                     \
  switch (dtype) {                                                       \
    case SWAPNET_F16: { using T = __half; __VA_ARGS__; break; }          \
    case SWAPNET_BF16: { using T = __nv_bfloat16; __VA_ARGS__; break; }  \
    default: SN_FAIL(SWAPNET_ERR_UNSUPPORTED, "decoder kernels: fp16 / bf16 only"); \
  }

int launch_embed(int dtype, const void* table, const int* ids, int tokens, int vocab, int d, void* out, int* err,
                 cudaStream_t s) {
  if ((d * 2) % 16 || ((uintptr_t)table | (uintptr_t)out) % 16)
    SN_FAIL(SWAPNET_ERR_MISALIGNED, "embedding rows must be 16-byte aligned");
  SN_DISPATCH16(dtype, T, return done(launch_pdl(embed_kernel<T>, dim3(tokens), dim3(256), 0, s,
                                                 static_cast<const T*>(table), ids, vocab, d,
                                                 static_cast<T*>(out), err), "embedding launch"));
  return SWAPNET_OK;
}

int launch_rmsnorm(int dtype, const void* x, const void* g, int rows, int d, float eps, void* y, cudaStream_t s) {
  const int vec = d % 8 == 0 && (((uintptr_t)x | (uintptr_t)g | (uintptr_t)y) & 15) == 0;
  SN_DISPATCH16(dtype, T, return done(launch_pdl(rmsnorm_kernel<T>, dim3(rows), dim3(kNormThreads), 0, s,
                                                 static_cast<const T*>(x), static_cast<const T*>(g), d, eps,
                                                 static_cast<T*>(y), vec), "rmsnorm launch"));
  return SWAPNET_OK;
}

int launch_attention(int dtype, void* q, const void* k, const void* v, void* kc, void* vc, const int* pos_ptr,
                     int tokens, int heads, int width, float theta, int max_seq, void* out, int* err,
                     cudaStream_t s) {
  if (width % heads || width / heads != kDh) SN_FAIL(SWAPNET_ERR_UNSUPPORTED, "attention: head width must be 128");
  SN_DISPATCH16(dtype, T, {
    if (((uintptr_t)q | (uintptr_t)k | (uintptr_t)v | (uintptr_t)kc | (uintptr_t)vc) & 15)
      SN_FAIL(SWAPNET_ERR_MISALIGNED, "attention: operands must be 16-byte aligned");
    // four heads and pairs per thread once that leaves a few warps for every SM
    const bool many = (int64_t)tokens * heads >= kRopeManyHeads;
    const int threads = many ? (heads + 3) / 4 * (kDh / 8) : heads * (kDh / 2);
    const dim3 g1((threads + 127) / 128, tokens);
    int rc = done(launch_pdl(many ? rope_append_kernel<T, 4, 4> : rope_append_kernel<T, 1, 1>, g1, dim3(128), 0, s,
                             static_cast<T*>(q), static_cast<const T*>(k), static_cast<const T*>(v),
                             static_cast<T*>(kc), static_cast<T*>(vc), pos_ptr, heads, kDh, theta, max_seq, err),
                  "rope launch");
    if (rc) return rc;
    if (attention_tc_supported(dtype, tokens, heads, width, max_seq))  // both contractions on the tensor cores
      return launch_attention_tc(dtype, q, kc, vc, pos_ptr, tokens, heads, width, max_seq, out, err, s);
    // decode: the visible keys split over a cluster of CTAs per (query, head)
    const SplitPlan sp = split_plan(max_seq);
    const size_t smem = attention_split_smem_bytes(sp.chunk);
    if (smem > 48 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(attention_split_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)smem);
      if (e != cudaSuccess) return done(e, "attention shared memory");
    }
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(sp.split, heads, tokens);
    cfg.blockDim = dim3(kSpThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = sp.split;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return done(cudaLaunchKernelEx(&cfg, attention_split_kernel<T>, static_cast<const T*>(q),
                                   static_cast<const T*>(kc), static_cast<const T*>(vc), pos_ptr, width, max_seq,
                                   sp.chunk, static_cast<T*>(out)),
                "attention launch");
  });
  return SWAPNET_OK;
}

int launch_argmax(int dtype, const void* x, int rows, int n, int* out, cudaStream_t s) {
  const int vec = n % 8 == 0 && ((uintptr_t)x & 15) == 0;
  SN_DISPATCH16(dtype, T, return done(launch_pdl(argmax_kernel<T>, dim3(rows), dim3(kArgThreads), 0, s,
                                                 static_cast<const T*>(x), n, out, vec), "argmax launch"));
  return SWAPNET_OK;
}

int launch_advance(int* pos_ptr, int n, cudaStream_t s) {
  return done(launch_pdl(advance_kernel, dim3(1), dim3(1), 0, s, pos_ptr, n), "position advance launch");
}

}  // namespace swapnet
