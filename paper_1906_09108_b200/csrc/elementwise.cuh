// Memory-bound kernels of the FDG module-step: batch-norm statistics / apply /
// backward, the classifier head, the shrink of the received delayed gradient
// (Eq. 15), the SGD-momentum update (Eq. 11), image ingest and dtype conversion.
//
// All tensors are NHWC, seen here as [rows = N*H*W][C].  T is the storage type
// (float or __nv_bfloat16); arithmetic, statistics and reductions are fp32 (final
// combination of per-block partial sums in fp64).  Every reduction has a fixed
// order, so results do not depend on scheduling.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "once_per_device.h"

namespace fdg {

// ------------------------------------------------ programmatic dependent launch --
// The kernels that follow one another in a module's chain (convolution, batch-norm apply, batch-norm
// backward apply) are launched with programmatic stream serialisation: the next kernel of the stream may be
// scheduled while this one still runs, does the part of its start-up that needs nothing from global
// memory (barriers, tensor-memory allocation, descriptor prefetch), and then blocks in grid_dependency_wait()
// until the preceding kernel has completed and its writes are visible.  Nothing may be read from or written
// to global memory before that wait.  grid_dependency_release() tells the scheduler that, as far as this
// block is concerned, the next kernel may start being scheduled (it fires once every block has called it or
// exited).  Both are no-ops in a kernel launched the ordinary way.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Launch with the attribute that allows the overlap described above.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Makes a setting of the current device (see OncePerDevice).  Setting a function attribute is no stream operation: a launch
// may be a recorded one.
template <typename Work>
inline cudaError_t once_per_device(OncePerDevice* once, Work work) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  return e != cudaSuccess ? e : once->run(dev, work);
}
template <typename Kernel>
inline cudaError_t set_smem_limit(Kernel kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// SMs of a B200.  Splits whose rows need scratch are planned for this number, not for the device's own: the size of the
// workspace is asked for without a device.
constexpr int kSms = 148;

// A batch norm with given statistics (inference) applied in the epilogue of the convolution that produces its input:
// the convolution's output is rounded to the storage type first, as if it had been stored, so that the result is that of
// bn_apply_kernel bit for bit.  stats null: none.
struct EpiAffine {
  const float* stats;       // mean[C], invstd[C]
  const float* gamma;
  const float* beta;
  int relu;
};

// ---------------------------------------------------------------- helpers ---
template <typename T> struct Vec;   // 16-byte vector of T
template <> struct Vec<float> {
  static constexpr int N = 4;
  float v[4];
};
template <> struct Vec<__nv_bfloat16> {
  static constexpr int N = 8;
  __nv_bfloat16 v[8];
};

__device__ __forceinline__ float to_f(float x) { return x; }
__device__ __forceinline__ float to_f(__nv_bfloat16 x) { return __bfloat162float(x); }
template <typename T> __device__ __forceinline__ T from_f(float x);
template <> __device__ __forceinline__ float from_f<float>(float x) { return x; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

// Loads VEC consecutive elements (VEC == 1 or a full 16-byte vector) as floats.
template <typename T, int VEC>
__device__ __forceinline__ void load_vec(const T* __restrict__ p, float (&out)[VEC]) {
  if constexpr (VEC == 1) {
    out[0] = to_f(p[0]);
  } else {
    static_assert(VEC * sizeof(T) == 16, "vector must be 16 bytes");
    uint4 raw = *reinterpret_cast<const uint4*>(p);
    const T* e = reinterpret_cast<const T*>(&raw);
#pragma unroll
    for (int i = 0; i < VEC; ++i) out[i] = to_f(e[i]);
  }
}
template <typename T, int VEC>
__device__ __forceinline__ void store_vec(T* __restrict__ p, const float (&in)[VEC]) {
  if constexpr (VEC == 1) {
    p[0] = from_f<T>(in[0]);
  } else {
    uint4 raw;
    T* e = reinterpret_cast<T*>(&raw);
#pragma unroll
    for (int i = 0; i < VEC; ++i) e[i] = from_f<T>(in[i]);
    *reinterpret_cast<uint4*>(p) = raw;
  }
}

// Running statistics of a batch norm, kept for inference beside the batch statistics of training:
// running[0..C) mean, running[C..2C) variance; each forward folds in the batch mean and the unbiased batch
// variance with weight `momentum` (null pointer: not kept).
struct RunningStats {
  float* running;
  float momentum;
  float unbias;      // M / (M - 1) for M values per channel
};
__device__ __forceinline__ void update_running(const RunningStats& r, int C, int c, float mean, float biased_var) {
  r.running[c] = (1.f - r.momentum) * r.running[c] + r.momentum * mean;
  r.running[C + c] = (1.f - r.momentum) * r.running[C + c] + r.momentum * (biased_var * r.unbias);
}

// ------------------------------------------------- channel reductions ------
// Sums over the rows of a [rows][C] tensor, per channel, in two launches: bn_sums_kernel leaves one row of NS * C sums per
// block, sums_finalize_kernel (or the apply kernel that consumes them, up to 128 channels) adds the rows in a fixed order.
// The first streams the operands: a block owns a contiguous range of rows, thread (r, cv) walks rows r, r + rp, ... of
// channel vector cv with kRedUnroll of them in flight, whole rows of the tensor at a time (a slab of 32 channels per block,
// with the block that finished last adding up, read 64-byte pieces and ended in a serial tail: 0.29 of the copy rate on a
// 42 MB tensor).
constexpr int kRedThreads = 512;
constexpr int kRedMaxBlocks = 148;
constexpr int kRedMaxSums = 3;
constexpr int kRedUnroll = 4;
constexpr int kRedMaxVecs = 256;      // channel vectors of a row that a block addresses

// Per-channel statistics record written by the forward and read by the backward.
// stats[0..C) = mean, stats[C..2C) = 1/sqrt(var+eps).

struct RedGeom {
  int rows, C, cv, rp, blocks, rows_per_block;
};
// `elem_bytes`: of the tensor.  bf16: every thread of the block, at least one full batch of rows each.  fp32 (the exact mode,
// a few layers of a network): half the threads and as few as two rows each, i.e. shorter chains of fp32 additions.
inline RedGeom red_geom(int rows, int C, int vec, size_t elem_bytes) {
  RedGeom g;
  g.rows = rows; g.C = C; g.cv = C / vec;
  g.rp = (elem_bytes == 4 ? kRedThreads / 2 : kRedThreads) / g.cv; if (g.rp < 1) g.rp = 1;
  const int least = g.rp * (elem_bytes == 4 ? 2 : kRedUnroll);
  const int want = (rows + least - 1) / least;
  g.blocks = want < 1 ? 1 : (want > kRedMaxBlocks ? kRedMaxBlocks : want);
  g.rows_per_block = (rows + g.blocks - 1) / g.blocks;
  return g;
}

// 16 raw bytes (or one element when VEC == 1) of T, converted to floats only when used, so that
// several loads can be in flight without holding their float images in registers.
template <typename T, int VEC> struct RawVec { uint4 q; };
template <typename T> struct RawVec<T, 1> { T q; };
template <typename T, int VEC> __device__ __forceinline__ RawVec<T, VEC> load_raw(const T* __restrict__ p) {
  RawVec<T, VEC> r;
  if constexpr (VEC == 1) r.q = p[0]; else r.q = *reinterpret_cast<const uint4*>(p);
  return r;
}
template <typename T, int VEC> __device__ __forceinline__ void raw_to_f(const RawVec<T, VEC>& r, float (&out)[VEC]) {
  if constexpr (VEC == 1) {
    out[0] = to_f(r.q);
  } else {
    const T* e = reinterpret_cast<const T*>(&r.q);
#pragma unroll
    for (int i = 0; i < VEC; ++i) out[i] = to_f(e[i]);
  }
}

// The ReLU gate of a backward pass: none (both null), the tensor itself (open where > 0), or its bits (bn_apply_kernel).
template <typename T> struct GateOf {
  const T* tensor;
  const unsigned char* bits;
};

// The gate of vector `vec` (VEC elements from element vec * VEC on) as bits.
template <typename T, int VEC> __device__ __forceinline__ unsigned int gate_bits_of(const GateOf<T>& g, size_t vec) {
  if (VEC == 8 && g.bits) return g.bits[vec];
  if (!g.tensor) return 0xffu;
  float m[VEC];
  raw_to_f<T, VEC>(load_raw<T, VEC>(g.tensor + vec * VEC), m);
  unsigned int b = 0;
#pragma unroll
  for (int i = 0; i < VEC; ++i) b |= (m[i] > 0.f ? 1u : 0u) << i;
  return b;
}

// KIND 1: sum x, sum x^2.  KIND 2: with dz = dy * [gate], sum dz, sum dz * xhat (xhat from x, stats).  KIND 3: also
// sum dz * xhat2 of a second normalised tensor sharing dz (the projection shortcut).
// partial[block][NS][C], NS = 2, 2, 3.
template <typename T, int VEC, int KIND>
__global__ void __launch_bounds__(kRedThreads, 1)
bn_sums_kernel(const T* __restrict__ dy, const GateOf<T> gate, const T* __restrict__ x, const float* __restrict__ stats,
               const T* __restrict__ x2, const float* __restrict__ stats2, RedGeom g, float* __restrict__ partial) {
  constexpr int NS = KIND == 3 ? 3 : 2;
  __shared__ float red[kRedThreads * VEC];                   // [rp][C] of one sum
  __shared__ double part[kRedThreads];                       // [nseg][C]
  const int tid = threadIdx.x, C = g.C;
  const int cvi = tid % g.cv, r = tid / g.cv;
  const bool active = r < g.rp;
  constexpr int U = KIND == 3 ? kRedUnroll / 2 : kRedUnroll;   // vectors in flight: what the registers hold
  grid_dependency_wait();
  float mean[KIND >= 2 ? VEC : 1], inv[KIND >= 2 ? VEC : 1], mean2[KIND == 3 ? VEC : 1], inv2[KIND == 3 ? VEC : 1];
  if constexpr (KIND >= 2) {
#pragma unroll
    for (int i = 0; i < VEC; ++i) {
      const int c = active ? cvi * VEC + i : 0;
      mean[i] = stats[c]; inv[i] = stats[C + c];
      if constexpr (KIND == 3) { mean2[i] = stats2[c]; inv2[i] = stats2[C + c]; }
    }
  }
  float sums[NS][VEC];
#pragma unroll
  for (int s = 0; s < NS; ++s)
#pragma unroll
    for (int i = 0; i < VEC; ++i) sums[s][i] = 0.f;
  struct Item { RawVec<T, VEC> d, v, v2; unsigned int open; };
  auto fetch = [&](size_t row, Item& it) {
    const size_t off = row * C + (size_t)cvi * VEC;
    it.v = load_raw<T, VEC>(x + off);
    if constexpr (KIND >= 2) {
      it.d = load_raw<T, VEC>(dy + off);
      it.open = gate_bits_of<T, VEC>(gate, off / VEC);
      if constexpr (KIND == 3) it.v2 = load_raw<T, VEC>(x2 + off);
    }
  };
  auto add = [&](const Item& it) {
    float v[VEC];
    raw_to_f<T, VEC>(it.v, v);
    if constexpr (KIND == 1) {
#pragma unroll
      for (int i = 0; i < VEC; ++i) { sums[0][i] += v[i]; sums[1][i] += v[i] * v[i]; }
    } else {
      float d[VEC], w[VEC];
      raw_to_f<T, VEC>(it.d, d);
      if constexpr (KIND == 3) raw_to_f<T, VEC>(it.v2, w);
#pragma unroll
      for (int i = 0; i < VEC; ++i) {
        const float dz = (it.open >> i & 1u) ? d[i] : 0.f;
        sums[0][i] += dz;
        sums[1][i] += dz * ((v[i] - mean[i]) * inv[i]);
        if constexpr (KIND == 3) sums[2][i] += dz * ((w[i] - mean2[i]) * inv2[i]);
      }
    }
  };
  if (active) {
    const int row0 = blockIdx.x * g.rows_per_block, row1 = min(row0 + g.rows_per_block, g.rows);
    int row = row0 + r;
    for (; row + (U - 1) * g.rp < row1; row += U * g.rp) {
      Item it[U];
#pragma unroll
      for (int u = 0; u < U; ++u) fetch((size_t)row + u * g.rp, it[u]);
#pragma unroll
      for (int u = 0; u < U; ++u) add(it[u]);
    }
    for (; row < row1; row += g.rp) { Item it; fetch(row, it); add(it); }
  }
  // A channel has rp sums: up to 16 threads share them (at 8 channels 512 sums are 32 + 16 fp64 additions in a row; one
  // thread per channel, 512 in a row, was most of the time of a small tensor's reduction).
  const int nseg = max(1, min(kRedThreads / C, min(g.rp, 16)));
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    __syncthreads();
    if (active) {
#pragma unroll
      for (int i = 0; i < VEC; ++i) red[r * C + cvi * VEC + i] = sums[s][i];
    }
    __syncthreads();
    for (int i = tid; i < nseg * C; i += kRedThreads) {
      const int seg = i / C, c = i - seg * C;
      double a = 0.0;
      for (int rr = seg; rr < g.rp; rr += nseg) a += (double)red[rr * C + c];
      if (nseg == 1) partial[(size_t)blockIdx.x * NS * C + s * C + c] = (float)a; else part[i] = a;
    }
    if (nseg == 1) continue;
    __syncthreads();
    for (int c = tid; c < C; c += kRedThreads) {
      double a = 0.0;
      for (int seg = 0; seg < nseg; ++seg) a += part[seg * C + c];
      partial[(size_t)blockIdx.x * NS * C + s * C + c] = (float)a;
    }
  }
}

// The totals of `nparts` rows partial[nparts][NS][C] and what they are for:
//   KIND 1  statistics: stats[0..C) = mean, stats[C..2C) = 1/sqrt(var + eps), and the running statistics;
//   KIND 2  out = the sums, o1 = dbeta, o2 = dgamma;   KIND 3  also o3 = dbeta2, o4 = dgamma2.
// A block takes 32 channels; its 32 warps take every 32nd row (a few loads each, all in flight), then warp w combines
// channel w: the order is fixed.  fp64 from here on.
template <int KIND>
__global__ void __launch_bounds__(1024) sums_finalize_kernel(const float* __restrict__ partial, int nparts, int C, double inv_count,
                                                             float eps, float* __restrict__ out, RunningStats run,
                                                             float* __restrict__ o1, float* __restrict__ o2,
                                                             float* __restrict__ o3, float* __restrict__ o4) {
  constexpr int NS = KIND == 3 ? 3 : 2;
  __shared__ double fin[NS][32][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = blockIdx.x * 32 + lane;
  grid_dependency_wait();                   // launched ahead of the end of the kernel that writes `partial`
  double t[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) t[s] = 0.0;
  if (c < C)
#pragma unroll 8
    for (int r = warp; r < nparts; r += 32) {
#pragma unroll
      for (int s = 0; s < NS; ++s) t[s] += (double)partial[((size_t)r * NS + s) * C + c];
    }
#pragma unroll
  for (int s = 0; s < NS; ++s) fin[s][warp][lane] = t[s];
  __syncthreads();
  const int cc = blockIdx.x * 32 + warp;
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    t[s] = fin[s][lane][warp];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t[s] += __shfl_xor_sync(0xffffffffu, t[s], o);
  }
  if (lane != 0 || cc >= C) return;
  if constexpr (KIND == 1) {
    const double mean = t[0] * inv_count;
    double var = t[1] * inv_count - mean * mean;
    if (var < 0.0) var = 0.0;
    out[cc] = (float)mean;
    out[C + cc] = (float)(1.0 / sqrt(var + (double)eps));
    if (run.running) update_running(run, C, cc, (float)mean, (float)var);
  } else {
    out[cc] = (float)t[0]; out[C + cc] = (float)t[1];
    o1[cc] = (float)t[0]; o2[cc] = (float)t[1];
    if constexpr (KIND == 3) { out[2 * C + cc] = (float)t[2]; o3[cc] = (float)t[0]; o4[cc] = (float)t[2]; }
  }
}
inline cudaError_t launch_stats_finalize(cudaStream_t st, const float* partial, int nparts, size_t rows, int C, float eps,
                                         float* stats, const RunningStats& run) {
  float* none = nullptr;
  return launch_chained(sums_finalize_kernel<1>, dim3((unsigned)((C + 31) / 32)), dim3(1024), 0, st, partial, nparts, C,
                        1.0 / (double)rows, eps, stats, run, none, none, none, none);
}

// Per-CTA partial sums left by a convolution epilogue, partial[nparts][2*C], to be added up by
// the kernel that consumes the totals (every block does it for itself: the partials are a few KB
// and sit in L2).  Fixed order: kEwThreads / (2C) threads share a (sum, channel) pair, each taking
// every nseg-th partial with 8 loads in flight; segment sums are added in segment order.
//   kind 1  totals are (sum x, sum x^2): out2c = (mean, 1/sqrt(var + eps))
//   kind 2  totals are the batch-norm backward's (sum dz, sum dz*xhat): out2c = the totals
struct PartialSums {
  const float* partial;     // null: nothing to add up (the totals are read from global memory instead)
  int nparts;
  int kind;
  float inv_count, eps;     // kind 1
  float* save0;             // block 0 stores out2c[0..C) here (kind 1: with save1 contiguous = stats[2C]; kind 2: dbeta)
  float* save1;             // and out2c[C..2C) here (kind 2: dgamma)
  RunningStats run;         // kind 1: block 0 also folds the batch statistics into the running ones
};
constexpr int kEwThreads = 256;

// The first eight rows of a thread's share, requested ahead of everything else an apply kernel loads.
__device__ __forceinline__ void fetch_partials(const PartialSums& ps, int C, float (&v)[8]) {
  const int pairs = 2 * C, nseg = kEwThreads / pairs, t = threadIdx.x % pairs, seg = threadIdx.x / pairs;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int b = seg + u * nseg;
    v[u] = (seg < nseg && b < ps.nparts) ? __ldcg(&ps.partial[(size_t)b * pairs + t]) : 0.f;
  }
}
// Fills out2c[2*C] (shared memory) from the partials; requires blockDim.x == kEwThreads and 2*C <= kEwThreads.  `v` as
// fetched above.
__device__ __forceinline__ void finalize_partials(const PartialSums& ps, int C, const float (&first)[8], float* out2c) {
  __shared__ double fin[kEwThreads];
  const int tid = threadIdx.x, pairs = 2 * C;
  const int nseg = kEwThreads / pairs;
  const int t = tid % pairs, seg = tid / pairs;
  double a = 0.0;
#pragma unroll
  for (int u = 0; u < 8; ++u) a += (double)first[u];
  if (seg < nseg)
    for (int b0 = seg + 8 * nseg; b0 < ps.nparts; b0 += 8 * nseg) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int b = b0 + u * nseg;
        v[u] = b < ps.nparts ? __ldcg(&ps.partial[(size_t)b * pairs + t]) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) a += (double)v[u];
    }
  fin[tid] = a;
  __syncthreads();
  if (tid < C) {
    double s0 = 0.0, s1 = 0.0;
    for (int q = 0; q < nseg; ++q) { s0 += fin[q * pairs + tid]; s1 += fin[q * pairs + C + tid]; }
    float o0, o1;
    if (ps.kind == 1) {
      const double mean = s0 * (double)ps.inv_count;
      double var = s1 * (double)ps.inv_count - mean * mean;
      if (var < 0.0) var = 0.0;
      o0 = (float)mean; o1 = (float)(1.0 / sqrt(var + (double)ps.eps));
      if (blockIdx.x == 0 && ps.run.running) update_running(ps.run, C, tid, (float)mean, (float)var);
    } else {
      o0 = (float)s0; o1 = (float)s1;
    }
    out2c[tid] = o0; out2c[C + tid] = o1;
    if (blockIdx.x == 0) { ps.save0[tid] = o0; ps.save1[tid] = o1; }
  }
  __syncthreads();
}

// N consecutive floats, by 16-byte loads where `vec` says the pointer allows it.
template <int N> __device__ __forceinline__ void load_consts(const float* p, bool vec, float (&v)[N]) {
  if constexpr (N % 4 == 0) {
    if (vec) {
#pragma unroll
      for (int j = 0; j < N; j += 4) {
        const float4 q = *reinterpret_cast<const float4*>(p + j);
        v[j] = q.x; v[j + 1] = q.y; v[j + 2] = q.z; v[j + 3] = q.w;
      }
      return;
    }
  }
#pragma unroll
  for (int j = 0; j < N; ++j) v[j] = p[j];
}

// ------------------------------------------------- batch norm, forward ------
// y = [relu]( gamma*(x-mean)*invstd + beta + residual ), residual = none (RES 0) | r (1) | BN_r(r) (2).
// The statistics come from `stats`, or are first formed from `ps.partial` (and saved to stats).
// The launcher makes the grid's thread count a multiple of the channel vectors per row, so a thread
// meets the same VEC channels in every iteration: their constants (mean, gamma * invstd, beta; the fp32 mode, whose results
// are compared at 1e-4 through many layers, keeps gamma and invstd apart) live in registers.  A
// thread's first batch of U vectors is requested right behind the partial sums, whose addition then hides its latency.
// `bits` (nullable; bf16 vectors only): one bit per element, set where y > 0 -- byte i holds those of vector i.  They are
// the ReLU gates of the backward pass at a sixteenth of the tensor's size.
constexpr int kEwUnroll = 4;
template <typename T, int VEC, int RES>
__global__ void __launch_bounds__(kEwThreads, RES == 2 ? 2 : 3)
bn_apply_kernel(const T* __restrict__ x, const float* __restrict__ stats,
                const float* __restrict__ gamma, const float* __restrict__ beta,
                const T* __restrict__ res, const float* __restrict__ res_stats,
                const float* __restrict__ res_gamma, const float* __restrict__ res_beta,
                int relu, int vec_consts, T* __restrict__ y, unsigned char* __restrict__ bits, size_t nvec, int C, PartialSums ps) {
  constexpr int U = RES == 2 ? 2 : kEwUnroll;
  __shared__ __align__(16) float s_stats[2 * 128];
  const int cv = C / VEC;
  const size_t gtid = blockIdx.x * (size_t)blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
  const int c0 = (int)(gtid % cv) * VEC;
  grid_dependency_wait();
  grid_dependency_release();
  float first[8];
  if (ps.partial) fetch_partials(ps, C, first);
  RawVec<T, VEC> xv[U], rv[RES ? U : 1];
  auto fetch = [&](size_t i) {
#pragma unroll
    for (int u = 0; u < U; ++u) xv[u] = load_raw<T, VEC>(x + (i + u * stride) * VEC);
    if constexpr (RES != 0) {
#pragma unroll
      for (int u = 0; u < U; ++u) rv[u] = load_raw<T, VEC>(res + (i + u * stride) * VEC);
    }
  };
  size_t i = gtid;
  bool full = i + (U - 1) * stride < nvec;
  if (full) fetch(i);
  constexpr bool EXACT = sizeof(T) == 4;
  float mean[VEC], ga[VEC], be[VEC], rmean[RES == 2 ? VEC : 1], rga[RES == 2 ? VEC : 1], rbe[RES == 2 ? VEC : 1];
  float inv[VEC], rinv[RES == 2 ? VEC : 1];
  const bool vc = vec_consts != 0;
  load_consts<VEC>(gamma + c0, vc, ga);
  load_consts<VEC>(beta + c0, vc, be);
  if constexpr (RES == 2) {
    load_consts<VEC>(res_gamma + c0, vc, rga);
    load_consts<VEC>(res_beta + c0, vc, rbe);
    load_consts<VEC>(res_stats + c0, vc, rmean);
    load_consts<VEC>(res_stats + C + c0, vc, rinv);
#pragma unroll
    for (int j = 0; j < VEC; ++j) if (!EXACT) rga[j] *= rinv[j];
  }
  const float* st = stats;
  if (ps.partial) { finalize_partials(ps, C, first, s_stats); st = s_stats; }
  load_consts<VEC>(st + c0, vc, mean);
  load_consts<VEC>(st + C + c0, vc, inv);
#pragma unroll
  for (int j = 0; j < VEC; ++j) if (!EXACT) ga[j] *= inv[j];
  auto one = [&](size_t at, const RawVec<T, VEC>& xq, const RawVec<T, VEC>& rq) {
    float v[VEC], r[VEC], o[VEC];
    raw_to_f<T, VEC>(xq, v);
    if constexpr (RES != 0) raw_to_f<T, VEC>(rq, r);
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
      float t = EXACT ? ga[j] * ((v[j] - mean[j]) * inv[j]) + be[j] : fmaf(v[j] - mean[j], ga[j], be[j]);
      if constexpr (RES == 1) t += r[j];
      if constexpr (RES == 2) t += EXACT ? rga[j] * ((r[j] - rmean[j]) * rinv[j]) + rbe[j] : fmaf(r[j] - rmean[j], rga[j], rbe[j]);
      o[j] = relu ? fmaxf(t, 0.f) : t;
    }
    if constexpr (VEC == 8) {
      // the gate is taken on the value as stored (a positive value below half the smallest bf16 number rounds to zero):
      // a stored bf16 is positive where its sign is clear and it is not zero
      uint32_t w[4];
      unsigned int m = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const __nv_bfloat162 q = __floats2bfloat162_rn(o[2 * j], o[2 * j + 1]);
        w[j] = *reinterpret_cast<const uint32_t*>(&q);
      }
      *reinterpret_cast<uint4*>(y + at * VEC) = make_uint4(w[0], w[1], w[2], w[3]);
      if (bits) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          m |= ((int)(w[j] << 16) > 0 ? 1u : 0u) << (2 * j);
          m |= ((int)(w[j] & 0xffff0000u) > 0 ? 1u : 0u) << (2 * j + 1);
        }
        bits[at] = (unsigned char)m;
      }
    } else {
      store_vec<T, VEC>(y + at * VEC, o);
    }
  };
  while (full) {
#pragma unroll
    for (int u = 0; u < U; ++u) one(i + u * stride, xv[u], rv[RES ? u : 0]);
    i += U * stride;
    full = i + (U - 1) * stride < nvec;
    if (full) fetch(i);
  }
  for (; i < nvec; i += stride) {
    const RawVec<T, VEC> xq = load_raw<T, VEC>(x + i * VEC);
    RawVec<T, VEC> rq = xq;
    if constexpr (RES != 0) rq = load_raw<T, VEC>(res + i * VEC);
    one(i, xq, rq);
  }
}

// ------------------------------------------------- batch norm, backward -----
// dx = gamma*invstd*(dz - s0/M - xhat*s1/M) [+ res] with dz = dy * [gate];  optionally the same for the second
// normalised tensor (dx2, TWO).  Written as  gi*dz - (x - mean)*k1 - k0  with gi = gamma*invstd, k1 = gi*invstd*s1/M,
// k0 = gi*s0/M: four constants per channel in registers (the fp32 mode keeps the first form).  First batch of loads ahead of the sums' addition as above.
template <typename T, int VEC, bool TWO>
__global__ void __launch_bounds__(kEwThreads, TWO ? 2 : 3)
bn_bwd_apply_kernel(const T* __restrict__ dy, const GateOf<T> gate, const T* __restrict__ x,
                    const float* __restrict__ stats, const float* __restrict__ gamma,
                    const float* __restrict__ sums, const T* __restrict__ x2,
                    const float* __restrict__ stats2, const float* __restrict__ gamma2,
                    const T* __restrict__ res, int vec_consts, T* __restrict__ dx, T* __restrict__ dx2,
                    size_t nvec, int C, float inv_m, PartialSums ps) {
  constexpr int U = 2;
  __shared__ __align__(16) float s_sums[2 * 128];
  const int cv = C / VEC;
  const size_t gtid = blockIdx.x * (size_t)blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
  const int c0 = (int)(gtid % cv) * VEC;
  grid_dependency_wait();
  grid_dependency_release();
  float first[8];
  if (ps.partial) fetch_partials(ps, C, first);
  RawVec<T, VEC> dv[U], xv[U];
  unsigned int open[U];
  auto fetch = [&](size_t i) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      dv[u] = load_raw<T, VEC>(dy + (i + u * stride) * VEC);
      xv[u] = load_raw<T, VEC>(x + (i + u * stride) * VEC);
      open[u] = gate_bits_of<T, VEC>(gate, i + u * stride);
    }
  };
  size_t i = gtid;
  bool full = i + (U - 1) * stride < nvec;
  if (full) fetch(i);
  const bool vc = vec_consts != 0;
  constexpr bool EXACT = sizeof(T) == 4;
  float mean[VEC], gi[VEC], k0[VEC], k1[VEC], mean2[TWO ? VEC : 1], gi2[TWO ? VEC : 1], k02[TWO ? VEC : 1], k12[TWO ? VEC : 1];
  float inv[VEC], inv2[TWO ? VEC : 1];
  auto consts = [&](const float* stv, const float* gav, const float* s0p, const float* s1p, float (&mu)[VEC], float (&iv)[VEC],
                    float (&g)[VEC], float (&a0)[VEC], float (&a1)[VEC]) {
    load_consts<VEC>(stv + c0, vc, mu);
    load_consts<VEC>(stv + C + c0, vc, iv);
    load_consts<VEC>(gav + c0, vc, g);
    load_consts<VEC>(s0p + c0, vc, a0);
    load_consts<VEC>(s1p + c0, vc, a1);
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
      g[j] *= iv[j];
      a0[j] *= inv_m; a1[j] *= inv_m;
      if (!EXACT) { a0[j] *= g[j]; a1[j] *= g[j] * iv[j]; }
    }
  };
  if (ps.partial) { finalize_partials(ps, C, first, s_sums); sums = s_sums; }
  consts(stats, gamma, sums, sums + C, mean, inv, gi, k0, k1);
  if constexpr (TWO) consts(stats2, gamma2, sums, sums + 2 * C, mean2, inv2, gi2, k02, k12);
  auto one = [&](size_t at, const RawVec<T, VEC>& dq, unsigned int op, const RawVec<T, VEC>& xq) {
    float d[VEC], v[VEC], v2[VEC], r[VEC], o[VEC], o2[VEC];
    raw_to_f<T, VEC>(dq, d);
    raw_to_f<T, VEC>(xq, v);
    if constexpr (TWO) load_vec<T, VEC>(x2 + at * VEC, v2);
    if (res) load_vec<T, VEC>(res + at * VEC, r);
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
      const float dz = (op >> j & 1u) ? d[j] : 0.f;
      const float t = EXACT ? gi[j] * (dz - k0[j] - (v[j] - mean[j]) * inv[j] * k1[j]) : fmaf(gi[j], dz, fmaf(mean[j] - v[j], k1[j], -k0[j]));
      o[j] = res ? t + r[j] : t;
      if constexpr (TWO) o2[j] = EXACT ? gi2[j] * (dz - k02[j] - (v2[j] - mean2[j]) * inv2[j] * k12[j]) : fmaf(gi2[j], dz, fmaf(mean2[j] - v2[j], k12[j], -k02[j]));
    }
    store_vec<T, VEC>(dx + at * VEC, o);
    if constexpr (TWO) store_vec<T, VEC>(dx2 + at * VEC, o2);
  };
  while (full) {
#pragma unroll
    for (int u = 0; u < U; ++u) one(i + u * stride, dv[u], open[u], xv[u]);
    i += U * stride;
    full = i + (U - 1) * stride < nvec;
    if (full) fetch(i);
  }
  for (; i < nvec; i += stride) {
    const RawVec<T, VEC> dq = load_raw<T, VEC>(dy + i * VEC), xq = load_raw<T, VEC>(x + i * VEC);
    one(i, dq, gate_bits_of<T, VEC>(gate, i), xq);
  }
}

// -------------------------------------------------------- small elementwise -
// out = scale * in  (the gradient-shrinking step, Eq. 15).
template <typename T, int VEC>
__global__ void scale_kernel(const T* __restrict__ in, T* __restrict__ out, float scale, size_t nvec) {
  grid_dependency_wait();
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nvec; i += (size_t)gridDim.x * blockDim.x) {
    float v[VEC];
    load_vec<T, VEC>(in + i * VEC, v);
#pragma unroll
    for (int j = 0; j < VEC; ++j) v[j] *= scale;
    store_vec<T, VEC>(out + i * VEC, v);
  }
}

// up[n][2p][2q][:] = dy[n][p][q][:], zero at the other pixels; dy [N][P][Q][C], up [N][2P][2Q][C], 16-byte vectors.
template <typename T, int VEC>
__global__ void upsample2_kernel(const T* __restrict__ dy, T* __restrict__ up, size_t nvec_up, int P, int Q, int C) {
  grid_dependency_wait();
  const int cv = C / VEC;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nvec_up; i += (size_t)gridDim.x * blockDim.x) {
    const int c = (int)(i % cv);
    size_t pix = i / cv;
    const int w = (int)(pix % (2 * Q)); pix /= 2 * Q;
    const int h = (int)(pix % (2 * P));
    const size_t n = pix / (2 * P);
    uint4 v = make_uint4(0, 0, 0, 0);
    if (((h | w) & 1) == 0) v = reinterpret_cast<const uint4*>(dy)[((n * P + (h >> 1)) * Q + (w >> 1)) * cv + c];
    reinterpret_cast<uint4*>(up)[i] = v;
  }
}

// Zero-padded shortcut of a block that changes the shape: out [N][P][Q][Co] = x [N][H][W][Ci] at every stride-th
// pixel, in channels lo .. lo+Ci-1 with lo = (Co - Ci)/2, zero elsewhere; and its backward, which puts the
// gated upstream gradient's middle channels back at those pixels of a zero [N][H][W][Ci] tensor.
template <typename T>
__global__ void pad_shortcut_kernel(const T* __restrict__ x, T* __restrict__ out, size_t rows_out, int P, int Q, int H, int W,
                                    int Ci, int Co, int stride) {
  grid_dependency_wait();
  const int lo = (Co - Ci) / 2;
  const size_t n = rows_out * (size_t)Co;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int c = (int)(i % Co);
    size_t pix = i / Co;
    const int q = (int)(pix % Q); pix /= Q;
    const int p = (int)(pix % P);
    const size_t img = pix / P;
    T v = from_f<T>(0.f);
    if (c >= lo && c < lo + Ci) v = x[((img * H + (size_t)p * stride) * W + (size_t)q * stride) * Ci + (c - lo)];
    out[i] = v;
  }
}
template <typename T>
__global__ void pad_shortcut_bwd_kernel(const T* __restrict__ dy, const T* __restrict__ y, T* __restrict__ dx, size_t rows_in,
                                        int P, int Q, int H, int W, int Ci, int Co, int stride) {
  grid_dependency_wait();
  const int lo = (Co - Ci) / 2;
  const size_t n = rows_in * (size_t)Ci;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int c = (int)(i % Ci);
    size_t pix = i / Ci;
    const int w = (int)(pix % W); pix /= W;
    const int h = (int)(pix % H);
    const size_t img = pix / H;
    T v = from_f<T>(0.f);
    if (h % stride == 0 && w % stride == 0) {
      const size_t o = ((img * P + h / stride) * Q + w / stride) * Co + lo + c;
      if (to_f(y[o]) > 0.f) v = dy[o];
    }
    dx[i] = v;
  }
}

// fp32 [rows][c_in] -> T [rows][c_out], channels c_in..c_out-1 zero (image ingest); labels copied alongside.
template <typename T>
__global__ void ingest_kernel(const float* __restrict__ img, T* __restrict__ out, size_t rows, int c_in, int c_out,
                              const int32_t* __restrict__ labels_in, int32_t* __restrict__ labels_out, int batch) {
  grid_dependency_wait();
  const size_t n = rows * (size_t)c_out;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const size_t row = i / c_out;
    const int c = (int)(i % c_out);
    out[i] = from_f<T>(c < c_in ? img[row * c_in + c] : 0.f);
  }
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i < batch; i += blockDim.x) labels_out[i] = labels_in[i];
}

// T [rows][c_src] -> fp32 [rows][c_dst] keeping the first c_dst channels (getters).
template <typename T>
__global__ void export_kernel(const T* __restrict__ in, float* __restrict__ out, size_t rows, int c_src, int c_dst) {
  const size_t n = rows * (size_t)c_dst;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const size_t row = i / c_dst;
    out[i] = to_f(in[row * c_src + (i % c_dst)]);
  }
}

// ------------------------------------------------------------------ head ----
// One block per sample: global average pool -> FC -> softmax cross-entropy, and the
// backward of all three down to the gradient of the pooled tensor's source.
//   x [B][HW][F] (T)   w [classes][F], b [classes] (fp32)
//   pooled [B][F], dlogits [B][classes], loss_n [B] (fp32 scratch for head_param_grad)
//   dx [B][HW][F] (T) = dpooled[f] / HW
// A label outside [0, classes) sets *bad_label and is treated as class 0.
// `groups` > 0 (F a multiple of the 16-byte vector, see head_groups): the sample is read and its gradient written in
// 16-byte vectors; `groups` sets of threads take every groups-th pixel and their partial sums are added in group
// order.  `groups` == 0: element by element, for any F.
template <typename T>
__global__ void head_fwd_bwd_kernel(const T* __restrict__ x, const float* __restrict__ w, const float* __restrict__ b,
                                    const int32_t* __restrict__ labels, int HW, int F, int classes, int batch, int groups,
                                    float* __restrict__ pooled, float* __restrict__ dlogits,
                                    float* __restrict__ loss_n, T* __restrict__ dx, int* __restrict__ bad_label) {
  grid_dependency_wait();
  constexpr int V = 16 / (int)sizeof(T);
  extern __shared__ __align__(16) float hs[];   // pooled[F] | dpooled[F] | partial[groups][F] | logits[classes]
  float* s_pool = hs;
  float* s_dpool = hs + F;
  float* s_part = s_dpool + F;
  float* s_logit = s_part + (size_t)groups * F;
  const int n = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
  const T* xn = x + (size_t)n * HW * F;
  if (groups > 0) {
    const int cols = F / V;
    for (int item = tid; item < groups * cols; item += nt) {
      const int g = item / cols, col = item - g * cols;
      float acc[V];
#pragma unroll
      for (int j = 0; j < V; ++j) acc[j] = 0.f;
#pragma unroll 4
      for (int p = g; p < HW; p += groups) {
        float v[V];
        load_vec<T, V>(xn + (size_t)p * F + col * V, v);
#pragma unroll
        for (int j = 0; j < V; ++j) acc[j] += v[j];
      }
#pragma unroll
      for (int j = 0; j < V; ++j) s_part[(size_t)g * F + col * V + j] = acc[j];
    }
    __syncthreads();
    for (int f = tid; f < F; f += nt) {
      float a = 0.f;
      for (int g = 0; g < groups; ++g) a += s_part[(size_t)g * F + f];
      a /= (float)HW;
      s_pool[f] = a;
      pooled[(size_t)n * F + f] = a;
    }
  } else {
    for (int f = tid; f < F; f += nt) {
      float a = 0.f;
#pragma unroll 8
      for (int p = 0; p < HW; ++p) a += to_f(xn[(size_t)p * F + f]);
      a /= (float)HW;
      s_pool[f] = a;
      pooled[(size_t)n * F + f] = a;
    }
  }
  __syncthreads();
  const int warp = tid >> 5, lane = tid & 31, nwarps = nt >> 5;
  for (int c = warp; c < classes; c += nwarps) {
    float a = 0.f;
    for (int f = lane; f < F; f += 32) a += w[(size_t)c * F + f] * s_pool[f];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) s_logit[c] = a + b[c];
  }
  __syncthreads();
  __shared__ float s_max, s_sum;
  int label = labels[n];
  if (label < 0 || label >= classes) { if (tid == 0) atomicExch(bad_label, 1); label = 0; }
  if (warp == 0) {                       // the lanes share the classes; the partial sums meet in a fixed butterfly
    float m = -INFINITY;
    for (int c = lane; c < classes; c += 32) m = fmaxf(m, s_logit[c]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    float s = 0.f;
    for (int c = lane; c < classes; c += 32) s += expf(s_logit[c] - m);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      s_max = m; s_sum = s;
      loss_n[n] = -(s_logit[label] - m - logf(s));
    }
  }
  __syncthreads();
  for (int c = tid; c < classes; c += nt) {
    float p = expf(s_logit[c] - s_max) / s_sum;
    float d = (p - (c == label ? 1.f : 0.f)) / (float)batch;
    s_logit[c] = d;
    dlogits[(size_t)n * classes + c] = d;
  }
  __syncthreads();
  for (int f = tid; f < F; f += nt) {
    float a = 0.f;
#pragma unroll 4
    for (int c = 0; c < classes; ++c) a += w[(size_t)c * F + f] * s_logit[c];
    s_dpool[f] = a / (float)HW;
  }
  __syncthreads();
  T* dxn = dx + (size_t)n * HW * F;
  if (groups > 0) {
    // the row of F gradients, packed once as T into the (now free) partial-sum area, then copied to every pixel
    T* s_row = reinterpret_cast<T*>(s_part);
    for (int f = tid; f < F; f += nt) s_row[f] = from_f<T>(s_dpool[f]);
    __syncthreads();
    const int cols = F / V;
    const uint4* row4 = reinterpret_cast<const uint4*>(s_row);
    uint4* dx4 = reinterpret_cast<uint4*>(dxn);
    for (int i = tid; i < HW * cols; i += nt) dx4[i] = row4[i % cols];
  } else {
    for (int i = tid; i < HW * F; i += nt) dxn[i] = from_f<T>(s_dpool[i % F]);
  }
}

constexpr int kHeadThreads = 256;
// Pixel groups of head_fwd_bwd_kernel for F features of `elem_bytes` each: 0 when F is not a whole number of
// 16-byte vectors, otherwise as many as fill the block (at most 8, and within the default shared-memory limit).
inline int head_groups(int F, int classes, int HW, size_t elem_bytes) {
  const int V = (int)(16 / elem_bytes);
  if (F % V != 0) return 0;
  int g = kHeadThreads / (F / V);
  if (g > 8) g = 8;
  if (g > HW) g = HW;
  if (g < 1) g = 1;
  while (g > 1 && ((size_t)(2 + g) * F + classes) * 4 > 40 * 1024) --g;
  return g;
}
inline size_t head_smem_bytes(int F, int classes, int groups) { return ((size_t)(2 + groups) * F + classes) * 4; }

// dW[c][f] = sum_n dlogits[n][c]*pooled[n][f], db[c] = sum_n dlogits[n][c].  Grid (classes, ceil(F / 32)), 128
// threads: a lane owns a feature, the four warps take every fourth sample and their partial sums are added in warp
// order.  Blocks (c, 0) also form db[c]; block (0, 0) reduces the loss (mean over the batch) and raises *nonfinite if
// it is NaN/Inf.
__global__ void head_param_grad_kernel(const float* __restrict__ pooled, const float* __restrict__ dlogits,
                                       const float* __restrict__ loss_n, int F, int classes, int batch,
                                       float* __restrict__ dW, float* __restrict__ db, float* __restrict__ loss,
                                       int* __restrict__ nonfinite) {
  grid_dependency_wait();
  __shared__ float s_part[4][32];
  const int c = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int f = blockIdx.y * 32 + lane;
  float a = 0.f;
  if (f < F) {
#pragma unroll 8
    for (int n = warp; n < batch; n += 4) a += dlogits[(size_t)n * classes + c] * pooled[(size_t)n * F + f];
  }
  s_part[warp][lane] = a;
  __syncthreads();
  if (warp == 0 && f < F) dW[(size_t)c * F + f] = ((s_part[0][lane] + s_part[1][lane]) + s_part[2][lane]) + s_part[3][lane];
  if (blockIdx.y != 0) return;
  // the sums over the batch: lanes take every 32nd sample, the partial sums meet in a fixed butterfly
  if (warp == 1) {
    float s = 0.f;
    for (int n = lane; n < batch; n += 32) s += dlogits[(size_t)n * classes + c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) db[c] = s;
  } else if (warp == 2 && c == 0) {
    double l = 0.0;
    for (int n = lane; n < batch; n += 32) l += (double)loss_n[n];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) {
      const float lf = (float)(l / (double)batch);
      *loss = lf;
      if (!isfinite(lf)) atomicExch(nonfinite, 1);
    }
  }
}

// The two launches of the head on stream `st` (arguments as the kernels').
template <typename T>
inline cudaError_t launch_head(cudaStream_t st, const T* x, const float* w, const float* b, const int32_t* labels, int HW,
                               int F, int classes, int batch, float* pooled, float* dlogits, float* loss_n, T* dx,
                               float* dW, float* db, float* loss, int* flags, bool second = true, bool first = true) {
  if (first) {
    int groups = head_groups(F, classes, HW, sizeof(T));
    if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(dx)) & 15) groups = 0;   // vectors need 16-byte alignment
    const cudaError_t e = launch_chained(head_fwd_bwd_kernel<T>, batch, kHeadThreads, head_smem_bytes(F, classes, groups), st,
                                         x, w, b, labels, HW, F, classes, batch, groups, pooled, dlogits, loss_n, dx, flags + 1);
    if (e != cudaSuccess) return e;
  }
  if (second) {
    return launch_chained(head_param_grad_kernel, dim3(classes, (F + 31) / 32), 128, 0, st, (const float*)pooled,
                          (const float*)dlogits, (const float*)loss_n, F, classes, batch, dW, db, loss, flags);
  }
  return cudaSuccess;
}

// ------------------------------------------------------------------- SGD ----
// g' = g + wd*theta ; v = mu*v + g' ; theta -= lr*v   (v starts at 0, so the first
// update gives v = g').  Also writes the copies of theta the kernels compute with into
// the next weight-version slot: fp32 always, bf16 when next16 is given.  g is left untouched.
// The learning rate is `lr`, or *lr_dev when that pointer is given (a recorded launch can then
// follow a schedule without being re-recorded).
__global__ void sgd_kernel(float* __restrict__ theta, float* __restrict__ v, const float* __restrict__ g,
                           float* __restrict__ next32, __nv_bfloat16* __restrict__ next16, size_t n, float lr,
                           const float* __restrict__ lr_dev, float mu, float wd) {
  grid_dependency_wait();
  if (lr_dev) lr = *lr_dev;
  const size_t n4 = n / 4;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
    float4 th = reinterpret_cast<float4*>(theta)[i];
    float4 vv = reinterpret_cast<float4*>(v)[i];
    const float4 gg = reinterpret_cast<const float4*>(g)[i];
    vv.x = mu * vv.x + (gg.x + wd * th.x); th.x -= lr * vv.x;
    vv.y = mu * vv.y + (gg.y + wd * th.y); th.y -= lr * vv.y;
    vv.z = mu * vv.z + (gg.z + wd * th.z); th.z -= lr * vv.z;
    vv.w = mu * vv.w + (gg.w + wd * th.w); th.w -= lr * vv.w;
    reinterpret_cast<float4*>(theta)[i] = th;
    reinterpret_cast<float4*>(v)[i] = vv;
    reinterpret_cast<float4*>(next32)[i] = th;
    if (next16) {
      __nv_bfloat162 lo = __floats2bfloat162_rn(th.x, th.y), hi = __floats2bfloat162_rn(th.z, th.w);
      uint2 pk;
      pk.x = *reinterpret_cast<unsigned int*>(&lo);
      pk.y = *reinterpret_cast<unsigned int*>(&hi);
      reinterpret_cast<uint2*>(next16)[i] = pk;
    }
  }
  if (blockIdx.x == 0)
    for (size_t i = n4 * 4 + threadIdx.x; i < n; i += blockDim.x) {
      float vv = mu * v[i] + (g[i] + wd * theta[i]);
      float th = theta[i] - lr * vv;
      v[i] = vv; theta[i] = th;
      next32[i] = th;
      if (next16) next16[i] = __float2bfloat16_rn(th);
    }
}

__global__ void set_scalar_kernel(float* dst, float value) { *dst = value; }

// fp32 -> T copy (refreshing the compute copies after fdg_set_params).
template <typename T>
__global__ void cast_kernel(const float* __restrict__ in, T* __restrict__ out, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    out[i] = from_f<T>(in[i]);
}

// ------------------------------------------------------------- inference ----
// Inference-mode statistics of all batch norms of a module in one launch: for table entry e,
// out[soff .. soff+C) = running mean, out[soff+C .. soff+2C) = 1/sqrt(running variance + eps).
struct EvalStatEntry { size_t roff, soff; int C; };
// All modules in one launch (blockIdx.y: the module; one per module stood between their passes: ResNet-110, K = 4, 1.6 % of a batch).
constexpr int kMaxModules = 64;
struct EvalStatModules {
  const float* running[kMaxModules];
  float* out[kMaxModules];
  const EvalStatEntry* table[kMaxModules];
  int entries[kMaxModules];
};
__global__ void bn_eval_stats_kernel(const __grid_constant__ EvalStatModules mods, float eps) {
  grid_dependency_wait();
  if ((int)blockIdx.x >= mods.entries[blockIdx.y]) return;
  const float* __restrict__ running = mods.running[blockIdx.y];
  float* __restrict__ out = mods.out[blockIdx.y];
  const EvalStatEntry e = mods.table[blockIdx.y][blockIdx.x];
  for (int c = threadIdx.x; c < e.C; c += blockDim.x) {
    out[e.soff + c] = running[e.roff + c];
    out[e.soff + e.C + c] = 1.f / sqrtf(running[e.roff + e.C + c] + eps);
  }
}

// Classifier in inference mode, one block per sample: global average pool -> FC -> logits (optional copy
// out) -> arg-max (lowest index among equal logits) compared with the label; *correct counts the matches.
template <typename T>
__global__ void head_eval_kernel(const T* __restrict__ x, const float* __restrict__ w, const float* __restrict__ b,
                                 const int32_t* __restrict__ labels, int HW, int F, int classes,
                                 float* __restrict__ logits_out, int* __restrict__ correct) {
  grid_dependency_wait();
  extern __shared__ float hs[];            // pooled[F] | logits[classes]
  float* s_pool = hs;
  float* s_logit = hs + F;
  const int n = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
  const T* xn = x + (size_t)n * HW * F;
  for (int f = tid; f < F; f += nt) {
    float a = 0.f;
    for (int p = 0; p < HW; ++p) a += to_f(xn[(size_t)p * F + f]);
    s_pool[f] = a / (float)HW;
  }
  __syncthreads();
  const int warp = tid >> 5, lane = tid & 31, nwarps = nt >> 5;
  for (int c = warp; c < classes; c += nwarps) {
    float a = 0.f;
    for (int f = lane; f < F; f += 32) a += w[(size_t)c * F + f] * s_pool[f];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) { s_logit[c] = a + b[c]; if (logits_out) logits_out[(size_t)n * classes + c] = a + b[c]; }
  }
  __syncthreads();
  if (tid == 0 && labels && correct) {
    int best = 0;
    for (int c = 1; c < classes; ++c) if (s_logit[c] > s_logit[best]) best = c;
    if (best == labels[n]) atomicAdd(correct, 1);
  }
}

// ---------------------------------------------------------- host launchers ---
// Shared by the module runtime and the operator-level entry points, so that both issue the same
// kernels in the same launch shapes.
inline int ew_blocks(size_t nvec) {
  size_t b = (nvec + 255) / 256;
  return (int)(b < 1 ? 1 : (b > 148 * 8 ? 148 * 8 : b));
}
template <typename T> constexpr int full_vec() { return 16 / sizeof(T); }

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// Floats of scratch a channel reduction over C channels may write (per-block partial sums).
inline size_t red_scratch_floats(int C) { return (size_t)kRedMaxBlocks * kRedMaxSums * C; }

// stats[0..C) = mean, stats[C..2C) = 1/sqrt(var + eps) of x [rows][C].
template <typename T>
inline cudaError_t launch_bn_stats(cudaStream_t st, const T* x, size_t rows, int C, float eps, float* stats,
                                   float* scratch, float* running = nullptr, float momentum = 0.f) {
  constexpr int V = full_vec<T>();
  const RunningStats run{running, momentum, rows > 1 ? (float)((double)rows / (double)(rows - 1)) : 1.f};
  const RedGeom g = red_geom((int)rows, C, C % V == 0 ? V : 1, sizeof(T));
  const T* no = nullptr;
  const float* nof = nullptr;
  const cudaError_t e = C % V == 0
      ? launch_chained(bn_sums_kernel<T, V, 1>, g.blocks, kRedThreads, 0, st, no, GateOf<T>{}, x, nof, no, nof, g, scratch)
      : launch_chained(bn_sums_kernel<T, 1, 1>, g.blocks, kRedThreads, 0, st, no, GateOf<T>{}, x, nof, no, nof, g, scratch);
  return e != cudaSuccess ? e : launch_stats_finalize(st, scratch, g.blocks, rows, C, eps, stats, run);
}

// Grid of the batch-norm apply kernels: what `nvec` vectors need, bounded by `cap` (0 = none), and such that
// the grid's thread count is a multiple of the `cv` channel vectors of a row (every thread then stays on the
// same channels).  Surplus blocks of a tiny tensor simply find no work.
inline int ew_grid_for_channels(size_t nvec, int cv, int cap) {
  int a = cv, b = kEwThreads;
  while (b) { const int t = a % b; a = b; b = t; }
  const int unit = cv / a;                       // blocks per period
  int blocks = ew_blocks((nvec + kEwUnroll - 1) / kEwUnroll);
  if (cap > 0 && blocks > cap) blocks = cap;
  blocks = blocks / unit * unit;
  return blocks < unit ? unit : blocks;
}

// y = [relu](BN(x) + residual).  `partial` != null: the statistics are not in `stats` yet; a convolution left
// `nparts` rows of per-CTA sums (sum x, sum x^2) there, which every block adds up first (block 0 saves the
// result to `stats`); `block_cap` then bounds the grid, since every block repeats that addition.
template <typename T>
inline cudaError_t launch_bn_apply(cudaStream_t st, const T* x, float* stats, const float* gamma, const float* beta,
                                   const T* res, const float* res_stats, const float* res_gamma, const float* res_beta,
                                   bool relu, T* y, size_t rows, int C, float eps, const float* partial, int nparts,
                                   int block_cap, float* running = nullptr, float momentum = 0.f, unsigned char* bits = nullptr) {
  constexpr int V = full_vec<T>();
  const size_t n = rows * C;
  PartialSums ps{};
  if (partial && nparts > 0) {
    if (2 * C > kEwThreads) return cudaErrorInvalidValue;
    ps.partial = partial; ps.nparts = nparts; ps.kind = 1; ps.inv_count = 1.f / (float)rows; ps.eps = eps;
    ps.save0 = stats; ps.save1 = stats + C;
    ps.run = RunningStats{running, momentum, rows > 1 ? (float)((double)rows / (double)(rows - 1)) : 1.f};
  }
  const int vc = aligned16(gamma) && aligned16(beta) && aligned16(stats) && aligned16(res_stats) && aligned16(res_gamma) &&
                 aligned16(res_beta) && C % 4 == 0;
  const bool vec = C % V == 0;
  const int blocks = ew_grid_for_channels(vec ? n / V : n, vec ? C / V : C, (vec && ps.partial) ? block_cap : 0);
#define FDG_APPLY(VV, R) launch_chained(bn_apply_kernel<T, VV, R>, blocks, kEwThreads, 0, st, x, stats, gamma, beta, res, res_stats, \
      res_gamma, res_beta, (int)relu, vc, y, VV == 8 ? bits : (unsigned char*)nullptr, n / VV, C, ps)
  if (vec) return res_stats ? FDG_APPLY(V, 2) : (res ? FDG_APPLY(V, 1) : FDG_APPLY(V, 0));
  return res_stats ? FDG_APPLY(1, 2) : (res ? FDG_APPLY(1, 1) : FDG_APPLY(1, 0));
#undef FDG_APPLY
}

// First half of the batch-norm backward: the per-channel sums of dz = dy*[gate] (and dz*xhat, dz*xhat2), which are also
// the parameter gradients.  Leaves the rows of partial sums in `scratch`; with *rows_left given and two sums of up to 128
// channels that is all (the apply kernel adds the rows), otherwise the totals go to `sums` [3*C] and the gradients.
template <typename T>
inline cudaError_t launch_bn_bwd_reduce(cudaStream_t st, const T* dy, const GateOf<T> gate, const T* x, const float* stats,
                                        const T* x2, const float* stats2, size_t rows, int C, float* sums,
                                        float* dgamma, float* dbeta, float* dgamma2, float* dbeta2, float* scratch,
                                        int* rows_left, uint64_t* launches) {
  constexpr int V = full_vec<T>();
  const bool two = x2 != nullptr, vec = C % V == 0;
  const RedGeom g = red_geom((int)rows, C, vec ? V : 1, sizeof(T));
#define FDG_RED(VV, K) launch_chained(bn_sums_kernel<T, VV, K>, g.blocks, kRedThreads, 0, st, dy, gate, x, stats, x2, stats2, g, scratch)
  cudaError_t e = vec ? (two ? FDG_RED(V, 3) : FDG_RED(V, 2)) : (two ? FDG_RED(1, 3) : FDG_RED(1, 2));
#undef FDG_RED
  ++*launches;
  if (rows_left) *rows_left = 0;
  if (e != cudaSuccess) return e;
  if (rows_left && !two && 2 * C <= kEwThreads) { *rows_left = g.blocks; return cudaSuccess; }
  ++*launches;
  const dim3 grid((unsigned)((C + 31) / 32));
  const RunningStats none{};
  return two ? launch_chained(sums_finalize_kernel<3>, grid, dim3(1024), 0, st, (const float*)scratch, g.blocks, C, 0.0, 0.f, sums, none, dbeta, dgamma, dbeta2, dgamma2)
             : launch_chained(sums_finalize_kernel<2>, grid, dim3(1024), 0, st, (const float*)scratch, g.blocks, C, 0.0, 0.f, sums, none, dbeta, dgamma, (float*)nullptr, (float*)nullptr);
}

// Second half: dx = gamma*invstd*(dz - s0/M - xhat*s1/M) [+ res] (and dx2 for the second normalised tensor).
// The sums come from `sums`, or, when `partial` != null, from `nparts` rows of per-CTA sums (sum dz, sum dz*xhat)
// left by the data-gradient kernel that produced dy (block 0 then also writes dbeta / dgamma).
template <typename T>
inline cudaError_t launch_bn_bwd_apply(cudaStream_t st, const T* dy, const GateOf<T> gate, const T* x, const float* stats,
                                       const float* gamma, const float* sums, const T* x2, const float* stats2,
                                       const float* gamma2, const T* res, T* dx, T* dx2, size_t rows, int C,
                                       const float* partial, int nparts, float* dgamma, float* dbeta, int block_cap) {
  constexpr int V = full_vec<T>();
  const size_t n = rows * C;
  const float inv_m = 1.f / (float)rows;
  PartialSums ps{};
  if (partial && nparts > 0) {
    if (2 * C > kEwThreads) return cudaErrorInvalidValue;
    ps.partial = partial; ps.nparts = nparts; ps.kind = 2; ps.save0 = dbeta; ps.save1 = dgamma;
  }
  const int vc = aligned16(stats) && aligned16(gamma) && aligned16(sums) && aligned16(stats2) && aligned16(gamma2) && C % 4 == 0;
  const bool vec = C % V == 0;
  const int blocks = ew_grid_for_channels(vec ? n / V : n, vec ? C / V : C, (vec && ps.partial) ? block_cap : 0);
#define FDG_BAPPLY(VV, TWO) launch_chained(bn_bwd_apply_kernel<T, VV, TWO>, blocks, kEwThreads, 0, st, dy, gate, x, stats, gamma, sums, x2, \
      stats2, gamma2, res, vc, dx, dx2, n / VV, C, inv_m, ps)
  if (vec) return dx2 ? FDG_BAPPLY(V, true) : FDG_BAPPLY(V, false);
  return dx2 ? FDG_BAPPLY(1, true) : FDG_BAPPLY(1, false);
#undef FDG_BAPPLY
}

template <typename T>
inline cudaError_t launch_scale(cudaStream_t st, const T* in, T* out, float s, size_t n) {
  constexpr int V = full_vec<T>();
  if (n % V == 0) return launch_chained(scale_kernel<T, V>, ew_blocks(n / V), 256, 0, st, in, out, s, n / V);
  return launch_chained(scale_kernel<T, 1>, ew_blocks(n), 256, 0, st, in, out, s, n);
}

inline cudaError_t launch_sgd(cudaStream_t st, float* theta, float* v, const float* g, float* next32,
                              __nv_bfloat16* next16, size_t n, float lr, const float* lr_dev, float mu, float wd) {
  size_t b = (n / 4 + 255) / 256;
  const int blocks = (int)(b < 1 ? 1 : (b > 148 * 8 ? 148 * 8 : b));
  return launch_chained(sgd_kernel, blocks, 256, 0, st, theta, v, g, next32, next16, n, lr, lr_dev, mu, wd);
}

template <typename T>
inline cudaError_t launch_ingest(cudaStream_t st, const float* img, T* out, size_t rows, int c_in, int c_out,
                                 const int32_t* labels_in, int32_t* labels_out, int batch) {
  return launch_chained(ingest_kernel<T>, ew_blocks(rows * c_out), 256, 0, st, img, out, rows, c_in, c_out, labels_in, labels_out, batch);
}

}  // namespace fdg
