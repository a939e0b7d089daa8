// 3x3 / pad 1 convolutions on the CUDA cores, register-tiled: what the exact fp32 mode runs on, and in bf16 storage the
// layers that the tensor cores do not take (the 3-channel stem).  conv_simt.cuh keeps the general implicit GEMM for
// other filter sizes and paddings.
//
// These layers are bound by fp32 multiply-adds (a 16-channel layer over 128 32x32 images: 8 us at the peak rate of
// 128 per SM and cycle, 3 us of memory traffic), so what counts is that almost every issued instruction is one.
//
// direct_conv_kernel (forward, data gradient).  A block takes TH output rows (or TI whole small images) and up to 32
// output channels; a thread 4 consecutive pixels of a row x NC channels.  The activation tile lies in shared memory
// channel by channel, so the 6 values that three filter taps of a row need are two vector loads and serve 12 * NC
// multiply-adds; the weights of a (channel, tap) are NC / 4 vector loads, the same address for the lanes that share
// channels.  The data gradient of a stride-1 layer is the same convolution with the filter turned by 180 degrees; that
// of a stride-2 layer reads dy spread out onto the input's pixel grid (the loader places it, nothing is materialised).
//
// direct_wgrad_kernel.  A block takes 32 x 32 channels at most and a share of the image rows; a thread 4 input x 4
// output channels of one filter row's three taps: walking along a row of pixels, one new vector of x and one of dy
// serve 48 multiply-adds.  Groups of threads take alternate rows; their sums are added in group order, the blocks'
// partial sums in block order (launch_wgrad_reduce), so the result does not depend on scheduling.  In bf16 storage (the
// stem and narrow projections) only a row's products are added in fp32; rows, groups and blocks are added in fp64.
#pragma once
#include "conv_simt.cuh"

namespace fdg {
namespace direct {

constexpr int kPx = 4;                   // pixels of a thread
constexpr int kKc = 16;                  // activation channels in shared memory at a time
constexpr int kMaxCb = 32;               // output channels of a block: with 64, a block of an 8x8 layer reads 9 KB of weights
                                         // for every KB of activations
constexpr int kPf = 6;                   // activation vectors a thread holds for the next tile while it multiplies this one
constexpr int kThreads = 256;

// Four consecutive elements as floats; elements from `live` on are zeros.
template <typename T, int VEC>
__device__ __forceinline__ void load4(const T* __restrict__ p, int live, float (&v)[4]) {
  if constexpr (VEC == 4) {
    if constexpr (sizeof(T) == 4) {
      const float4 q = *reinterpret_cast<const float4*>(p);
      v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else {
      const uint2 q = *reinterpret_cast<const uint2*>(p);
      const T* e = reinterpret_cast<const T*>(&q);
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = to_f(e[i]);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = i < live ? to_f(p[i]) : 0.f;
  }
}

// x / d for 0 <= x < 2^20 with inv = 1.0f / d (exact: the half keeps the product away from whole numbers).
__device__ __forceinline__ int div_small(int x, float inv) { return (int)(((float)x + 0.5f) * inv); }

struct ConvParams {
  int N, Hi, Wi, Ck;        // activation tensor and its channels (forward: x, Ci; data gradient: dy, Co)
  int P, Q, Cn;             // output tensor [N][P][Q][Cn]
  int up;                   // 1, or 2: the activation's pixels lie at the even positions of a grid twice as fine
  int TH, TI;               // output rows (per image) and images per tile
  int segs;                 // 4-pixel segments per row
  int row_tiles, tiles;     // tiles per image (1 when TI > 1), tiles in all
  int rows_in, pitch, plane;// activation tile: rows per image, floats per row, floats per channel
  int cb, cgs;              // output channels of a block, thread columns cb / NC
  int wvec;                 // the weights can be read four at a time
  int vec;                  // the output-shaped tensors are 16-byte aligned and Cn is a multiple of 4
};

// A per-channel reduction over what the kernel stores, one row of 2 * Cn floats per blockIdx.x (modes as in the
// tensor-core kernels: 1 = sum v, sum v^2; 2 = the sums of the batch-norm backward that v feeds).
template <typename T> struct Reduce {
  int mode;
  const T* mask;
  const T* xprev;
  const float* pstats;
  float* partial;
};

template <typename T, int VEC, int STRIDE, int NC, bool FLIP>
__global__ void __launch_bounds__(kThreads, 2)
direct_conv_kernel(ConvParams p, const T* __restrict__ act, const T* __restrict__ wgt, T* __restrict__ out,
                   const T* __restrict__ res, const T* __restrict__ res_mask, Reduce<T> red, EpiAffine aff) {
  grid_dependency_wait();
  extern __shared__ __align__(16) float dc_smem[];
  float* sa = dc_smem;                                       // [kKc][plane]
  float* sw = dc_smem + kKc * p.plane;                       // [kKc][9][cb]
  const int tid = threadIdx.x;
  const int cg = tid % p.cgs, sid = tid / p.cgs;             // thread column, segment of the tile
  const int n_segs = p.TI * p.TH * p.segs;
  const bool active = sid < n_segs;
  const int ti = sid / (p.TH * p.segs), th = (sid / p.segs) % p.TH, sg = sid % p.segs;
  const int n0 = blockIdx.y * p.cb, c0 = n0 + cg * NC;       // first output channel of the block, of this thread
  const int chunks = (p.Ck + kKc - 1) / kKc;
  const int win = p.Wi * p.up, hin = p.Hi * p.up;            // size of the grid the filter slides over
  const float* a_base = sa + ((ti * p.rows_in + th * STRIDE) * p.pitch + sg * kPx * STRIDE);
  float s0[NC], s1[NC];
#pragma unroll
  for (int j = 0; j < NC; ++j) s0[j] = s1[j] = 0.f;

  // activations of one (tile, chunk): items = (pixel of the bordered tile, 4-channel group).  The first kPf * kThreads of
  // them are requested one step ahead into registers (`fetch`), so that their latency runs beside the multiplication;
  // where they lie in the tile and in the tensor is worked out once.
  const int cols = win + 2;
  const int kv = min(kKc, (p.Ck + 3) & ~3) / 4;              // 4-channel groups of a chunk (the last may have fewer channels)
  const int items = p.TI * p.rows_in * cols * kv;
  const float inv_cols = 1.f / (float)cols, inv_rows = 1.f / (float)p.rows_in, inv_kv = 1.f / (float)kv;
  struct Item { int s_off, g_off, row; };                    // row = (image << 16) | row of the tile; < 0: a border column
  auto item_of = [&](int i) {
    Item it;
    const int px = div_small(i, inv_kv), g4 = i - px * kv;
    const int rr = div_small(px, inv_cols), col = px - rr * cols;
    const int im = div_small(rr, inv_rows), lr = rr - im * p.rows_in;
    it.s_off = 4 * g4 * p.plane + rr * p.pitch + col;
    const int w = col - 1;
    const bool ok = w >= 0 && w < win && (p.up == 1 || (w & 1) == 0);
    it.row = ok ? (im << 16) | lr : -1;
    it.g_off = (p.up == 1 ? ((im * p.Hi + lr - 1) * p.Wi + w) : (im * p.Hi * p.Wi + (w >> 1))) * p.Ck + 4 * g4;
    return it;
  };
  auto load_item = [&](int tile, int ch, const Item& it, int i, float (&v)[4]) {
    v[0] = v[1] = v[2] = v[3] = 0.f;
    const int img0 = (tile / p.row_tiles) * p.TI, row0 = (tile % p.row_tiles) * p.TH;
    const int im = it.row >> 16, h = row0 * STRIDE + (it.row & 0xffff) - 1;
    if (it.row < 0 || h < 0 || h >= hin || img0 + im >= p.N) return;
    const int k0 = ch * kKc;
    if (VEC == 4 && k0 + kKc > p.Ck && k0 + 4 * (i - div_small(i, inv_kv) * kv) >= p.Ck) return;   // past the last channel
    const T* base = act + ((size_t)img0 * p.Hi + (p.up == 1 ? row0 * STRIDE : 0)) * (size_t)p.Wi * p.Ck + k0;
    int off = it.g_off;
    if (p.up == 2) { if (h & 1) return; off += (h >> 1) * p.Wi * p.Ck; }
    load4<T, VEC>(base + off, VEC == 4 ? 4 : p.Ck - k0 - 4 * (i - div_small(i, inv_kv) * kv), v);
  };
  auto store_item = [&](const Item& it, const float (&v)[4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) sa[it.s_off + j * p.plane] = v[j];
  };
  float pf[kPf][4];
  Item pfi[kPf];
#pragma unroll
  for (int u = 0; u < kPf; ++u) pfi[u] = item_of(tid + u * kThreads);
  auto fetch = [&](int tile, int ch) {
#pragma unroll
    for (int u = 0; u < kPf; ++u)
      if (tid + u * kThreads < items) load_item(tile, ch, pfi[u], tid + u * kThreads, pf[u]);
  };
  if ((int)blockIdx.x < p.tiles) fetch(blockIdx.x, 0);

  for (int tile = blockIdx.x; tile < p.tiles; tile += gridDim.x) {
    const int img0 = (tile / p.row_tiles) * p.TI, row0 = (tile % p.row_tiles) * p.TH;
    float acc[kPx][NC];
#pragma unroll
    for (int i = 0; i < kPx; ++i)
#pragma unroll
      for (int j = 0; j < NC; ++j) acc[i][j] = 0.f;
    for (int ch = 0; ch < chunks; ++ch) {
      const int k0 = ch * kKc, kc = min(kKc, p.Ck - k0);
      __syncthreads();                                       // the previous chunk has been multiplied
#pragma unroll
      for (int u = 0; u < kPf; ++u)
        if (tid + u * kThreads < items) store_item(pfi[u], pf[u]);
      for (int i = tid + kPf * kThreads; i < items; i += kThreads) {
        float v[4];
        const Item it = item_of(i);
        load_item(tile, ch, it, i, v);
        store_item(it, v);
      }
      // weights: sw[channel][tap][output channel]; they stay where one chunk holds all channels
      if (chunks > 1 || tile == (int)blockIdx.x) {
        const int c4 = p.cb >> 2, kw = (kc + 3) / 4, wn = FLIP ? kc * 9 * c4 : kw * 9 * p.cb;
        for (int i0 = tid; i0 < wn; i0 += 4 * kThreads) {
          float v[4][4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * kThreads;
            v[u][0] = v[u][1] = v[u][2] = v[u][3] = 0.f;
            if (i >= wn) continue;
            if (FLIP) {                                      // w[k][8 - tap][n]: four output channels
              const int kt = i / c4, n = (i - kt * c4) * 4, k = kt / 9, tap = kt - 9 * k;
              if (n0 + n < p.Cn) {
                const T* src = wgt + ((size_t)(k0 + k) * 9 + 8 - tap) * p.Cn + n0 + n;
                if (p.wvec) load4<T, 4>(src, 4, v[u]); else load4<T, 1>(src, p.Cn - n0 - n, v[u]);
              }
            } else {                                         // w[n][tap][k]: four activation channels
              const int vt = i / p.cb, n = i - vt * p.cb, g4 = vt / 9, tap = vt - 9 * g4;
              if (n0 + n < p.Cn) {
                const T* src = wgt + ((size_t)(n0 + n) * 9 + tap) * p.Ck + k0 + 4 * g4;
                if (p.wvec) load4<T, 4>(src, 4, v[u]); else load4<T, 1>(src, kc - 4 * g4, v[u]);
              }
            }
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * kThreads;
            if (i >= wn) continue;
            if (FLIP) {
              *reinterpret_cast<float4*>(sw + 4 * i) = make_float4(v[u][0], v[u][1], v[u][2], v[u][3]);
            } else {
              const int vt = i / p.cb, n = i - vt * p.cb, g4 = vt / 9, tap = vt - 9 * g4;
#pragma unroll
              for (int j = 0; j < 4; ++j) sw[((4 * g4 + j) * 9 + tap) * p.cb + n] = v[u][j];
            }
          }
        }
      }
      {                                                      // the next step's activations
        int nt = tile, nc = ch + 1;
        if (nc == chunks) { nc = 0; nt += gridDim.x; }
        if (nt < p.tiles) fetch(nt, nc);
      }
      __syncthreads();
      if (active) {
        for (int k = 0; k < kc; ++k) {
          const float* ap = a_base + k * p.plane;
          const float* wp = sw + k * 9 * p.cb + cg * NC;
#pragma unroll
          for (int r = 0; r < 3; ++r) {
            constexpr int WIN = (kPx - 1) * STRIDE + 3;      // 6 or 9 values
            float a[WIN];
            const float4 q0 = *reinterpret_cast<const float4*>(ap + r * p.pitch);
            a[0] = q0.x; a[1] = q0.y; a[2] = q0.z; a[3] = q0.w;
            if constexpr (STRIDE == 1) {
              const float2 q1 = *reinterpret_cast<const float2*>(ap + r * p.pitch + 4);
              a[4] = q1.x; a[5] = q1.y;
            } else {
              const float4 q1 = *reinterpret_cast<const float4*>(ap + r * p.pitch + 4);
              a[4] = q1.x; a[5] = q1.y; a[6] = q1.z; a[7] = q1.w;
              a[8] = ap[r * p.pitch + 8];
            }
#pragma unroll
            for (int s = 0; s < 3; ++s) {
              float w[NC];
#pragma unroll
              for (int j = 0; j < NC; j += 4) {
                const float4 q = *reinterpret_cast<const float4*>(wp + (r * 3 + s) * p.cb + j);
                w[j] = q.x; w[j + 1] = q.y; w[j + 2] = q.z; w[j + 3] = q.w;
              }
#pragma unroll
              for (int i = 0; i < kPx; ++i)
#pragma unroll
                for (int j = 0; j < NC; ++j) acc[i][j] = fmaf(a[i * STRIDE + s], w[j], acc[i][j]);
            }
          }
        }
      }
    }
    // ---- store (+ residual), sums of the stored values
    const int n = img0 + ti, h = row0 + th;
    if (active && n < p.N && h < p.P && c0 < p.Cn) {
      const int live = p.Cn - c0;
#pragma unroll
      for (int i = 0; i < kPx; ++i) {
        const int q = sg * kPx + i;
        if (q >= p.Q) break;
        const size_t base = (((size_t)n * p.P + h) * p.Q + q) * p.Cn + c0;
#pragma unroll
        for (int j = 0; j < NC; j += 4) {
          if (j >= live) break;
          float v[4] = {acc[i][j], acc[i][j + 1], acc[i][j + 2], acc[i][j + 3]};
          const bool vec = p.vec != 0;
          if (aff.stats) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              if (j + e >= live) break;
              const int c = c0 + j + e;
              const float x = to_f(from_f<T>(v[e])) - aff.stats[c], g = aff.gamma[c], iv = aff.stats[p.Cn + c];
              v[e] = sizeof(T) == 4 ? g * (x * iv) + aff.beta[c] : fmaf(x, g * iv, aff.beta[c]);
            }
          }
          if (res) {
            float rv[4], mv[4] = {1.f, 1.f, 1.f, 1.f};
            if (vec) load4<T, 4>(res + base + j, 4, rv); else load4<T, 1>(res + base + j, live - j, rv);
            if (res_mask) { if (vec) load4<T, 4>(res_mask + base + j, 4, mv); else load4<T, 1>(res_mask + base + j, live - j, mv); }
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] += mv[e] > 0.f ? rv[e] : 0.f;
          }
          T o[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) o[e] = from_f<T>(aff.relu ? fmaxf(v[e], 0.f) : v[e]);
          if (vec) {
            if constexpr (sizeof(T) == 4) *reinterpret_cast<float4*>(out + base + j) = *reinterpret_cast<const float4*>(o);
            else *reinterpret_cast<uint2*>(out + base + j) = *reinterpret_cast<const uint2*>(o);
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) if (j + e < live) out[base + j + e] = o[e];
          }
          if (red.mode == 1) {
#pragma unroll
            for (int e = 0; e < 4; ++e) { const float t = to_f(o[e]); s0[j + e] += t; s1[j + e] += t * t; }
          } else if (red.mode == 2) {                        // only with vector-sized channel counts
            float mv[4], xv[4];
            load4<T, 4>(red.mask + base + j, 4, mv);
            load4<T, 4>(red.xprev + base + j, 4, xv);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float dz = mv[e] > 0.f ? to_f(o[e]) : 0.f;
              s0[j + e] += dz;
              s1[j + e] += dz * ((xv[e] - red.pstats[c0 + j + e]) * red.pstats[p.Cn + c0 + j + e]);
            }
          }
        }
      }
    }
  }
  if (red.mode) {
    // this block's sums: every segment's thread leaves its own in shared memory; kThreads / (2 * cb) threads share a
    // (sum, channel) pair, each taking every parts-th segment, and their totals are added in order
    __syncthreads();
    float* buf = dc_smem;                                    // [segments][2][cb]; see conv_smem_bytes
    __shared__ double part[kThreads];
    if (active) {
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        buf[(sid * 2 + 0) * p.cb + cg * NC + j] = s0[j];
        buf[(sid * 2 + 1) * p.cb + cg * NC + j] = s1[j];
      }
    }
    __syncthreads();
    const int pairs = 2 * p.cb, parts = kThreads / pairs;
    const int t = tid % pairs, pt = tid / pairs;
    double a = 0.0;
    if (pt < parts)
      for (int s = pt; s < n_segs; s += parts) a += (double)buf[s * pairs + t];
    part[tid] = a;
    __syncthreads();
    if (pt == 0) {
      for (int q = 1; q < parts; ++q) a += part[q * pairs + t];
      const int stat = t / p.cb, c = t - stat * p.cb;
      if (n0 + c < p.Cn) red.partial[(size_t)blockIdx.x * 2 * p.Cn + (size_t)stat * p.Cn + n0 + c] = (float)a;
    }
  }
}

// Rows of partial sums a launch may leave (its blocks along x): what the callers' buffers hold.
constexpr int kMaxRows = FDG_CONV_PARTIAL_ROWS;

inline bool conv_supported(const ConvGeom& g, bool dgrad) {
  if (g.R != 3 || g.S != 3 || g.pad != 1) return false;
  if (g.stride == 1) { if (g.P != g.H || g.Q != g.W) return false; }
  else if (g.stride == 2) {
    if (g.H % 2 || g.W % 2 || g.P != g.H / 2 || g.Q != g.W / 2) return false;
  } else return false;
  return (dgrad ? g.W : g.Q) <= 64 && g.W <= 64;
}

constexpr size_t kConvSmemMax = 160 * 1024;
inline ConvParams conv_params(const ConvGeom& g, bool dgrad, int nc) {
  ConvParams p{};
  const int stride = dgrad ? 1 : g.stride;
  p.N = g.N;
  p.Hi = dgrad ? g.P : g.H; p.Wi = dgrad ? g.Q : g.W; p.Ck = dgrad ? g.Co : g.Ci;
  p.P = dgrad ? g.H : g.P; p.Q = dgrad ? g.W : g.Q; p.Cn = dgrad ? g.Ci : g.Co;
  p.up = dgrad ? g.stride : 1;
  p.segs = (p.Q + kPx - 1) / kPx;
  // output channels of a block: equal shares of at most kMaxCb, whole thread columns
  const int blocks_n = (p.Cn + kMaxCb - 1) / kMaxCb;
  p.cb = ((p.Cn + blocks_n - 1) / blocks_n + nc - 1) / nc * nc;
  p.cgs = p.cb / nc;
  // rows: what fills the block and fits shared memory, in equal shares of an image; whole images where one does not
  // fill a block
  int rows = kThreads / p.cgs / p.segs;
  if (rows < 1) rows = 1;
  p.pitch = ((p.segs * kPx - 1) * stride + 3 + 3) / 4 * 4;
  if (p.pitch < p.Wi * p.up + 2) p.pitch = (p.Wi * p.up + 2 + 3) / 4 * 4;
  while (rows > 1 && (size_t)kKc * (rows * stride + 2) * p.pitch * 4 > 96 * 1024) rows /= 2;
  if (rows >= p.P) { p.TH = p.P; p.TI = std::max(1, std::min(rows / p.P, p.N / kSms)); }
  else { const int t = (p.P + rows - 1) / rows; p.TH = (p.P + t - 1) / t; p.TI = 1; }
  p.rows_in = (p.TH - 1) * stride + 3;
  // Every image of a tile has border rows of its own, which the bound above does not count: images of one or two rows
  // take up to three times the shared memory of their output rows.
  while (p.TI > 1 && ((size_t)kKc * (p.TI * p.rows_in * p.pitch + 4) + (size_t)kKc * 9 * p.cb) * 4 > kConvSmemMax) --p.TI;
  p.row_tiles = (p.P + p.TH - 1) / p.TH;
  p.tiles = ((p.N + p.TI - 1) / p.TI) * p.row_tiles;
  p.plane = p.TI * p.rows_in * p.pitch;
  if (p.plane % 8 == 0) p.plane += 4;                        // 4-channel groups of a warp's stores on different banks
  return p;
}
inline size_t conv_smem_bytes(const ConvParams& p) {
  const size_t tiles = (size_t)kKc * p.plane + (size_t)kKc * 9 * p.cb;
  const size_t sums = (size_t)p.TI * p.TH * p.segs * 2 * p.cb;
  return (tiles > sums ? tiles : sums) * 4;
}

template <typename T, int VEC, int STRIDE, int NC, bool FLIP>
inline cudaError_t conv_launch_one(cudaStream_t st, const ConvParams& p, int grid, const T* act, const T* wgt, T* out,
                                   const T* res, const T* mask, const Reduce<T>& red, const EpiAffine& aff) {
  auto kernel = direct_conv_kernel<T, VEC, STRIDE, NC, FLIP>;
  static OncePerDevice once;
  const cudaError_t e = once_per_device(&once, [&]() { return set_smem_limit(kernel, kConvSmemMax); });
  if (e != cudaSuccess) return e;
  return launch_chained(kernel, dim3(grid, (p.Cn + p.cb - 1) / p.cb), dim3(kThreads), conv_smem_bytes(p), st, p, act, wgt, out, res, mask, red, aff);
}

// y = conv3x3(x, w) [+ res], or (dgrad) dx = conv^T(dy, w) [+ res * [mask > 0]].  `red` (nullable) asks for the rows of
// sums described at Reduce, *nparts receives their number.
template <typename T>
inline cudaError_t launch_conv(cudaStream_t st, const ConvGeom& g, bool dgrad, const T* act, const T* wgt, T* out, const T* res,
                               const T* mask, const Reduce<T>* red, int* nparts, uint64_t* launches,
                               const EpiAffine* affine = nullptr) {
  // With 8 channels per thread 8 shared-memory loads serve 96 multiply-adds, with 4 channels 5 serve 48; 4 where 8 would
  // leave an SM fewer than four warps (fp32, 128 images, 8 / 4 channels per thread: 16 channels on 32x32, 14 warps per SM,
  // 22.3 / 24.9 us; 32 on 16x16, 7 warps, 25.3 / 24.2; 64 on 8x8, 3.5 warps, 46.4 / 30.9).  (Packed two-wide multiply-adds were
  // tried: the moves that form their operand pairs go through the same pipe, no gain.)
  const long pixels4 = (long)g.N * (dgrad ? g.H : g.P) * (((dgrad ? g.W : g.Q) + kPx - 1) / kPx);
  const int cn = dgrad ? g.Ci : g.Co;
  const bool wide = cn % 8 == 0 && pixels4 * (cn / 8) >= (long)kSms * 128;
  ConvParams p = conv_params(g, dgrad, wide ? 8 : 4);
  p.wvec = g.Ci % 4 == 0 && (reinterpret_cast<uintptr_t>(wgt) & 15) == 0;   // contiguous along Ci either way
  p.vec = cn % 4 == 0 && ((reinterpret_cast<uintptr_t>(out) | reinterpret_cast<uintptr_t>(res) | reinterpret_cast<uintptr_t>(mask) |
                           (red ? reinterpret_cast<uintptr_t>(red->mask) | reinterpret_cast<uintptr_t>(red->xprev) : 0)) & 15) == 0;
  if (red && red->mode == 2 && !p.vec) red = nullptr;
  int grid = p.tiles;
  const int cap = red ? kMaxRows : 4 * kSms;
  if (grid > cap) { const int per = (grid + cap - 1) / cap; grid = (grid + per - 1) / per; }
  const bool vec = p.Ck % 4 == 0 && (reinterpret_cast<uintptr_t>(act) & 15) == 0;
  Reduce<T> r{};
  if (red) r = *red;
  const EpiAffine a = affine ? *affine : EpiAffine{};
  if (nparts) *nparts = red ? grid : 0;
  ++*launches;
#define FDG_DC(V, S, C, F) return conv_launch_one<T, V, S, C, F>(st, p, grid, act, wgt, out, res, mask, r, a)
  if (dgrad) {
    if (vec) { if (wide) FDG_DC(4, 1, 8, true); FDG_DC(4, 1, 4, true); }
    if (wide) FDG_DC(1, 1, 8, true);
    FDG_DC(1, 1, 4, true);
  }
  if (g.stride == 1) {
    if (vec) { if (wide) FDG_DC(4, 1, 8, false); FDG_DC(4, 1, 4, false); }
    if (wide) FDG_DC(1, 1, 8, false);
    FDG_DC(1, 1, 4, false);
  }
  if (vec) { if (wide) FDG_DC(4, 2, 8, false); FDG_DC(4, 2, 4, false); }
  if (wide) FDG_DC(1, 2, 8, false);
  FDG_DC(1, 2, 4, false);
#undef FDG_DC
}

// ------------------------------------------------------------- weight gradient --
constexpr int kWgCi = 32, kWgCo = 32;        // channels of a block at most
constexpr size_t kWgradSmemMax = 176 * 1024;  // what a block may use: one group of 192 threads with fp64 sums takes up to 170 KB
struct WgradParams {
  int N, H, W, Ci, P, Q, Co;
  int cib, cob, ci_blocks;      // channels per block (multiples of 4), blocks along ci
  int ct, ot, tt;               // 4-channel groups, threads of one row group: ct * ot * R
  int rg, threads;              // row groups, threads of the block
  int TH, strips, units;        // dy rows per step, steps per image, steps in all
  int xrow, rows_x;             // floats per x row in shared memory, x rows per step
  int splits;                   // blocks along the pixels
};

template <typename T> constexpr bool kByRow = sizeof(T) == 2;         // rows are added in fp64

template <typename T, int VECX, int VECY, int R, int STRIDE>
__global__ void __launch_bounds__(kThreads)
direct_wgrad_kernel(WgradParams p, const T* __restrict__ x, const T* __restrict__ dy, float* __restrict__ partial) {
  grid_dependency_wait();
  constexpr int PAD = R == 3 ? 1 : 0;
  constexpr bool BY_ROW = kByRow<T>;
  extern __shared__ __align__(16) float dw_smem[];
  float* sx = dw_smem;                                       // [rows_x][W + 2 * PAD][cib], rows padded to xrow
  float* sy = dw_smem + p.rows_x * p.xrow;                   // [TH][Q][cob]
  // By rows: the groups leave their row's products in ex[value][thread] (a value per tap, output and input channel of a
  // thread), and the block's fp64 totals [value][thread of a group] are divided among all threads: in the registers of the
  // thread that multiplies they would halve the blocks of an SM (stem of 128 32x32 images: 26.9 us, this way 13.3).
  float* ex = sy + p.TH * p.Q * p.cob;
  double* total = reinterpret_cast<double*>(ex + p.rg * p.tt * 16 * R);
  const int tid = threadIdx.x;
  const int ci0 = (blockIdx.y % p.ci_blocks) * p.cib, co0 = (blockIdx.y / p.ci_blocks) * p.cob;
  const int grp = tid / p.tt, t = tid - grp * p.tt;          // row group, thread of the tile
  const int c = t % p.ct, o = (t / p.ct) % p.ot, r = t / (p.ct * p.ot);
  const bool active = grp < p.rg;
  const int cols = p.W + 2 * PAD;
  float acc[R][4][4];                                        // [tap of the row][output channel][input channel]
#pragma unroll
  for (int s = 0; s < R; ++s)
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[s][i][j] = 0.f;
  if (BY_ROW && active) for (int v = grp; v < 16 * R; v += p.rg) total[v * p.tt + t] = 0.0;
  const float inv_ct = 1.f / (float)p.ct, inv_ot = 1.f / (float)p.ot, inv_cols = 1.f / (float)cols;
  for (int u = blockIdx.x; u < p.units; u += gridDim.x) {
    const int n = u / p.strips, p0 = (u - n * p.strips) * p.TH;
    const int rows = min(p.TH, p.P - p0);
    __syncthreads();
    const T* xn = x + (size_t)n * p.H * p.W * p.Ci;
    const T* yn = dy + (size_t)n * p.P * p.Q * p.Co;
    // (four vectors in flight per thread)
    const int xitems = p.rows_x * cols * p.ct, yitems = rows * p.Q * p.ot;
    for (int i0 = tid; i0 < xitems; i0 += 4 * p.threads) {
      float q[4][4];
      int at[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int i = i0 + k * p.threads;
        q[k][0] = q[k][1] = q[k][2] = q[k][3] = 0.f;
        at[k] = -1;
        if (i >= xitems) continue;
        const int px = div_small(i, inv_ct), v = i - px * p.ct;
        const int rr = div_small(px, inv_cols), col = px - rr * cols;
        const int h = p0 * STRIDE + rr - PAD, w = col - PAD;
        at[k] = rr * p.xrow + col * p.cib + 4 * v;
        if (h >= 0 && h < p.H && w >= 0 && w < p.W && ci0 + 4 * v < p.Ci)
          load4<T, VECX>(xn + ((size_t)h * p.W + w) * p.Ci + ci0 + 4 * v, p.Ci - ci0 - 4 * v, q[k]);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (at[k] >= 0) *reinterpret_cast<float4*>(sx + at[k]) = make_float4(q[k][0], q[k][1], q[k][2], q[k][3]);
    }
    for (int i0 = tid; i0 < yitems; i0 += 4 * p.threads) {
      float q[4][4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int i = i0 + k * p.threads;
        q[k][0] = q[k][1] = q[k][2] = q[k][3] = 0.f;
        const int px = div_small(i, inv_ot), v = i - px * p.ot;
        if (i < yitems && co0 + 4 * v < p.Co)
          load4<T, VECY>(yn + ((size_t)p0 * p.Q + px) * p.Co + co0 + 4 * v, p.Co - co0 - 4 * v, q[k]);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (i0 + k * p.threads < yitems)
          *reinterpret_cast<float4*>(sy + 4 * (i0 + k * p.threads)) = make_float4(q[k][0], q[k][1], q[k][2], q[k][3]);
    }
    __syncthreads();
    auto add_row = [&](int row) {
      const float* xp = sx + (row * STRIDE + r) * p.xrow + 4 * c;
      const float* yp = sy + row * p.Q * p.cob + 4 * o;
      float4 w0, w1, w2;                                     // x at the taps of this pixel
      auto xat = [&](int px) { return *reinterpret_cast<const float4*>(xp + px * p.cib); };
      if constexpr (R == 3) {
        if constexpr (STRIDE == 1) { w1 = xat(0); w2 = xat(1); } else w2 = xat(0);
      }
#pragma unroll 4
      for (int q = 0; q < p.Q; ++q) {
        const float4 d = *reinterpret_cast<const float4*>(yp + q * p.cob);
        if constexpr (R == 3) {
          if constexpr (STRIDE == 1) { w0 = w1; w1 = w2; w2 = xat(q + 2); }
          else { w0 = w2; w1 = xat(2 * q + 1); w2 = xat(2 * q + 2); }
        } else {
          w0 = xat(q * STRIDE);
        }
        const float dv[4] = {d.x, d.y, d.z, d.w};
        const float xv[3][4] = {{w0.x, w0.y, w0.z, w0.w}, {w1.x, w1.y, w1.z, w1.w}, {w2.x, w2.y, w2.z, w2.w}};
#pragma unroll
        for (int s = 0; s < R; ++s)
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[s][i][j] = fmaf(dv[i], xv[s][j], acc[s][i][j]);
      }
    };
    if constexpr (!BY_ROW) {
      if (active)
        for (int row = grp; row < rows; row += p.rg) add_row(row);
    } else {
      for (int row0 = 0; row0 < rows; row0 += p.rg) {
#pragma unroll
        for (int s = 0; s < R; ++s)
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[s][i][j] = 0.f;
        if (row0) __syncthreads();                           // the row before has been added (the first: behind the tiles' barriers)
        if (active && row0 + grp < rows) add_row(row0 + grp);
        if (active) {
#pragma unroll
          for (int s = 0; s < R; ++s)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j) ex[((s * 4 + i) * 4 + j) * (p.rg * p.tt) + tid] = acc[s][i][j];
        }
        __syncthreads();
        if (active)
          for (int v = grp; v < 16 * R; v += p.rg) {
            const float* e = ex + v * p.rg * p.tt + t;
            double a = total[v * p.tt + t];
#pragma unroll 4
            for (int g = 0; g < p.rg; ++g) a += (double)e[g * p.tt];
            total[v * p.tt + t] = a;
          }
      }
    }
  }
  if constexpr (BY_ROW) {
    if (!active) return;
    float* dst = partial + (size_t)blockIdx.x * p.Co * R * R * p.Ci;
    for (int v = grp; v < 16 * R; v += p.rg) {
      const int s = v >> 4, co = co0 + 4 * o + ((v >> 2) & 3), ci = ci0 + 4 * c + (v & 3);
      if (co < p.Co && ci < p.Ci) dst[(((size_t)co * R + r) * R + s) * p.Ci + ci] = (float)total[v * p.tt + t];
    }
  } else {
    // the row groups' sums, added in group order through shared memory
    for (int g = 1; g < p.rg; ++g) {
      __syncthreads();
      if (grp == g) {
#pragma unroll
        for (int s = 0; s < R; ++s)
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) dw_smem[((s * 4 + i) * 4 + j) * p.tt + t] = acc[s][i][j];
      }
      __syncthreads();
      if (grp == 0) {
#pragma unroll
        for (int s = 0; s < R; ++s)
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[s][i][j] += dw_smem[((s * 4 + i) * 4 + j) * p.tt + t];
      }
    }
    if (grp == 0) {
      float* dst = partial + (size_t)blockIdx.x * p.Co * R * R * p.Ci;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int co = co0 + 4 * o + i;
        if (co >= p.Co) continue;
#pragma unroll
        for (int s = 0; s < R; ++s)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int ci = ci0 + 4 * c + j;
            if (ci < p.Ci) dst[(((size_t)co * R + r) * R + s) * p.Ci + ci] = acc[s][i][j];
          }
      }
    }
  }
}

inline bool wgrad_direct_supported(const ConvGeom& g) {
  if (g.R == 3) { if (!conv_supported(g, false)) return false; }
  else if (g.R != 1 || g.S != 1 || g.pad != 0 || g.stride > 2 || g.W > 64) return false;
  return true;
}
// Bytes of shared memory of a block: tiles of `rows` rows of dy; the groups' sums over them (one group's at a time) or, by
// rows, behind them (all groups', and the totals).
inline size_t wgrad_smem(const WgradParams& p, int R, int stride, int rows, bool by_row) {
  const size_t tile = (((size_t)(rows - 1) * stride + R) * p.xrow + (size_t)rows * p.Q * p.cob) * 4;
  const size_t values = (size_t)p.tt * 16 * R, sums = p.rg > 1 ? values * 4 : 0;
  return by_row ? tile + values * (4 * p.rg + 8) : (tile > sums ? tile : sums);
}
inline WgradParams wgrad_params(const ConvGeom& g, bool by_row) {
  WgradParams p{};
  p.N = g.N; p.H = g.H; p.W = g.W; p.Ci = g.Ci; p.P = g.P; p.Q = g.Q; p.Co = g.Co;
  p.ci_blocks = (g.Ci + kWgCi - 1) / kWgCi;
  const int co_blocks = (g.Co + kWgCo - 1) / kWgCo;
  p.cib = ((g.Ci + p.ci_blocks - 1) / p.ci_blocks + 3) / 4 * 4;
  p.cob = ((g.Co + co_blocks - 1) / co_blocks + 3) / 4 * 4;
  p.ct = p.cib / 4; p.ot = p.cob / 4; p.tt = p.ct * p.ot * g.R;
  p.rg = std::min(kThreads / p.tt, 16);
  while (p.rg > 1 && g.P % p.rg && p.rg > g.P / 2) --p.rg;      // rows of an image in whole turns where that costs few threads
  if (p.rg > 4 && g.P % p.rg) p.rg = 4;
  if (p.rg > g.P) p.rg = g.P;
  if (p.rg < 1) p.rg = 1;
  const int pad = g.R == 3 ? 1 : 0;
  p.xrow = (g.W + 2 * pad) * p.cib + (p.cib <= 16 ? 16 : 0);     // rows of a warp's taps on different banks
  // A step holds a row of dy (and its rows of x) for every group: wide rows of many channels leave room for fewer groups.
  // One group always fits, with the four rows that it may take below.
  while (p.rg > 1 && wgrad_smem(p, g.R, g.stride, p.rg, by_row) > kWgradSmemMax) --p.rg;
  p.threads = (p.rg * p.tt + 31) / 32 * 32;
  // rows per step: whole turns of the row groups, about four rows within 40 KB of shared memory, in equal shares of an
  // image (every step reads two rows of x more than it has rows of dy)
  const int row_floats = p.xrow * g.stride + g.Q * p.cob;
  const int turns = std::max(1, std::min(4 / p.rg, 10 * 1024 / row_floats / p.rg));
  p.strips = (g.P + turns * p.rg - 1) / (turns * p.rg);
  p.TH = (g.P + p.strips - 1) / p.strips;
  p.units = g.N * p.strips;
  p.rows_x = (p.TH - 1) * g.stride + g.R;
  // Blocks along the pixels: the number that leaves the busiest SM the fewest steps (up to two blocks share an SM), as long as
  // the partial sums stay below about twice the operands (they are written and read again).  A block alone on its SM waits
  // for its loads: fp32, 16 channels, 128 images of 32x32, 28.7 us on 148 blocks of 7 steps, 22.3 us on 296 of 4, i.e. 1.47
  // times as long a step; 512 images 107 us (28 steps) and 73.4 us (14), 1.46.  Counted as 1.3: with 1.47 the 64-channel
  // layers would take 208 blocks instead of 148, 26.9 us instead of 27.0, and 40 % more partial sums.
  const int pairs = p.ci_blocks * co_blocks;
  const size_t outs = (size_t)g.Co * g.R * g.R * g.Ci;
  const size_t operands = (size_t)g.N * ((size_t)g.H * g.W * g.Ci + (size_t)g.P * g.Q * g.Co);
  int most = (int)std::min<size_t>(std::max<size_t>(2 * operands / outs, 1), (size_t)p.units);
  most = std::min(most, std::max(1, 2 * kSms / pairs));
  int best = 1;
  long best_cost = -1;
  for (int sp = 1; sp <= most; ++sp) {
    const int per = (p.units + sp - 1) / sp;
    if ((p.units + per - 1) / per != sp) continue;
    const int blocks_per_sm = (sp * pairs + kSms - 1) / kSms;
    const long cost = (long)per * blocks_per_sm * (blocks_per_sm == 1 ? 13 : 10);
    if (best_cost < 0 || cost < best_cost) { best = sp; best_cost = cost; }
  }
  p.splits = best;
  return p;
}
inline size_t wgrad_direct_scratch_elems(const ConvGeom& g, bool by_row) {
  return wgrad_direct_supported(g) ? (size_t)wgrad_params(g, by_row).splits * g.Co * g.R * g.R * g.Ci : 0;
}

template <typename T, int VX, int VY, int R, int STRIDE>
inline cudaError_t wgrad_launch_one(cudaStream_t st, const WgradParams& p, const T* x, const T* dy, float* dst) {
  auto kernel = direct_wgrad_kernel<T, VX, VY, R, STRIDE>;
  static OncePerDevice once;
  const cudaError_t e = once_per_device(&once, [&]() { return set_smem_limit(kernel, kWgradSmemMax); });
  if (e != cudaSuccess) return e;
  const int pairs = p.ci_blocks * ((p.Co + p.cob - 1) / p.cob);
  return launch_chained(kernel, dim3(p.splits, pairs), dim3(p.threads), wgrad_smem(p, R, STRIDE, p.TH, kByRow<T>), st, p, x, dy, dst);
}

// dw [Co][R][R][Ci] (fp32) from x and dy; `scratch` of wgrad_direct_scratch_elems floats.
template <typename T>
inline cudaError_t launch_wgrad(cudaStream_t st, const ConvGeom& g, const T* x, const T* dy, float* scratch, float* dw,
                                uint64_t* launches) {
  const WgradParams p = wgrad_params(g, kByRow<T>);
  float* dst = p.splits == 1 ? dw : scratch;
  const bool vx = g.Ci % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0;
  const bool vy = g.Co % 4 == 0 && (reinterpret_cast<uintptr_t>(dy) & 15) == 0;
  cudaError_t e;
  ++*launches;
#define FDG_DW(R, S) (vx ? (vy ? wgrad_launch_one<T, 4, 4, R, S>(st, p, x, dy, dst) : wgrad_launch_one<T, 4, 1, R, S>(st, p, x, dy, dst)) \
                         : (vy ? wgrad_launch_one<T, 1, 4, R, S>(st, p, x, dy, dst) : wgrad_launch_one<T, 1, 1, R, S>(st, p, x, dy, dst)))
  if (g.R == 3) e = g.stride == 1 ? FDG_DW(3, 1) : FDG_DW(3, 2);
  else e = g.stride == 1 ? FDG_DW(1, 1) : FDG_DW(1, 2);
#undef FDG_DW
  if (e != cudaSuccess || p.splits == 1) return e;
  ++*launches;
  typedef std::conditional_t<kByRow<T>, double, float> Sum;
  return launch_wgrad_reduce<Sum>(st, scratch, dw, (size_t)g.Co * g.R * g.R * g.Ci, p.splits);
}

}  // namespace direct
}  // namespace fdg
