// Runs of identity blocks (conv, batch norm, ReLU, conv, batch norm, shortcut, ReLU; 16, 32 or 64 channels in and out, stride 1)
// as ONE launch per pass: forward of training, forward of inference, and the backward pass up to the weight gradients.
//
// What bounds such a layer alone is not its arithmetic (a 16-channel layer over 128 images: 1.3 us of HBM, 0.8 us of tensor
// instructions on all SMs) but the launches around it: convolution and batch norm cannot share a launch without a wait of all
// images for the statistics, so each layer was two launches that start cold, load their images, and store them again.
// Here a CTA keeps its images for the whole run:
//   - the operand of the tensor instructions stays in shared memory; a batch norm's apply writes the next layer's operand in
//     place, beside the copy in global memory that the backward pass (or the weight gradients) will read;
//   - a convolution's output (rounded to bf16) goes from tensor memory into the operand's place, whose instructions are done
//     by then: the apply reads it there;
//   - what the CTAs must know of one another is 2 * C sums per layer: every CTA publishes its own as (value, tag) words and
//     reads all of them (publish and collect below).  The launch is cooperative: its CTAs are resident together, and several such launches
//     on different streams run side by side (measured: 4 launches of 32 CTAs take the time of one; an exchange costs 1.1 us).  Those
//     of one context always fit the device together (chain_plan.h: fit_device); those of two contexts at work on one device at the
//     same time may not, and then a launch waits until all of its CTAs find room, which is what a cooperative launch promises.
// Measured, 128 images of 32x32x16 on 64 CTAs: a layer's forward pass 8 us, its backward pass up to the weight gradient 11 us
// (convolution and apply by themselves: 13 us, and 20 to 25); ResNet-56 with K = 2 1.09 -> 0.78 ms per iteration, an inference
// batch of ResNet-110 0.79 -> 0.41 ms.  What bounds a layer now: the exchange (2.5 us with the CTAs' skew) and the latencies of
// an epilogue of 16 warps (42 % of the issue slots), then the tensor instructions (1 us per image).  640 threads leave the epilogue
// 104 registers: 13 of the 18 variants spill, the backward ones of 12 to 16 bytes with 88 to 108 bytes of loads (16 channels in
// four streams: none), the others 4 to 8 with 20 to 28 (64 channels: none).
// The tensor instructions are those of conv_rows.cuh: an accumulator row is a group of G = 64 / C neighbouring pixels (128
// bytes), a tile 16 image rows x 8 groups.  Pixel i of a group has the columns from (G - 1 - i) * C on: in this order the
// filter taps a window position needs are neighbours in memory, and the nine taps are kept once (9 * C * C values).
//
// Roles by warp: 0..1 issue instructions (alternate tiles), 2..3 bring the weights of the next layer (and, in the backward pass,
// ask for the saved tensors two layers ahead into L2), 4..19 epilogue: a thread has 8 channels of two pixels of every part of
// a tile.  Every wait is bounded; after one that ran out the roles run to their ends without waiting any more (barriers among
// them stay matched) and the CTA raises an error word.
#pragma once
#include <type_traits>

#include "chain_plan.h"
#include "conv_rows.cuh"

namespace fdg {
namespace chain {

using namespace fdg::tc;
using rows::Window;

constexpr int kIssuers = 2, kLoaders = 2;
constexpr int kFirstEpi = 4;                      // a warpgroup of its own for the issuers: it gives its registers to the others
constexpr int kIssuerRegs = 56, kEpiRegs = 104;  // of 96 each at launch: 128 * 56 + 512 * 104 <= 640 * 96
constexpr int kThreads = 32 * kFirstEpi + kEpiThreads;
constexpr uint32_t kPollLimit = 1u << 20;        // an exchange: about a second

// Where the run's tensors are.  Layer l belongs to block l / 2; a block's four tensors (conv1 output, ReLU(BN1), conv2 output,
// block output) lie `t_step` apart, its two gate tensors `q_step`; blocks `b_step` apart.
struct Tensors {
  __nv_bfloat16* t0;          // first block's conv1 output
  size_t t_step, b_step;      // elements
  unsigned char* q0;          // gates as bits of the first block's ReLU(BN1) (null: not kept)
  size_t q_step;              // bytes
  float* stats;               // mean[C], 1/sqrt(var + eps)[C] of layer 0's batch norm
  size_t st_step;             // floats from layer to layer
  const __nv_bfloat16* w;     // filters of layer 0, [C][9][C] (backward: flipped and transposed)
  size_t w_step;              // elements from layer to layer
  const float* gamma;         // of layer 0; the shift C floats behind
  size_t p_step;              // floats from layer to layer
};
struct TrainArgs {
  const __nv_bfloat16* x;     // the run's input
  float* running;             // running statistics of layer 0 (2 * C floats per layer)
  float momentum, unbias, eps;
  double inv_count;
};
struct BackwardArgs {
  __nv_bfloat16* dy;          // gradient of the last block's output; overwritten by itself and those of the blocks below it, gated
  __nv_bfloat16* dx;          // gradient of the run's input
  __nv_bfloat16* dc;          // [layers] gradients of the convolution outputs
  size_t dc_step;
  float* dgamma;              // of layer 0 (dbeta C floats behind), p_step from layer to layer
  float inv_m;
  // the batch-norm backward in front of the run, if its sums are wanted (null: not): gates, normalised tensor, mean and
  // 1/sqrt(var + eps); one row of 2 * C sums per CTA
  const unsigned char* out_gate;
  const __nv_bfloat16* out_x;
  const float* out_stats;
  float* out_partial;
  // copies for an inspection of the pass (null: none): gradients of ReLU(BN1) and of the block inputs, by block
  __nv_bfloat16* keep_a;
  __nv_bfloat16* keep_x;
  size_t keep_step;
};
// Published sums: [CTAs][2][2 * C] words of (tag << 32 | value); `epoch` counts the exchanges of this module, so that no tag occurs
// twice.
struct Exchange {
  unsigned long long* words;
  unsigned int* epoch;
};

__device__ __forceinline__ void st_word(unsigned long long* p, uint32_t tag, float v) {
  const unsigned long long w = ((unsigned long long)tag << 32) | __float_as_uint(v);
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ unsigned long long ld_word(const unsigned long long* p) {
  unsigned long long w;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  return w;
}
// Waits until the words of CTAs b0, b0 + stride, .. (eight of them, those below n; `pitch` words apart) carry `tag`: false when
// the limit is hit or another role has raised *abort_flag.
__device__ __forceinline__ bool poll_words(unsigned long long (&v)[8], const unsigned long long* words, size_t pitch, int b0, int stride, int n,
                                           uint32_t tag, volatile int* abort_flag, uint32_t limit = kPollLimit) {
  for (uint32_t i = 0; ; ++i) {
    bool all = true;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int b = b0 + u * stride;
      v[u] = b < n ? ld_word(words + (size_t)b * pitch) : (unsigned long long)tag << 32;
      all = all && (uint32_t)(v[u] >> 32) == tag;
    }
    if (all) return true;
    if ((i & 63u) == 63u && *abort_flag) return false;
    if (i == limit) { *abort_flag = 1; return false; }
  }
}
// Two warps wait as the kernels do: one, with their bounded wait, on a barrier that nothing ever arrives at, the other, with the
// bounded poll of an exchange, for a word that carries no tag.  After `limit` polls each gives up, and when both have, that is
// reported the way the kernels report it.  Nothing is in flight and no tensor memory is held when the kernel leaves.  Lets the
// host-side handling of a wait that ran out be exercised without making a real kernel misbehave.
__global__ void wait_probe_kernel(uint32_t limit, const unsigned long long* untagged, int* error_word) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int flags[2];
  if (threadIdx.x == 0) {
    flags[0] = flags[1] = 0;
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0) mbar_wait(&bar, 0, &flags[0], limit);
  if (threadIdx.x >= 32) {
    unsigned long long v[8];
    poll_words(v, untagged, 0, 0, 1, 8, 1u, &flags[1], limit);
  }
  __syncthreads();
  if (*(volatile int*)&flags[0] && *(volatile int*)&flags[1] && threadIdx.x == 0 && error_word) atomicExch(error_word, 1);
}
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory"); }
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// A wait that is skipped once any role of the CTA has given up.
__device__ __forceinline__ bool chain_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  if (mbar_try_wait(bar, parity)) return true;
  if (*abort_flag) return false;
  return mbar_wait(bar, parity, abort_flag);
}

// The instructions of one tile (see rows::issue_tile; the filter taps of a window position are neighbours here).
template <int C>
__device__ __forceinline__ void issue_tile(uint32_t leader, uint32_t d, uint32_t a_lo, uint32_t a_hi, uint32_t row_units, uint32_t b_lo, uint32_t b_hi) {
  using Wd = Window<C>;
  constexpr int first = Wd::G == 1 ? 0 : 1;
#pragma unroll
  for (int r = 0; r < 3; ++r, a_lo += row_units) {
#pragma unroll
    for (int jj = 0; jj < Wd::J; ++jj) {
      const int j = Wd::G == 4 ? (jj == 0 ? 1 : jj == 1 ? 4 : jj == 2 ? 0 : jj == 5 ? 5 : jj - 1)
                               : (Wd::G == 2 ? (jj == 0 ? 1 : jj == 1 ? 0 : jj) : jj);
      const bool overwrite = r == 0 && (j == first || (Wd::G == 4 && j == 4));
      const int n = (Wd::i1(j) - Wd::i0(j) + 1) * C;
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);
      const uint32_t a = a_lo + (uint32_t)((128 + (j - 1) * C * 2) >> 4);
      const uint32_t b = b_lo + (uint32_t)(((r * 3 + j - Wd::i1(j)) * (C * C * 2)) >> 4);
#pragma unroll
      for (int k = 0; k < C / 16; ++k)
        rows::mma_lohi(leader, d + (uint32_t)((Wd::G - 1 - Wd::i1(j)) * C), a + 2 * k, a_hi, b + 2 * k, b_hi, idesc, (overwrite && k == 0) ? 0u : 1u);
    }
  }
}

// 16 items per lane; afterwards the first N items of a lane are sums over the lanes that differ from it in the bits taken, of
// the items from the returned one on.  Bits taken: 16, 8 and, for N = 2, 4 and, for N = 1, 2.
template <int N> __device__ __forceinline__ int column_reduce(float (&q)[16], int lane) {
  int item = 0;
#pragma unroll
  for (int off = 16, n = 8; n >= N; off >>= 1, n >>= 1) {
    const bool upper = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const float send = upper ? q[i] : q[i + n];
      const float keep = upper ? q[i + n] : q[i];
      q[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
    item += upper ? n : 0;
  }
  return item;
}
__device__ __forceinline__ float inverse_sqrt(double v) {
  float r;
  if (v > 1e-30 && v < 1e30 && inverse_sqrt_from(v, rsqrtf((float)v), r)) return r;
  return (float)(1.0 / sqrt(v));
}
// Arithmetic on two values at a time: what an apply costs is its instructions (51 per value written one by one, four warps a
// scheduler).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 two(float lo, float hi) { f32x2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi)); return r; }
__device__ __forceinline__ void split(f32x2 v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) { f32x2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) { f32x2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
__device__ __forceinline__ f32x2 widen(uint32_t w) { return two(rows::bf_lo(w), rows::bf_hi(w)); }
__device__ __forceinline__ uint32_t narrow(f32x2 v) { float lo, hi; split(v, lo, hi); return rows::pack_bf(lo, hi); }
__device__ __forceinline__ uint32_t relu2(uint32_t w) {
  uint32_t r;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(w), "r"(0u));
  return r;
}
// The gates of 8 stored values as a byte: set where positive (see bn_apply_kernel).
__device__ __forceinline__ uint32_t gates_of(const uint32_t (&y)[4]) {
  uint32_t m[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) asm("set.gt.u32.bf16x2 %0, %1, %2;" : "=r"(m[q]) : "r"(y[q]), "r"(0u));
  const uint32_t t = (m[0] & 0x00020001u) | (m[1] & 0x00080004u) | (m[2] & 0x00200010u) | (m[3] & 0x00800040u);
  return (t | (t >> 16)) & 0xffu;
}
// A byte of gates as masks of four words of two values.  Bits 0..3 times the constant are the top bits of bytes 0..3.
__device__ __forceinline__ void gate_masks(uint32_t bits, uint32_t (&m)[4]) {
  const uint32_t lo = (bits & 15u) * 0x10204080u, hi = (bits >> 4) * 0x10204080u;
  asm("prmt.b32 %0, %1, %1, 0x9988;" : "=r"(m[0]) : "r"(lo));
  asm("prmt.b32 %0, %1, %1, 0xBBAA;" : "=r"(m[1]) : "r"(lo));
  asm("prmt.b32 %0, %1, %1, 0x9988;" : "=r"(m[2]) : "r"(hi));
  asm("prmt.b32 %0, %1, %1, 0xBBAA;" : "=r"(m[3]) : "r"(hi));
}
// A thread's two places.
struct Px { uint4 v[2]; };
__device__ __forceinline__ void unpack(const uint4& p, uint32_t (&w)[4]) { w[0] = p.x; w[1] = p.y; w[2] = p.z; w[3] = p.w; }
__device__ __forceinline__ uint4 pack4(const uint32_t (&w)[4]) { return make_uint4(w[0], w[1], w[2], w[3]); }
__device__ __forceinline__ void load8(const float* p, f32x2 (&v)[4]) {
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
  v[0] = two(a.x, a.y); v[1] = two(a.z, a.w); v[2] = two(b.x, b.y); v[3] = two(b.z, b.w);
}
// S: tiles the epilogue works on at once.  A scheduler has the four warps that may read one quarter of tensor memory; with S = 4
// each takes a tile of its own, with 2 a pair shares one, with 1 all four do.
template <int C, int PASS, int S>
__global__ void __launch_bounds__(kThreads, 1)
chain_kernel(const __grid_constant__ CUtensorMap map_x, const Geom p, const Tensors ts, const TrainArgs fa, const BackwardArgs ba,
             const Exchange ex, int* __restrict__ error_word) {
  using Wd = Window<C>;
  constexpr int G = Wd::G;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t issued[kIssuers];      // nothing of the issuer's is in flight
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* w_smem = smem + (size_t)p.images * p.a_bytes;
  double* part = reinterpret_cast<double*>(w_smem + (size_t)p.w_stages * p.w_bytes);      // [kEpiThreads]
  float* sums = reinterpret_cast<float*>(part + kEpiThreads);                              // [kEpiWarps][C / 8][16]
  float* cst = sums + kEpiWarps * 2 * C;                                                      // [2][5][C] constants of a batch norm
  uint64_t* bars = reinterpret_cast<uint64_t*>(cst + 2 * 5 * C);
  uint64_t* a_full = bars;                          // [images]  loaded
  uint64_t* a_ready = a_full + kAccSlots;           // [images]  rewritten by the epilogue
  uint64_t* acc_full = a_ready + kAccSlots;         // [tiles]   accumulator complete
  uint64_t* w_full = acc_full + kAccSlots;          // [w_stages]
  uint64_t* w_empty = w_full + 2;                   // [w_stages]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(w_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  uint32_t* epoch_smem = tmem_slot + 2;
  Tile* tab = reinterpret_cast<Tile*>(tmem_slot + 4);                                     // [kAccSlots]

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int step = (int)gridDim.x;
  const int images = (p.N - 1 - (int)blockIdx.x) / step + 1;           // the grid has at most N CTAs
  const int tiles = images * p.tpi;
  if (threadIdx.x < (unsigned)(3 * kAccSlots + 4)) {
    const int i = threadIdx.x;
    const uint32_t count = i < kAccSlots ? 1 : (i < 2 * kAccSlots ? p.tpi * kEpiWarps / S : (i < 3 * kAccSlots ? 1 : (i < 3 * kAccSlots + 2 ? kLoaders : kIssuers)));
    mbar_init(bars + i, count);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x >= 96 && (int)threadIdx.x - 96 < tiles) {
    const int t = (int)threadIdx.x - 96, j = t / p.tpi, k = t - j * p.tpi, rbk = k / p.cb, cbk = k - rbk * p.cb;
    Tile q;
    q.g = (uint32_t)((((size_t)(blockIdx.x + j * step) * p.H + rbk * kTileRows) * p.WG + cbk * kTileGroups) * 64);
    q.s = (uint32_t)j * p.a_bytes + (uint32_t)(rbk * kTileRows * (kTileGroups * p.cb + 2) + cbk * kTileGroups) * 128u;
    q.rows = (uint16_t)min(p.H - rbk * kTileRows, kTileRows); q.groups = (uint16_t)min(p.WG - cbk * kTileGroups, kTileGroups);
    q.image = (uint16_t)j; q.first = (uint16_t)(j * p.tpi);
    tab[t] = q;
  }
  if (threadIdx.x == 64) {
    *abort_flag = 0;
    for (int i = 0; i < kIssuers; ++i) mbar_init(&issued[i], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_x)) : "memory");
    if (PASS != INFER) *epoch_smem = *ex.epoch;
  }
  if (PASS == BACKWARD) {                           // the operand is written by the epilogue: its borders once, here
    for (uint32_t o = threadIdx.x * 16; o < (uint32_t)images * p.a_bytes; o += kThreads * 16) *reinterpret_cast<uint4*>(smem + o) = make_uint4(0, 0, 0, 0);
    halo::fence_proxy_async();
  }
  if (warp == 0) tmem_alloc(tmem_slot, kAccSlots * 64);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);

  if (warp < kFirstEpi) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kIssuerRegs));
    if (warp < kIssuers) {
    const uint32_t leader = lane == 0 ? 1u : 0u;
    const uint32_t row_units = p.row_bytes >> 4;
    int ws = 0;
    uint32_t wph = 0;
    bool ok = true;                                 // after a wait that ran out nothing more is issued
    for (int s = 0; s < p.layers; ++s) {
      ok = chain_wait(&w_full[ws], wph, abort_flag) && ok;
      const uint64_t b_desc = smem_desc_kmajor(smem_u32(w_smem + (size_t)ws * p.w_bytes), C * 2);
      int t = 0;
      for (int j = 0; j < images; ++j) {
        if (PASS != BACKWARD && s == 0) ok = chain_wait(&a_full[j], 0, abort_flag) && ok;
        else ok = chain_wait(&a_ready[j], (uint32_t)(PASS == BACKWARD ? s : s - 1) & 1u, abort_flag) && ok;
        tc_fence_after();
        const uint64_t a_img = smem_desc_kmajor_sbo(smem_u32(smem + (size_t)j * p.a_bytes), 128, p.row_bytes);
        for (int rbk = 0; rbk < p.rb; ++rbk)
          for (int cbk = 0; cbk < p.cb; ++cbk, ++t) {
            if (t % kIssuers != warp || !ok) continue;
            issue_tile<C>(leader, tmem_base + (uint32_t)t * 64u, (uint32_t)a_img + (uint32_t)rbk * (kTileRows * row_units) + (uint32_t)cbk * 64u,
                          (uint32_t)(a_img >> 32), row_units, (uint32_t)b_desc, (uint32_t)(b_desc >> 32));
            rows::commit_by(leader, &acc_full[t]);
          }
      }
      if (ok) rows::commit_by(leader, &w_empty[ws]);
      if (++ws == p.w_stages) { ws = 0; wph ^= 1u; }
    }
    rows::commit_by(leader, &issued[warp]);
    } else {
      // shared memory: [tap][c_out] rows of C channels, swizzled; global memory: [c_out][tap][C]
      constexpr uint32_t mask = C == 64 ? 7u : (C == 32 ? 3u : 1u);
      constexpr int kPieces = C / 8;                // 16-byte pieces of a row
      const int lt = (warp - kIssuers) * 32 + lane;
      const uint32_t img_elems = (uint32_t)(p.H * p.W) * C;
      auto ask = [&](int l) {                       // the saved tensors of batch norm l, into L2
        if (l < 0 || lt >= images) return;
        const size_t n = (size_t)((int)blockIdx.x + lt * step);
        halo::prefetch_l2_bulk(ts.t0 + (size_t)(l >> 1) * ts.b_step + ((l & 1) ? 2 * ts.t_step : 0) + n * img_elems, img_elems * 2);
        if (img_elems % 128 == 0)
          halo::prefetch_l2_bulk(ts.q0 + (size_t)(l >> 1) * ts.b_step * 2 + ((l & 1) ? ts.q_step : 0) + n * (img_elems / 8), img_elems / 8);
      };
      if (PASS == BACKWARD) ask(p.layers - 2);
      int ws = 0;
      uint32_t wph = 0;
      for (int s = 0; s < p.layers; ++s) {
        const int l = PASS == BACKWARD ? p.layers - 1 - s : s;
        if (s >= p.w_stages) chain_wait(&w_empty[ws], wph ^ 1u, abort_flag);
        const uint32_t dst = smem_u32(w_smem + (size_t)ws * p.w_bytes);
        const __nv_bfloat16* src = ts.w + (size_t)l * ts.w_step;
        for (int i = lt; i < 9 * C * kPieces; i += 32 * kLoaders) {
          const int r = i / kPieces, pc = i - r * kPieces, tap = r / C, co = r - tap * C;
          const uint32_t o = (uint32_t)i * 16;
          cp_async16(dst + (o ^ (((o >> 7) & mask) << 4)), src + (co * 9 + tap) * C + pc * 8);
        }
        if (PASS == BACKWARD) ask(l - 2);
        asm volatile("cp.async.wait_all;" ::: "memory");
        halo::fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(&w_full[ws]);
        if (++ws == p.w_stages) { ws = 0; wph ^= 1u; }
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kEpiRegs));
    const int etid = threadIdx.x - 32 * kFirstEpi;
    const int ewarp = warp - kFirstEpi, lane_grp = warp & 3;
    // 4 / S warps share 32 accumulator rows of a tile: four image rows x 8 groups.  As a READER a warp has S * 16 of their
    // columns, a thread one row of them (what tensor memory hands out); at its PLACES a warp has S of the image rows, a thread 16
    // bytes (8 channels) of two groups of each, so that an access to any tensor covers whole 128-byte lines.  Between the two go
    // 16-byte pieces of the operand's own shared memory, whose instructions are done by then.  (With a row per lane for the
    // global accesses too, the apply of a tile of 16 channels took 3100 cycles, against 900 for its tensor instructions.)
    const int stream = (ewarp >> 2) / (4 / S), part0 = (ewarp >> 2) % (4 / S) * S;      // tiles stream, stream + S, ..; parts part0 ..
    const int c0 = (lane & 7) * 8 % C;              // places: first channel
    const int dr0 = lane_grp * 4 + part0, dg = lane >> 3;                // first image row; group (and the one four further on)
    const int dra = lane_grp * 4 + (lane >> 3), dga = lane & 7;          // reader: image row and group
    const uint32_t taddr = tmem_base + ((uint32_t)(lane_grp * 32) << 16) + (uint32_t)part0 * 16u;
    const uint32_t epoch = PASS != INFER ? *epoch_smem : 0u;
    if (PASS != BACKWARD && etid == 0)
      for (int j = 0; j < images; ++j) {
        mbar_expect_tx(&a_full[j], p.a_tx);
        tma_load_4d(smem + (size_t)j * p.a_bytes, &map_x, &a_full[j], 0, -1, -1, (int)blockIdx.x + j * step);
      }
    // Relative to a tile: elements of a tensor, bytes of the operands (a tile and an image start at a multiple of 8 lines, so the
    // swizzle of a line does not depend on them).
    const uint32_t row_elems = (uint32_t)p.WG * 64u, pitch = (uint32_t)(kTileGroups * p.cb + 2);
    const uint32_t e_off = (uint32_t)dr0 * row_elems + (uint32_t)dg * 64u + (uint32_t)(lane & 7) * 8u;
    const uint32_t line0 = (uint32_t)(dr0 + 1) * pitch + (uint32_t)dg + 1u, linea = (uint32_t)(dra + 1) * pitch + (uint32_t)dga + 1u;
    const uint32_t sbase = smem_u32(smem);
    auto place_smem = [&](const Tile& t, int part, int i) -> uint32_t {
      const uint32_t line = line0 + (uint32_t)part * pitch + 4u * (uint32_t)i;
      return sbase + t.s + line * 128u + ((((uint32_t)lane & 7u) ^ (line & 7u)) << 4);
    };
    auto reader_smem = [&](const Tile& t, int part, int i) -> uint32_t {
      const int col = (part0 + part) * 16;
      const uint32_t piece = (uint32_t)(((G - 1 - col / C) * C + col % C) >> 3) + (uint32_t)i;
      return sbase + t.s + linea * 128u + ((piece ^ (linea & 7u)) << 4);
    };

    // This thread's two places of a part in a tensor; one outside the image reads element 0 instead.  Loads are unconditional: under
    // a condition their results were merged, i.e. waited for, where they are issued (a tile of the backward apply: 2500 cycles of 3600).
    struct At { uint32_t e[2]; bool ok[2]; };
    auto place = [&](const Tile& t, int part) {
      At a;
      const bool row = dr0 + part < t.rows;
      a.ok[0] = row && dg < t.groups; a.ok[1] = row && dg + 4 < t.groups;
      const uint32_t e = t.g + e_off + (uint32_t)part * row_elems;
      a.e[0] = a.ok[0] ? e : 0u; a.e[1] = a.ok[1] ? e + 256u : 0u;
      return a;
    };
    // The place that comes after part `part` of tile t in this warp's order (behind the last one: the last one again).
    auto place_after = [&](int t, int part) {
      const int nt = part + 1 < S ? t : (t + S < tiles ? t + S : t);
      return place(tab[nt], part + 1 < S ? part + 1 : (t + S < tiles ? 0 : part));
    };
    auto load = [&](const __nv_bfloat16* t, const At& a, Px& x) {
#pragma unroll
      for (int i = 0; i < 2; ++i) x.v[i] = *reinterpret_cast<const uint4*>(t + a.e[i]);
    };
    auto store = [&](__nv_bfloat16* t, const At& a, int i, const uint32_t (&y)[4]) { *reinterpret_cast<uint4*>(t + a.e[i]) = pack4(y); };
    auto gates = [&](const unsigned char* bits, const At& a, uint32_t (&m)[2]) {
#pragma unroll
      for (int i = 0; i < 2; ++i) m[i] = (uint32_t)bits[a.e[i] >> 3];
    };
    auto sts = [&](uint32_t at, const uint32_t* y) {
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(y[0]), "r"(y[1]), "r"(y[2]), "r"(y[3]) : "memory");
    };
    auto lds = [&](uint32_t at, uint32_t* y) {
      asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(y[0]), "=r"(y[1]), "=r"(y[2]), "=r"(y[3]) : "r"(at) : "memory");
    };
    auto to_operand = [&](const Tile& t, int part, int i, const uint32_t (&y)[4]) { sts(place_smem(t, part, i), y); };
    auto from_operand = [&](const Tile& t, int part, uint32_t (&y)[2][4]) { lds(place_smem(t, part, 0), y[0]); lds(place_smem(t, part, 1), y[1]); };
    auto tile_sync = [&]() {                        // the warps of a tile's quarter
      if (S == 4) __syncwarp();
      else asm volatile("bar.sync %0, %1;" ::"r"(2 + lane_grp * S + stream), "n"(128 / S) : "memory");
    };
    // All instructions that read the tile's image are done.
    auto wait_image = [&](const Tile& t, uint32_t ph) {
      for (int q = 0; q < p.tpi; ++q) chain_wait(&acc_full[t.first + q], ph, abort_flag);
      tc_fence_after();
    };
    // The accumulator of tile t, rounded to bf16, into the operand's place (ADD: added to what is there first).
    auto to_smem = [&](auto is_add, int t, const Tile& tl) {
      constexpr bool ADD = decltype(is_add)::value;
      const bool ok = dra < tl.rows && dga < tl.groups;
#pragma unroll
      for (int part = 0; part < S; ++part) {
        uint32_t r[8], v[16];
        if (ADD) { lds(reader_smem(tl, part, 0), r); lds(reader_smem(tl, part, 1), r + 4); }
        __syncwarp();
        tmem_ld16(taddr + (uint32_t)t * 64u + (uint32_t)part * 16u, v);
        tmem_ld_wait();
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const f32x2 a = two(__uint_as_float(v[2 * q]), __uint_as_float(v[2 * q + 1]));
          r[q] = narrow(ADD ? add2(a, widen(r[q])) : a);
        }
        if (ok) { sts(reader_smem(tl, part, 0), r); sts(reader_smem(tl, part, 1), r + 4); }
      }
      tile_sync();
    };
    auto tile_done = [&](const Tile& t) {           // this warp's share of the tile's operand is written
      tc_fence_before();
      halo::fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(&a_ready[t.image]);
    };

    // Sums: `run` holds this thread's, 8 channels each of two statistics.  warp_sums leaves the warp's in shared memory, cta_sum
    // adds the warps in order, publish makes this CTA's known, collect adds everybody's.  What else a layer needs meanwhile is
    // issued between the two.  Barriers of the epilogue warps: one in warp_sums, one in collect, one behind the use of the totals.
    auto warp_sums = [&](const f32x2 (&run2)[8]) {
      float run[16];
#pragma unroll
      for (int q = 0; q < 8; ++q) split(run2[q], run[2 * q], run[2 * q + 1]);
      constexpr int N = C == 64 ? 4 : (C == 32 ? 2 : 1);                 // pieces with the same channels are lanes 4 (and 2) apart
      const int item = column_reduce<N>(run, lane);
      float* d = sums + ewarp * 2 * C + (c0 >> 3) * 16 + item;
#pragma unroll
      for (int i = 0; i < N; ++i) d[i] = run[i];
      epi_sync();
    };
    auto cta_sum = [&](int i) -> float {            // sum i: statistic i / C of channel i % C
      const int stat = i / C, c = i - stat * C;
      const float* d = sums + (c >> 3) * 16 + stat * 8 + (c & 7);
      float a = 0.f;
#pragma unroll
      for (int w = 0; w < kEpiWarps; ++w) a += d[w * 2 * C];
      return a;
    };
    auto words_of = [&](int number) { return ex.words + (size_t)(number & 1) * 2 * C; };
    auto publish = [&](int number, float own) {     // `own`: this CTA's sum etid, for etid < 2 * C
      if (etid < 2 * C) st_word(words_of(number) + (size_t)blockIdx.x * 4 * C + etid, epoch + 1u + (uint32_t)number, own);
    };
    // First thread (sum etid % (2 * C), segment etid / (2 * C)) adds every kSegs-th CTA's word; then a warp has C / 16 channels:
    // lane (channel, statistic, segment).  A channel's leader ends up with its totals.  (A CTA's words lie in a row of their own:
    // with all CTAs' words of a sum side by side an exchange took twice as long.)
    constexpr int kSegs = kEpiThreads / (2 * C);
    const int chan = ewarp * (C / 16) + lane / (2 * kSegs);
    const bool leader = lane % (2 * kSegs) == 0;
    auto collect = [&](int number, double& s0, double& s1) {
      const uint32_t tag = epoch + 1u + (uint32_t)number;
      const unsigned long long* mine = words_of(number) + etid % (2 * C);
      double a = 0.0;
      for (int b0 = etid / (2 * C); b0 < step; b0 += 8 * kSegs) {
        unsigned long long v[8];
        poll_words(v, mine, 4 * C, b0, kSegs, step, tag, abort_flag);
#pragma unroll
        for (int u = 0; u < 8; ++u) a += (double)__uint_as_float((uint32_t)v[u]);
      }
      part[etid] = a;
      epi_sync();
      a = part[lane % kSegs * (2 * C) + lane / kSegs % 2 * C + chan];
#pragma unroll
      for (int o = kSegs / 2; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      s0 = a;
      s1 = __shfl_down_sync(0xffffffffu, a, kSegs);
    };

    if constexpr (PASS != BACKWARD) {
      if (PASS == INFER && etid < C) {
        cst[etid] = -ts.stats[etid]; cst[C + etid] = ts.gamma[etid] * ts.stats[C + etid]; cst[2 * C + etid] = ts.gamma[C + etid];
      }
      // the apply: the convolution's output, normalised, the shortcut, ReLU; the next layer's operand in its place
      auto apply = [&](auto is_second, const float* k, uint32_t ph, bool last, const __nv_bfloat16* res, __nv_bfloat16* out, unsigned char* bits) {
        constexpr bool second = decltype(is_second)::value;
        if (stream >= tiles) return;
        f32x2 mu[4], ga[4], be[4];                  // the mean negated
        load8(k + c0, mu); load8(k + C + c0, ga); load8(k + 2 * C + c0, be);
        At at = place(tab[stream], 0);
        Px r;
        if (second) load(res, at, r);
        for (int t = stream; t < tiles; t += S) {
          const Tile tl = tab[t];
          if (PASS == INFER) {
            wait_image(tl, ph);
            to_smem(std::false_type{}, t, tl);
          }
#pragma unroll
          for (int part = 0; part < S; ++part) {
            uint32_t y[2][4];
            from_operand(tl, part, y);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              uint32_t rw[4];
              if (second) unpack(r.v[i], rw);
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                f32x2 v = fma2(add2(widen(y[i][q]), mu[q]), ga[q], be[q]);
                if (second) v = add2(v, widen(rw[q]));
                y[i][q] = relu2(narrow(v));
              }
            }
            const At here = at;
            at = place_after(t, part);
            if (second) load(res, at, r);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              if (!here.ok[i]) continue;
              if (!last) to_operand(tl, part, i, y[i]);
              if (PASS == TRAIN || second) store(out, here, i, y[i]);
              if (PASS == TRAIN) bits[here.e[i] >> 3] = (unsigned char)gates_of(y[i]);
            }
          }
          if (!last) tile_done(tl);
        }
      };
      for (int l = 0; l < p.layers; ++l) {
        const bool second = (l & 1) != 0, last = l == p.layers - 1;
        const size_t blk = (size_t)(l >> 1) * ts.b_step;
        __nv_bfloat16* conv_out = ts.t0 + blk + (second ? 2 * ts.t_step : 0);
        __nv_bfloat16* act_out = conv_out + ts.t_step;
        const __nv_bfloat16* res = l < 2 ? fa.x : ts.t0 + blk - ts.b_step + 3 * ts.t_step;
        unsigned char* bits = PASS == TRAIN ? ts.q0 + blk * 2 + (second ? ts.q_step : 0) : nullptr;
        float* k = cst + (l & 1) * 5 * C;
        const float* gamma = ts.gamma + (size_t)l * ts.p_step;
        float* stats = ts.stats + (size_t)l * ts.st_step;
        const uint32_t ph = (uint32_t)l & 1u;
        if constexpr (PASS == TRAIN) {
          f32x2 run[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) run[i] = 0ull;
          for (int t = stream; t < tiles; t += S) {
            const Tile tl = tab[t];
            wait_image(tl, ph);
            to_smem(std::false_type{}, t, tl);
#pragma unroll
            for (int part = 0; part < S; ++part) {
              const At at = place(tl, part);
              uint32_t y[2][4];
              from_operand(tl, part, y);
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                if (!at.ok[i]) continue;
                store(conv_out, at, i, y[i]);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                  const f32x2 v = widen(y[i][q]);
                  run[q] = add2(run[q], v); run[4 + q] = fma2(v, v, run[4 + q]);
                }
              }
            }
          }
          warp_sums(run);
          publish(l, etid < 2 * C ? cta_sum(etid) : 0.f);
          const float ga = gamma[chan], be = gamma[C + chan];
          float* run_at = fa.running + (size_t)l * 2 * C + chan;
          const bool keeper = blockIdx.x == 0 && leader;
          const float rmean = keeper ? run_at[0] : 0.f, rvar = keeper ? run_at[C] : 0.f;      // see update_running
          double s0, s1;
          collect(l, s0, s1);
          if (leader) {
            const double mean = s0 * fa.inv_count;
            double var = s1 * fa.inv_count - mean * mean;
            if (var < 0.0) var = 0.0;
            const float mu = (float)mean, inv = inverse_sqrt(var + (double)fa.eps);
            k[chan] = -mu; k[C + chan] = ga * inv; k[2 * C + chan] = be;
            if (keeper) {
              stats[chan] = mu; stats[C + chan] = inv;
              run_at[0] = (1.f - fa.momentum) * rmean + fa.momentum * mu;
              run_at[C] = (1.f - fa.momentum) * rvar + fa.momentum * ((float)var * fa.unbias);
            }
          }
          epi_sync();
        } else {
          // The next layer's constants: requested now, put down when this layer's first convolution is done (every warp is done
          // with the layer before then, and with its constants).
          float n0 = 0.f, n1 = 0.f, n2 = 0.f;
          if (!last && etid < C) {
            const float* sn = stats + ts.st_step;
            const float* gn = gamma + ts.p_step;
            n0 = -sn[etid]; n1 = gn[etid] * sn[C + etid]; n2 = gn[C + etid];
          }
          epi_sync();
          wait_image(tab[0], ph);
          if (!last && etid < C) {
            float* kn = cst + ((l + 1) & 1) * 5 * C;
            kn[etid] = n0; kn[C + etid] = n1; kn[2 * C + etid] = n2;
          }
        }
        if (second) apply(std::true_type{}, k, ph, last, res, act_out, bits);
        else apply(std::false_type{}, k, ph, last, nullptr, act_out, bits);
      }
      if (PASS == TRAIN && blockIdx.x == 0 && etid == 0) *ex.epoch = epoch + (uint32_t)p.layers;
    } else {
      // ---- backward: batch norm l = layers-1 .. 0, each followed by its convolution's data gradient
      f32x2 run[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) run[i] = 0ull;
      const int top = p.layers - 1;
      auto conv_out_of = [&](int l) { return ts.t0 + (size_t)(l >> 1) * ts.b_step + ((l & 1) ? 2 * ts.t_step : 0); };
      auto bits_of = [&](int l) { return ts.q0 + (size_t)(l >> 1) * ts.b_step * 2 + ((l & 1) ? ts.q_step : 0); };
      // y <- y * [gate], its sum and that of y * (x - mean); `mu`: the mean negated
      auto gate_and_add = [&](uint32_t (&y)[4], uint32_t km, const uint4& x, const f32x2 (&mu)[4]) {
        uint32_t xw[4], m[4];
        unpack(x, xw);
        gate_masks(km, m);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          y[q] &= m[q];
          const f32x2 d = widen(y[q]);
          run[q] = add2(run[q], d);
          run[4 + q] = fma2(d, add2(widen(xw[q]), mu[q]), run[4 + q]);
        }
      };
      // constants, two sets: -mean, invstd, gamma * invstd, -k0, -k1 of the batch norm whose sums are being formed
      if (etid < C) {
        const float* st = ts.stats + (size_t)top * ts.st_step;
        float* k = cst + (top & 1) * 5 * C;
        k[etid] = -st[etid]; k[C + etid] = st[C + etid];
      }
      epi_sync();
      // The gradient of the last block's output: gated (the operand's place has it, and `dy` in place of itself for the shortcut),
      // with the sums of that block's second batch norm.
      {
        const __nv_bfloat16* x = conv_out_of(top);
        const unsigned char* bits = bits_of(top);
        f32x2 mu[4];
        load8(cst + (top & 1) * 5 * C + c0, mu);
        for (int t = stream; t < tiles; t += S) {
          const Tile tl = tab[t];
#pragma unroll
          for (int part = 0; part < S; ++part) {
            const At at = place(tl, part);
            Px d, v;
            uint32_t km[2];
            load(ba.dy, at, d); load(x, at, v); gates(bits, at, km);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              if (!at.ok[i]) continue;
              uint32_t y[4];
              unpack(d.v[i], y);
              gate_and_add(y, km[i], v.v[i], mu);
              to_operand(tl, part, i, y);
              store(ba.dy, at, i, y);
            }
          }
        }
      }
      // the gradient of convolution l's output, as operand (in the place of the gradient it is formed from) and to memory
      auto apply = [&](const float* k, const __nv_bfloat16* x, __nv_bfloat16* dc, Px& v) {
        f32x2 mu[4], k1[4];
        load8(k + c0, mu); load8(k + 4 * C + c0, k1);
        for (int t = stream; t < tiles; t += S) {
          const Tile tl = tab[t];
#pragma unroll
          for (int part = 0; part < S; ++part) {
            uint32_t y[2][4];
            from_operand(tl, part, y);
            f32x2 gi[4], k0[4];
            load8(k + 2 * C + c0, gi); load8(k + 3 * C + c0, k0);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              uint32_t xw[4];
              unpack(v.v[i], xw);
#pragma unroll
              for (int q = 0; q < 4; ++q) y[i][q] = narrow(fma2(gi[q], widen(y[i][q]), fma2(add2(widen(xw[q]), mu[q]), k1[q], k0[q])));
            }
            load(x, place_after(t, part), v);
            const At here = place(tl, part);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              if (!here.ok[i]) continue;
              to_operand(tl, part, i, y[i]);
              store(dc, here, i, y[i]);
            }
          }
          tile_done(tl);
        }
      };
      // The data gradient of convolution l (first of a block: + the shortcut's gradient, gated already; stored for the block below,
      // gated again, or as it is where it leaves the run), and the sums of the batch norm that it meets.
      auto finish = [&](auto is_second, uint32_t ph, const float* mean, const __nv_bfloat16* x, const unsigned char* bits, bool leaves,
                        __nv_bfloat16* out, __nv_bfloat16* keep) {
        constexpr bool second = decltype(is_second)::value;
        f32x2 mu[4];
        load8(mean + c0, mu);
#pragma unroll
        for (int i = 0; i < 8; ++i) run[i] = 0ull;
        if (stream >= tiles) return;
        At at = place(tab[stream], 0);
        Px v;
        uint32_t km[2];
        load(x, at, v); gates(bits, at, km);
        for (int t = stream; t < tiles; t += S) {
          const Tile tl = tab[t];
          wait_image(tl, ph);
          if (!second) {
#pragma unroll
            for (int part = 0; part < S; ++part) {
              const At a = place(tl, part);
#pragma unroll
              for (int i = 0; i < 2; ++i) if (a.ok[i]) cp_async16(place_smem(tl, part, i), ba.dy + a.e[i]);
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            tile_sync();
            to_smem(std::true_type{}, t, tl);
          } else {
            to_smem(std::false_type{}, t, tl);
          }
#pragma unroll
          for (int part = 0; part < S; ++part) {
            uint32_t y[2][4];
            from_operand(tl, part, y);
            const At here = at;
            at = place_after(t, part);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              if (!here.ok[i]) continue;
              if (keep) store(keep, here, i, y[i]);
              if (!second && leaves) store(out, here, i, y[i]);
              gate_and_add(y[i], km[i], v.v[i], mu);
              if (!second && !leaves) store(out, here, i, y[i]);
              to_operand(tl, part, i, y[i]);
            }
            load(x, at, v); gates(bits, at, km);
          }
        }
      };
      for (int s = 0; s < p.layers; ++s) {
        const int l = top - s;
        const bool second = (l & 1) != 0;           // the block's second convolution
        float* k = cst + (l & 1) * 5 * C;
        const uint32_t ph = (uint32_t)s & 1u;
        // -- totals of batch norm l; constants of the next one (l - 1, or the one in front of the run)
        warp_sums(run);
        float own = 0.f;
        if (etid < 2 * C) {
          own = cta_sum(etid);
          if (etid >= C) own *= k[etid];            // invstd of channel etid - C
        }
        publish(s, own);
        Px v;                                       // the apply's first operand
        load(conv_out_of(l), place(tab[stream < tiles ? stream : 0], 0), v);
        float nmean = 0.f, ninv = 0.f;
        const float ga = ts.gamma[(size_t)l * ts.p_step + chan];
        const float* nst = l > 0 ? ts.stats + (size_t)(l - 1) * ts.st_step : ba.out_stats;
        if (nst) { nmean = nst[chan]; ninv = nst[C + chan]; }
        double s0, s1;
        collect(s, s0, s1);
        float* kn = cst + ((l + 1) & 1) * 5 * C;
        if (leader) {
          const float inv = k[C + chan], gi = ga * inv;
          const float t0 = (float)s0, t1 = (float)s1;
          k[2 * C + chan] = gi; k[3 * C + chan] = -(t0 * ba.inv_m * gi); k[4 * C + chan] = -(t1 * ba.inv_m * (gi * inv));
          kn[chan] = -nmean; kn[C + chan] = ninv;
          if (blockIdx.x == 0) {
            float* dg = ba.dgamma + (size_t)l * ts.p_step;
            dg[chan] = t1; dg[C + chan] = t0;
          }
        }
        epi_sync();
        __nv_bfloat16* dc = ba.dc + (size_t)l * ba.dc_step;
        // the last convolution's sums go to the batch norm in front of the run; where none are wanted they are formed and dropped
        const __nv_bfloat16* x = l > 0 ? conv_out_of(l - 1) : (ba.out_partial ? ba.out_x : conv_out_of(0));
        const unsigned char* bits = l > 0 ? bits_of(l - 1) : (ba.out_partial ? ba.out_gate : bits_of(0));
        const size_t kept = (size_t)(l >> 1) * ba.keep_step;
        apply(k, conv_out_of(l), dc, v);
        if (second) finish(std::true_type{}, ph, kn, x, bits, false, nullptr, ba.keep_a ? ba.keep_a + kept : nullptr);
        else finish(std::false_type{}, ph, kn, x, bits, l == 0, l > 0 ? ba.dy : ba.dx, ba.keep_x ? ba.keep_x + kept : nullptr);
      }
      if (ba.out_partial) {
        warp_sums(run);
        if (etid < 2 * C) {
          float a = cta_sum(etid);
          if (etid >= C) a *= cst[5 * C + etid];    // invstd of the batch norm in front of the run: set (0 + 1) & 1
          ba.out_partial[(size_t)blockIdx.x * 2 * C + etid] = a;
        }
      }
      if (blockIdx.x == 0 && etid == 0) *ex.epoch = epoch + (uint32_t)p.layers;
    }
  }

  // Teardown.  After an abort copies towards this CTA's shared memory may still be in flight, and instructions that read it and
  // write tensor memory: give their barriers a bounded chance to complete before that memory is given back.
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) {
      if (error_word) atomicExch(error_word, 1);
      auto settle = [](uint64_t* bar) { for (uint32_t i = 0; i < (1u << 16) && !mbar_try_wait(bar, 0); ++i) {} };
      if (PASS != BACKWARD)
        for (int j = 0; j < images; ++j) settle(&a_full[j]);
      for (int i = 0; i < kIssuers; ++i) settle(&issued[i]);
    }
    __syncthreads();
  }
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kAccSlots * 64);
  }
}

// ----------------------------------------------------------------- host side ---
typedef void (*ChainKernel)(CUtensorMap, Geom, Tensors, TrainArgs, BackwardArgs, Exchange, int*);
template <int C> inline ChainKernel kernel_of(int pass, int streams) {
  if (pass == INFER) return streams == 2 ? chain_kernel<C, INFER, 2> : chain_kernel<C, INFER, 1>;
  if (pass == TRAIN) return streams == 4 ? chain_kernel<C, TRAIN, 4> : chain_kernel<C, TRAIN, 2>;
  return streams == 4 ? chain_kernel<C, BACKWARD, 4> : chain_kernel<C, BACKWARD, 2>;
}
inline ChainKernel kernel_of(int C, int pass, int streams) {
  return C == 16 ? kernel_of<16>(pass, streams) : (C == 32 ? kernel_of<32>(pass, streams) : kernel_of<64>(pass, streams));
}
inline cudaError_t set_attrs(int dev) {
  static OncePerDevice once;
  return once.run(dev, []() {
    cudaError_t e = cudaSuccess;
    for (int c = 16; c <= 64; c *= 2)
      for (int pass = 0; pass < 3; ++pass)
        for (int st = 1; st <= 4 && e == cudaSuccess; st *= 2) e = set_smem_limit(kernel_of(c, pass, st), kSmemLimit);
    return e;
  });
}
inline cudaError_t launch(cudaStream_t st, int C, int pass, const CUtensorMap& map_x, const Geom& p, const Tensors& ts, const TrainArgs& fa,
                          const BackwardArgs& ba, const Exchange& ex, int* error_word) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)chain_ctas(p)); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = chain_smem_bytes(p, C); cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at; cfg.numAttrs = pass == INFER ? 0 : 1;                  // the images of an inference pass do not meet
  return cudaLaunchKernelEx(&cfg, kernel_of(C, pass, chain_streams(p, pass)), map_x, p, ts, fa, ba, ex, error_word);
}

}  // namespace chain
}  // namespace fdg
