// 3x3 / stride 1 / pad 1 convolutions of the narrow layers that keep their width (16, 32 or 64 channels in and out) on the
// sm_100a tensor cores: forward and data gradient of nearly every layer of a 6n+2 network.
//
// What bounds such a layer is not its arithmetic but the number of tensor instructions and what surrounds them: an
// instruction of M = 128 holds the pipe about 47 cycles however small N is, so N = 16 (one accumulator row per pixel)
// wastes five sixths of it.  Here an accumulator row is a GROUP of G = 64 / C neighbouring pixels of an image row, i.e.
// 128 bytes of the tensor, and has 64 columns: column i * C + co is channel co of the group's pixel i.
//   - The operand of window position j (pixel G*g - 1 + j, j = 0 .. G+1) is the same shared-memory tile read from a
//     start address j pixels further on; it contributes to the pixels i with 0 <= j - i <= 2, through the filter tap
//     s = j - i, so one instruction of N = (number of such i) * C covers up to three taps.  The weights of the pixels lie
//     one after the other: block (r, j) = the filters of taps (r, j - i) for those i in turn.
//   - Per 128 groups: 18 instructions for 512 pixels at 16 channels (72 before), 24 for 256 at 32 (36), 36 for 128 at 64.
// A tile is 16 image rows x 8 groups; in shared memory an image lies row by row, each row with one group of zeros on
// either side (out-of-bounds groups and rows are the hardware's zero fill: the padding), so that the 8-row groups of the
// operand are one image row apart whatever the image's width.  Tiles reach over the image's edge where its sides are no
// multiples (28x28: 7 of 8 groups, 28 of 32 rows); what lies outside is never stored and not counted.
//
// Epilogue: a tile of the output is 128 rows of 128 bytes in every tensor of its shape, so everything it reads or writes
// per element goes through shared memory in swizzled 16 KB tiles moved by TMA: the residual, the tensor a following
// batch-norm backward normalised, and the output, which overwrites one of them in place.  ReLU gates are bits (one per
// element, 8 bytes per row), written by the batch-norm kernels beside the activations.  Every thread takes 16 columns of a
// row (16 channels of one pixel) of every tile and keeps their per-channel sums in registers to the end.
//
// Roles by warp: 0..1 issue instructions (alternate tiles), 2 loads images, 3 moves the epilogue's tiles, 4..19 epilogue (and
// the weights' loads): four groups of four warps.  Every wait is bounded; on time-out the CTA raises an error word.
#pragma once
#include "conv_halo.cuh"

namespace fdg {
namespace rows {

using namespace fdg::tc;

constexpr int kIssuers = 2;
constexpr int kLoadWarp = 2, kOpWarp = 3, kFirstEpi = 4;
constexpr int kEpiGroups = 4;
constexpr int kEpiWarps = 4 * kEpiGroups;
constexpr int kThreads = 32 * (kFirstEpi + kEpiWarps);
constexpr int kAccSlots = 8;                     // accumulators of 64 columns
constexpr uint32_t kTileBytes = 128 * 128;       // an epilogue tile
constexpr int kTileRows = 16, kTileGroups = 8;

struct RowsParams {
  int N, H, W, WG;            // image; groups per row (W / G)
  int rb, cb, tpi;            // tiles of an image: row blocks, column blocks, rb * cb
  uint32_t row_bytes;         // shared memory of one image row: (8 * cb + 2) groups
  uint32_t a_bytes;           // one image, multiple of 1 KiB
  uint32_t a_tx;              // bytes its load writes
  uint32_t b_bytes;           // weights, multiple of 1 KiB
  int a_stages, op_stages;
  int n_ops;                  // operand tiles per epilogue tile: residual, normalised tensor
};

// A gate per element, as bits (8 bytes per group: bit c = column c) or as the tensor itself.
struct Gate {
  const unsigned char* bits;
  const __nv_bfloat16* tensor;
};
// What an epilogue does besides (template parameter MODE): 0 nothing; sums: 1 sum v, sum v^2, 2 sum dz, sum dz * xhat with
// dz = v * [gate]; 3 the batch norm that follows, with given statistics (inference), before the residual.
struct EpiParams {
  EpiAffine affine;           // MODE 3
  Gate res_gate;              // residual counts where the gate is set (both null: everywhere)
  Gate gate;                  // MODE 2
  const float* pstats;        // MODE 2: mean[C], invstd[C]
  float* partial;             // [gridDim.x][2 * C]
};

__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, const void* src, int c0, int c1, int c2, int c3) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
               ::"l"(map), "r"(smem_u32(src)), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// The gates of 16 elements from the tensor itself.
__device__ __forceinline__ uint32_t gate16_tensor(const __nv_bfloat16* p) {
  uint32_t m = 0;
  const uint4 q0 = *reinterpret_cast<const uint4*>(p), q1 = *reinterpret_cast<const uint4*>(p + 8);
  const __nv_bfloat16* e0 = reinterpret_cast<const __nv_bfloat16*>(&q0);
  const __nv_bfloat16* e1 = reinterpret_cast<const __nv_bfloat16*>(&q1);
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    m |= (__bfloat162float(e0[e]) > 0.f ? 1u : 0u) << e;
    m |= (__bfloat162float(e1[e]) > 0.f ? 1u : 0u) << (8 + e);
  }
  return m;
}

// The weight blocks: per filter row r, window position j the pixels i in [max(0, j-2), min(G-1, j)].
template <int C> struct Window {
  static constexpr int G = 64 / C;
  static constexpr int J = G + 2;
  __host__ __device__ static constexpr int i0(int j) { return j > 2 ? j - 2 : 0; }
  __host__ __device__ static constexpr int i1(int j) { return j < G - 1 ? j : G - 1; }
  __host__ __device__ static constexpr int blocks_before(int j) { int n = 0; for (int q = 0; q < j; ++q) n += i1(q) - i0(q) + 1; return n; }
  static constexpr int per_row = 3 * G;                       // blocks of a filter row: every pixel meets three taps
  static constexpr uint32_t block_bytes = C * C * 2;
};

// The instructions of one tile, fully unrolled.  The first ones of the tile (accumulate = 0) cover disjoint columns and
// together all 64: window positions 1 and 4 at G = 4, position 1 at G = 2, position 0 at G = 1.  A descriptor's low word
// holds the start address in 16-byte units: moving an operand is a 32-bit add, the high words never change.  The whole
// warp walks the loop (`leader` is one of its lanes), so that descriptors stay in uniform registers: with one lane alone
// in a branch, an instruction left every 138 cycles.
__device__ __forceinline__ void mma_lohi(uint32_t leader, uint32_t d, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                         uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .b64 a, b;\n\t"
      "mov.b64 a, {%1, %2};\n\tmov.b64 b, {%3, %4};\n\t"
      "setp.ne.b32 p, %6, 0;\n\tsetp.ne.b32 q, %7, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n\t}"
      ::"r"(d), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate), "r"(leader) : "memory");
}
__device__ __forceinline__ void commit_by(uint32_t leader, uint64_t* bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
      ::"r"(smem_u32(bar)), "r"(leader) : "memory");
}
template <int C>
__device__ __forceinline__ void issue_tile(uint32_t leader, uint32_t d, uint32_t a_lo, uint32_t a_hi, uint32_t row_units, uint32_t b_lo, uint32_t b_hi) {
  using Wd = Window<C>;
  constexpr int first = Wd::G == 1 ? 0 : 1;
#pragma unroll
  for (int r = 0; r < 3; ++r, a_lo += row_units) {
#pragma unroll
    for (int jj = 0; jj < Wd::J; ++jj) {
      // order: the overwriting positions come first
      const int j = Wd::G == 4 ? (jj == 0 ? 1 : jj == 1 ? 4 : jj == 2 ? 0 : jj == 5 ? 5 : jj - 1)
                               : (Wd::G == 2 ? (jj == 0 ? 1 : jj == 1 ? 0 : jj) : jj);
      const bool overwrite = r == 0 && (j == first || (Wd::G == 4 && j == 4));
      const int n = (Wd::i1(j) - Wd::i0(j) + 1) * C;
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);
      const uint32_t a = a_lo + (uint32_t)((128 + (j - 1) * C * 2) >> 4);
      const uint32_t b = b_lo + (uint32_t)(((r * Wd::per_row + Wd::blocks_before(j)) * Wd::block_bytes) >> 4);
#pragma unroll
      for (int k = 0; k < C / 16; ++k)
        mma_lohi(leader, d + (uint32_t)(Wd::i0(j) * C), a + 2 * k, a_hi, b + 2 * k, b_hi, idesc, (overwrite && k == 0) ? 0u : 1u);
    }
  }
}

// Walks a CTA's tiles in order, with the stage and the accumulator slot of each and the phase of their barriers: all by
// additions (a division per tile and thread costs more here than the tile's arithmetic).
struct Walk {
  int n, rbk, cbk;            // image, row block, column block
  int s, slot;                // stage of the epilogue ring, accumulator slot
  uint32_t sph, aph;          // their phases
  __device__ __forceinline__ explicit Walk(int first) : n(first), rbk(0), cbk(0), s(0), slot(0), sph(0), aph(0) {}
  __device__ __forceinline__ void next(const RowsParams& p, int step) {
    if (++cbk == p.cb) { cbk = 0; if (++rbk == p.rb) { rbk = 0; n += step; } }
    if (++s == p.op_stages) { s = 0; sph ^= 1; }
    if (++slot == kAccSlots) { slot = 0; aph ^= 1; }
  }
};

__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
__device__ __forceinline__ uint32_t pack_bf(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

template <int C, int MODE, bool RES>
__global__ void __launch_bounds__(kThreads, 1)
conv_rows_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_w,
                 const __grid_constant__ CUtensorMap map_out, const __grid_constant__ CUtensorMap map_res,
                 const __grid_constant__ CUtensorMap map_x, RowsParams p, EpiParams e, int* __restrict__ error_word) {
  using Wd = Window<C>;
  constexpr int kOps = (RES ? 1 : 0) + (MODE == 2 ? 1 : 0);
  constexpr uint32_t op_bytes = (kOps > 1 ? kOps : 1) * kTileBytes;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* w_smem = smem + (size_t)p.a_stages * p.a_bytes;
  uint8_t* op_smem = w_smem + p.b_bytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(op_smem + (size_t)p.op_stages * op_bytes);
  uint64_t* a_full = bars;                         // [a_stages]   image landed
  uint64_t* a_empty = a_full + p.a_stages;         // [a_stages]   image multiplied
  uint64_t* w_full = a_empty + p.a_stages;         // weights landed
  uint64_t* acc_full = w_full + 1;                 // [kAccSlots]  accumulator complete
  uint64_t* acc_empty = acc_full + kAccSlots;      // [kAccSlots]  accumulator read
  uint64_t* op_ready = acc_empty + kAccSlots;      // [op_stages]  operand tiles landed, output tile may be written
  uint64_t* tile_done = op_ready + p.op_stages;    // [op_stages]  output tile written
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tile_done + p.op_stages);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* sums = reinterpret_cast<float*>(tmem_slot + 2);        // [kEpiWarps][32]; 16-byte aligned (the barriers are odd in number)
  float* mean = sums + kEpiWarps * 32;                          // [3][C]: mean, invstd (MODE 2); mean, gamma * invstd, beta

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int step = (int)gridDim.x;
  const int images = ((int)blockIdx.x < p.N) ? (p.N - 1 - (int)blockIdx.x) / step + 1 : 0;
  const int tiles = images * p.tpi;
  // Everything up to the barrier needs nothing of the preceding kernel and may run beside it.
  if (warp == kFirstEpi) {                         // one barrier per lane (they lie in a row; at most 31 of them)
    const int e_first = 2 * p.a_stages + 1 + kAccSlots, t_first = e_first + kAccSlots + p.op_stages;
    if (lane < t_first + p.op_stages) {
      uint32_t count = 1;
      if (lane >= p.a_stages && lane < 2 * p.a_stages) count = kIssuers;
      if ((lane >= e_first && lane < e_first + kAccSlots) || lane >= t_first) count = kEpiWarps;
      mbar_init(bars + lane, count);
    }
    if (lane == 31) *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  } else if (threadIdx.x == 32 * kLoadWarp) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_a)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_w)) : "memory");
  } else if (threadIdx.x == 32 * kOpWarp) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_out)) : "memory");
    if (RES) asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_res)) : "memory");
    if (MODE == 2) asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_x)) : "memory");
  }
  if (warp == 0) tmem_alloc(tmem_slot, kAccSlots * 64);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  grid_dependency_wait();                          // from here on the preceding kernel's results may be read
  if (MODE == 3) grid_dependency_release();        // inference: one stream, nothing else wants the places of the next kernel

  if (warp >= kFirstEpi && lane == 0) {
    // The weight blocks, a few by each epilogue warp (one thread takes 150 cycles per request: 36 of them one after the
    // other were a third of a launch)
    for (int b = warp - kFirstEpi; b < 3 * Wd::per_row; b += kEpiWarps) {
      const int r = b / Wd::per_row;
      int q = b - r * Wd::per_row, j = 0;
      while (q > Wd::i1(j) - Wd::i0(j)) { q -= Wd::i1(j) - Wd::i0(j) + 1; ++j; }
      tma_load_2d(w_smem + (uint32_t)b * Wd::block_bytes, &map_w, w_full, (r * 3 + j - (Wd::i0(j) + q)) * C, 0);
    }
  }
  __syncwarp();                                    // the warp-wide instructions below want the warp together
  if (warp < kIssuers) {
    {
      const uint32_t leader = lane == 0 ? 1u : 0u;
      bool ok = mbar_wait(w_full, 0, abort_flag);
      tc_fence_after();
      const uint64_t b_desc = smem_desc_kmajor(smem_u32(w_smem), C * 2);
      const uint32_t row_units = p.row_bytes >> 4;
      Walk wk((int)blockIdx.x);
      int t = 0, as = 0;
      uint32_t aph = 0;
      for (int im = 0; ok && im < images; ++im) {
        if (!mbar_wait(&a_full[as], aph, abort_flag)) break;
        tc_fence_after();
        const uint64_t a_img = smem_desc_kmajor_sbo(smem_u32(smem + (size_t)as * p.a_bytes), 128, p.row_bytes);
        for (int k = 0; k < p.tpi; ++k, ++t, wk.next(p, 0)) {
          if (t % kIssuers != warp) continue;
          if (t >= kAccSlots) {
            if (!mbar_wait(&acc_empty[wk.slot], wk.aph ^ 1u, abort_flag)) { ok = false; break; }
            tc_fence_after();
          }
          issue_tile<C>(leader, tmem_base + (uint32_t)wk.slot * 64u, (uint32_t)a_img + (uint32_t)wk.rbk * (kTileRows * row_units) + (uint32_t)wk.cbk * 64u,
                        (uint32_t)(a_img >> 32), row_units, (uint32_t)b_desc, (uint32_t)(b_desc >> 32));
          commit_by(leader, &acc_full[wk.slot]);
        }
        if (ok) commit_by(leader, &a_empty[as]);
        if (++as == p.a_stages) { as = 0; aph ^= 1; }
      }
    }
  } else if (warp == kLoadWarp) {
    if (lane == 0) {
      mbar_expect_tx(w_full, (uint32_t)(3 * Wd::per_row) * Wd::block_bytes);
      int ls = 0;
      uint32_t lph = 0;
      for (int im = 0; im < images; ++im) {
        if (im >= p.a_stages && !mbar_wait(&a_empty[ls], lph ^ 1u, abort_flag)) break;
        mbar_expect_tx(&a_full[ls], p.a_tx);
        tma_load_4d(smem + (size_t)ls * p.a_bytes, &map_a, &a_full[ls], 0, -1, -1, (int)blockIdx.x + im * step);
        if (++ls == p.a_stages) { ls = 0; lph ^= 1; }
      }
    }
  } else if (warp == kOpWarp) {
    if (lane == 0) {
      // The epilogue's tiles: operands in, output out.  Tile t uses stage t % op_stages; a stage is handed out again when
      // the store that read it has finished reading.
      auto hand_out = [&](const Walk& w) {
        if (kOps == 0) { mbar_arrive(&op_ready[w.s]); return; }
        uint8_t* dst = op_smem + (size_t)w.s * op_bytes;
        mbar_expect_tx(&op_ready[w.s], (uint32_t)kOps * kTileBytes);
        if (RES) { tma_load_4d(dst, &map_res, &op_ready[w.s], 0, w.cbk * kTileGroups, w.rbk * kTileRows, w.n); dst += kTileBytes; }
        if (MODE == 2) tma_load_4d(dst, &map_x, &op_ready[w.s], 0, w.cbk * kTileGroups, w.rbk * kTileRows, w.n);
      };
      Walk in((int)blockIdx.x), out((int)blockIdx.x);
      int handed = 0;
      for (; handed < p.op_stages && handed < tiles; ++handed) { hand_out(in); in.next(p, step); }
      for (int t = 0; t < tiles; ++t) {
        if (!mbar_wait(&tile_done[out.s], out.sph, abort_flag)) break;
        tma_store_4d(&map_out, op_smem + (size_t)out.s * op_bytes, 0, out.cbk * kTileGroups, out.rbk * kTileRows, out.n);
        bulk_commit();
        out.next(p, step);
        if (handed < tiles) { bulk_wait_read(); hand_out(in); in.next(p, step); ++handed; }
      }
      bulk_wait_read();
    }
  } else if (warp >= kFirstEpi) {
    const int lane_grp = warp & 3;                 // tensor-memory lanes 32 * (warp % 4) ..
    const int group = (warp - kFirstEpi) >> 2;
    const int col = group * 16;                    // this thread's columns: 16 channels of one pixel of the group
    const int c0 = col % C;                        // its first channel
    const int row = lane_grp * 32 + lane;          // accumulator row = row of an epilogue tile
    const int dr = row >> 3, dg = row & 7;
    const uint32_t o0 = ((col >> 3) ^ dg) << 4, o1 = (((col >> 3) + 1) ^ dg) << 4;   // its two 16-byte pieces of a swizzled line
    const uint32_t taddr = tmem_base + ((uint32_t)(lane_grp * 32) << 16) + (uint32_t)col;
    if (MODE >= 2) {
      if (MODE == 2) {
        for (int i = threadIdx.x - 32 * kFirstEpi; i < 2 * C; i += 32 * kEpiWarps) mean[i] = e.pstats[i];
      } else {                                     // mean, gamma * invstd, beta
        for (int i = threadIdx.x - 32 * kFirstEpi; i < C; i += 32 * kEpiWarps) {
          mean[i] = e.affine.stats[i]; mean[C + i] = e.affine.gamma[i] * e.affine.stats[C + i]; mean[2 * C + i] = e.affine.beta[i];
        }
      }
      asm volatile("bar.sync 1, %0;" ::"n"(32 * kEpiWarps) : "memory");
    }
    constexpr bool kSums = MODE == 1 || MODE == 2;
    float run[kSums ? 32 : 1];
#pragma unroll
    for (int i = 0; i < (kSums ? 32 : 1); ++i) run[i] = 0.f;
    Walk wk((int)blockIdx.x);
    for (int t = 0; t < tiles; ++t, wk.next(p, step)) {
      const int h = wk.rbk * kTileRows + dr, g = wk.cbk * kTileGroups + dg;
      const bool valid = h < p.H && g < p.WG;
      uint32_t rm = 0xffffu, km = 0u;              // gates of this thread's 16 elements
      if ((RES || MODE == 2) && valid) {
        const size_t grp_index = ((size_t)wk.n * p.H + h) * p.WG + g;
        if (RES) {
          if (e.res_gate.bits) rm = *reinterpret_cast<const uint16_t*>(e.res_gate.bits + grp_index * 8 + (col >> 3));
          else if (e.res_gate.tensor) rm = gate16_tensor(e.res_gate.tensor + grp_index * 64 + col);
        }
        if (MODE == 2) {
          if (e.gate.bits) km = *reinterpret_cast<const uint16_t*>(e.gate.bits + grp_index * 8 + (col >> 3));
          else km = gate16_tensor(e.gate.tensor + grp_index * 64 + col);
        }
      }
      if (!mbar_wait(&op_ready[wk.s], wk.sph, abort_flag)) break;
      uint8_t* line = op_smem + (uint32_t)wk.s * op_bytes + row * 128;      // output, in place of the first operand
      uint4 r0, r1, x0, x1;
      if (RES) { r0 = *reinterpret_cast<const uint4*>(line + o0); r1 = *reinterpret_cast<const uint4*>(line + o1); }
      if (MODE == 2) {
        const uint8_t* xline = line + (RES ? kTileBytes : 0);
        x0 = *reinterpret_cast<const uint4*>(xline + o0); x1 = *reinterpret_cast<const uint4*>(xline + o1);
      }
      if (!mbar_wait(&acc_full[wk.slot], wk.aph, abort_flag)) break;
      __syncwarp();
      tc_fence_after();
      uint32_t v[16];
      tmem_ld16(taddr + (uint32_t)wk.slot * 64u, v);
      tmem_ld_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[wk.slot]);                 // the values are in registers
      if (MODE == 3) {                             // on the value as it would have been stored: bn_apply_kernel's result
        const float* mu = mean + c0;
#pragma unroll
        for (int q = 0; q < 16; q += 4) {
          const float4 m = *reinterpret_cast<const float4*>(mu + q), g = *reinterpret_cast<const float4*>(mu + C + q),
                       b = *reinterpret_cast<const float4*>(mu + 2 * C + q);
          v[q] = __float_as_uint(fmaf(__bfloat162float(__float2bfloat16_rn(__uint_as_float(v[q]))) - m.x, g.x, b.x));
          v[q + 1] = __float_as_uint(fmaf(__bfloat162float(__float2bfloat16_rn(__uint_as_float(v[q + 1]))) - m.y, g.y, b.y));
          v[q + 2] = __float_as_uint(fmaf(__bfloat162float(__float2bfloat16_rn(__uint_as_float(v[q + 2]))) - m.z, g.z, b.z));
          v[q + 3] = __float_as_uint(fmaf(__bfloat162float(__float2bfloat16_rn(__uint_as_float(v[q + 3]))) - m.w, g.w, b.w));
        }
      }
      if (RES) {
        const uint32_t rw[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          v[2 * q] = __float_as_uint(__uint_as_float(v[2 * q]) + ((rm & (1u << (2 * q))) ? bf_lo(rw[q]) : 0.f));
          v[2 * q + 1] = __float_as_uint(__uint_as_float(v[2 * q + 1]) + ((rm & (2u << (2 * q))) ? bf_hi(rw[q]) : 0.f));
        }
      }
      if (MODE == 3 && e.affine.relu) {
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q] = __float_as_uint(fmaxf(__uint_as_float(v[q]), 0.f));
      }
      uint32_t y[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) y[q] = pack_bf(__uint_as_float(v[2 * q]), __uint_as_float(v[2 * q + 1]));
      *reinterpret_cast<uint4*>(line + o0) = make_uint4(y[0], y[1], y[2], y[3]);
      *reinterpret_cast<uint4*>(line + o1) = make_uint4(y[4], y[5], y[6], y[7]);
      halo::fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tile_done[wk.s]);                    // this warp's part of the output tile is written
      // the sums are those of the values as stored
      if (MODE == 1) {
        if (valid) {
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const float a = bf_lo(y[q]), b = bf_hi(y[q]);
            run[2 * q] += a; run[16 + 2 * q] = fmaf(a, a, run[16 + 2 * q]);
            run[2 * q + 1] += b; run[17 + 2 * q] = fmaf(b, b, run[17 + 2 * q]);
          }
        }
      } else if (MODE == 2) {
        const uint32_t xw[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
        const float* mu = mean + c0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float a = (km & (1u << (2 * q))) ? bf_lo(y[q]) : 0.f, b = (km & (2u << (2 * q))) ? bf_hi(y[q]) : 0.f;
          run[2 * q] += a; run[16 + 2 * q] = fmaf(a, bf_lo(xw[q]) - mu[2 * q], run[16 + 2 * q]);
          run[2 * q + 1] += b; run[17 + 2 * q] = fmaf(b, bf_hi(xw[q]) - mu[2 * q + 1], run[17 + 2 * q]);
        }
      }
    }
    if constexpr (kSums) {
      transpose_reduce32(run, lane);               // lane l: item l of this warp's 32 rows (channel l % 16, sum l / 16)
      sums[(warp - kFirstEpi) * 32 + lane] = run[0];
    }
  }

  // Teardown.  After an abort, TMA copies may still be in flight towards this CTA's shared memory: give every barrier
  // that was armed a bounded chance to complete before leaving.
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) {
      if (error_word) atomicExch(error_word, 1);
      for (int s = 0; s < p.a_stages + p.op_stages + 1; ++s) {
        uint64_t* b = s < p.a_stages ? &a_full[s] : (s == p.a_stages ? w_full : &op_ready[s - p.a_stages - 1]);
        for (uint32_t i = 0; i < (1u << 16); ++i)
          if (mbar_try_wait(b, 0) || mbar_try_wait(b, 1)) break;
      }
    }
    __syncthreads();
  }
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kAccSlots * 64);
  }
  if ((MODE == 1 || MODE == 2) && !*abort_flag) {
    // this CTA's sums, warps in order: the warps of group q hold the 16 channels from (16 * q) % C
    for (int i = threadIdx.x; i < 2 * C; i += kThreads) {
      const int stat = i / C, c = i - stat * C, item = (c & 15) + 16 * stat;
      float a = 0.f;
#pragma unroll
      for (int q = 0; q < kEpiGroups; ++q) {
        if ((q * 16) % C != (c & ~15)) continue;
#pragma unroll
        for (int w = 0; w < 4; ++w) a += sums[(q * 4 + w) * 32 + item];
      }
      if (MODE == 2 && stat == 1) a *= mean[C + c];
      e.partial[(size_t)blockIdx.x * 2 * C + i] = a;
    }
  }
}

// ----------------------------------------------------------------- host side ---
constexpr size_t kSmemLimit = 226 * 1024;
inline size_t fixed_smem(int a_stages, int op_stages) {
  return (size_t)(2 * a_stages + 1 + 2 * kAccSlots + 2 * op_stages) * 8 + 16 + (size_t)kEpiWarps * 32 * 4 + 3 * 64 * 4 + 1024;
}
// `per_cta` images per CTA at most, `n_ops` operand tiles; a_stages = 0 where the shape is not covered.
inline RowsParams rows_params(int N, int H, int W, int C, int per_cta, int n_ops) {
  RowsParams p{};
  const int G = 64 / C;
  p.N = N; p.H = H; p.W = W; p.WG = W / G;
  p.rb = (H + kTileRows - 1) / kTileRows; p.cb = (p.WG + kTileGroups - 1) / kTileGroups; p.tpi = p.rb * p.cb;
  p.row_bytes = (uint32_t)(kTileGroups * p.cb + 2) * 128;
  p.a_bytes = halo::round_up_u32((uint32_t)(p.rb * kTileRows + 2) * p.row_bytes, 1024);
  p.a_tx = (uint32_t)(H + 2) * p.row_bytes;
  p.b_bytes = (uint32_t)(9 * G) * (uint32_t)(C * C * 2);
  p.n_ops = n_ops;
  const size_t op = (size_t)(n_ops > 1 ? n_ops : 1) * kTileBytes;
  const int tiles = per_cta * p.tpi;
  // Two images in flight (the next one lands while this one is multiplied), then epilogue tiles: at least two, up to four.
  for (int as = per_cta > 1 ? 2 : 1; as >= 1; --as) {
    const size_t used = (size_t)as * p.a_bytes + p.b_bytes + fixed_smem(3, 4);
    int os = used < kSmemLimit ? (int)((kSmemLimit - used) / op) : 0;
    os = os > 4 ? 4 : os;
    if (os > tiles) os = tiles;
    if (os < 1 || (os < 2 && tiles > 1 && as > 1)) continue;
    p.a_stages = as; p.op_stages = os;
    if (as == 2 && per_cta > 2 && used + (size_t)os * op + p.a_bytes <= kSmemLimit) p.a_stages = 3;
    break;
  }
  return p;
}
inline size_t rows_smem_bytes(const RowsParams& p) {
  return (size_t)p.a_stages * p.a_bytes + p.b_bytes + (size_t)p.op_stages * (p.n_ops > 1 ? p.n_ops : 1) * kTileBytes +
         fixed_smem(p.a_stages, p.op_stages);
}
inline bool rows_supported(int N, int H, int W, int Ck, int Cn) {
  if (Ck != Cn || (Ck != 16 && Ck != 32 && Ck != 64) || N < 1) return false;
  const int G = 64 / Ck;
  if (W % G || H + 2 > 256 || W / G + 2 > 256) return false;
  const RowsParams p = rows_params(N, H, W, Ck, 4, 2);
  return p.a_stages > 0 && p.a_tx < (1u << 20);
}

// A [N][H][W][C] tensor as rows of 128-byte groups: box of `box_g` groups x `box_h` rows of one image.
inline cudaError_t make_group_map(const void* t, int N, int H, int W, int C, int box_g, int box_h, CUtensorMap* map) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return cudaErrorNotSupported;
  const int G = 64 / C;
  cuuint64_t dims[4] = {64u, (cuuint64_t)(W / G), (cuuint64_t)H, (cuuint64_t)N};
  cuuint64_t strides[3] = {128u, (cuuint64_t)W * C * 2, (cuuint64_t)H * W * C * 2};
  cuuint32_t box[4] = {64u, (cuuint32_t)box_g, (cuuint32_t)box_h, 1u};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  if (enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(t), dims, strides, box, estr,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  return cudaSuccess;
}

typedef void (*RowsKernel)(CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, RowsParams, EpiParams, int*);
template <int C> inline RowsKernel kernel_of(int mode, bool res) {
  if (mode == 1) return res ? conv_rows_kernel<C, 1, true> : conv_rows_kernel<C, 1, false>;
  if (mode == 3) return res ? conv_rows_kernel<C, 3, true> : conv_rows_kernel<C, 3, false>;
  if (mode == 2) return res ? conv_rows_kernel<C, 2, true> : conv_rows_kernel<C, 2, false>;
  return res ? conv_rows_kernel<C, 0, true> : conv_rows_kernel<C, 0, false>;
}
inline RowsKernel kernel_of(int C, int mode, bool res) {
  return C == 16 ? kernel_of<16>(mode, res) : (C == 32 ? kernel_of<32>(mode, res) : kernel_of<64>(mode, res));
}

inline cudaError_t set_attrs(int dev) {
  static OncePerDevice once;
  return once.run(dev, []() {
    cudaError_t e = cudaSuccess;
    for (int c = 16; c <= 64; c *= 2)
      for (int mode = 0; mode < 4; ++mode)
        for (int res = 0; res < 2 && e == cudaSuccess; ++res) e = set_smem_limit(kernel_of(c, mode, res != 0), kSmemLimit);
    return e;
  });
}

}  // namespace rows
}  // namespace fdg
