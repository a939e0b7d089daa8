// Chooses the kernel for one convolution: the tcgen05 tensor-core kernels for bf16 3x3
// stride-1 convolutions whose shape they cover, the CUDA-core implicit GEMM otherwise.
#pragma once
#include <algorithm>
#include <cstring>
#include <map>
#include <vector>

#include "conv_direct.cuh"
#include "conv_simt.cuh"
#include "conv_tc.cuh"
#include "conv_halo.cuh"
#include "conv_rows.cuh"
#include "conv_chain.cuh"
#include "wgrad_wide.cuh"
#include "elementwise.cuh"

namespace fdg {

typedef __nv_bfloat16 bf16_t;

// Tensor maps are pure functions of (pointer, shape, box); the runtime cycles through a
// fixed set of buffers, so they are encoded once and looked up afterwards.
struct TensorMapCache {
  struct Key {
    const void* ptr; int d[8];
    bool operator<(const Key& o) const { return std::memcmp(this, &o, sizeof(Key)) < 0; }
  };
  std::map<Key, CUtensorMap> maps;
  int device = 0, sm_count = 0;   // the device the cache is for; 0 SMs: not asked yet (cached_sm_count)
  int share = 1;        // kernels expected to run side by side (one per module stream): a launch takes
                        // about sm_count / share CTAs and walks its tiles with them
  int wgrad_side_cap = 0;   // upper bound of the pixel split of a weight gradient issued beside the stream that
                            // needs its inputs' other consumers (0 = none), see halo::wgrad_ctas
};

inline int cached_sm_count(TensorMapCache* cache) {
  if (cache->sm_count == 0) {
    cudaGetDevice(&cache->device);
    cudaDeviceGetAttribute(&cache->sm_count, cudaDevAttrMultiProcessorCount, cache->device);
  }
  return cache->sm_count;
}
inline int cached_device(TensorMapCache* cache) { cached_sm_count(cache); return cache->device; }

inline bool tc_eligible(const ConvGeom& g) {
  return g.R == 3 && g.S == 3 && g.stride == 1 && g.pad == 1 && g.P == g.H && g.Q == g.W &&
         tc::conv_tc_supported(g.N, g.H, g.W, g.Ci, g.Co, (size_t)g.N * g.P * g.Q);
}

// Runs D = conv3x3(act, wgt) on the tensor cores.  `Ck`/`Cn` are the GEMM-K and GEMM-N channel
// counts (forward: Ci/Co; data gradient: Co/Ci with the flipped weight copy).
inline cudaError_t run_conv_tc(cudaStream_t st, TensorMapCache* cache, int N, int H, int W, int Ck, int Cn,
                               const bf16_t* act, const bf16_t* wgt, bf16_t* out, const bf16_t* res,
                               const bf16_t* res_mask, int* err_dev, int sub = 1, int taps = 9, int act_sub = 1,
                               float* stat_partial = nullptr, int* ctas_out = nullptr, const EpiAffine* affine = nullptr, int s2 = 0) {
  const int sm_count = cached_sm_count(cache);
  tc::ConvTcParams p = tc::conv_tc_params(N, H, W, Ck, Cn, taps, cache->share, s2);
  p.sub = sub;
  if (s2 == 0) p.act_sub = act_sub;
  TensorMapCache::Key ka, kb;
  std::memset(&ka, 0, sizeof(ka)); std::memset(&kb, 0, sizeof(kb));
  ka.ptr = act; ka.d[0] = 1; ka.d[1] = N; ka.d[2] = H; ka.d[3] = W; ka.d[4] = Ck; ka.d[5] = p.kc; ka.d[6] = p.patch; ka.d[7] = p.act_sub;
  kb.ptr = wgt; kb.d[0] = 2; kb.d[1] = Ck; kb.d[2] = Cn; kb.d[3] = p.kc; kb.d[4] = p.n_tile; kb.d[5] = taps;
  auto ia = cache->maps.find(ka), ib = cache->maps.find(kb);
  if (ia == cache->maps.end() || ib == cache->maps.end()) {
    CUtensorMap ma, mb;
    cudaError_t e = tc::conv_tc_make_maps(p, act, wgt, &ma, &mb);
    if (e != cudaSuccess) return e;
    ia = cache->maps.insert({ka, ma}).first;
    ib = cache->maps.insert({kb, mb}).first;
  }
  const cudaError_t e = tc::conv_tc_set_attrs(cached_device(cache));
  if (e != cudaSuccess) return e;
  tc::ActMaps maps;
  for (int q = 0; q < 4; ++q) maps.m[q] = ia->second;
  for (int q = 1; q < 4 && s2 == 1; ++q) {       // the other parities of x [N][2H][2W][Ck]
    ka.ptr = act + ((size_t)(q >> 1) * 2 * W + (q & 1)) * Ck;
    auto iq = cache->maps.find(ka);
    if (iq == cache->maps.end()) {
      CUtensorMap mq, unused;
      const cudaError_t eq = tc::conv_tc_make_maps(p, ka.ptr, wgt, &mq, &unused);
      if (eq != cudaSuccess) return eq;
      iq = cache->maps.insert({ka, mq}).first;
    }
    maps.m[q] = iq->second;
  }
  return tc::conv_tc_launch(st, p, maps, ib->second, out, res, res_mask, err_dev, sm_count, stat_partial, ctas_out, affine);
}


// ---- halo-tile kernels (16/32/64-channel layers) ------------------------------------------
inline bool halo_shape(const ConvGeom& g) {
  return g.R == 3 && g.S == 3 && g.stride == 1 && g.pad == 1 && g.P == g.H && g.Q == g.W;
}
// forward: K channels = Ci, N channels = Co; data gradient: the other way round
inline bool halo_fprop_eligible(const ConvGeom& g) { return halo_shape(g) && halo::fwd_supported(g.N, g.H, g.W, g.Ci, g.Co); }
inline bool halo_dgrad_eligible(const ConvGeom& g) { return halo_shape(g) && halo::fwd_supported(g.N, g.H, g.W, g.Co, g.Ci); }
inline bool halo_wgrad_eligible(const ConvGeom& g) { return halo_shape(g) && halo::wgrad_supported(g.N, g.H, g.W, g.Ci, g.Co); }

// A 3x3 / stride 2 / pad 1 convolution on even image sizes runs exactly, on the output grid, forward and data gradient
// (conv_tc.cuh: ActMaps).  Its weight gradient is the stride-1 one taken with dy spread onto the even pixels of a zero
// tensor of the input's size: four times the arithmetic.
inline bool halo_s2_shape(const ConvGeom& g) {
  return g.R == 3 && g.S == 3 && g.stride == 2 && g.pad == 1 && g.H % 2 == 0 && g.W % 2 == 0 && g.P == g.H / 2 && g.Q == g.W / 2;
}
inline bool s2_planned(const ConvGeom& g, int Ck, int Cn) {
  return (tc::conv_tc_supported(g.N, g.H, g.W, Ck, Cn, (size_t)g.N * g.P * g.Q) || halo::fwd_supported(g.N, g.H, g.W, Ck, Cn)) &&
         tc::conv_tc_supported(g.N, g.P, g.Q, Ck, Cn, (size_t)g.N * g.P * g.Q);
}
// (H and W, not P and Q: images of more than 128 columns, or 254 where the halo kernel covers the channels, stay with the CUDA
// cores, as their workspaces were planned)
inline bool tc_s2_fprop_eligible(const ConvGeom& g) { return halo_s2_shape(g) && s2_planned(g, g.Ci, g.Co); }
inline bool tc_s2_dgrad_eligible(const ConvGeom& g) { return halo_s2_shape(g) && s2_planned(g, g.Co, g.Ci); }
// with the sums of the batch-norm backward that dx feeds: those are formed by the halo kernel, at full resolution from a spread-out dy
// (an operator-level call may ask for them; the module-step does without)
inline bool halo_s2_dgrad_sums_eligible(const ConvGeom& g) { return halo_s2_shape(g) && halo::fwd_supported(g.N, g.H, g.W, g.Co, g.Ci) && g.Ci <= 64; }
inline bool halo_s2_wgrad_eligible(const ConvGeom& g) { return halo_s2_shape(g) && halo::wgrad_supported(g.N, g.H, g.W, g.Ci, g.Co); }
// 1x1 convolutions without padding (projection shortcuts), stride 1 or 2: one "tap" of the per-tap kernel on the output
// grid; a stride-2 forward reads the even pixels of x as a strided tensor, a stride-2 data gradient writes dx at the
// even pixels (dx is cleared first).
inline bool tc_1x1_shape(const ConvGeom& g) {
  return g.R == 1 && g.S == 1 && g.pad == 0 && (g.stride == 1 || (g.stride == 2 && g.H % 2 == 0 && g.W % 2 == 0)) &&
         g.P == g.H / g.stride && g.Q == g.W / g.stride;
}
inline bool tc_1x1_fprop_eligible(const ConvGeom& g) { return tc_1x1_shape(g) && tc::conv_tc_supported(g.N, g.P, g.Q, g.Ci, g.Co, (size_t)g.N * g.P * g.Q); }
inline bool tc_1x1_dgrad_eligible(const ConvGeom& g) { return tc_1x1_shape(g) && tc::conv_tc_supported(g.N, g.P, g.Q, g.Co, g.Ci, (size_t)g.N * g.P * g.Q); }
// wide layers: the exact-tile weight-gradient kernel (stride 2 with dy spread onto the input grid; 1x1 filters on the output grid)
// (layers under 128 channels stay with the halo-tile kernel where it covers them)
inline bool wide_wgrad_eligible(const ConvGeom& g) {
  return halo_shape(g) && wide::wide_supported(g.N, g.H, g.W, g.Ci, g.Co) && ((g.Ci >= 128 && g.Co >= 128) || !halo_wgrad_eligible(g));
}
inline bool wide_s2_wgrad_eligible(const ConvGeom& g) {
  return halo_s2_shape(g) && wide::wide_supported(g.N, g.H, g.W, g.Ci, g.Co) && ((g.Ci >= 128 && g.Co >= 128) || !halo_s2_wgrad_eligible(g));
}
// Projections of fewer than 64 channels on a side stay with direct_wgrad_kernel, which adds their rows in fp64: tensor
// memory truncates at every instruction, an error that grows with a CTA's pixels, and a narrow projection gives few CTAs.
// 128 images, error against 64 bits and time, tensor cores / CUDA cores: 16 -> 32 on 32x32, stride 2: 1.0e-6, 15.4 us /
// 4.2e-8, 10.7 us; 32 -> 64 on 16x16: 2.5e-7, 9.3 us / 3.9e-8, 11.1 us; 16 -> 160 on 32x32: 4.4e-6, 40.6 us / 5.0e-8,
// 49.5 us; 2048 images of the first: 1.9e-5, 139 us / 4.3e-8, 93 us.  With 64 channels or more on both sides it is arithmetic,
// where the tensor cores are the faster by 4 to 25 times: 64 -> 128 on 32x32, stride 2: 1.0e-6, 15.7 us / 4.2e-8, 70 us.
inline bool wide_1x1_wgrad_eligible(const ConvGeom& g) {
  return tc_1x1_shape(g) && g.Ci >= 64 && g.Co >= 64 && wide::wide_supported(g.N, g.P, g.Q, g.Ci, g.Co, 1);
}

inline cudaError_t cached_tile_map(TensorMapCache* cache, const void* act, int N, int H, int W, int C, int G,
                                   const CUtensorMap** out, int boxC = 0) {
  if (boxC == 0) boxC = C;
  TensorMapCache::Key k;
  std::memset(&k, 0, sizeof(k));
  k.ptr = act; k.d[0] = 3; k.d[1] = N; k.d[2] = H; k.d[3] = W; k.d[4] = C; k.d[5] = G; k.d[6] = boxC;
  auto it = cache->maps.find(k);
  if (it == cache->maps.end()) {
    CUtensorMap m;
    cudaError_t e = halo::make_tile_map(act, N, H, W, C, G, &m, boxC);
    if (e != cudaSuccess) return e;
    it = cache->maps.insert({k, m}).first;
  }
  *out = &it->second;
  return cudaSuccess;
}
inline cudaError_t cached_weight_map(TensorMapCache* cache, const void* wgt, int Ck, int Cn, const CUtensorMap** out) {
  TensorMapCache::Key k;
  std::memset(&k, 0, sizeof(k));
  k.ptr = wgt; k.d[0] = 4; k.d[1] = Ck; k.d[2] = Cn;
  auto it = cache->maps.find(k);
  if (it == cache->maps.end()) {
    CUtensorMap m;
    cudaError_t e = halo::make_weight_map(wgt, Ck, Cn, &m);
    if (e != cudaSuccess) return e;
    it = cache->maps.insert({k, m}).first;
  }
  *out = &it->second;
  return cudaSuccess;
}

// out = conv3x3(act, wgt) [+ res * [mask > 0]]; act [N][H][W][Ck], wgt [Cn][9*Ck], out [N][H][W][Cn].
// `red` (nullable, Cn <= 64 only) asks for a per-channel reduction in the epilogue; its `partial`
// must hold 2*Cn floats per CTA; *ctas_out receives the number of CTAs, i.e. of partial rows.
inline bool halo_reduce_ok(int Cn) { return Cn <= 64; }
inline cudaError_t run_conv_halo(cudaStream_t st, TensorMapCache* cache, int N, int H, int W, int Ck, int Cn,
                                 const bf16_t* act, const bf16_t* wgt, bf16_t* out, const bf16_t* res,
                                 const bf16_t* res_mask, int* err_dev, const halo::EpiReduce* red = nullptr,
                                 int* ctas_out = nullptr) {
  int sms = cached_sm_count(cache) / (cache->share > 0 ? cache->share : 1);
  if (sms < 16) sms = 16;
  const halo::FwdParams p = halo::fwd_params(N, H, W, Ck, Cn, sms);
  const CUtensorMap *mx, *mw;
  cudaError_t e = cached_tile_map(cache, act, N, H, W, Ck, p.G, &mx);
  if (e == cudaSuccess) e = cached_weight_map(cache, wgt, Ck, Cn, &mw);
  if (e == cudaSuccess) e = halo::set_smem_attrs(cached_device(cache));
  if (e != cudaSuccess) return e;
  // the fewest CTAs that keep the number of tiles of the busiest one at ceil(tiles / sms)
  const int per_cta = (p.tiles + sms - 1) / sms;
  const int grid = (p.tiles + per_cta - 1) / per_cta;
  halo::EpiReduce r{};
  if (red) { if (!halo_reduce_ok(Cn)) return cudaErrorInvalidValue; r = *red; }
  if (ctas_out) *ctas_out = grid;
  return launch_chained(halo::conv_halo_kernel, grid, halo::kConvThreads, halo::fwd_smem_bytes(p), st, *mx, *mw, p, out, res, res_mask, r, err_dev);
}

// The same contract for layers of equal width (rows::conv_rows_kernel).  `res_bits`: the residual's gate as bits (or null:
// `res_mask`, or none).
inline bool rows_eligible(const ConvGeom& g) { return halo_shape(g) && rows::rows_supported(g.N, g.H, g.W, g.Ci, g.Co); }
inline cudaError_t cached_group_map(TensorMapCache* cache, const void* t, int N, int H, int W, int C, int box_g, int box_h,
                                    const CUtensorMap** out) {
  TensorMapCache::Key k;
  std::memset(&k, 0, sizeof(k));
  k.ptr = t; k.d[0] = 6; k.d[1] = N; k.d[2] = H; k.d[3] = W; k.d[4] = C; k.d[5] = box_g; k.d[6] = box_h;
  auto it = cache->maps.find(k);
  if (it == cache->maps.end()) {
    CUtensorMap m;
    cudaError_t e = rows::make_group_map(t, N, H, W, C, box_g, box_h, &m);
    if (e != cudaSuccess) return e;
    it = cache->maps.insert({k, m}).first;
  }
  *out = &it->second;
  return cudaSuccess;
}
inline cudaError_t run_conv_rows(cudaStream_t st, TensorMapCache* cache, int N, int H, int W, int C, const bf16_t* act,
                                 const bf16_t* wgt, bf16_t* out, const bf16_t* res, const bf16_t* res_mask,
                                 const unsigned char* res_bits, int* err_dev, const halo::EpiReduce* red, int* ctas_out,
                                 const EpiAffine* affine = nullptr) {
  int sms = cached_sm_count(cache) / (cache->share > 0 ? cache->share : 1);
  if (sms < 16) sms = 16;
  // the fewest CTAs that keep the number of images of the busiest one at ceil(N / sms)
  const int per_cta = (N + sms - 1) / sms, grid = (N + per_cta - 1) / per_cta;
  rows::EpiParams e{};
  const int mode = affine ? 3 : (red ? red->mode : 0);
  if (affine) e.affine = *affine;
  e.res_gate = rows::Gate{res_bits, res_bits ? nullptr : res_mask};
  if (red) {
    e.gate = rows::Gate{red->mask_bits, red->mask_bits ? nullptr : red->mask};
    e.pstats = red->pstats; e.partial = red->partial;
  }
  const int n_ops = (res ? 1 : 0) + (mode == 2 ? 1 : 0);
  const rows::RowsParams p = rows::rows_params(N, H, W, C, per_cta, n_ops);
  const CUtensorMap *ma, *mw, *mo, *mr, *mx;
  cudaError_t er = cached_group_map(cache, act, N, H, W, C, rows::kTileGroups * p.cb + 2, H + 2, &ma);
  if (er == cudaSuccess) er = cached_weight_map(cache, wgt, C, C, &mw);
  if (er == cudaSuccess) er = cached_group_map(cache, out, N, H, W, C, rows::kTileGroups, rows::kTileRows, &mo);
  mr = mx = mo;
  if (er == cudaSuccess && res) er = cached_group_map(cache, res, N, H, W, C, rows::kTileGroups, rows::kTileRows, &mr);
  if (er == cudaSuccess && mode == 2) er = cached_group_map(cache, red->xprev, N, H, W, C, rows::kTileGroups, rows::kTileRows, &mx);
  if (er == cudaSuccess) er = rows::set_attrs(cached_device(cache));
  if (er != cudaSuccess) return er;
  if (ctas_out) *ctas_out = grid;
  return launch_chained(rows::kernel_of(C, mode, res != nullptr), grid, rows::kThreads, rows::rows_smem_bytes(p), st, *ma, *mw, *mo, *mr, *mx, p, e, err_dev);
}

// dw[Co][3][3][Ci] (fp32) from x [N][H][W][Ci] and dy [N][H][W][Co]; `scratch` holds the per-CTA partials
// (halo::wgrad_scratch_elems floats).  Two launches: the tensor-core kernel and the fixed-order sum.
inline cudaError_t run_wgrad_halo(cudaStream_t st, TensorMapCache* cache, int N, int H, int W, int Ci, int Co,
                                  const bf16_t* x, const bf16_t* dy, float* dw, float* scratch, int* err_dev,
                                  bool side = false) {
  halo::WgradParams p = halo::wgrad_params(N, H, W, Ci, Co);
  const CUtensorMap *mx, *my;
  cudaError_t e = cached_tile_map(cache, x, N, H, W, Ci, p.G, &mx, p.kcx);
  if (e == cudaSuccess) e = cached_tile_map(cache, dy, N, H, W, Co, p.G, &my, p.kcy);
  if (e == cudaSuccess) e = halo::set_smem_attrs(cached_device(cache));
  if (e != cudaSuccess) return e;
  const int ctas = halo::wgrad_ctas(p, side ? cache->wgrad_side_cap : 0);
  halo::WgradMaps<1> maps;
  maps.x[0] = *mx; maps.y[0] = *my;
  e = launch_chained(halo::wgrad_halo_kernel<1>, dim3(ctas, halo::wgrad_pairs(p)), dim3(halo::kFwdThreads), halo::wgrad_smem_bytes(p), st,
                     maps, p, halo::GroupScratch{scratch, 1, nullptr}, err_dev);
  if (e != cudaSuccess) return e;
  const size_t n = (size_t)Co * 9 * Ci;
  if (n >= ((size_t)1 << 17) && ctas <= 8)        // large filters, few partials: four outputs per thread, partials in turn
    return launch_chained(wide::wgrad_wide_sum_kernel, dim3((unsigned)((n / 4 + 255) / 256)), dim3(256), 0, st,
                          reinterpret_cast<const float4*>(scratch), reinterpret_cast<float4*>(dw), n / 4, ctas);
  return launch_chained(halo::wgrad_halo_reduce_kernel, dim3((unsigned)((n + 31) / 32)), dim3(256), 0, st, (const float*)scratch, dw, n, ctas);
}
// The weight gradients of `layers` layers of one shape (c_in = c_out = C), two launches for as many of them as the two pieces of scratch
// (floats in each) hold partial sums of (at least one): x[i], dy[i] -> dw + i * dw_step.
inline size_t wgrad_group_scratch_elems(int N, int H, int W, int C, int layers, int cap) {
  return (size_t)std::min(layers, halo::kWgradLayers) * halo::wgrad_ctas(halo::wgrad_params(N, H, W, C, C), cap) * C * 9 * C;
}
inline cudaError_t run_wgrad_group(cudaStream_t st, TensorMapCache* cache, int N, int H, int W, int C, int layers, const bf16_t* const* x,
                                   const bf16_t* const* dy, float* dw, size_t dw_step, float* const (&scratch)[2], const size_t (&scratch_floats)[2], int* err_dev, int cap,
                                   uint64_t* launches) {
  halo::WgradParams p = halo::wgrad_params(N, H, W, C, C);
  cudaError_t e = halo::set_smem_attrs(cached_device(cache));
  const int ctas = halo::wgrad_ctas(p, cap);
  p.stages = 1;                                   // two CTAs per SM instead
  const size_t n = (size_t)C * 9 * C;
  const size_t hold0 = scratch_floats[0] / (n * ctas), hold1 = scratch_floats[1] / (n * ctas);
  const int most = (int)std::min<size_t>(halo::kWgradLayers, hold0 + hold1);
  if (most < 1) return cudaErrorInvalidValue;
  const halo::GroupScratch parts_at{scratch[0], (int)std::min<size_t>(hold0, halo::kWgradLayers), scratch[1]};
  const int parts = (layers + most - 1) / most, group = (layers + parts - 1) / parts;
  for (int l0 = 0; l0 < layers && e == cudaSuccess; l0 += group) {
    const int nl = std::min(group, layers - l0);
    halo::WgradMaps<halo::kWgradLayers> maps;
    for (int i = 0; i < halo::kWgradLayers && e == cudaSuccess; ++i) {
      const CUtensorMap *mx, *my;
      const int l = l0 + (i < nl ? i : 0);
      e = cached_tile_map(cache, x[l], N, H, W, C, p.G, &mx, p.kcx);
      if (e == cudaSuccess) e = cached_tile_map(cache, dy[l], N, H, W, C, p.G, &my, p.kcy);
      if (e == cudaSuccess) { maps.x[i] = *mx; maps.y[i] = *my; }
    }
    if (e != cudaSuccess) return e;
    e = launch_chained(halo::wgrad_halo_kernel<halo::kWgradLayers>, dim3(ctas, halo::wgrad_pairs(p), nl), dim3(halo::kFwdThreads),
                       halo::wgrad_smem_bytes(p), st, maps, p, parts_at, err_dev);
    if (e == cudaSuccess)
      e = launch_chained(halo::wgrad_group_sum_kernel, dim3((unsigned)((n / 2 + 127) / 128), nl), dim3(128), 0, st,
                         parts_at, dw + (size_t)l0 * dw_step, (int)(n / 2), ctas, dw_step);
    *launches += 2;
  }
  return e;
}

// The same contract for wide layers and 1x1 filters (wide::wgrad_wide_kernel; scratch of wide::wide_scratch_elems
// floats).  R = 1: H, W are the output grid and `x_sub` the stride (2: x is [N][2H][2W][Ci], read at its even pixels).
inline cudaError_t cached_slab_map(TensorMapCache* cache, const void* act, int N, int H, int W, int C, int box_w, int box_h,
                                   const CUtensorMap** out, int sub = 1) {
  TensorMapCache::Key k;
  std::memset(&k, 0, sizeof(k));
  k.ptr = act; k.d[0] = 5; k.d[1] = N; k.d[2] = H; k.d[3] = W; k.d[4] = C; k.d[5] = box_w; k.d[6] = box_h; k.d[7] = sub;
  auto it = cache->maps.find(k);
  if (it == cache->maps.end()) {
    CUtensorMap m;
    cudaError_t e = wide::make_slab_map(act, N, H, W, C, box_w, box_h, &m, sub);
    if (e != cudaSuccess) return e;
    it = cache->maps.insert({k, m}).first;
  }
  *out = &it->second;
  return cudaSuccess;
}
inline cudaError_t run_wgrad_wide(cudaStream_t st, TensorMapCache* cache, int N, int H, int W, int Ci, int Co,
                                  const bf16_t* x, const bf16_t* dy, float* dw, float* scratch, int* err_dev, int R = 3,
                                  int x_sub = 1) {
  const wide::WideParams p = wide::wide_params(N, H, W, Ci, Co, cached_sm_count(cache), R, cache->share);
  const CUtensorMap *mx, *my;
  cudaError_t e = cached_slab_map(cache, x, N, H, W, Ci, p.xw, p.S, &mx, x_sub);
  if (e == cudaSuccess) e = cached_slab_map(cache, dy, N, H, W, Co, p.Wk, p.S, &my);
  if (e == cudaSuccess) e = wide::wide_set_attrs(cached_device(cache));
  if (e != cudaSuccess) return e;
  const dim3 grid(p.co_blocks * p.ci_chunks * p.rdim, p.splits);
  auto kernel = R == 3 ? wide::wgrad_wide_kernel<3> : wide::wgrad_wide_kernel<1>;
  e = launch_chained(kernel, grid, dim3(wide::kWideThreads), wide::wide_smem_bytes(p), st, *mx, *my, p, scratch, err_dev);
  if (e != cudaSuccess) return e;
  const size_t n4 = (size_t)Co * R * R * Ci / 4;                 // Ci is a multiple of 8
  // the sum's launch overlaps the tail of the kernel above; it waits for that kernel before it reads
  return launch_chained(wide::wgrad_wide_sum_kernel, dim3((unsigned)((n4 + 255) / 256)), dim3(256), 0, st,
                        reinterpret_cast<const float4*>(scratch), reinterpret_cast<float4*>(dw), n4, p.splits);
}

// Does the data gradient of this convolution read the flipped/transposed weight copy?
inline bool dgrad_uses_flipped(const ConvGeom& g) {
  return rows_eligible(g) || halo_dgrad_eligible(g) || tc_eligible(g) || tc_s2_dgrad_eligible(g) || tc_1x1_dgrad_eligible(g);
}
// Does the stride-2 weight gradient of this convolution run on the tensor cores, given a spread-out copy of dy?
inline bool s2_uses_spread_dy(const ConvGeom& g) { return (halo_s2_wgrad_eligible(g) || wide_s2_wgrad_eligible(g)) && g.Co % 8 == 0; }
// Has a module's workspace room for that copy?  Also where only the data gradient runs on the tensor cores: a saved state holds it.
inline bool s2_has_spread_room(const ConvGeom& g) { return s2_uses_spread_dy(g) || (tc_s2_dgrad_eligible(g) && g.Co % 8 == 0); }

// fp32 scratch elements a weight-gradient call may need (bf16 storage: whichever kernel is chosen).
inline size_t conv_wgrad_scratch_elems(bool bf16_storage, const ConvGeom& g) {
  size_t n = std::max(wgrad_scratch_elems(g), direct::wgrad_direct_scratch_elems(g, bf16_storage));
  if (bf16_storage && (halo_wgrad_eligible(g) || halo_s2_wgrad_eligible(g)))
    n = std::max(n, halo::wgrad_scratch_elems(g.N, g.H, g.W, g.Ci, g.Co));
  if (bf16_storage && (wide_wgrad_eligible(g) || wide_s2_wgrad_eligible(g)))
    n = std::max(n, wide::wide_scratch_elems(g.N, g.H, g.W, g.Ci, g.Co));
  if (bf16_storage && wide_1x1_wgrad_eligible(g))
    n = std::max(n, wide::wide_scratch_elems(g.N, g.P, g.Q, g.Ci, g.Co, 1));
  return n;
}

// ---- the CUDA-core kernels, either storage type: register-tiled for 3x3 filters with padding 1 (weight gradient: also
// 1x1), the general implicit GEMM for the rest ----
// `red` (nullable) asks for per-channel sums of the output; they are formed where the consumer can add the rows up (at
// most 128 channels, whole vectors), *nparts = 0 tells the caller they were not.
template <typename T>
inline cudaError_t cuda_core_conv(cudaStream_t st, const ConvGeom& g, bool dgrad, const T* act, const T* w, T* out, const T* res,
                                  const T* mask, const direct::Reduce<T>* red, int* nparts, uint64_t* launches,
                                  const EpiAffine* affine = nullptr) {
  if (nparts) *nparts = 0;
  if (direct::conv_supported(g, dgrad)) {
    const int cn = dgrad ? g.Ci : g.Co;
    const bool sums = red && red->mode != 0 && cn % 4 == 0 && 2 * cn <= kEwThreads;
    return direct::launch_conv<T>(st, g, dgrad, act, w, out, res, mask, sums ? red : nullptr, nparts, launches, affine);
  }
  if (dgrad) return launch_conv_simt<T, CONV_DGRAD>(st, g, act, w, out, nullptr, nullptr, res, mask, launches);
  return launch_conv_simt<T, CONV_FPROP>(st, g, act, w, out, nullptr, nullptr, res, mask, launches);
}
template <typename T>
inline cudaError_t cuda_core_wgrad(cudaStream_t st, const ConvGeom& g, const T* x, const T* dy, float* scratch, float* dw,
                                   uint64_t* launches) {
  if (direct::wgrad_direct_supported(g)) return direct::launch_wgrad<T>(st, g, x, dy, scratch, dw, launches);
  return launch_conv_simt<T, CONV_WGRAD>(st, g, x, dy, (T*)nullptr, scratch, dw, (const T*)nullptr, (const T*)nullptr, launches);
}

// ---- one convolution operator in bf16 storage: which kernel, in which launch shape ------------------
// Used by the module runtime and by the operator-level entry points alike.  `launches` counts kernels.

// dy [N][P][Q][Co] of a stride-2 convolution spread onto the even pixels of a zero [N][H][W][Co] tensor `up`.
inline cudaError_t bf16_spread_dy(cudaStream_t st, const ConvGeom& g, const bf16_t* dy, bf16_t* up, uint64_t* launches) {
  const size_t nvec = (size_t)g.N * g.H * g.W * g.Co / 8;
  ++*launches;
  return launch_chained(upsample2_kernel<bf16_t, 8>, ew_blocks(nvec), 256, 0, st, dy, up, nvec, g.P, g.Q, g.Co);
}

// y = conv(x, w) [+ res].  `red` (mode 1) asks for the per-CTA sums of y and y^2; *nparts receives the number
// of rows left in red->partial, 0 when the chosen kernel forms none.
// Where the statistics of y go when a wide layer's kernel forms their partial sums (WideStats): `partial` holds one
// row of 2 * Co floats per CTA; with `stats` set, the totals are finalised right behind the convolution (mean and
// 1/sqrt(var + eps) over `rows` values per channel, running statistics included) and *nparts = -1 tells the caller
// that nothing is left to do; without, *nparts = the rows left in `partial`.
struct WideStats {
  float* partial; size_t partial_floats;
  float* stats; size_t rows; float eps;
  float* running; float momentum;
};
inline bool wide_stats_ok(TensorMapCache* cache, const ConvGeom& g, const WideStats* ws) {
  return ws && ws->partial && g.Co <= tc::kStatChunks * 16 && (size_t)cached_sm_count(cache) * 2 * g.Co <= ws->partial_floats;
}
inline cudaError_t finish_wide_stats(cudaStream_t st, const ConvGeom& g, const WideStats* ws, int ctas, int* nparts,
                                     uint64_t* launches) {
  if (!ws->stats) { if (nparts) *nparts = ctas; return cudaSuccess; }
  const RunningStats run{ws->running, ws->momentum, ws->rows > 1 ? (float)((double)ws->rows / (double)(ws->rows - 1)) : 1.f};
  ++*launches;
  if (nparts) *nparts = -1;
  return launch_stats_finalize(st, ws->partial, ctas, ws->rows, g.Co, ws->eps, ws->stats, run);
}

// Can the kernel this forward convolution takes apply a batch norm in its epilogue (`affine`)?
inline bool bf16_fprop_affine_ok(const ConvGeom& g) {
  if (rows_eligible(g)) return true;
  if (halo_fprop_eligible(g)) return false;
  if (tc_eligible(g) || tc_s2_fprop_eligible(g) || tc_1x1_fprop_eligible(g)) return 3 * g.Co <= tc::kStatFloats;
  return direct::conv_supported(g, false);
}
inline cudaError_t bf16_conv_fprop(cudaStream_t st, TensorMapCache* cache, const ConvGeom& g, const bf16_t* x,
                                   const bf16_t* w, bf16_t* y, const bf16_t* res, const halo::EpiReduce* red, int* nparts,
                                   int* err_dev, uint64_t* launches, const WideStats* ws = nullptr, const EpiAffine* affine = nullptr) {
  if (nparts) *nparts = 0;
  if (rows_eligible(g)) {
    ++*launches;
    const bool fuse = red && red->mode == 1;
    int ctas = 0;
    const cudaError_t e = run_conv_rows(st, cache, g.N, g.H, g.W, g.Ci, x, w, y, res, nullptr, nullptr, err_dev, fuse ? red : nullptr, &ctas, affine);
    if (fuse && nparts) *nparts = ctas;
    return e;
  }
  if (halo_fprop_eligible(g)) {
    ++*launches;
    const bool fuse = red && red->mode == 1 && halo_reduce_ok(g.Co);
    int ctas = 0;
    cudaError_t e = run_conv_halo(st, cache, g.N, g.H, g.W, g.Ci, g.Co, x, w, y, res, nullptr, err_dev, fuse ? red : nullptr, &ctas);
    if (fuse && nparts) *nparts = ctas;
    return e;
  }
  if (tc_eligible(g) || tc_s2_fprop_eligible(g)) {
    ++*launches;
    const int s2 = g.stride == 2 ? 1 : 0;
    if (s2 && red && red->mode == 1 && 2 * g.Co <= kEwThreads && (!ws || ws->stats)) {      // narrow: the batch norm behind it adds the rows up
      int ctas = 0;
      const cudaError_t e = run_conv_tc(st, cache, g.N, g.P, g.Q, g.Ci, g.Co, x, w, y, res, nullptr, err_dev, 1, 9, 1, red->partial, &ctas, nullptr, s2);
      if (nparts) *nparts = ctas;
      return e;
    }
    if (wide_stats_ok(cache, g, ws)) {
      int ctas = 0;
      const cudaError_t e = run_conv_tc(st, cache, g.N, g.P, g.Q, g.Ci, g.Co, x, w, y, res, nullptr, err_dev, 1, 9, 1, ws->partial, &ctas, nullptr, s2);
      return e != cudaSuccess ? e : finish_wide_stats(st, g, ws, ctas, nparts, launches);
    }
    return run_conv_tc(st, cache, g.N, g.P, g.Q, g.Ci, g.Co, x, w, y, res, nullptr, err_dev, 1, 9, 1, nullptr, nullptr, affine, s2);
  }
  if (tc_1x1_fprop_eligible(g)) {
    ++*launches;
    if (wide_stats_ok(cache, g, ws)) {
      int ctas = 0;
      const cudaError_t e = run_conv_tc(st, cache, g.N, g.P, g.Q, g.Ci, g.Co, x, w, y, res, nullptr, err_dev, 1, 1, g.stride, ws->partial, &ctas);
      return e != cudaSuccess ? e : finish_wide_stats(st, g, ws, ctas, nparts, launches);
    }
    return run_conv_tc(st, cache, g.N, g.P, g.Q, g.Ci, g.Co, x, w, y, res, nullptr, err_dev, 1, 1, g.stride, nullptr, nullptr, affine);
  }
  const direct::Reduce<bf16_t> r = red ? direct::Reduce<bf16_t>{red->mode, nullptr, nullptr, nullptr, red->partial} : direct::Reduce<bf16_t>{};
  return cuda_core_conv(st, g, false, x, w, y, res, (const bf16_t*)nullptr, red ? &r : nullptr, nparts, launches, affine);
}

// dx = conv^T(dy, w) [+ res * [mask > 0]].  `wflip` is the flipped/transposed weight copy (null: CUDA cores);
// `red` (mode 2) asks for the sums of the batch-norm backward that dx feeds; a stride-2 layer forms them given `dy_up`, the
// spread-out dy (nullable).
inline cudaError_t bf16_conv_dgrad(cudaStream_t st, TensorMapCache* cache, const ConvGeom& g, const bf16_t* dy,
                                   const bf16_t* w, const bf16_t* wflip, const bf16_t* dy_up, bf16_t* dx, const bf16_t* res,
                                   const bf16_t* mask, const halo::EpiReduce* red, int* nparts, int* err_dev,
                                   uint64_t* launches, const unsigned char* mask_bits = nullptr) {
  if (nparts) *nparts = 0;
  if (wflip && rows_eligible(g)) {
    ++*launches;
    const bool fuse = red && red->mode == 2;
    int ctas = 0;
    const cudaError_t e = run_conv_rows(st, cache, g.N, g.H, g.W, g.Ci, dy, wflip, dx, res, mask, mask_bits, err_dev, fuse ? red : nullptr, &ctas);
    if (fuse && nparts) *nparts = ctas;
    return e;
  }
  const bool s2_sums = wflip && dy_up && red && red->mode == 2 && halo_s2_dgrad_sums_eligible(g);
  if ((wflip && halo_dgrad_eligible(g)) || s2_sums) {
    ++*launches;
    const bool fuse = red && red->mode == 2 && halo_reduce_ok(g.Ci);
    int ctas = 0;
    cudaError_t e = run_conv_halo(st, cache, g.N, g.H, g.W, g.Co, g.Ci, s2_sums ? dy_up : dy, wflip, dx, res, mask, err_dev, fuse ? red : nullptr, &ctas);
    if (fuse && nparts) *nparts = ctas;
    return e;
  }
  if (wflip && tc_eligible(g)) {
    ++*launches;
    return run_conv_tc(st, cache, g.N, g.H, g.W, g.Co, g.Ci, dy, wflip, dx, res, mask, err_dev);
  }
  if (wflip && tc_s2_dgrad_eligible(g)) {
    ++*launches;
    return run_conv_tc(st, cache, g.N, g.P, g.Q, g.Co, g.Ci, dy, wflip, dx, res, mask, err_dev, 1, 9, 1, nullptr, nullptr, nullptr, 2);
  }
  if (wflip && tc_1x1_dgrad_eligible(g) && (g.stride == 1 || (!res && !mask))) {
    // stride 2: only the even pixels of dx receive a gradient; the rest of dx is cleared first
    if (g.stride == 2) {
      const cudaError_t e = cudaMemsetAsync(dx, 0, (size_t)g.N * g.H * g.W * g.Ci * sizeof(bf16_t), st);
      if (e != cudaSuccess) return e;
    }
    ++*launches;
    return run_conv_tc(st, cache, g.N, g.P, g.Q, g.Co, g.Ci, dy, wflip, dx, res, mask, err_dev, g.stride == 2 ? 3 : 1, 1, 1);
  }
  const direct::Reduce<bf16_t> r = red ? direct::Reduce<bf16_t>{red->mode, red->mask, red->xprev, red->pstats, red->partial} : direct::Reduce<bf16_t>{};
  return cuda_core_conv(st, g, true, dy, w, dx, res, mask, red ? &r : nullptr, nparts, launches);
}

// dw (fp32) from x and dy; `scratch` of conv_wgrad_scratch_elems floats; `side`: bound the pixel split by
// cache->wgrad_side_cap (a weight gradient issued beside the chain that needs the SMs more).
inline cudaError_t bf16_conv_wgrad(cudaStream_t st, TensorMapCache* cache, const ConvGeom& g, const bf16_t* x,
                                   const bf16_t* dy, const bf16_t* dy_up, float* dw, float* scratch, int* err_dev,
                                   bool side, uint64_t* launches) {
  if ((dy_up && wide_s2_wgrad_eligible(g)) || wide_wgrad_eligible(g)) {
    *launches += 2;
    return run_wgrad_wide(st, cache, g.N, g.H, g.W, g.Ci, g.Co, x, wide_wgrad_eligible(g) ? dy : dy_up, dw, scratch, err_dev);
  }
  if (wide_1x1_wgrad_eligible(g)) {
    *launches += 2;
    return run_wgrad_wide(st, cache, g.N, g.P, g.Q, g.Ci, g.Co, x, dy, dw, scratch, err_dev, 1, g.stride);
  }
  if (dy_up && halo_s2_wgrad_eligible(g)) {
    *launches += 2;
    return run_wgrad_halo(st, cache, g.N, g.H, g.W, g.Ci, g.Co, x, dy_up, dw, scratch, err_dev, side);
  }
  if (halo_wgrad_eligible(g)) {
    *launches += 2;
    return run_wgrad_halo(st, cache, g.N, g.H, g.W, g.Ci, g.Co, x, dy, dw, scratch, err_dev, side);
  }
  return cuda_core_wgrad(st, g, x, dy, scratch, dw, launches);
}

}  // namespace fdg
