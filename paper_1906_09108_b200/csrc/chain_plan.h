// Launch shapes of the runs of identity blocks (conv_chain.cuh) and arithmetic of theirs that the host can run too.
#pragma once
#include <math.h>
#include <stddef.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

namespace fdg {
namespace chain {

constexpr int kEpiWarps = 16, kEpiThreads = 32 * kEpiWarps;
constexpr int kAccSlots = 8;                     // accumulators of 128 rows x 64 columns: all of tensor memory
constexpr int kTileRows = 16, kTileGroups = 8;   // a tile: image rows, groups of 64 / C pixels
constexpr int kMaxCtas = 148;
enum Pass { TRAIN = 0, INFER = 1, BACKWARD = 2 };

struct Geom {
  int N, H, W, WG;            // image; groups per row (W / G)
  int rb, cb, tpi;            // tiles of an image: row blocks, column blocks, rb * cb
  int images;                 // per CTA at most; images * tpi <= kAccSlots
  int layers;                 // convolutions of the run (two per block)
  uint32_t row_bytes;         // shared memory of one image row: (8 * cb + 2) groups
  uint32_t a_bytes;           // one image, multiple of 1 KiB
  uint32_t a_tx;              // bytes its load writes
  uint32_t w_bytes;           // nine taps, multiple of 1 KiB
  int w_stages;
};

// A tile: its first element in a tensor of the layers' shape, its place in the operands, how much of it lies inside the image,
// its image and that image's first tile.
struct __align__(16) Tile { uint32_t g, s; uint16_t rows, groups, image, first; };

inline uint32_t round_up(uint32_t x, uint32_t a) { return (x + a - 1) / a * a; }
constexpr size_t kSmemLimit = 226 * 1024;
// Two CTAs of such launches must never share an SM: both want all of tensor memory, and each may hold it while the other's
// launch waits for a CTA elsewhere.  Their registers forbid it already (640 threads of 96); their shared memory does too.
constexpr size_t kSmemLeast = 120 * 1024;
inline size_t fixed_smem(int C) {
  return (size_t)kEpiThreads * 8 + (size_t)kEpiWarps * 2 * C * 4 + (size_t)2 * 5 * C * 4 + (3 * kAccSlots + 4) * 8 + 16 + kAccSlots * sizeof(Tile) + 1024;
}
// Launch shape: about `sms` CTAs; images = 0 where the shape is not covered.  A CTA holds its images' operands and accumulators.
inline Geom chain_geom(int N, int H, int W, int C, int layers, int sms, int pass) {
  Geom p{};
  const int G = 64 / C;
  p.N = N; p.H = H; p.W = W; p.WG = W / G; p.layers = layers;
  p.rb = (H + kTileRows - 1) / kTileRows; p.cb = (p.WG + kTileGroups - 1) / kTileGroups; p.tpi = p.rb * p.cb;
  p.row_bytes = (uint32_t)(kTileGroups * p.cb + 2) * 128;
  p.a_bytes = round_up((uint32_t)(p.rb * kTileRows + 2) * p.row_bytes, 1024);
  p.a_tx = (uint32_t)(H + 2) * p.row_bytes;
  p.w_bytes = round_up((uint32_t)(9 * C * C * 2), 1024);
  const size_t left = kSmemLimit - fixed_smem(C) - p.w_bytes;
  int most = (int)std::min<size_t>(left / p.a_bytes, (size_t)(kAccSlots / p.tpi));
  const int want = (N + sms - 1) / sms;
  if (most > want) most = want;
  p.images = most;
  if (most < 1) return p;
  p.w_stages = pass == INFER && (size_t)most * p.a_bytes + 2 * (size_t)p.w_bytes + fixed_smem(C) <= kSmemLimit ? 2 : 1;
  return p;
}
inline int chain_ctas(const Geom& p) { return (p.N + p.images - 1) / p.images; }
inline size_t exchange_words(int N, int C) { return (size_t)2 * std::min(N, kMaxCtas) * 2 * C; }      // for any launch of a run
inline size_t chain_smem_bytes(const Geom& p, int C) {
  return std::max(kSmemLeast, (size_t)p.images * p.a_bytes + (size_t)p.w_stages * p.w_bytes + fixed_smem(C));
}
inline bool chain_supported(int N, int H, int W, int C) {
  if ((C != 16 && C != 32 && C != 64) || N < 1) return false;
  const int G = 64 / C;
  if (W % G || H + 2 > 256 || W / G + 2 > 256 || kTileGroups * ((W / G + kTileGroups - 1) / kTileGroups) + 2 > 256) return false;
  const Geom p = chain_geom(N, H, W, C, 2, kMaxCtas, TRAIN);
  return p.images >= 1 && p.a_tx < (1u << 20) && chain_ctas(p) <= kMaxCtas;
}

// Runs of all modules, and whether each trains as one launch per pass.  A module has one such launch on the device at a time, but
// the modules' launches go side by side, and CTAs that wait for one another must all be resident: a launch takes the device's SMs
// as if every other module had its largest one there.
struct Run { int module, blocks, N, H, W, C; bool launch; };
constexpr int kLeastShare = 16;                  // a module's share of the SMs is not taken to be smaller
inline int module_share(int sms, int modules) { return std::max(kLeastShare, sms / std::max(1, modules)); }
inline int run_ctas(const Run& r, int share) {
  int most = 0;
  for (int pass : {TRAIN, BACKWARD}) {
    const Geom p = chain_geom(r.N, r.H, r.W, r.C, 2, share, pass);
    if (p.images < 1) return kMaxCtas + 1;
    most = std::max(most, chain_ctas(p));
  }
  return most;
}
inline bool within_share(int ctas, int share) { return 5 * ctas <= 8 * share; }
// `modules`: how many have streams of their own (1: all on one stream, each launch has the device to itself).
// A launch's CTAs exceed its module's share where shared memory or the accumulators cap its images per CTA (128 images of 40x40x16:
// 128 CTAs at any share).  Beyond 8/5 of the share a run goes layer by layer: the other modules then wait for SMs, and one image per
// CTA gains little.  (ms per iteration, by runs / layer by layer.  K = 4, 18 blocks a stage: 150 images of 32x32x16, 1.03 shares,
// 1.24 / 1.62; 40x40x16, 48 images, 1.3 shares, 1.02 / 1.36, 56 images, 1.5 shares, 1.30 / 1.44, 72 images, 1.9 shares, 1.82 / 1.65;
// K = 4, 128 images, 1.7 shares: 20x20x32 1.40 / 1.34, 32x32x32 1.064 / 1.045; K = 2, 24x24x64, 1.7 shares, 1.64 / 1.53.)
// Where the modules' largest launches together still want more than `sms`, those runs go as launches that hold the most blocks within
// it (what a block gains hardly depends on its shape): the best sum over the modules of the blocks in runs of at most so many CTAs.
inline void fit_device(std::vector<Run>& runs, int modules, int sms) {
  const int share = module_share(sms, modules);
  std::vector<int> ctas;
  for (Run& r : runs) {
    ctas.push_back(run_ctas(r, share));
    r.launch = ctas.back() <= std::min(sms, kMaxCtas) && (modules <= 1 || within_share(ctas.back(), share));
  }
  if (modules <= 1) return;
  std::vector<std::vector<int>> best(modules + 1, std::vector<int>(sms + 1, 0)), limit = best;
  for (int k = 0; k < modules; ++k)
    for (int have = 0; have <= sms; ++have) {
      best[k + 1][have] = best[k][have];
      for (size_t i = 0; i < runs.size(); ++i) {
        if (runs[i].module != k || !runs[i].launch || ctas[i] > have) continue;
        int blocks = best[k][have - ctas[i]];
        for (size_t j = 0; j < runs.size(); ++j) blocks += runs[j].module == k && runs[j].launch && ctas[j] <= ctas[i] ? runs[j].blocks : 0;
        if (blocks > best[k + 1][have]) { best[k + 1][have] = blocks; limit[k + 1][have] = ctas[i]; }
      }
    }
  for (int k = modules - 1, have = sms; k >= 0; --k) {
    const int most = limit[k + 1][have];
    for (size_t i = 0; i < runs.size(); ++i) if (runs[i].module == k && ctas[i] > most) runs[i].launch = false;
    have -= most;
  }
}

// 1 / sqrt(v) in fp64, rounded to fp32, to the last bit: a fp32 approximation `seed` within 2^-21 of it and one Newton step in fp64
// leave a relative error below 1.5 * 2^-42 and rounding; where everything within 2^-40 rounds to the same fp32 value that is the
// result, else (one argument in about 2^16) false, and the caller divides.  A seventh of the time of the fp64 square root
// and division that every layer would wait for.
__host__ __device__ inline bool inverse_sqrt_from(double v, float seed, float& r) {
  const double y = (double)seed, z = y * fma(-0.5 * v * y, y, 1.5), d = z * 0x1p-40;
  r = (float)(z + d);
  return r == (float)(z - d);
}

// Tiles at once: as many as share the CTA's tiles evenly (inference, few tiles: at most 2; the others at least 2).
// (ms a logging interval, ResNet-56 K = 2 / its K = 3 on 28x28 / ResNet-110 K = 4 / ResNet-1202 K = 4: by this rule 6.28 / 4.27 / 9.82 / 27.26;
// training and backward 2 and 2 everywhere 6.22 / 4.25 / 9.72 / 26.54, 2 and 4 6.46 / 4.43 / 9.79 / 27.86, 4 and 2 6.27 / 4.31 / 9.89 / 26.94,
// 4 and 4 6.56 / 4.53 / 9.82 / 28.72.  Eight batches of inference, 1 / 2 everywhere: ResNet-110 3.42 / 3.22, 128 images of 40x40 1.89 / 1.77, one image
// 1.06 / 1.03.)
inline int chain_streams(const Geom& p, int pass) {
  const int tiles = p.images * p.tpi;
  if (pass == INFER) return tiles % 2 == 0 ? 2 : 1;
  return tiles % 4 == 0 || tiles == 3 || tiles > 6 ? 4 : 2;
}

}  // namespace chain
}  // namespace fdg
