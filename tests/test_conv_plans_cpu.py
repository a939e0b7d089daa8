"""Launch plans without a GPU: whatever shape the dispatcher hands to the CUDA-core convolutions, the launch they plan stays
within the shared memory that the kernels are given and covers the whole problem; and the split of the wide weight
gradients bounds what an accumulator adds up.  A small host program made from the library's own headers walks the
shapes."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1906_09108_b200", "csrc")

PROLOGUE = r"""
#include <cstdio>
#include <cstring>
#include <cuda.h>
#include "fdg_ops.h"
#include "chain_plan.h"
#include "conv_direct.cuh"
#include "wgrad_wide.cuh"
using namespace fdg;
static int bad = 0;
static void report(const char* what, const ConvGeom& g, size_t bytes) {
  if (bad++ < 10) printf("%s N=%d %dx%d %d->%d R=%d stride=%d: %zu\n", what, g.N, g.H, g.W, g.Ci, g.Co, g.R, g.stride, bytes);
}
template <typename F> static void shapes(F f) {
  const int chans[] = {1, 4, 5, 8, 16, 24, 32, 33, 64}, batches[] = {1, 128, 600, 2368};
  for (int N : batches) for (int R = 1; R <= 3; R += 2) for (int s = 1; s <= 2; ++s)
    for (int H = 1; H <= 70; H += H < 18 ? 1 : 5) for (int W = 1; W <= 64; W += W < 18 ? 1 : 3)
      for (int ci : chans) for (int co : chans) {
        const int P = (H + 2 * (R / 2) - R) / s + 1, Q = (W + 2 * (R / 2) - R) / s + 1;
        f(ConvGeom{N, H, W, ci, P, Q, co, R, R, s, R / 2});
      }
}
"""


def _run(tmp_path, body):
    src = tmp_path / "plans.cu"
    src.write_text(PROLOGUE + "int main() {\n" + body + "\n  return bad != 0;\n}\n")
    exe = str(tmp_path / "plans")
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", CSRC, "-I",
                    os.path.join(os.path.dirname(os.path.dirname(CSRC)), "include"), "-o", exe, str(src)], check=True,
                   capture_output=True)
    res = subprocess.run([exe], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout


def test_weight_gradient_plans_fit_shared_memory(tmp_path):
    _run(tmp_path, r"""
  shapes([](const ConvGeom& g) {
    if (!direct::wgrad_direct_supported(g)) return;
    for (int by_row = 0; by_row < 2; ++by_row) {
      const direct::WgradParams p = direct::wgrad_params(g, by_row != 0);
      const size_t bytes = direct::wgrad_smem(p, g.R, g.stride, p.TH, by_row != 0);
      if (bytes > direct::kWgradSmemMax) report("shared memory", g, bytes);
      if (p.rg < 1 || p.rg * p.tt > p.threads || p.threads > direct::kThreads) report("threads", g, (size_t)p.threads);
      if (p.rows_x != (p.TH - 1) * g.stride + g.R) report("rows of x", g, (size_t)p.rows_x);
      if (p.TH < 1 || p.TH * p.strips < g.P || p.units != g.N * p.strips || p.splits < 1) report("rows", g, (size_t)p.TH);
    }
  });""")


def test_forward_and_data_gradient_plans_fit_shared_memory(tmp_path):
    _run(tmp_path, r"""
  shapes([](const ConvGeom& g) {
    for (int dgrad = 0; dgrad < 2; ++dgrad) {
      if (!direct::conv_supported(g, dgrad != 0)) continue;
      for (int nc = 4; nc <= 8; nc += 4) {
        const direct::ConvParams p = direct::conv_params(g, dgrad != 0, nc);
        const size_t bytes = direct::conv_smem_bytes(p);
        if (bytes > direct::kConvSmemMax) report("shared memory", g, bytes);
        if (p.TI * p.TH * p.segs * p.cgs > direct::kThreads) report("threads", g, (size_t)(p.TI * p.TH * p.segs * p.cgs));
        if (p.TI < 1 || p.TH < 1 || p.TH * p.row_tiles < p.P || (long)p.tiles * p.TI < (long)g.N * p.row_tiles) report("tiles", g, (size_t)p.tiles);
        if ((long)p.TI * p.rows_in * (p.Wi * p.up + 2) * 4 >= 1 << 20) report("items", g, (size_t)p.TI);   // div_small's range
      }
    }
  });""")


def test_a_share_of_the_gpu_lengthens_no_long_accumulation(tmp_path):
    """An accumulator's rounding error grows with its instructions: sharing the SMs may bring them up to 256, beyond that
    the split is the whole GPU's; and never finer than that one, for which the scratch is sized."""
    _run(tmp_path, r"""
  const int chans[] = {8, 64, 128, 160, 256, 320, 512, 640};
  for (int R = 1; R <= 3; R += 2) for (int N : {1, 8, 128, 2048}) for (int H : {4, 6, 8, 13, 16, 24, 32, 64})
    for (int ci : chans) for (int co : chans) {
      const ConvGeom g{N, H, H, ci, H, H, co, R, R, 1, R / 2};
      if (!wide::wide_supported(N, H, H, ci, co, R)) continue;
      const wide::WideParams whole = wide::wide_params(N, H, H, ci, co, 148, R);
      for (int share = 1; share <= 16; ++share) {
        const wide::WideParams p = wide::wide_params(N, H, H, ci, co, 148, R, share);
        auto steps = [](const wide::WideParams& q) {      // instructions with pixels in them
          const int rows = q.S < q.H ? q.S : q.H;
          return (q.slabs + q.splits - 1) / q.splits * ((rows * q.Wk + 15) / 16);
        };
        if (p.splits < 1 || p.splits > whole.splits) report("splits", g, (size_t)p.splits);
        if (steps(p) > 256 && steps(p) > steps(whole)) report("instructions", g, (size_t)steps(p));
      }
    }""")


def test_runs_of_blocks_fit_an_sm_and_the_device(tmp_path):
    """Every launch shape of a run holds its images' operands and accumulators, covers the batch with CTAs that can be resident
    together, and keeps a CTA's tiles below the slots; more than half of an SM's shared memory, so that two never share one."""
    _run(tmp_path, r"""
  for (int C = 16; C <= 64; C *= 2) for (int N : {1, 2, 31, 97, 128, 148, 149, 160, 600, 1184}) for (int H = 1; H <= 70; ++H) for (int W = 1; W <= 70; ++W) {
    const ConvGeom g{N, H, W, C, H, W, C, 3, 3, 1, 1};
    if (!chain::chain_supported(N, H, W, C)) continue;
    for (int share = 1; share <= 16; ++share) for (int pass = 0; pass < 3; ++pass) {
      const chain::Geom p = chain::chain_geom(N, H, W, C, 2, 148 / share < 16 ? 16 : 148 / share, pass);
      const size_t bytes = chain::chain_smem_bytes(p, C);
      const int ctas = chain::chain_ctas(p), st = chain::chain_streams(p, pass);
      if (bytes > chain::kSmemLimit || 2 * bytes <= 228 * 1024) report("shared memory", g, bytes);
      if (p.images < 1 || p.images * p.tpi > chain::kAccSlots) report("accumulators", g, (size_t)p.images);
      if (ctas < 1 || ctas > chain::kMaxCtas || ctas > N || (long)ctas * p.images < N) report("CTAs", g, (size_t)ctas);
      if (p.rb * chain::kTileRows < H || p.cb * chain::kTileGroups * (64 / C) < W || p.WG * (64 / C) != W) report("tiles", g, (size_t)p.tpi);
      if ((size_t)(p.rb * chain::kTileRows + 2) * p.row_bytes > p.a_bytes || p.a_bytes % 1024 || p.w_bytes % 1024) report("operands", g, p.a_bytes);
      if ((size_t)p.w_bytes < (size_t)18 * C * C || p.w_stages < 1 || p.w_stages > 2 || (pass != chain::INFER && p.w_stages != 1)) report("weights", g, p.w_bytes);
      if (pass == chain::INFER ? st > 2 : st < 2) report("streams", g, (size_t)st);
    }
  }""")


def test_runs_of_all_modules_fit_the_device_together(tmp_path):
    """CTAs of a run wait for one another: whatever the modules' runs are, the launches that may meet want no more SMs than there
    are, none is given up where all fit, and the shape each is launched with is the one that was counted."""
    _run(tmp_path, r"""
  unsigned seed = 1;
  auto pick = [&](int n) { seed = seed * 1664525u + 1013904223u; return (int)((seed >> 8) % (unsigned)n); };
  for (int it = 0; it < 40000; ++it) {
    const int modules = 1 + pick(16), sms = pick(4) ? 148 : 16 + pick(133), N = 1 + pick(pick(2) ? 160 : 600), side = 4 * (1 + pick(16)), share = chain::module_share(sms, modules);
    std::vector<chain::Run> runs;
    for (int k = 0; k < modules; ++k)
      for (int j = pick(4); j > 0; --j) {
        const int down = pick(3), C = 16 << pick(3), H = side >> down;
        if (H >= 1 && chain::chain_supported(N, H, H, C)) runs.push_back(chain::Run{k, 1 + pick(20), N, H, H, C, false});
      }
    std::vector<int> all(modules, 0), on(modules, 0);
    bool alone = true;
    chain::fit_device(runs, modules, sms);
    for (const chain::Run& r : runs) {
      const int n = chain::run_ctas(r, share);
      for (int pass : {chain::TRAIN, chain::BACKWARD}) {
        const chain::Geom p = chain::chain_geom(r.N, r.H, r.W, r.C, 2, share, pass);
        if (p.images < 1 || chain::chain_ctas(p) > n) report("counted", ConvGeom{r.N, r.H, r.W, r.C, r.H, r.W, r.C, 3, 3, 1, 1}, (size_t)n);
      }
      all[r.module] = std::max(all[r.module], n);
      if (r.launch) on[r.module] = std::max(on[r.module], n);
      alone = alone && n <= sms && (modules == 1 || chain::within_share(n, share));
    }
    int want = 0, have = 0;
    for (int k = 0; k < modules; ++k) { want += all[k]; have += on[k]; }
    const ConvGeom g{N, side, side, modules, side, side, sms, 3, 3, 1, 1};
    if (have > sms) report("together", g, (size_t)have);
    for (const chain::Run& r : runs) {
      const int n = chain::run_ctas(r, share);
      if (r.launch && modules > 1 && !chain::within_share(n, share)) report("beyond its share", g, (size_t)n);
      if (r.launch) continue;
      if (alone && (want <= sms || modules == 1)) report("given up", g, (size_t)want);
      if (modules > 1 && chain::within_share(n, share) && have - on[r.module] + std::max(on[r.module], n) <= sms) report("left out", g, (size_t)have);
    }
  }
  // 128 images: two modules of 40x40x16 (128 CTAs each), four or three of 32x32x32 (64 each), four of 16x16x64 (43 each) and of 32x32x16 (32 each)
  struct { int n, side, C, kept; } known[] = {{2, 40, 16, 0}, {4, 32, 32, 0}, {3, 32, 32, 2}, {4, 16, 64, 3}, {4, 32, 16, 4}};
  for (auto& q : known) {
    std::vector<chain::Run> runs;
    for (int k = 0; k < q.n; ++k) runs.push_back(chain::Run{k, 4, 128, q.side, q.side, q.C, false});
    chain::fit_device(runs, q.n, 148);
    int kept = 0;
    for (const chain::Run& r : runs) kept += r.launch;
    if (kept != q.kept) report("kept", ConvGeom{128, q.side, q.side, q.C, q.side, q.side, q.C, 3, 3, 1, 1}, (size_t)kept);
  }
  // the most blocks, not the most modules: 64 + 64 CTAs hold 4 + 2 + 2 of them, 43 + 43 and 64 + 43 at most 7
  std::vector<chain::Run> runs = {{0, 4, 128, 32, 32, 32, false}, {1, 2, 128, 32, 32, 32, false}, {1, 2, 128, 16, 16, 64, false}, {2, 3, 128, 16, 16, 64, false}};
  chain::fit_device(runs, 3, 148);
  if (!runs[0].launch || !runs[1].launch || !runs[2].launch || runs[3].launch) report("most blocks", ConvGeom{128, 32, 32, 32, 32, 32, 32, 3, 3, 1, 1}, 0);""")


def test_a_run_s_inverse_square_root_is_the_64_bit_one_rounded(tmp_path):
    """1 / sqrt(v) of a run's batch norms: what the short way returns is (float)(1.0 / sqrt(v)) to the last bit, with a seed as far
    off as an fp32 approximation may be (4 units; rsqrtf promises 2), for ordinary arguments and for those whose result lies
    next to the middle of two fp32 values; and nearly every ordinary argument takes it."""
    _run(tmp_path, r"""
  unsigned long long seed = 1;
  auto next = [&]() { seed = seed * 6364136223846793005ull + 1442695040888963407ull; return (double)(seed >> 11) / 9007199254740992.0; };
  auto units = [](float x, int n) { unsigned u; memcpy(&u, &x, 4); u += n; memcpy(&x, &u, 4); return x; };
  const ConvGeom none{};
  long taken = 0, all = 0;
  for (int it = 0; it < 2000000; ++it) {
    const bool tie = it & 1;
    double v = exp2(next() * 120.0 - 60.0);
    if (tie) {
      const float f = (float)(1.0 / sqrt(v));
      const double middle = 0.5 * ((double)f + (double)units(f, 1));
      v = 1.0 / (middle * middle) * (1.0 + (next() - 0.5) * exp2(-36.0 - 16.0 * next()));
    }
    const float want = (float)(1.0 / sqrt(v)), s = units((float)(1.0 / sqrt((double)(float)v)), (int)(next() * 9.0) - 4);
    float r;
    const bool ok = chain::inverse_sqrt_from(v, s, r);
    if (ok && r != want) report("last bit", none, (size_t)it);
    if (!tie) { ++all; taken += ok; }
  }
  if (all - taken > all / 10000) report("taken", none, (size_t)(all - taken));""")
