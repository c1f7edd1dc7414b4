// Channel tile of the tensor-core convolutions (host code only, no CUDA: the rules are tested without a GPU).
#pragma once
#include <algorithm>

namespace lp {

// Fewest tiles of at most 256 channels with the least padding.
inline void pick_n_tile(int Cout, int& n_tile, int& n_tiles) {
  int best_nt = 0, best_tile = 0, best_waste = 1 << 30;
  const int lo = (Cout + 255) / 256;
  for (int nt = lo; nt <= lo + 3; ++nt) {
    int tile = (Cout + nt - 1) / nt;
    tile = (tile + 15) / 16 * 16;
    if (tile > 256) continue;
    const int waste = nt * tile - Cout;
    if (waste < best_waste) { best_waste = waste; best_nt = nt; best_tile = tile; }
  }
  n_tile = best_tile;
  n_tiles = best_nt;
}

struct ConvTileQuery {
  int Cout, m_tiles, sm_count;
  int k_mmas;        // K = 16 slices of a tile
  int epilogue;      // 0 plain, 1 with statistics, 2 with a shortcut
  bool wide_epi;     // eight epilogue warps at 256 channels
};

// Cycles of the busiest CTA.  A tile costs its MMAs (0.46 a column each, at least 82, or 75 where two accumulators
// alternate: a pipeline stage of narrow MMAs takes that long with its waits and operand reads) and its epilogue, which runs
// beside the next tile's MMAs; the first tile's MMAs, the last epilogue and 3800 cycles of start and end are not hidden.
// The constants are fitted to 2334 timings of launches alone on the machine (3x3 and 1x1 layers of 64 to 2048 channels, 5 to
// 56 pixels wide, 1 to 128 images, plain, with statistics and with a shortcut, every tile of 64 to 256 columns): of the 531
// choices among them the fastest tile takes 0.828 of the time of pick_n_tile's in the geometric mean, the estimate's choice
// 0.831, and it is at most 3 % slower than pick_n_tile's anywhere.  (The first form of this estimate, 33 cycles for a narrow
// MMA and 20 a column for every epilogue, took 64 columns where 160 or 256 are faster: 320 -> 320 channels, 128 images of
// 16x16 with statistics, 63.7 us instead of 50.6; 64 -> 256, 32 images of 56x56 with a shortcut, 51.0 instead of 29.2.)
inline double conv_tile_cycles(const ConvTileQuery& q, int tile) {
  static const double column[2][3] = {{29.0, 33.0, 25.0}, {28.0, 32.0, 18.0}};   // [eight warps][epilogue]
  const long long tiles = (long long)q.m_tiles * ((q.Cout + tile - 1) / tile);
  const double per = (double)((tiles + q.sm_count - 1) / q.sm_count);
  const bool pair = q.m_tiles >= 2 && 2 * tiles >= 3 * std::min<long long>(tiles, q.sm_count);
  const double mma = q.k_mmas * std::max(pair ? 75.0 : 82.0, tile * 0.46);
  const double epi = 1250.0 + tile * column[q.wide_epi && tile == 256 ? 1 : 0][q.epilogue];
  return 3800.0 + mma + epi + (per - 1.0) * std::max(mma, epi);
}

// What SM time is worth beside the length of a launch, where modules run side by side: a launch of length t on a share s of the
// SMs costs t (1 + w s).  `step_flops`: convolutions of the modules in one training step (not those of the AuxNets).  Steps of little work are as long as their chains of
// launches, and narrower tiles shorten a launch of few CTAs (8 CTAs of 256 channels took 40 to 46 us of ResNet-50's last module
// on 12 images of 176x176); steps of much work are bound by the SM time that narrow tiles waste.  us per step for w = none, 1,
// 2, 4, 8, 16: ResNet-34 on 3 images of 256x176 (0.06 TFLOP) 781, 683, 640, 638, 642, 674, on 25 of 128x160 with recursive
// AuxNets and distillation (0.22) 1234, 1159, 1158, 1196, 1232, 1232; ResNet-50 on 12 of 176x176 (0.18) 1405, 1369, 1360, 1361,
// 1370, 1410, on 19 with distillation (0.29) 2130, 2091, 2086, 2090, 2106, 2134, on 32 of 224x224 (0.79) 3303, 3358, 3332, 3325,
// 3306, 3308.  Where the cubic goes beyond 16 it is as good as infinite: against a limit of 16, ResNet-50 on 32 of 224x224 (w = 79)
// 3240 and 3239, ResNet-34 on 64 of them (w in the hundreds) 2875 and 2872, WRN-28-10 on 128 of 32x32 (w = 10 000) 4690 and 4682.
// The rule does not know the number of modules: with one module, which only its own weight gradients run beside, w = 0 would be
// right for some networks (WRN-28-10 on 16 images 1530 -> 1435) and wrong for others (ResNet-34 on 8 of 160x160 1295 -> 1408).
// Tiles of 64 columns also select the two-per-SM instantiation for small layers, which conv_tile_cycles() takes for the other one.
inline double sm_time_worth(double step_flops) {
  const double x = step_flops / 0.25e12;
  return 2.5 * std::max(1.0, x * x * x);
}

// Channel tile of least cost: `worth` = 0 for a launch that has the machine to itself, sm_time_worth() beside other modules.  The
// widest tiles leave SMs idle where there are few pixel tiles (74 CTAs of 256 channels on 37 images of 12x16).  A narrower tile
// has to be estimated 2 % cheaper.
inline void pick_n_tile_by_cost(const ConvTileQuery& q, double worth, int& n_tile, int& n_tiles) {
  const auto cost = [&](int tile) {
    const long long tiles = (long long)q.m_tiles * ((q.Cout + tile - 1) / tile);
    return conv_tile_cycles(q, tile) * (1.0 + worth * (double)std::min<long long>(tiles, q.sm_count) / q.sm_count);
  };
  pick_n_tile(q.Cout, n_tile, n_tiles);
  const int widest = n_tile, lo = (q.Cout + 255) / 256;
  double best = cost(widest);
  for (int nt = lo; nt <= 8 * lo; ++nt) {
    const int tile = ((q.Cout + nt - 1) / nt + 31) / 32 * 32;
    if (tile > 256 || tile < 64 || tile == widest) continue;
    const double t = cost(tile);
    if (t < best * 0.98) { best = t; n_tile = tile; n_tiles = (q.Cout + tile - 1) / tile; }
  }
}

}  // namespace lp
