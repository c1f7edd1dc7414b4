// Which fp32 convolutions take the tiled kernels of conv_f32.cuh (host code only, no CUDA: tested without a GPU).  The tiled
// kernels take any 1x1 or 3x3 filter; the direct ones of conv_simt.cuh are faster where a tile's 16 x 16 channels are mostly
// padding and the launch is large, and for the 1x1 stride-1 input gradient of launches that fill the machine.  Measured over
// 1378 shapes alone on the machine: fp32 forward and input gradient on either kernel, 4 to 512 channels, 1 to 128 images.
// (With the tiled kernels everywhere: 4 -> 64 channels, 3x3, 64 images of 32x32, 48.3 us instead of 22.6; the input gradient
// of 128 -> 128, 1x1, 64 images of 28x28, 205 instead of 135.)
#pragma once
#include <algorithm>

namespace lp {

struct F32Conv { int N, H, W, cin, OH, OW, cout, R, stride; };

// few_channel_kernel: the direct kernel would be the one with the filter bank in shared memory.  (No machine size in it:
// whether the batch-norm statistics come with the convolution is part of the plan, which is made without a device.)
inline bool f32_forward_on_tiles(const F32Conv& c, bool few_channel_kernel) {
  const long long tiles = (long long)c.N * ((c.OH + 7) / 8) * ((c.OW + 7) / 8);
  if (c.cin <= 4 && few_channel_kernel) return tiles < (c.R == 1 ? 256 : 512);
  if (c.cin <= 8 && c.R == 1 && c.cin * c.cout <= 64) return tiles < 256;
  if (c.cin * c.cout <= 16) return tiles < 1024;
  return true;
}

// Estimated microseconds of both kernels.  Tiled: waves of four blocks an SM, each as long as its 16-channel chunks take.
// Direct (one pixel x 4 channels a thread, 2048 threads an SM): a latency of one pass over C_out, then throughput, lower
// once the weights (64 KB and more) leave the L1 cache.
inline bool f32_dgrad_on_tiles(const F32Conv& c, int sm_count) {
  const long long tiles = (long long)c.N * ((c.H + 7) / 8) * ((c.W + 7) / 8);
  if (c.R == 3) return !(c.stride == 1 && c.cin * c.cout <= 16 && tiles >= 1024);
  if (c.stride != 1 || (c.cin < 16 && c.cin * c.cout > 128)) return true;
  const double fill = (double)c.N * c.H * c.W * (c.cin / 4) / (2048.0 * sm_count);
  const double l1 = c.cin * c.cout <= 16384 ? 1.0 : 1.9;
  const double direct = 3.6 + 0.148 * c.cout + std::max(0.0, fill - 0.36) * (2.8 + 0.174 * l1 * c.cout);
  const long long blocks = tiles * ((c.cin + 15) / 16);
  const double waves = blocks <= 2LL * sm_count ? 0.6 : (double)((blocks + 4LL * sm_count - 1) / (4LL * sm_count));
  const double tiled = 1.9 + waves * (1.28 + 0.103 * c.cout);
  return direct >= 0.95 * tiled;
}

}  // namespace lp
