// fp32 convolutions on the CUDA cores: 1x1 and 3x3 filters, stride 1 or 2, channel counts that are multiples of 4.
// (The tensor cores have no mode that keeps all 24 bits of an fp32 operand, so the fp32 path multiplies with FFMA.)
//
// Forward and input gradient are one kernel, an implicit GEMM over a list of taps: a block produces an 8x8 pixel
// tile x 16 output channels; the activation patch of the tile (with the taps' reach) and the taps' weights of 16
// input channels are staged in shared memory by cp.async, two chunks deep.  A lane owns one tile row (8 pixels) x 4
// output channels, so that 12 16-byte shared-memory loads feed 128 FFMA; the block's warps split the (tap, four
// input channels) items of a chunk among themselves and add up their tiles through shared memory at the end.
// Splitting K over warps instead of pixels keeps an SM's schedulers busy where a layer has few tiles: the 64-channel
// 8x8 layers of a batch of 32 are 128 blocks, one per SM.  A stride-2 input gradient runs its four parity classes
// (each a stride-1 convolution over a subset of the taps) as blockIdx.z.
//
// The direct kernels these replace read x and w with scalar loads straight from L2 (one output pixel x 4 channels a
// thread, neighbouring threads C_in apart in w).  Measured on the ResNet-56 shapes at a batch of 32 (16 / 32 / 64
// channels, 75 M multiply-adds a launch): forward 93 -> 14 us, input gradient 57 -> 13, weight gradient 125 -> 9.5;
// the step 12.2 -> 1.40 ms.  They are latency-bound now (2 to 4 us of FFMA in a launch): the first chunk of weights is
// fetched before the preceding kernel ends and the set-up loops are rolled (21 -> 15 KB of code), 1.40 -> 1.35 ms.
#pragma once
#include "common.cuh"

namespace lp {

struct ConvF32Params {
  const float* act;            // [N][aH][aW][aC]
  const float* w;              // fp32 masters [C_out][taps][C_in] of the convolution
  const float* addend;         // nullable; geometry of out, may alias it
  float* out;
  double* stats;               // nullable; [2*Cout] per-channel sum and sum of squares of out (forward only)
  int aH, aW, aC;
  int OHl, OWl;                // logical output grid (of a class)
  int in_step;                 // input coordinate = logical * in_step + tap offset
  int out_H, out_W, Cout;      // physical output tensor
  int os;                      // physical pixel = logical * os + class offset
  int wtaps;                   // taps of the weight tensor
  int tiles_w, tiles_h;
  int ncls;
  int cls_oh[4], cls_ow[4];
  int cls_ntaps[4], cls_tap0[4];
  int cls_dh0[4], cls_dw0[4];  // smallest tap offsets of the class: the patch starts there
  int tap_dh[9], tap_dw[9], tap_w[9];
  int PH, PW;                  // patch size of the largest class
  int row_pitch;               // floats between patch rows: = 4 mod 32, so that the 8 tile rows of a load sit in different banks
  int w_pitch;                 // floats between weight rows (16 x taps + 4)
  int stage_floats, w_off;     // one stage: patch, then weights
};

__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool valid) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// KS: warps of the block, each working on its share of a chunk's (tap, channel quad) items
template <int KS, bool kDgrad>
__global__ void __launch_bounds__(32 * KS)
conv_f32_tile_kernel(const __grid_constant__ ConvF32Params p) {
  extern __shared__ __align__(16) float smf[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cls = blockIdx.z;
  const int co0 = blockIdx.y * 16;
  int t = blockIdx.x;
  const int tw = t % p.tiles_w;
  t /= p.tiles_w;
  const int th = t % p.tiles_h;
  const int n = t / p.tiles_h;
  const int w0 = tw * 8, h0 = th * 8;
  const int ntaps = p.cls_ntaps[cls], tap0 = p.cls_tap0[cls];
  const int dh0 = p.cls_dh0[cls], dw0 = p.cls_dw0[cls];
  const int nchunks = ntaps ? (p.aC + 15) >> 4 : 0;

  // (the loops of the block's set-up are kept rolled: they run a few times, and unrolled code would first have to be fetched)
  auto load_patch = [&](int c) {
    float* a = smf + (c & 1) * p.stage_floats;
    const int c0 = c * 16;
    const int ih0 = h0 * p.in_step + dh0, iw0 = w0 * p.in_step + dw0;
#pragma unroll 1
    for (int r = warp; r < p.PH; r += KS) {
      const int ih = ih0 + r;
      const bool row_ok = ih >= 0 && ih < p.aH;
#pragma unroll 1
      for (int l = lane; l < p.PW * 4; l += 32) {
        const int iw = iw0 + (l >> 2), ci = c0 + 4 * (l & 3);
        const bool ok = row_ok && iw >= 0 && iw < p.aW && ci < p.aC;
        const float* src = ok ? p.act + (((long long)n * p.aH + ih) * p.aW + iw) * p.aC + ci : p.act;
        cp_async16(a + r * p.row_pitch + 4 * l, src, ok);
      }
    }
  };
  // weights in their own order: rows of 16 input channels per (output channel, tap), or (input gradient) rows of
  // 16 output channels per (input channel, tap)
  auto load_weights = [&](int c) {
    float* wb = smf + (c & 1) * p.stage_floats + p.w_off;
    const int c0 = c * 16;
#pragma unroll 1
    for (int r = warp; r < 16; r += KS) {
#pragma unroll 1
      for (int l = lane; l < ntaps * 4; l += 32) {
        const int tap = p.tap_w[tap0 + (l >> 2)], v = 4 * (l & 3);
        bool ok;
        const float* src = p.w;
        if (kDgrad) {
          ok = c0 + r < p.aC && co0 + v < p.Cout;
          if (ok) src += ((long long)(c0 + r) * p.wtaps + tap) * p.Cout + co0 + v;
        } else {
          ok = co0 + r < p.Cout && c0 + v < p.aC;
          if (ok) src += ((long long)(co0 + r) * p.wtaps + tap) * p.aC + c0 + v;
        }
        cp_async16(wb + r * p.w_pitch + 4 * l, src, ok);
      }
    }
  };
  // the first weights were written at least one kernel before the preceding one: on their way before its end
  if (nchunks) load_weights(0);
  pdl_wait();
  pdl_launch_dependents();

  const int row = lane >> 2, cg = lane & 3;
  float acc[8][4];
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[j][k] = 0.f;

  if (nchunks) load_patch(0);
  cp_async_commit();
#pragma unroll 1
  for (int c = 0; c < nchunks; ++c) {
    if (c + 1 < nchunks) {
      load_patch(c + 1);
      load_weights(c + 1);
      cp_async_commit();
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const float* a = smf + (c & 1) * p.stage_floats + row * p.in_step * p.row_pitch;
    const float* wb = smf + (c & 1) * p.stage_floats + p.w_off;
    const int nq = min(4, (p.aC - c * 16) >> 2);   // quads of real input channels
    const int items = ntaps * nq;
#pragma unroll 1
    for (int it = warp; it < items; it += KS) {
      const int tp = nq == 4 ? it >> 2 : it / nq;
      const int q = it - tp * nq;
      const float* ap = a + (p.tap_dh[tap0 + tp] - dh0) * p.row_pitch + (p.tap_dw[tap0 + tp] - dw0) * 16 + 4 * q;
      float4 wv[4];
      if (kDgrad) {   // wv[k]: output channels 4*cg .. +3 of input channel 4*q + k
        const float* wp = wb + 4 * q * p.w_pitch + tp * 16 + 4 * cg;
#pragma unroll
        for (int k = 0; k < 4; ++k) wv[k] = *reinterpret_cast<const float4*>(wp + k * p.w_pitch);
      } else {        // wv[k]: input channels 4*q .. +3 of output channel cg + 4*k
        const float* wp = wb + cg * p.w_pitch + tp * 16 + 4 * q;
#pragma unroll
        for (int k = 0; k < 4; ++k) wv[k] = *reinterpret_cast<const float4*>(wp + 4 * k * p.w_pitch);
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float4 av = *reinterpret_cast<const float4*>(ap + j * p.in_step * 16);
        if (kDgrad) {
          acc[j][0] = fmaf(av.x, wv[0].x, acc[j][0]); acc[j][1] = fmaf(av.x, wv[0].y, acc[j][1]);
          acc[j][2] = fmaf(av.x, wv[0].z, acc[j][2]); acc[j][3] = fmaf(av.x, wv[0].w, acc[j][3]);
          acc[j][0] = fmaf(av.y, wv[1].x, acc[j][0]); acc[j][1] = fmaf(av.y, wv[1].y, acc[j][1]);
          acc[j][2] = fmaf(av.y, wv[1].z, acc[j][2]); acc[j][3] = fmaf(av.y, wv[1].w, acc[j][3]);
          acc[j][0] = fmaf(av.z, wv[2].x, acc[j][0]); acc[j][1] = fmaf(av.z, wv[2].y, acc[j][1]);
          acc[j][2] = fmaf(av.z, wv[2].z, acc[j][2]); acc[j][3] = fmaf(av.z, wv[2].w, acc[j][3]);
          acc[j][0] = fmaf(av.w, wv[3].x, acc[j][0]); acc[j][1] = fmaf(av.w, wv[3].y, acc[j][1]);
          acc[j][2] = fmaf(av.w, wv[3].z, acc[j][2]); acc[j][3] = fmaf(av.w, wv[3].w, acc[j][3]);
        } else {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            acc[j][k] = fmaf(av.x, wv[k].x, acc[j][k]);
            acc[j][k] = fmaf(av.y, wv[k].y, acc[j][k]);
            acc[j][k] = fmaf(av.z, wv[k].z, acc[j][k]);
            acc[j][k] = fmaf(av.w, wv[k].w, acc[j][k]);
          }
        }
      }
    }
    __syncthreads();
  }

  // The warps' tiles are added up: red[warp][pixel][16 channels], 16 bytes per pixel and lane group for the input
  // gradient, single words for the forward kernel (its lanes own every fourth channel).  The pixel pitch of 20
  // floats spreads the 8 rows of a store over the banks.
  constexpr int kPix = 20;
  float* red = smf + warp * 64 * kPix;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    float* rp = red + (row * 8 + j) * kPix;
    if (kDgrad) {
      *reinterpret_cast<float4*>(rp + 4 * cg) = make_float4(acc[j][0], acc[j][1], acc[j][2], acc[j][3]);
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) rp[cg + 4 * k] = acc[j][k];
    }
  }
  __syncthreads();
  // thread -> (pixel, four channels): 256 of them
  float s[4] = {0.f, 0.f, 0.f, 0.f}, q2[4] = {0.f, 0.f, 0.f, 0.f};
  const int v = threadIdx.x & 3;
  const int c = co0 + 4 * v;
#pragma unroll 1
  for (int px = threadIdx.x >> 2; px < 64; px += 8 * KS) {
    const int oh = h0 + (px >> 3), ow = w0 + (px & 7);
    const int ph = oh * p.os + p.cls_oh[cls], pw = ow * p.os + p.cls_ow[cls];
    if (oh >= p.OHl || ow >= p.OWl || ph >= p.out_H || pw >= p.out_W || c >= p.Cout) continue;
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < KS; ++k) {
      const float4 u = *reinterpret_cast<const float4*>(smf + (k * 64 + px) * kPix + 4 * v);
      o.x += u.x; o.y += u.y; o.z += u.z; o.w += u.w;
    }
    const long long at = (((long long)n * p.out_H + ph) * p.out_W + pw) * p.Cout + c;
    if (p.addend) {
      const float4 u = *reinterpret_cast<const float4*>(p.addend + at);
      o.x += u.x; o.y += u.y; o.z += u.z; o.w += u.w;
    }
    *reinterpret_cast<float4*>(p.out + at) = o;
    if (!kDgrad) {
      s[0] += o.x; s[1] += o.y; s[2] += o.z; s[3] += o.w;
      q2[0] = fmaf(o.x, o.x, q2[0]); q2[1] = fmaf(o.y, o.y, q2[1]); q2[2] = fmaf(o.z, o.z, q2[2]); q2[3] = fmaf(o.w, o.w, q2[3]);
    }
  }
  if (!kDgrad && p.stats) {
    // batch-norm statistics of the tile: lanes of the same channel quad, then the warps, then one double atomic each
#pragma unroll
    for (int j = 0; j < 4; ++j)
      for (int o = 4; o < 32; o <<= 1) {
        s[j] += __shfl_xor_sync(0xffffffffu, s[j], o);
        q2[j] += __shfl_xor_sync(0xffffffffu, q2[j], o);
      }
    __syncthreads();
    if (lane < 4) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        smf[warp * 32 + 4 * lane + j] = s[j];
        smf[warp * 32 + 16 + 4 * lane + j] = q2[j];
      }
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      float a = 0.f;
      for (int k = 0; k < KS; ++k) a += smf[k * 32 + threadIdx.x];
      const int ch = co0 + (threadIdx.x & 15);
      if (ch < p.Cout) atomicAdd(p.stats + (threadIdx.x >> 4) * p.Cout + ch, (double)a);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Weight gradient.  A block owns 16 input x 16 output channels, all taps, and a range of pixel tiles (8x8 output
// pixels; x patch and dy tile staged by cp.async two tiles deep).  A thread owns one filter row r, four input and
// four output channels, and every fourth row of a tile: along a row it slides a window of R x positions, so that two
// (stride 1) or three 16-byte loads per pixel feed 16 R FFMA.  The four row lanes are added in shared memory, the
// blocks with vector reductions into dw (zeroed by the caller).
// ---------------------------------------------------------------------------------------------
struct WgradF32Params {
  const float* x;              // [N][H][W][Cin]
  const float* dy;             // [N][OH][OW][Cout]
  float* dw;                   // [Cout][R*R][Cin]
  int H, W, Cin, OH, OW, Cout, pad;
  int tiles_w, tiles_h, tiles; // 8x8 pixel tiles of all images
  int co_tiles;
  int vec_red;                 // dw is 16-byte aligned
};

template <int R, int S>
struct WgradF32Cfg {
  static constexpr int kUnits = R * 16;                    // (filter row, ci quad, co quad)
  static constexpr int kLanes = R == 3 ? 4 : 8;            // row lanes
  static constexpr int kThreads = kUnits * kLanes;         // 192 or 128
  static constexpr int PW = 7 * S + R, PH = 7 * S + R;
  static constexpr int kRow = PW * 16 + ((PW & 1) ? 0 : 16);   // = 16 mod 32: two filter rows of a warp in different banks
  static constexpr int kStage = PH * kRow + 64 * 16;
  static constexpr int kRed = kLanes * kUnits * (16 * R + 4);
  static constexpr size_t kSmem = sizeof(float) * (size_t)(2 * kStage > kRed ? 2 * kStage : kRed);
};

__device__ __forceinline__ void red_add_v4(float* p, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1,%2,%3,%4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

template <int R, int S>
__global__ void __launch_bounds__(WgradF32Cfg<R, S>::kThreads)
wgrad_f32_tile_kernel(const __grid_constant__ WgradF32Params p) {
  using C = WgradF32Cfg<R, S>;
  extern __shared__ __align__(16) float smf[];
  pdl_wait();
  pdl_launch_dependents();
  const int tid = threadIdx.x;
  const int ci0 = (blockIdx.y / p.co_tiles) * 16, co0 = (blockIdx.y % p.co_tiles) * 16;
  const int t_begin = (int)(((long long)p.tiles * blockIdx.x) / gridDim.x);
  const int t_end = (int)(((long long)p.tiles * (blockIdx.x + 1)) / gridDim.x);

  auto load_tile = [&](int tile, int buf) {
    float* xb = smf + buf * C::kStage;
    float* db = xb + C::PH * C::kRow;
    int t = tile;
    const int tw = t % p.tiles_w;
    t /= p.tiles_w;
    const int th = t % p.tiles_h;
    const int n = t / p.tiles_h;
    const int ih0 = th * 8 * S - p.pad, iw0 = tw * 8 * S - p.pad;
    for (int i = tid; i < C::PH * C::PW * 4; i += C::kThreads) {
      const int r = i / (C::PW * 4), l = i - r * (C::PW * 4);
      const int ih = ih0 + r, iw = iw0 + (l >> 2), ci = ci0 + 4 * (l & 3);
      const bool ok = ih >= 0 && ih < p.H && iw >= 0 && iw < p.W && ci < p.Cin;
      cp_async16(xb + r * C::kRow + 4 * l, ok ? p.x + (((long long)n * p.H + ih) * p.W + iw) * p.Cin + ci : p.x, ok);
    }
    for (int i = tid; i < 256; i += C::kThreads) {
      const int oh = th * 8 + (i >> 5), ow = tw * 8 + ((i >> 2) & 7), co = co0 + 4 * (i & 3);
      const bool ok = oh < p.OH && ow < p.OW && co < p.Cout;
      cp_async16(db + 4 * i, ok ? p.dy + (((long long)n * p.OH + oh) * p.OW + ow) * p.Cout + co : p.dy, ok);
    }
    cp_async_commit();
  };

  const int unit = tid % C::kUnits, rl = tid / C::kUnits;
  const int qi = unit & 3, qo = (unit >> 2) & 3, fr = unit >> 4;
  float acc[R][4][4];   // [filter column][output channel][input channel]
#pragma unroll
  for (int s = 0; s < R; ++s)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int k = 0; k < 4; ++k) acc[s][j][k] = 0.f;

  if (t_begin < t_end) load_tile(t_begin, 0);
  for (int t = t_begin; t < t_end; ++t) {
    const int buf = (t - t_begin) & 1;
    if (t + 1 < t_end) {
      load_tile(t + 1, buf ^ 1);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const float* xb = smf + buf * C::kStage + 4 * qi;
    const float* db = smf + buf * C::kStage + C::PH * C::kRow + 4 * qo;
    for (int row = rl; row < 8; row += C::kLanes) {
      const float* xr = xb + (row * S + fr) * C::kRow;
      const float* dr = db + row * 8 * 16;
      float4 win[R];
#pragma unroll
      for (int s = 0; s < R; ++s) win[s] = *reinterpret_cast<const float4*>(xr + s * 16);
#pragma unroll
      for (int px = 0; px < 8; ++px) {
        const float4 d = *reinterpret_cast<const float4*>(dr + px * 16);
        const float dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
        for (int s = 0; s < R; ++s) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            acc[s][j][0] = fmaf(dv[j], win[s].x, acc[s][j][0]);
            acc[s][j][1] = fmaf(dv[j], win[s].y, acc[s][j][1]);
            acc[s][j][2] = fmaf(dv[j], win[s].z, acc[s][j][2]);
            acc[s][j][3] = fmaf(dv[j], win[s].w, acc[s][j][3]);
          }
        }
        if (px < 7) {   // slide by S positions
#pragma unroll
          for (int s = 0; s < R; ++s) {
            if (s + S < R) win[s] = win[(s + S) % R];
            else win[s] = *reinterpret_cast<const float4*>(xr + ((px + 1) * S + s) * 16);
          }
        }
      }
    }
    __syncthreads();
  }

  constexpr int kPitch = 16 * R + 4;
  float* mine = smf + (rl * C::kUnits + unit) * kPitch;
#pragma unroll
  for (int s = 0; s < R; ++s)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      *reinterpret_cast<float4*>(mine + (s * 4 + j) * 4) = make_float4(acc[s][j][0], acc[s][j][1], acc[s][j][2], acc[s][j][3]);
  __syncthreads();
  // output (filter row, filter column, output channel, ci quad)
  for (int o = tid; o < C::kUnits * R * 4; o += C::kThreads) {
    const int u = o / (R * 4), sj = o - u * (R * 4);
    const int s = sj >> 2, j = sj & 3;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int l = 0; l < C::kLanes; ++l) {
      const float4 w = *reinterpret_cast<const float4*>(smf + (l * C::kUnits + u) * kPitch + sj * 4);
      v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
    }
    const int ci = ci0 + 4 * (u & 3), co = co0 + 4 * ((u >> 2) & 3) + j, r = u >> 4;
    if (ci >= p.Cin || co >= p.Cout) continue;
    float* d = p.dw + ((long long)co * (R * R) + r * R + s) * p.Cin + ci;
    if (p.vec_red) {
      red_add_v4(d, v.x, v.y, v.z, v.w);
    } else {
      atomicAdd(d, v.x); atomicAdd(d + 1, v.y); atomicAdd(d + 2, v.z); atomicAdd(d + 3, v.w);
    }
  }
}

}  // namespace lp
