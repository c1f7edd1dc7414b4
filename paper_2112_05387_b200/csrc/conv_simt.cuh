// Direct (CUDA-core) convolution kernels: any filter size, stride, padding and channel count.
// They carry the fp32 workload (tensor cores have no true-fp32 mode) and the few bf16 shapes
// the tensor-core path does not take (3-channel stems).  fp32 accumulation throughout;
// weights are the fp32 masters w[co][r][s][ci], rounded to the activation type as they are read
// so that both convolution paths of a bf16 network contract the same operands.
// fp32 results are added up in partial sums (per filter position, four channels at a time or in four chains), as the tiled
// kernels do: one chain over all terms was up to twice as far from the exact sum (input gradient of 128 -> 128, 1x1: 2.0e-7
// against 1.1e-7).
#pragma once
#include "common.cuh"

namespace lp {

struct ConvGeom {
  int N, H, W, Cin;      // input
  int OH, OW, Cout;      // output
  int R, S, stride, pad;
};

// y[n,oh,ow,co..co+3] = sum_{r,s,ci} w[co][r][s][ci] * x[n, oh*st+r-p, ow*st+s-p, ci]  (+ addend)
template <typename T>
__global__ void conv_fwd_simt_kernel(const T* __restrict__ x, const float* __restrict__ w, const T* __restrict__ addend,
                                     T* __restrict__ y, ConvGeom g) {
  constexpr bool kPartial = sizeof(T) == 4;
  const int CG = g.Cout >> 2;
  const long long total = (long long)g.N * g.OH * g.OW * CG;
  const long long tap_stride = (long long)g.R * g.S * g.Cin;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int co = (int)(i % CG) * 4;
    long long p = i / CG;
    const int ow = (int)(p % g.OW);
    long long q = p / g.OW;
    const int oh = (int)(q % g.OH);
    const int n = (int)(q / g.OH);
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int r = 0; r < g.R; ++r) {
      const int ih = oh * g.stride + r - g.pad;
      if (ih < 0 || ih >= g.H) continue;
      for (int s = 0; s < g.S; ++s) {
        const int iw = ow * g.stride + s - g.pad;
        if (iw < 0 || iw >= g.W) continue;
        const T* xp = x + (((long long)n * g.H + ih) * g.W + iw) * g.Cin;
        const float* wp = w + ((long long)co * g.R * g.S + (r * g.S + s)) * g.Cin;
        float part[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) part[j] = kPartial ? 0.f : acc[j];
        for (int ci = 0; ci < g.Cin; ++ci) {
          const float xv = to_f(xp[ci]);
#pragma unroll
          for (int j = 0; j < 4; ++j) part[j] += xv * round_storage<T>(__ldg(wp + j * tap_stride + ci));
          if (kPartial && (ci & 3) == 3) {
#pragma unroll
            for (int j = 0; j < 4; ++j) { acc[j] += part[j]; part[j] = 0.f; }
          }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[j] = kPartial ? acc[j] + part[j] : part[j];
      }
    }
    const long long o = p * g.Cout + co;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float v = acc[j];
      if (addend) v += to_f(addend[o + j]);
      from_f(y[o + j], v);
    }
  }
}

// dx[n,ih,iw,ci..ci+3] = sum_{r,s,co : (ih+p-r) % st == 0 ...} dy[n,(ih+p-r)/st,(iw+p-s)/st,co] * w[co][r][s][ci]
template <typename T>
__global__ void conv_dgrad_simt_kernel(const T* __restrict__ dy, const float* __restrict__ w,
                                       const T* __restrict__ addend, T* __restrict__ dx, ConvGeom g) {
  const int CG = g.Cin >> 2;
  const long long total = (long long)g.N * g.H * g.W * CG;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int ci = (int)(i % CG) * 4;
    long long p = i / CG;
    const int iw = (int)(p % g.W);
    long long q = p / g.W;
    const int ih = (int)(q % g.H);
    const int n = (int)(q / g.H);
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int r = 0; r < g.R; ++r) {
      const int th = ih + g.pad - r;
      if (th < 0 || th % g.stride) continue;
      const int oh = th / g.stride;
      if (oh >= g.OH) continue;
      for (int s = 0; s < g.S; ++s) {
        const int tw = iw + g.pad - s;
        if (tw < 0 || tw % g.stride) continue;
        const int ow = tw / g.stride;
        if (ow >= g.OW) continue;
        const T* dp = dy + (((long long)n * g.OH + oh) * g.OW + ow) * g.Cout;
        const float* wp = w + (long long)(r * g.S + s) * g.Cin + ci;
        int co = 0;
        if constexpr (sizeof(T) == 4) {
          float part[4][4] = {};
          for (; co + 4 <= g.Cout; co += 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const float d = to_f(dp[co + u]);
              const float4 wv = __ldg(reinterpret_cast<const float4*>(wp + (long long)(co + u) * g.R * g.S * g.Cin));
              part[u][0] += d * wv.x; part[u][1] += d * wv.y; part[u][2] += d * wv.z; part[u][3] += d * wv.w;
            }
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[j] += (part[0][j] + part[1][j]) + (part[2][j] + part[3][j]);
        }
        for (; co < g.Cout; ++co) {
          const float d = to_f(dp[co]);
          const float4 wv = __ldg(reinterpret_cast<const float4*>(wp + (long long)co * g.R * g.S * g.Cin));
          acc[0] += d * round_storage<T>(wv.x);
          acc[1] += d * round_storage<T>(wv.y);
          acc[2] += d * round_storage<T>(wv.z);
          acc[3] += d * round_storage<T>(wv.w);
        }
      }
    }
    const long long o = p * g.Cin + ci;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float v = acc[j];
      if (addend) v += to_f(addend[o + j]);
      from_f(dx[o + j], v);
    }
  }
}

// dw[co][r][s][ci] += sum over the block's pixel chunk of dy[n,oh,ow,co] * x[n,oh*st+r-p,ow*st+s-p,ci]
// grid.x: chunks of output elements, grid.y: pixel chunks; dw must be zero before the launch.
template <typename T>
__global__ void conv_wgrad_simt_kernel(const T* __restrict__ x, const T* __restrict__ dy, float* __restrict__ dw,
                                       ConvGeom g, int pixels_per_chunk) {
  const int n_out = g.Cout * g.R * g.S * g.Cin;
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= n_out) return;
  const int ci = o % g.Cin;
  int t = o / g.Cin;
  const int s = t % g.S;
  t /= g.S;
  const int r = t % g.R;
  const int co = t / g.R;
  const long long npix = (long long)g.N * g.OH * g.OW;
  long long p0 = (long long)blockIdx.y * pixels_per_chunk;
  long long p1 = p0 + pixels_per_chunk;
  if (p1 > npix) p1 = npix;
  int ow = (int)(p0 % g.OW);
  long long q = p0 / g.OW;
  int oh = (int)(q % g.OH);
  int n = (int)(q / g.OH);
  float acc = 0.f;
  for (long long p = p0; p < p1; ++p) {
    const int ih = oh * g.stride + r - g.pad, iw = ow * g.stride + s - g.pad;
    if (ih >= 0 && ih < g.H && iw >= 0 && iw < g.W)
      acc += to_f(dy[p * g.Cout + co]) * to_f(x[(((long long)n * g.H + ih) * g.W + iw) * g.Cin + ci]);
    if (++ow == g.OW) {
      ow = 0;
      if (++oh == g.OH) {
        oh = 0;
        ++n;
      }
    }
  }
  atomicAdd(&dw[o], acc);
}

// ---------------------------------------------------------------------------------------------
// Few input channels (the 3-channel stems and the first AuxNet convolution): K = R*S*Cin is tiny,
// so the whole filter bank fits in shared memory.  A thread produces CPT output channels of one
// pixel: one activation load and CPT/4 broadcast reads of the filter bank feed CPT multiply-adds.
// Same operands as the generic kernels (weights rounded to the activation type, fp32 accumulation).
// ---------------------------------------------------------------------------------------------
// kPartial: a filter position at a time is added up by itself (fp32 layers that the tiled kernel would take too, at a CPT of 32 at
// most: 127 registers, two blocks an SM).
template <typename T, int CPT, bool kPartial = false>
__global__ void __launch_bounds__(256)
conv_fwd_fewch_kernel(const T* __restrict__ x, const float* __restrict__ w, T* __restrict__ y, ConvGeom g) {
  constexpr int V = VecT<T>::N;
  extern __shared__ float ws[];            // [K][Cout], K = R*S*Cin
  const int K = g.R * g.S * g.Cin;
  for (int i = threadIdx.x; i < K * g.Cout; i += blockDim.x) {
    const int k = i / g.Cout, co = i % g.Cout;
    ws[i] = round_storage<T>(w[(long long)co * K + k]);
  }
  __syncthreads();
  const int CG = g.Cout / CPT;
  const long long total = (long long)g.N * g.OH * g.OW * CG;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int cg = (int)(i % CG);
    const long long p = i / CG;
    const int ow = (int)(p % g.OW);
    const long long q = p / g.OW;
    const int oh = (int)(q % g.OH);
    const int n = (int)(q / g.OH);
    float sum[kPartial ? CPT : 1], acc[CPT];
#pragma unroll
    for (int j = 0; j < CPT; ++j) acc[j] = 0.f;
    for (int r = 0; r < g.R; ++r) {
      const int ih = oh * g.stride + r - g.pad;
      if (ih < 0 || ih >= g.H) continue;
      for (int s = 0; s < g.S; ++s) {
        const int iw = ow * g.stride + s - g.pad;
        if (iw < 0 || iw >= g.W) continue;
        if constexpr (kPartial) {
#pragma unroll
          for (int j = 0; j < CPT; ++j) { sum[j] = acc[j]; acc[j] = 0.f; }
        }
        const T* xp = x + (((long long)n * g.H + ih) * g.W + iw) * g.Cin;
        const float* wr = ws + (r * g.S + s) * g.Cin * g.Cout + cg * CPT;
        for (int ci = 0; ci < g.Cin; ++ci) {
          const float xv = to_f(xp[ci]);
#pragma unroll
          for (int j4 = 0; j4 < CPT; j4 += 4) {
            const float4 wv = *reinterpret_cast<const float4*>(wr + ci * g.Cout + j4);
            acc[j4] += xv * wv.x; acc[j4 + 1] += xv * wv.y; acc[j4 + 2] += xv * wv.z; acc[j4 + 3] += xv * wv.w;
          }
        }
        if constexpr (kPartial) {
#pragma unroll
          for (int j = 0; j < CPT; ++j) acc[j] += sum[j];
        }
      }
    }
#pragma unroll
    for (int j = 0; j < CPT; j += V) stv(y + p * g.Cout + cg * CPT + j, *reinterpret_cast<float(*)[V]>(&acc[j]));
  }
}

// ---------------------------------------------------------------------------------------------
// 3x3 convolutions (pad 1, stride 1 or 2) of bf16 images of three channels: the stems and first AuxNet convolutions.  A block
// works on tiles of 32 columns x TH rows of the output; the input patch is staged in shared memory as fp32, one plane per
// channel (and per parity of the column, stride 2), so that the lanes of a warp, the tile's columns, read 32 neighbouring words.
// ---------------------------------------------------------------------------------------------
struct ImageTiles {
  int N, H, W, OH, OW, Cout, TH, tiles_w, tiles_h, tiles;
};
constexpr int kImgCols = 34;      // words of a plane's row
__host__ __device__ constexpr int image_patch_rows(int TH, int stride) { return (TH - 1) * stride + 3; }
__host__ __device__ constexpr int image_patch_floats(int TH, int stride) { return image_patch_rows(TH, stride) * 3 * stride * kImgCols; }
template <int kStride>
__device__ __forceinline__ int image_at(int row, int c, int col) {
  return ((row * 3 + c) * kStride + (kStride == 2 ? col & 1 : 0)) * kImgCols + (kStride == 2 ? col >> 1 : col);
}
template <int kStride>
__device__ __forceinline__ void image_stage(const ImageTiles& g, const bf16* __restrict__ x, float* patch, int n, int oh0, int ow0) {
  constexpr int COLS = 31 * kStride + 3, E = (COLS * 3 + 31) / 32;
  const int rows = image_patch_rows(g.TH, kStride), warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ih0 = oh0 * kStride - 1, iw0 = ow0 * kStride - 1;
  // a lane keeps its elements of a row (every 32nd: the same channels and columns in every row)
  int to[E];
  uint32_t in = 0;
#pragma unroll
  for (int u = 0; u < E; ++u) {
    const int e = lane + 32 * u, col = e / 3, c = e - col * 3;
    to[u] = e < COLS * 3 ? image_at<kStride>(0, c, col) : -1;
    if (e < COLS * 3 && iw0 + col >= 0 && iw0 + col < g.W) in |= 1u << u;
  }
#pragma unroll 1
  for (int r = warp; r < rows; r += blockDim.x >> 5) {
    const int ih = ih0 + r;
    const bf16* xp = x + ((long long)(n * g.H + ih) * g.W + iw0) * 3 + lane;
    const uint32_t ok = ih >= 0 && ih < g.H ? in : 0u;
    float v[E];
#pragma unroll
    for (int u = 0; u < E; ++u) v[u] = (ok >> u) & 1 ? to_f(xp[32 * u]) : 0.f;
    float* row = patch + r * 3 * kStride * kImgCols;
#pragma unroll
    for (int u = 0; u < E; ++u)
      if (to[u] >= 0) row[to[u]] = v[u];
  }
}
__device__ __forceinline__ uint64_t pair_of(float lo, float hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ void pair_fma(uint64_t& acc, uint64_t a, uint64_t b) {   // two multiply-adds in one instruction
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

// Forward, with the statistics of the batch norm that follows.  A thread computes four rows of its column x 8 output channels:
// a weight (broadcast) serves four pixels, an input value three filter rows.  conv_fwd_fewch_kernel, one pixel a thread, waits
// for its reads of the filter bank, and the statistics were another launch (with them, timed alone, that kernel and this one:
// 20.9 and 12.4 us on 128 images of 32x32, 16 channels, 50.4 and 22.2 with 40; 86 and 72 on 32 of 224x224, 64 channels, stride
// 2; 55 and 45 on 64 with 16).  Statistics are summed over the values as stored, in a thread, over the warp and the block, then
// in double.
template <int kStride>
__global__ void __launch_bounds__(256)
image_conv_kernel(const bf16* __restrict__ x, const float* __restrict__ w, bf16* __restrict__ y, double* __restrict__ stats,
                  const ImageTiles g) {
  constexpr int P = 4, CPT = 8, K = 27, ROWS = (P - 1) * kStride + 3;
  extern __shared__ float sm[];                 // weights [K][Cout], sums [2 * Cout], input patch
  float *ws = sm, *sums = sm + K * g.Cout, *patch = sums + 2 * g.Cout;
  for (int i = threadIdx.x; i < K * g.Cout; i += 256) {
    const int co = i / K, k = i - co * K;
    ws[k * g.Cout + co] = round_storage<bf16>(w[i]);
  }
  for (int i = threadIdx.x; i < 2 * g.Cout; i += 256) sums[i] = 0.f;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int CG = g.Cout / CPT, items = CG * (g.TH / P);
  float s[CPT], q[CPT];
  int stat_co = -1;
#pragma unroll
  for (int j = 0; j < CPT; ++j) s[j] = q[j] = 0.f;
  const auto flush = [&]() {
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
      s[j] = warp_sum(s[j]);
      q[j] = warp_sum(q[j]);
      if (lane == 0) {
        atomicAdd(&sums[stat_co + j], s[j]);
        atomicAdd(&sums[g.Cout + stat_co + j], q[j]);
      }
      s[j] = q[j] = 0.f;
    }
  };
#pragma unroll 1
  for (int t = blockIdx.x; t < g.tiles; t += gridDim.x) {
    const int tw = t % g.tiles_w, t2 = t / g.tiles_w, th = t2 % g.tiles_h, n = t2 / g.tiles_h;
    const int oh0 = th * g.TH, ow0 = tw * 32;
    __syncthreads();                            // the previous tile has been read
    image_stage<kStride>(g, x, patch, n, oh0, ow0);
    __syncthreads();
#pragma unroll 1
    for (int item = warp; item < items; item += 8) {
      const int co0 = item % CG * CPT, h0 = item / CG * P;
      if (oh0 + h0 >= g.OH) break;
      uint64_t acc[P][CPT / 2];
#pragma unroll
      for (int a = 0; a < P; ++a)
#pragma unroll
        for (int j = 0; j < CPT / 2; ++j) acc[a][j] = 0;
#pragma unroll 1
      for (int k = 0; k < 9; ++k) {             // (filter column, input channel)
        const int fc = k / 3, c = k - fc * 3;
        float v[ROWS];
#pragma unroll
        for (int i = 0; i < ROWS; ++i) v[i] = patch[image_at<kStride>(h0 * kStride + i, c, lane * kStride + fc)];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          const float* wr = ws + (r * 9 + k) * g.Cout + co0;
          const float4 wa = *reinterpret_cast<const float4*>(wr), wb = *reinterpret_cast<const float4*>(wr + 4);
          const uint64_t w2[4] = {pair_of(wa.x, wa.y), pair_of(wa.z, wa.w), pair_of(wb.x, wb.y), pair_of(wb.z, wb.w)};
#pragma unroll
          for (int a = 0; a < P; ++a) {
            const uint64_t v2 = pair_of(v[a * kStride + r], v[a * kStride + r]);
#pragma unroll
            for (int j = 0; j < CPT / 2; ++j) pair_fma(acc[a][j], v2, w2[j]);
          }
        }
      }
      if (stats && co0 != stat_co) {            // (a warp's channels rarely change)
        if (stat_co >= 0) flush();
        stat_co = co0;
      }
      const int ow = ow0 + lane;
      if (ow < g.OW) {
        bf16* yp = y + ((long long)(n * g.OH + oh0 + h0) * g.OW + ow) * g.Cout + co0;
#pragma unroll
        for (int a = 0; a < P; ++a) {
          if (oh0 + h0 + a >= g.OH) break;
          uint32_t o[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            float lo, hi;
            asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(acc[a][j]));
            o[j] = pack_bf16x2(lo, hi);
            lo = __uint_as_float(o[j] << 16); hi = __uint_as_float(o[j] & 0xFFFF0000u);
            s[2 * j] += lo; s[2 * j + 1] += hi;
            q[2 * j] = fmaf(lo, lo, q[2 * j]); q[2 * j + 1] = fmaf(hi, hi, q[2 * j + 1]);
          }
          *reinterpret_cast<uint4*>(yp + (long long)a * g.OW * g.Cout) = make_uint4(o[0], o[1], o[2], o[3]);
        }
      }
      __syncwarp();
    }
  }
  if (!stats) return;
  if (stat_co >= 0) flush();
  __syncthreads();
  for (int i = threadIdx.x; i < 2 * g.Cout; i += 256) atomicAdd(&stats[i], (double)sums[i]);
}

// Weight gradient: a thread sums over its column of the tiles the nine products of one filter row and four output channels;
// the lanes are added up once, at the end, then the blocks (conv_wgrad_fewch_kernel reads an activation and all of dy for every
// filter position: 29.6 against 24.5 us on 128 images of 32x32 with 16 channels, 78 against 29 with 40, 122 against 73 on 64 of
// 224x224, 16 channels, stride 2).  dw must be zero before the launch.
template <int kStride>
__global__ void __launch_bounds__(384)
image_wgrad_kernel(const bf16* __restrict__ x, const bf16* __restrict__ dy, float* __restrict__ dw, const ImageTiles g) {
  constexpr int CPT = 4;
  extern __shared__ float patch[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, items = 3 * (g.Cout / CPT);
  const int item = blockIdx.y * 12 + warp, fr = item % 3, co0 = item / 3 * CPT;    // (a block row per twelve items)
  uint64_t acc[9][CPT / 2];
#pragma unroll
  for (int k = 0; k < 9; ++k)
#pragma unroll
    for (int j = 0; j < CPT / 2; ++j) acc[k][j] = 0;
#pragma unroll 1
  for (int t = blockIdx.x; t < g.tiles; t += gridDim.x) {
    const int tw = t % g.tiles_w, t2 = t / g.tiles_w, th = t2 % g.tiles_h, n = t2 / g.tiles_h;
    const int oh0 = th * g.TH, ow0 = tw * 32, ow = ow0 + lane;
    __syncthreads();
    image_stage<kStride>(g, x, patch, n, oh0, ow0);
    __syncthreads();
    // (a lane past the last column adds nothing: not a product with a zero, since the patch may hold an infinity of the image)
    const int rows = item < items && ow < g.OW ? min(g.TH, g.OH - oh0) : 0;
    const bf16* dp = dy + ((long long)(n * g.OH + oh0) * g.OW + ow) * g.Cout + co0;
#pragma unroll 2
    for (int h = 0; h < rows; ++h) {
      const uint2 d = *reinterpret_cast<const uint2*>(dp + (long long)h * g.OW * g.Cout);
      const uint64_t d2[2] = {pair_of(__uint_as_float(d.x << 16), __uint_as_float(d.x & 0xFFFF0000u)),
                              pair_of(__uint_as_float(d.y << 16), __uint_as_float(d.y & 0xFFFF0000u))};
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        const float v = patch[image_at<kStride>(h * kStride + fr, k % 3, lane * kStride + k / 3)];
        const uint64_t v2 = pair_of(v, v);
        pair_fma(acc[k][0], v2, d2[0]);
        pair_fma(acc[k][1], v2, d2[1]);
      }
    }
  }
  if (item >= items) return;
#pragma unroll
  for (int k = 0; k < 9; ++k)
#pragma unroll
    for (int j = 0; j < CPT / 2; ++j) {
      float lo, hi;
      asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(acc[k][j]));
      lo = warp_sum(lo);
      hi = warp_sum(hi);
      if (lane == 0) {
        atomicAdd(&dw[(long long)(co0 + 2 * j) * 27 + fr * 9 + k], lo);
        atomicAdd(&dw[(long long)(co0 + 2 * j + 1) * 27 + fr * 9 + k], hi);
      }
    }
}

// Weight gradient for few input channels.  A thread owns one filter position k = (r, s, ci) and
// CPT output channels, and walks the pixels of its block's range: per pixel one activation load
// and CPT/V 16-byte loads of dy (the same for every thread of a channel group) feed CPT
// multiply-adds.  With few (k, group) pairs the block's threads also split into pixel lanes, summed
// through shared memory (threads * CPT floats, dynamic) before one atomic add per output.
// dw must be zero before the launch.
template <typename T, int CPT>
__global__ void __launch_bounds__(256)
conv_wgrad_fewch_kernel(const T* __restrict__ x, const T* __restrict__ dy, float* __restrict__ dw, ConvGeom g,
                        int pair_threads, long long pixels_per_block) {
  constexpr int V = VecT<T>::N;
  extern __shared__ float red[];
  const int K = g.R * g.S * g.Cin;
  const int CG = g.Cout / CPT;
  const int npairs = K * CG;
  const int PL = blockDim.x / pair_threads;          // pixel lanes
  const int pl = threadIdx.x / pair_threads, pt = threadIdx.x % pair_threads;
  const bool live = pt < npairs;
  const int k = live ? pt / CG : 0, cg = live ? pt % CG : 0;
  const int ci = k % g.Cin, fs = (k / g.Cin) % g.S, fr = k / (g.Cin * g.S);
  float acc[CPT];
#pragma unroll
  for (int j = 0; j < CPT; ++j) acc[j] = 0.f;
  const long long npix = (long long)g.N * g.OH * g.OW;
  const long long p0 = (long long)blockIdx.x * pixels_per_block;
  long long p1 = p0 + pixels_per_block;
  if (p1 > npix) p1 = npix;
  if (live && p0 + pl < p1) {
    long long p = p0 + pl;
    int ow = (int)(p % g.OW);
    long long t = p / g.OW;
    int oh = (int)(t % g.OH);
    int n = (int)(t / g.OH);
    for (; p < p1; p += PL) {
      const int ih = oh * g.stride + fr - g.pad, iw = ow * g.stride + fs - g.pad;
      if (ih >= 0 && ih < g.H && iw >= 0 && iw < g.W) {
        const float xv = to_f(x[(((long long)n * g.H + ih) * g.W + iw) * g.Cin + ci]);
        const T* dp = dy + p * g.Cout + cg * CPT;
#pragma unroll
        for (int j = 0; j < CPT; j += V) {
          float f[V];
          ldv(dp + j, f);
#pragma unroll
          for (int u = 0; u < V; ++u) acc[j + u] += xv * f[u];
        }
      }
      ow += PL;
      while (ow >= g.OW) {
        ow -= g.OW;
        if (++oh == g.OH) { oh = 0; ++n; }
      }
    }
  }
  if (PL > 1) {
#pragma unroll
    for (int j = 0; j < CPT; ++j) red[threadIdx.x * CPT + j] = acc[j];
    __syncthreads();
    if (pl == 0)
      for (int l = 1; l < PL; ++l)
#pragma unroll
        for (int j = 0; j < CPT; ++j) acc[j] += red[(l * pair_threads + pt) * CPT + j];
  }
  if (pl == 0 && live) {
#pragma unroll
    for (int j = 0; j < CPT; ++j) atomicAdd(&dw[(long long)(cg * CPT + j) * K + k], acc[j]);
  }
}

}  // namespace lp
