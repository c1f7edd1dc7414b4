// 3x3 stride-1 convolutions with 16, 32 or 64 channels on both sides (forward and input gradient), with the batch
// norms around them taken along.
//
// What bounds such a layer is not a unit of the machine but the number of steps: a launch moves a few MB and multiplies
// for less than two microseconds, and one residual block was ten such launches in a row (convolution, batch norm,
// convolution, batch norm + shortcut; reduction, batch-norm backward, input gradient, twice), each with its own start-up
// and its own trip through memory, and a convolution of 16 channels issued 36 MMAs of N = 16 per 512 pixels.  Here
//
//  * g = 64 / C neighbouring pixels of an image row are one "group" of 64 channels (the same memory, seen as an image of
//    W / g columns and 64 channels).  A 3x3 convolution over pixels is then a 3x3 convolution over groups whose 64 x 64
//    weight blocks hold the taps (the three pixels an output pixel reads lie in its own group or at the near edge of a
//    neighbour); the K = 16 slices that hold no tap are left out: 18 MMAs of N = 64 per 128 groups at 16 channels, 24 at
//    32, 36 at 64.  All layers become the same 128 x 64 tile over rows of 128 bytes;
//  * the weights of all slices (36 to 72 KB) are fetched once per CTA, before the preceding kernel has finished;
//  * the operand tile with its halo arrives by TMA.  Where the operand is not a stored tensor it is PRODUCED in place by
//    the warps -- normalised, rounded to bf16 as the separate kernel did, zeroed outside the image -- and its inner part
//    written to memory for the kernels that need the tensor itself (shortcut, weight gradient):
//      kMode 1  relu(bn(y))         kMode 2  bn(y) + shortcut        kMode 3  batch-norm backward from (dy, y);
//  * the epilogue takes the statistics of the next batch norm (forward) or the reduction pass of the next batch-norm
//    backward (input gradient) as column sums over the staged output tile, which leaves by a TMA store.
//
// A residual block is four launches in a row instead of ten (ResNet-56 on 128 images 1202 -> 785 us per step, ResNet-110
// 2127 -> 1455; with the rolled loops of the other kernels 738 and 1343).  A CTA runs most of its code once or twice, so fetching
// instructions costs as much as executing them: loops are kept rolled and whole tiles are moved by single copies (an
// unrolled version with the loads in registers, 2.5 times the code, took 1.5 times as long per launch).  For the same
// reason nothing is pipelined inside a CTA: beside it run the kernels of the other modules' streams (a launch takes one CTA
// per SM at most; registers and, up to 32 channels, shared memory leave room for a CTA of another launch).
//
// Tile geometry: M row r of a tile sits at box position (r / 8) * S + r % 8 (rows of 128 bytes; box dimensions W, image,
// H with P = BW + 2 columns).  S = P and BW = 8: eight columns per row group; S = 8: the box rows are taken as one run,
// halo columns included (their results are dropped), which wastes less where the width is 9 to 14 groups.  A tap is a row
// offset into the box, as in conv_tc.cuh (the 128-byte swizzle is a function of the address).
#pragma once
#include "common.cuh"
#include "conv_tc.cuh"
#include "tc_ptx.cuh"

namespace lp {
namespace tc {

constexpr int kThinWarps = 8;
constexpr int kThinThreads = 32 * kThinWarps;
constexpr int kThinMaxBoxRows = 256;
constexpr int kThinBoxBytesW = 64 * 128;           // one weight box: 64 output columns x 64 K columns

struct ConvThinParams {
  int N, H, Wg;                  // images, rows, groups per row
  int BW, BH, BNI, P, S;         // tile (groups, rows, images), box columns, box rows between 8-row groups of M
  int box_rows, tile_rows;       // rows of the operand box; of an output tile
  int tiles_w, tiles_h, tiles;
  FastDiv fd_w, fd_h, fd_P, fd_BNI, fd_TP;   // fd_TP: columns of the output tile's rows (BW, or P where S = 8)
  int C;                         // channels of a pixel (16, 32, 64)
  int n_mma, n_wbox;
  uint16_t a_off[36];            // operand start of MMA i inside the box, in units of 16 bytes
  uint32_t a_offset, b_offset, b2_offset, tail_offset;   // operand box; second box / shortcut tile; reduction tile; rest
  uint32_t idesc;
  uint64_t desc_a, desc_b;
  // operand production (kMode 1..3)
  BnArgs bn;
  const float* bn_dgamma;        // kMode 3: sums of the reduction pass
  const float* bn_dbeta;
  int bn_relu;                   // kMode 3: a ReLU followed the batch norm
  bf16* pre_out;                 // the produced tensor
  // epilogue
  int has_addend;                // kBwd
  double* stats;                 // !kBwd, nullable: [2*C]
  int has_red;                   // kBwd: the output is the dy of a batch-norm backward whose reduction pass is taken here
  BnArgs red_bn;
  float* red_dgamma;
  float* red_dbeta;
  int red_relu;
  int* err;
};

struct ThinSmemTail {
  uint64_t full, aux_full, acc_full, w_full;
  uint32_t tmem_base;
  int abort_flag;
  float4 kconst[64];             // batch norm of the operand: scale, shift and, kMode 3, the factors of x and 1; column c at
                                 // (c % 8) * 8 + c / 8, the order the producing threads read
  float4 rconst[64];             // reduction pass: scale, shift, mean, rstd per column
  float4 red[kThinWarps][32];    // column sums of a warp's rows: two columns x two kinds
};

// tmIn0 / tmIn1: first and second tensor of the operand (boxes with halo); tmB: weights; tmAdd / tmRed: shortcut and
// normalised tensor of the reduction pass (output tiles); tmOut: output.
template <int kMode, bool kBwd>
__global__ void __launch_bounds__(kThinThreads, 2)
conv_thin_kernel(const __grid_constant__ CUtensorMap tmIn0, const __grid_constant__ CUtensorMap tmIn1,
                 const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmAdd,
                 const __grid_constant__ CUtensorMap tmRed, const __grid_constant__ CUtensorMap tmOut,
                 const __grid_constant__ ConvThinParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  ThinSmemTail* tail = reinterpret_cast<ThinSmemTail*>(smem + p.tail_offset);
  volatile int* abort_flag = &tail->abort_flag;
  const int wt = threadIdx.x, warp = wt >> 5, lane = wt & 31;
  const int t_begin = (int)(((long long)p.tiles * blockIdx.x) / gridDim.x);
  const int t_end = (int)(((long long)p.tiles * (blockIdx.x + 1)) / gridDim.x);

  if (wt == 0) {
    mbar_init(&tail->full, 1);
    mbar_init(&tail->aux_full, 1);
    mbar_init(&tail->acc_full, 1);
    tail->abort_flag = 0;
    fence_barrier_init();
    prefetch_tmap(&tmIn0);
    if (kMode >= 2) prefetch_tmap(&tmIn1);
  } else if (wt == 32) {
    // the weights were written at least one kernel before the preceding one: they may be fetched before its end
    mbar_init(&tail->w_full, 1);
    fence_barrier_init();
    mbar_expect_tx(&tail->w_full, (uint32_t)(p.n_wbox * kThinBoxBytesW));
#pragma unroll 1
    for (int i = 0; i < p.n_wbox; ++i) tma_load_2d(smem + i * kThinBoxBytesW, &tmB, &tail->w_full, i * 64, 0);
  }
  if (warp == 2) {
    tmem_alloc(&tail->tmem_base, 64);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait();
  pdl_launch_dependents();
  const uint32_t tmem_base = tail->tmem_base;
  uint8_t* box = smem + p.a_offset;         // operand; later the staged output tile
  uint8_t* box2 = smem + p.b_offset;        // second tensor of the operand; later the shortcut's tile
  bool failed = false;
  float s0 = 0.f, s1 = 0.f, q0 = 0.f, q1 = 0.f;   // columns 2 * lane and 2 * lane + 1, over this warp's rows

#pragma unroll 1
  for (int t = t_begin; t < t_end; ++t) {
    const uint32_t ph = (uint32_t)(t - t_begin) & 1;
    int q1_, tw, tn, th;
    fd_divmod(t, p.fd_w, q1_, tw);
    fd_divmod(q1_, p.fd_h, tn, th);
    const int w0 = tw * p.BW, h0 = th * p.BH, n0 = tn * p.BNI;
    if (t > t_begin) {
      tc_fence_before();
      __syncthreads();                      // everything of the previous tile has been read
      tc_fence_after();
    }
    if (wt == 0) {
      mbar_expect_tx(&tail->full, (uint32_t)((kMode >= 2 ? 2 : 1) * p.box_rows * 128));
      tma_load_4d(box, &tmIn0, &tail->full, 0, w0 - 1, n0, h0 - 1);
      if (kMode >= 2) tma_load_4d(box2, &tmIn1, &tail->full, 0, w0 - 1, n0, h0 - 1);
    }
    if (t == t_begin) {
      // constants of the two batch norms, one thread per column (they repeat every C columns)
      if ((kMode || kBwd) && warp >= 6) {
        const int col = wt - 192, c = col & (p.C - 1);
        if constexpr (kMode != 0) {
          float mean, rstd;
          bn_mean_rstd(p.bn.stats[c], p.bn.stats[p.C + c], p.bn.inv_count, p.bn.eps, mean, rstd);
          float4 k = make_float4(p.bn.gamma[c] * rstd, 0.f, 0.f, 0.f);
          k.y = p.bn.beta[c] - mean * k.x;
          if constexpr (kMode == 3) {       // dx = k.x * dy_m + k.z * x + k.w, as in bn_bwd_apply_kernel
            const float invM = (float)p.bn.inv_count;
            const float mb = p.bn_dbeta[c] * invM, mg = p.bn_dgamma[c] * invM;
            k.z = -k.x * rstd * mg;
            k.w = -k.x * mb - k.z * mean;
          }
          tail->kconst[(col & 7) * 8 + (col >> 3)] = k;
        }
        if (kBwd && p.has_red) {
          float mean, rstd;
          bn_mean_rstd(p.red_bn.stats[c], p.red_bn.stats[p.C + c], p.red_bn.inv_count, p.red_bn.eps, mean, rstd);
          const float sa = p.red_bn.gamma[c] * rstd;
          tail->rconst[col] = make_float4(sa, p.red_bn.beta[c] - mean * sa, mean, rstd);
        }
      }
      if (kMode || kBwd) __syncthreads();
    }
    if constexpr (kMode != 0) {
      // operand: thread = 16-byte piece `chunk` (a fixed group of 8 columns) of every 32nd row of the box
      const int chunk = wt & 7;
      float k0[8], k1[8], k2[kMode == 3 ? 8 : 1], k3[kMode == 3 ? 8 : 1];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float4 k = tail->kconst[j * 8 + chunk];
        k0[j] = k.x; k1[j] = k.y;
        if constexpr (kMode == 3) { k2[j] = k.z; k3[j] = k.w; }
      }
      failed |= !mbar_wait_warp(&tail->full, ph, abort_flag);
#pragma unroll 1
      for (int r = wt >> 3; r < p.box_rows; r += 32) {
        int q, lw, lh, ln;
        fd_divmod(r, p.fd_P, q, lw);
        fd_divmod(q, p.fd_BNI, lh, ln);
        const int w = w0 - 1 + lw, n = n0 + ln, h = h0 - 1 + lh;
        uint4* at = reinterpret_cast<uint4*>(box + r * 128 + ((chunk ^ (r & 7)) << 4));
        uint4 o = make_uint4(0u, 0u, 0u, 0u);
        if ((unsigned)w < (unsigned)p.Wg && (unsigned)h < (unsigned)p.H && n < p.N) {
          float f[8], y[8];
          cvt_raw(*at, f);
          if constexpr (kMode == 1) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              y[j] = fmaf(f[j], k0[j], k1[j]);
              y[j] = y[j] > 0.f ? y[j] : 0.f;
            }
          } else {
            float x[8];
            cvt_raw(*reinterpret_cast<const uint4*>(box2 + r * 128 + ((chunk ^ (r & 7)) << 4)), x);
            if constexpr (kMode == 2) {
#pragma unroll
              for (int j = 0; j < 8; ++j) y[j] = fmaf(f[j], k0[j], k1[j]) + x[j];
            } else {
              if (p.bn_relu) {
#pragma unroll
                for (int j = 0; j < 8; ++j) f[j] = fmaf(x[j], k0[j], k1[j]) > 0.f ? f[j] : 0.f;
              }
#pragma unroll
              for (int j = 0; j < 8; ++j) y[j] = fmaf(k0[j], f[j], fmaf(k2[j], x[j], k3[j]));
            }
          }
          o = make_uint4(pack_bf16x2(y[0], y[1]), pack_bf16x2(y[2], y[3]), pack_bf16x2(y[4], y[5]), pack_bf16x2(y[6], y[7]));
          if (lw >= 1 && lw <= p.BW && lh >= 1 && lh <= p.BH)
            *reinterpret_cast<uint4*>(p.pre_out + ((long long)(n * p.H + h) * p.Wg + w) * 64 + chunk * 8) = o;
        }
        *at = o;
      }
      fence_proxy_async();                  // the tile is read by the tensor core, box2 rewritten by a copy
      __syncthreads();
    }
    if (warp == 0) {
      if (kMode == 0) failed |= !mbar_wait_warp(&tail->full, ph, abort_flag);
      if (t == t_begin) failed |= !mbar_wait_warp(&tail->w_full, 0, abort_flag);
      tc_fence_after();
      const uint64_t ad0 = smem_desc(p.desc_a, smem_u32(box)), bd0 = smem_desc(p.desc_b, smem_u32(smem));
      if (elect_one()) {
#pragma unroll 6
        for (int i = 0; i < p.n_mma; ++i)
          mma_bf16(tmem_base, ad0 + p.a_off[i], bd0 + (uint64_t)((i >> 2) * (kThinBoxBytesW >> 4) + (i & 3) * 2), p.idesc,
                   i ? 1u : 0u);
        mma_commit(&tail->acc_full);
      }
      __syncwarp();
    } else if (kBwd && wt == 32 && (p.has_addend | p.has_red)) {
      mbar_expect_tx(&tail->aux_full, (uint32_t)((p.has_addend + p.has_red) * p.tile_rows * 128));
      if (p.has_addend) tma_load_4d(box2, &tmAdd, &tail->aux_full, 0, w0, n0, h0);
      if (p.has_red) tma_load_4d(smem + p.b2_offset, &tmRed, &tail->aux_full, 0, w0, n0, h0);
    }
    // epilogue: thread = one row of the tile, half of its 64 columns
    const int row = (warp & 3) * 32 + lane, half = warp >> 2;
    bool valid;
    {
      int q, lw, lh, ln;
      fd_divmod(row, p.fd_TP, q, lw);
      fd_divmod(q, p.fd_BNI, lh, ln);
      valid = lw < p.BW && lh < p.BH && w0 + lw < p.Wg && h0 + lh < p.H && n0 + ln < p.N;
    }
    if (kBwd && (p.has_addend | p.has_red)) failed |= !mbar_wait_warp(&tail->aux_full, ph, abort_flag);
    failed |= !mbar_wait_warp(&tail->acc_full, ph, abort_flag);
    tc_fence_after();
    uint32_t raw[32];
    tmem_ld32_issue(tmem_base + half * 32 + ((uint32_t)((warp & 3) * 32) << 16), raw);
    tmem_ld_wait();
    tmem_ld_fence(raw);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t at = row * 128 + (((half * 4 + u) ^ (row & 7)) << 4);
      float v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(raw[8 * u + j]);
      if (kBwd && p.has_addend) {
        float f[8];
        cvt_raw(*reinterpret_cast<const uint4*>(box2 + at), f);
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] += f[j];
      }
      uint4 o = make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]), pack_bf16x2(v[6], v[7]));
      if (!valid) o = make_uint4(0u, 0u, 0u, 0u);
      *reinterpret_cast<uint4*>(box + at) = o;
    }
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    if (wt == 0) {
      tma_store_4d(&tmOut, box, 0, w0, n0, h0);    // (parts of the box outside the tensor are not written)
      bulk_commit_group();
    }
    // column sums of the tensor as stored: lane = two columns, warp = 16 rows
    if (kBwd ? p.has_red != 0 : p.stats != nullptr) {
      float4 ka, kb;
      if (kBwd) { ka = tail->rconst[2 * lane]; kb = tail->rconst[2 * lane + 1]; }
      const int r_end = min(warp * 16 + 16, p.tile_rows);
#pragma unroll 4
      for (int r = warp * 16; r < r_end; ++r) {
        const uint32_t at = r * 128 + (((lane >> 2) ^ (r & 7)) << 4) + (lane & 3) * 4;
        const uint32_t d2 = *reinterpret_cast<const uint32_t*>(box + at);
        float lo = __uint_as_float(d2 << 16), hi = __uint_as_float(d2 & 0xFFFF0000u);
        if constexpr (kBwd) {
          const uint32_t x2 = *reinterpret_cast<const uint32_t*>(smem + p.b2_offset + at);
          const float xlo = __uint_as_float(x2 << 16), xhi = __uint_as_float(x2 & 0xFFFF0000u);
          if (p.red_relu) {
            lo = fmaf(xlo, ka.x, ka.y) > 0.f ? lo : 0.f;
            hi = fmaf(xhi, kb.x, kb.y) > 0.f ? hi : 0.f;
          }
          q0 = fmaf(lo, xlo - ka.z, q0); q1 = fmaf(hi, xhi - kb.z, q1);
        } else {
          q0 = fmaf(lo, lo, q0); q1 = fmaf(hi, hi, q1);
        }
        s0 += lo; s1 += hi;
      }
    }
    if (wt == 0) bulk_wait_read(0);
  }
  // column sums of the CTA: the g places of a channel, then the warps
  if (kBwd ? p.has_red != 0 : p.stats != nullptr) {
#pragma unroll 1
    for (int o = p.C >> 1; o < 32; o <<= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, o); s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      q0 += __shfl_xor_sync(0xffffffffu, q0, o); q1 += __shfl_xor_sync(0xffffffffu, q1, o);
    }
    tail->red[warp][lane] = make_float4(s0, s1, q0, q1);
    __syncthreads();
    if (wt < 2 * p.C) {
      const int kind = wt >= p.C ? 1 : 0, c = wt - kind * p.C;
      float a = 0.f;
#pragma unroll
      for (int w = 0; w < kThinWarps; ++w) a += reinterpret_cast<const float*>(&tail->red[w][c >> 1])[kind * 2 + (c & 1)];
      if constexpr (kBwd) {
        if (kind) atomicAdd(&p.red_dgamma[c], a * tail->rconst[c].w);
        else atomicAdd(&p.red_dbeta[c], a);
      } else {
        atomicAdd(&p.stats[wt], (double)a);
      }
    }
  }

  if (failed) {
    *abort_flag = 1;
    atomicExch(p.err, 1);
#pragma unroll 1
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);   // copies and MMAs in flight land before the memory is released
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {            // (the same for all threads: set before the barrier)
    if (!failed)
  #pragma unroll 1
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
    __syncthreads();
  }
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 64);
  }
}

// fp32 weight gradients of grouped layers, folded back: dwg[(p_out, co)][tap][(p_in, ci)] (the gradient of the 64 x 64
// blocks) -> dw[co][r][s][ci], the sum of the g places a tap has in them.
struct FoldEntry {
  float* dwg;
  float* dw;
  int C;
};
__global__ void __launch_bounds__(256)
wgrad_fold_kernel(const FoldEntry* __restrict__ tab) {
  const FoldEntry e = tab[blockIdx.x];
  const int g = 64 / e.C, total = 9 * e.C * e.C;
  for (int i = blockIdx.y * 256 + threadIdx.x; i < total; i += gridDim.y * 256) {
    const int ci = i % e.C;
    const int t = (i / e.C) % 9;
    const int co = i / (9 * e.C);
    const int r = t / 3, s = t % 3;
    float a = 0.f;
    for (int po = 0; po < g; ++po) {
      const int pi = po + s - 1;                       // pixel read, counted from the output pixel's group
      const int dx = pi < 0 ? 0 : (pi >= g ? 2 : 1);
      a += e.dwg[((po * e.C + co) * 9 + r * 3 + dx) * 64 + (pi + g * (1 - dx)) * e.C + ci];
    }
    e.dw[i] = a;
  }
}

}  // namespace tc
}  // namespace lp
