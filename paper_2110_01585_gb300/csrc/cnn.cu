// Learned warm start: the building blocks of a small fully convolutional network
// (3x3 convolutions on the torus with bias and ReLU, their backward pass, the
// Adam step, the training loss) and nothing else.  The paper has no
// counterpart; its EP sweeps correct whatever the network's output gets wrong.
//
// Arrays are float32 NCHW.  The convolution is a direct one on CUDA cores in FP32,
// bound by its FP32 FMAs (18 cin per pixel and output against 4 (cin + cout) bytes): a
// thread keeps four pixels x 16 outputs in registers as packed pairs of outputs, reads
// six inputs and twelve float4 of weights (one address per warp) from shared memory per
// channel and row of taps and does 96 packed FMAs with them.  The weight gradient keeps
// 2 outputs x 9 taps of one input channel per thread and walks over the pixels; its sums
// are reduced in a fixed order (no atomics), so training is deterministic.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <mutex>

#include "internal.cuh"

namespace eptv {

namespace {

constexpr int kMaxOut = 32;   // output channels per launch
constexpr int kWarmOut = 6;   // network outputs: mean residual, five site log-precisions

__device__ __forceinline__ int wrapi(int v, int n) {
  if (v >= 0 && v < n) return v;  // the common cases without a division
  if (v < 0 && v >= -n) return v + n;
  if (v >= n && v < 2 * n) return v - n;
  v %= n;
  return v < 0 ? v + n : v;
}

// 4-byte asynchronous copy to shared memory; zeros when ok is false (nothing is read).
__device__ __forceinline__ void cp4(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(ok ? 4 : 0)
               : "memory");
}
__device__ __forceinline__ void cp16(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(ok ? 16 : 0)
               : "memory");
}
// Rows of planes of width w starting at p hold whole aligned float4.
__device__ __forceinline__ bool rows_vec4(const float* p, int w) {
  return (w & 3) == 0 && (reinterpret_cast<uintptr_t>(p) & 15) == 0;
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Forward: y[n, o] = b[o] + sum_c sum_tap w[o, c, tap] x[n, c, shifted by tap], ReLU optional.
// Input gradient (kGrad): dx[n, c] = sum_o sum_tap w[o, c, 8 - tap] g[n, o, shifted by tap],
// i.e. the same with the roles of the channels exchanged and the taps reversed.  Every
// output sums its channels and taps in order with one FMA each, starting from the bias.
//
// A block computes a tile of 32 x kRowsT pixels, all output channels: lane l of a warp has
// pixels 4 (l & 7) .. + 3 of row l >> 3 of the warp's four rows; the warps of one tile share
// it between groups of CO outputs.  kCC input channels at a time are staged by
// asynchronous copies, with a one-pixel circular halo, while the block computes on the
// previous ones; the weights as [channel][tap][output] with a pitch of kOut + 4, which
// keeps the transposing copies to four-way bank conflicts.
// Measured at 32 -> 32 channels, 8 images of 128^2 (2.4 GFLOP), forward pass: 127 us with one
// pixel x 32 outputs per thread (a weight load per four unpacked FMAs), 64 here, of the
// 31 that the FMAs alone take; half of the issued instructions are FMAs.
constexpr int kTW = 32;       // tile width
constexpr int kPitch = kTW + 8;  // columns x0 - 4 .. x0 + 35: whole float4 of the image's rows

template <int CO, int kGroups, bool kGrad>
__global__ void __launch_bounds__(128, 4) conv3x3_kernel(int cin, int cout, int H, int W, const float* __restrict__ x,
                                                         const float* __restrict__ w, const float* __restrict__ b,
                                                         int relu, float* __restrict__ y) {
  constexpr int kRowsT = 16 / kGroups;       // tile rows: four per warp
  constexpr int kCC = kGroups == 2 ? 8 : 4;  // input channels per stage
  constexpr int kOut = CO * kGroups, kWp = kOut + 4;
  __shared__ __align__(16) float xs[2][kCC][kRowsT + 2][kPitch];
  __shared__ __align__(16) float ws[2][kCC * 9 * kWp];
  const int n = blockIdx.z;
  const int tiles_x = (W + kTW - 1) / kTW;
  const int x0 = (int)(blockIdx.x % tiles_x) * kTW, y0 = (int)(blockIdx.x / tiles_x) * kRowsT;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = warp % kGroups, o0 = grp * CO;
  const int qx = 4 * (lane & 7), qy = (warp / kGroups) * 4 + (lane >> 3);
  const long long plane = (long long)H * W;
  const float* xn = x + (long long)n * cin * plane;
  const bool vec_in = rows_vec4(x, W);
  auto stage = [&](int c0, int buf) {
    const int cc = min(kCC, cin - c0);
    const int rows = cc * (kRowsT + 2);
    const float* xc = xn + (long long)c0 * plane;
    if (vec_in) {
      for (int i = threadIdx.x; i < rows * (kPitch / 4); i += 128) {
        const int cr = i / (kPitch / 4), v = i % (kPitch / 4), c = cr / (kRowsT + 2), r = cr % (kRowsT + 2);
        cp16(&xs[buf][c][r][4 * v],
             xc + c * plane + (long long)wrapi(y0 - 1 + r, H) * W + wrapi(x0 - 4 + 4 * v, W), true);
      }
    } else {
      const int q0 = wrapi(x0 - 1 + lane, W), q1 = wrapi(x0 + 31 + (lane & 1), W);
      for (int i = warp; i < rows; i += 4) {
        const int c = i / (kRowsT + 2), r = i % (kRowsT + 2);
        const float* row = xc + c * plane + (long long)wrapi(y0 - 1 + r, H) * W;
        cp4(&xs[buf][c][r][3 + lane], row + q0, true);
        if (lane < 2) cp4(&xs[buf][c][r][35 + lane], row + q1, true);
      }
    }
    if (kGrad) {
      // w[c0 + c][o][tap], tap reversed: contiguous in (o, tap) for one c
      for (int i = threadIdx.x; i < kCC * 9 * kOut; i += 128) {
        const int c = i / (9 * kOut), e = i % (9 * kOut), o = e / 9;
        const bool ok = o < cout && c < cc;
        cp4(&ws[buf][(9 * c + 8 - e % 9) * kWp + o], w + (ok ? (long long)(c0 + c) * cout * 9 + e : 0), ok);
      }
    } else {
      // w[o][c0 + c][tap]: contiguous in (c, tap) for one o
      int o = threadIdx.x / (9 * kCC), e = threadIdx.x % (9 * kCC);
#pragma unroll 3
      for (; o < kOut;) {
        const bool ok = o < cout && e < 9 * cc;
        cp4(&ws[buf][e * kWp + o], w + (ok ? ((long long)o * cin + c0) * 9 + e : 0), ok);
        o += 128 / (9 * kCC);
        e += 128 % (9 * kCC);
        if (e >= 9 * kCC) {
          e -= 9 * kCC;
          ++o;
        }
      }
    }
    cp_commit();
  };
  float2 acc[4][CO / 2];
#pragma unroll
  for (int o = 0; o < CO / 2; ++o) {
    const int oa = o0 + 2 * o;
    const float2 bo = make_float2(b && oa < cout ? b[oa] : 0.0f, b && oa + 1 < cout ? b[oa + 1] : 0.0f);
#pragma unroll
    for (int p = 0; p < 4; ++p) acc[p][o] = bo;
  }
  stage(0, 0);
  int buf = 0;
  for (int c0 = 0; c0 < cin; c0 += kCC, buf ^= 1) {
    const int cc = min(kCC, cin - c0);
    if (c0 + kCC < cin) {
      stage(c0 + kCC, buf ^ 1);
      cp_wait<1>();
    } else {
      cp_wait<0>();
    }
    __syncthreads();
    for (int c = 0; c < cc; ++c) {
#pragma unroll
      for (int ky = 0; ky < 3; ++ky) {
        const float* row = &xs[buf][c][qy + ky][qx];  // columns x - 4 .. x + 7 of pixels x .. x + 3
        const float4 xa = *reinterpret_cast<const float4*>(row + 4);
        const float xv[6] = {row[3], xa.x, xa.y, xa.z, xa.w, row[8]};
#pragma unroll
        for (int kx = 0; kx < 3; ++kx) {
          const float4* wv = reinterpret_cast<const float4*>(&ws[buf][(c * 9 + 3 * ky + kx) * kWp + o0]);
#pragma unroll
          for (int o4 = 0; o4 < CO / 4; ++o4) {
            const float4 q = wv[o4];
#pragma unroll
            for (int p = 0; p < 4; ++p) {
              const float2 xx = make_float2(xv[p + kx], xv[p + kx]);
              acc[p][2 * o4] = __ffma2_rn(make_float2(q.x, q.y), xx, acc[p][2 * o4]);
              acc[p][2 * o4 + 1] = __ffma2_rn(make_float2(q.z, q.w), xx, acc[p][2 * o4 + 1]);
            }
          }
        }
      }
    }
    __syncthreads();
  }
  const int gy = y0 + qy, gx = x0 + qx;
  if (gy >= H || gx >= W) return;
  const bool vec = (W & 3) == 0 && (reinterpret_cast<uintptr_t>(y) & 15) == 0;  // then gx + 3 < W
#pragma unroll
  for (int o = 0; o < CO; ++o) {
    if (o0 + o >= cout) break;
    float v[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      v[p] = o & 1 ? acc[p][o / 2].y : acc[p][o / 2].x;
      if (relu) v[p] = fmaxf(v[p], 0.0f);
    }
    float* out = y + ((long long)n * cout + o0 + o) * plane + (long long)gy * W + gx;
    if (vec) {
      *reinterpret_cast<float4*>(out) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int p = 0; p < 4; ++p)
        if (gx + p < W) out[p] = v[p];
    }
  }
}

// Weight and bias gradients:
//   part[blk][o][c][tap] = sum_p g[o, p] x[c, p shifted by tap], part[blk][cout*cin*9 + o] = sum_p g[o, p]
// over the tiles of 16 x 16 pixels that block blockIdx.x takes (every gridDim.x-th), for
// the input channels 32 blockIdx.y .. + 31.  g = dy, masked by y > 0 when the layer had a
// ReLU (y = max(z, 0) > 0 iff z > 0); with gout the masked gradient is also written there,
// for the input gradient.  Thread: the pair of outputs 2 (t & 15), channel t >> 4; four
// pixels of a tile's row at a time share the inputs of their taps, so they cost seven loads
// and 36 packed FMAs.  The next tile's x, dy and y arrive by asynchronous copies
// meanwhile; dy and y are turned into the masked gradient, pixel-major, between tiles.
// A tile's sums are FP32; their sum over the block's tiles is FP64, as is the reduction over
// blocks (a pair of FP32 sums with TwoSum holds fewer bits and makes NaN of an infinite
// tile sum; it took 10 us less, the FP64 additions being two per clock and SM).
// Measured at 32 -> 32 channels, 8 images of 128^2: 145 us with one output and channel per
// thread and a pass for the mask (23 us) before, 94 here; the reduction 78 -> 6.5 us.
constexpr int kT = 16;        // tile side (pixels)
constexpr int kDwThreads = 512;
constexpr int kDwPitch = kT + 8;  // columns x0 - 4 .. x0 + 19
constexpr int kDwXs = 32 * (kT + 2) * kDwPitch;  // inputs of a tile
constexpr int kDwG = kT * kT * kMaxOut;          // gradients of a tile
constexpr int kDwSmem = (2 * kDwXs + 3 * kDwG) * 4;

__global__ void __launch_bounds__(kDwThreads) conv3x3_dw_kernel(int cin, int cout, int H, int W, int tiles_x,
                                                                long long n_tiles, const float* __restrict__ x,
                                                                const float* __restrict__ dy,
                                                                const float* __restrict__ y, float* __restrict__ gout,
                                                                double* __restrict__ part) {
  extern __shared__ __align__(16) float dw_smem[];
  float* gs = dw_smem;             // [kT * kT][kMaxOut], the outputs of pixel p rotated by 4 p
  float* rg = gs + kDwG;           // dy and y as they lie in memory: [output][pixel]
  float* ry = rg + kDwG;
  float* xs2 = ry + kDwG;          // two of [32][kT + 2][kDwPitch]
  const int og = threadIdx.x & 15, c = threadIdx.x >> 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c0 = 32 * blockIdx.y, cc = min(32, cin - c0);
  const long long plane = (long long)H * W;
  const long long tiles = (long long)tiles_x * ((H + kT - 1) / kT);
  const bool vecx = rows_vec4(x, W), vecg = rows_vec4(dy, W) && (!y || rows_vec4(y, W));
  auto stage = [&](long long tile, int buf) {
    const long long n = tile / tiles, tt = tile % tiles;
    const int x0 = (int)(tt % tiles_x) * kT, y0 = (int)(tt / tiles_x) * kT;
    float* xs = xs2 + buf * kDwXs;
    const float* xc = x + (n * cin + c0) * plane;
    if (vecx) {
      for (int i = threadIdx.x; i < 32 * (kT + 2) * (kDwPitch / 4); i += kDwThreads) {
        const int cr = i / (kDwPitch / 4), v = i % (kDwPitch / 4), ch = cr / (kT + 2), r = cr % (kT + 2);
        const bool ok = ch < cc;
        cp16(xs + cr * kDwPitch + 4 * v,
             xc + (ok ? ch : 0) * plane + (long long)wrapi(y0 - 1 + r, H) * W + wrapi(x0 - 4 + 4 * v, W), ok);
      }
    } else {
      const int gq = wrapi(x0 - 1 + min(lane, kT + 1), W);  // 18 lanes a row (the rest of a warp idles)
      for (int i = warp; i < 32 * (kT + 2); i += kDwThreads / 32) {
        const int ch = i / (kT + 2), r = i % (kT + 2);
        const bool ok = ch < cc;
        const float* row = xc + (ok ? ch : 0) * plane + (long long)wrapi(y0 - 1 + r, H) * W;
        if (lane < kT + 2) cp4(xs + i * kDwPitch + 3 + lane, row + gq, ok);
      }
    }
    // dy and y, zero outside the image
    if (vecg) {
      for (int i = threadIdx.x; i < kMaxOut * kT * (kT / 4); i += kDwThreads) {
        const int o = i / (kT * (kT / 4)), e = i % (kT * (kT / 4));
        const int gx = x0 + 4 * (e % (kT / 4)), gy = y0 + e / (kT / 4);
        const bool ok = o < cout && gx < W && gy < H;
        const long long at = ok ? (n * cout + o) * plane + (long long)gy * W + gx : 0;
        cp16(rg + 4 * i, dy + at, ok);
        if (y) cp16(ry + 4 * i, y + at, ok);
      }
    } else {
      for (int i = threadIdx.x; i < kMaxOut * kT * kT; i += kDwThreads) {
        const int o = i / (kT * kT), e = i % (kT * kT);
        const int gx = x0 + e % kT, gy = y0 + e / kT;
        const bool ok = o < cout && gx < W && gy < H;
        const long long at = ok ? (n * cout + o) * plane + (long long)gy * W + gx : 0;
        cp4(rg + i, dy + at, ok);
        if (y) cp4(ry + i, y + at, ok);
      }
    }
    cp_commit();
  };
  double2 sum[9], bsum = make_double2(0.0, 0.0);
#pragma unroll
  for (int k = 0; k < 9; ++k) sum[k] = make_double2(0.0, 0.0);
  int buf = 0;
  if (blockIdx.x < n_tiles) stage(blockIdx.x, 0);
  for (long long tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, buf ^= 1) {
    cp_wait<0>();
    __syncthreads();  // the tile has landed, and the previous one is done with gs
    {
      const long long n = tile / tiles, tt = tile % tiles;
      const int x0 = (int)(tt % tiles_x) * kT, y0 = (int)(tt / tiles_x) * kT;
      // one pixel and half of the outputs per thread
      const int p = threadIdx.x % (kT * kT), gx = x0 + p % kT, gy = y0 + p / kT;
      const bool put = gout && gx < W && gy < H;
      const int oh = threadIdx.x / (kT * kT) * (kMaxOut / 2);
#pragma unroll 8
      for (int o = oh; o < oh + kMaxOut / 2; ++o) {
        float v = rg[o * (kT * kT) + p];
        if (y && !(ry[o * (kT * kT) + p] > 0.0f)) v = 0.0f;
        gs[p * kMaxOut + ((o + 4 * p) & 31)] = v;
        if (put && o < cout) gout[(n * cout + o) * plane + (long long)gy * W + gx] = v;
      }
    }
    __syncthreads();
    if (tile + gridDim.x < n_tiles) stage(tile + gridDim.x, buf ^ 1);
    const float* xs = xs2 + buf * kDwXs;
    float2 acc[9], bacc = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 9; ++k) acc[k] = make_float2(0.f, 0.f);
    for (int r = 0; r < kT; ++r) {
      const float* xr = xs + (c * (kT + 2) + r) * kDwPitch;
      float pv[3];   // column left of the current four pixels, then their own columns
      float4 v[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        pv[k] = xr[k * kDwPitch + 3];
        v[k] = *reinterpret_cast<const float4*>(xr + k * kDwPitch + 4);
      }
#pragma unroll
      for (int a = 0; a < kT / 4; ++a) {
        float2 g[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int p = r * kT + 4 * a + q;
          g[q] = *reinterpret_cast<const float2*>(gs + p * kMaxOut + ((2 * og + 4 * p) & 31));
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const float4 nx = *reinterpret_cast<const float4*>(xr + k * kDwPitch + 4 * a + 8);
          const float e[6] = {pv[k], v[k].x, v[k].y, v[k].z, v[k].w, nx.x};
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int t = 0; t < 3; ++t)
              acc[3 * k + t] = __ffma2_rn(g[q], make_float2(e[q + t], e[q + t]), acc[3 * k + t]);
          pv[k] = v[k].w;
          v[k] = nx;
        }
        if (c == 0) {
#pragma unroll
          for (int q = 0; q < 4; ++q) bacc = __fadd2_rn(bacc, g[q]);
        }
      }
    }
    if (tile == blockIdx.x) {
#pragma unroll
      for (int k = 0; k < 9; ++k) sum[k] = make_double2((double)acc[k].x, (double)acc[k].y);
      bsum = make_double2((double)bacc.x, (double)bacc.y);
    } else {
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        sum[k].x += (double)acc[k].x;
        sum[k].y += (double)acc[k].y;
      }
      if (c == 0) {
        bsum.x += (double)bacc.x;
        bsum.y += (double)bacc.y;
      }
    }
  }
  const long long stride = (long long)cout * cin * 9 + cout;
  double* out = part + blockIdx.x * stride;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int o = 2 * og + e;
    if (o >= cout) break;
    if (c < cc) {
#pragma unroll
      for (int k = 0; k < 9; ++k) out[((long long)o * cin + c0 + c) * 9 + k] = e ? sum[k].y : sum[k].x;
    }
    if (c == 0 && c0 == 0) out[(long long)cout * cin * 9 + o] = e ? bsum.y : bsum.x;
  }
}

// dst[i] = sum over blocks of part[blk][i] in FP64: 32 entries per block, its eight warps take
// every eighth partial and their sums are added in order.
__global__ void __launch_bounds__(256) reduce_parts_kernel(const double* part, long long stride, int nblk, float* dw,
                                                           float* db, long long nw) {
  __shared__ double red[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long i = blockIdx.x * 32ll + lane;
  double s = 0.0;
  if (i < stride)
    for (int k = w; k < nblk; k += 8) s += part[k * stride + i];
  red[w][lane] = s;
  __syncthreads();
  if (w || i >= stride) return;
#pragma unroll
  for (int u = 1; u < 8; ++u) s += red[u][lane];
  if (i < nw) dw[i] = (float)s;
  else db[i - nw] = (float)s;
}

__global__ void adam_kernel(long long count, float* p, const float* g, float* m, float* v,
                            float lr, float b1, float b2, float eps, float c1, float c2) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// Targets of the warm start from a labelled EP state: out0 -> mean - y and
// out[1 + s] -> log(tau_s) + log(xi) for the five sites s.  dout = dL/dout of
// L = mean over images and pixels of w_mu (out0 - t0)^2 + (1/5) sum_s (out[1+s] - t[1+s])^2;
// loss += block sums.
__global__ void warmstart_loss_kernel(int n, long long hw, const float* out, const float* y,
                                      const float* mean, const float* tau, const float* log_xi,
                                      float w_mu, float* dout, double* loss) {
  const double inv = 1.0 / ((double)n * hw);
  double s = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)n * hw;
       i += (long long)gridDim.x * blockDim.x) {
    const long long img = i / hw, p = i - img * hw;
    const float* o = out + img * kWarmOut * hw + p;
    float* d = dout + img * kWarmOut * hw + p;
    const float r0 = o[0] - (mean[i] - y[i]);
    d[0] = (float)(2.0 * w_mu * r0 * inv);
    double acc = (double)w_mu * r0 * r0;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const float t = logf(tau[(img * 5 + k) * hw + p]) + log_xi[img];
      const float r = o[(1 + k) * hw] - t;
      d[(1 + k) * hw] = (float)(0.4 * r * inv);
      acc += 0.2 * (double)r * r;
    }
    s += acc;
  }
  __shared__ double red[256];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int k = blockDim.x / 2; k > 0; k >>= 1) {
    if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicAdd(loss, red[0] * inv);
}

inline int ew_grid(long long n) {
  long long b = (n + 255) / 256;
  return (int)(b < 1 ? 1 : (b > 65536 ? 65536 : b));
}

bool conv_args_ok(int n, int cin, int cout, int h, int w) {
  return n >= 1 && cin >= 1 && cout >= 1 && cout <= kMaxOut && h >= 1 && w >= 1 &&
         (long long)n * (cin > cout ? cin : cout) * h * w < (1ll << 40);
}

inline ep_tv_status launch_status() {
  return cudaGetLastError() == cudaSuccess ? EP_TV_OK : EP_TV_ERR_CUDA;
}

long long tiles(int h, int w) { return (long long)((w + kT - 1) / kT) * ((h + kT - 1) / kT); }

// Blocks of the weight gradient: one per tile up to one per SM of a 152-SM GPU (one is
// resident; every block writes one partial gradient).
int dw_blocks(long long n_tiles) { return (int)(n_tiles < 152 ? n_tiles : 152); }

// Raises the weight gradient's dynamic shared-memory limit (once per device).
bool dw_smem_ok() {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  std::lock_guard<std::mutex> lock(mu);
  if (!done[dev])
    done[dev] = cudaFuncSetAttribute(conv3x3_dw_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDwSmem) == cudaSuccess;
  return done[dev];
}

// Whether the ranges a .. a + na - 1 and b .. b + nb - 1 share memory.
bool overlap(const float* a, long long na, const float* b, long long nb) {
  const uintptr_t a0 = (uintptr_t)a, b0 = (uintptr_t)b;
  return a0 < b0 + sizeof(float) * (size_t)nb && b0 < a0 + sizeof(float) * (size_t)na;
}

// Output groups and tile shape by the number of output channels: 8 or 16 outputs per thread
// with tiles of 16 rows, or two groups of 16 with tiles of 8 (the same 128 threads).
template <bool kGrad>
void launch_conv(int n, int cin, int cout, int h, int w, const float* x, const float* weight, const float* bias, int relu,
                 float* y, cudaStream_t s) {
  const unsigned gx = (w + kTW - 1) / kTW, g16 = gx * ((h + 15) / 16), g8 = gx * ((h + 7) / 8);
  if (cout <= 8)
    conv3x3_kernel<8, 1, kGrad><<<dim3(g16, 1, n), 128, 0, s>>>(cin, cout, h, w, x, weight, bias, relu, y);
  else if (cout <= 16)
    conv3x3_kernel<16, 1, kGrad><<<dim3(g16, 1, n), 128, 0, s>>>(cin, cout, h, w, x, weight, bias, relu, y);
  else
    conv3x3_kernel<16, 2, kGrad><<<dim3(g8, 1, n), 128, 0, s>>>(cin, cout, h, w, x, weight, bias, relu, y);
}

}  // namespace
}  // namespace eptv

using namespace eptv;

extern "C" {

ep_tv_status ep_tv_conv3x3_forward(int32_t n, int32_t cin, int32_t cout, int32_t height,
                                   int32_t width, const float* x, const float* weight,
                                   const float* bias, int32_t relu, float* y, void* cuda_stream) {
  if (!conv_args_ok(n, cin, cout, height, width) || !x || !weight || !y || x == y) return EP_TV_ERR_ARG;
  if (n > 65535) return EP_TV_ERR_ARG;
  launch_conv<false>(n, cin, cout, height, width, x, weight, bias, relu != 0, y, (cudaStream_t)cuda_stream);
  return launch_status();
}

size_t ep_tv_conv3x3_backward_work(int32_t n, int32_t cin, int32_t cout, int32_t height,
                                   int32_t width) {
  if (!conv_args_ok(n, cin, cout, height, width)) return 0;
  const long long stride = (long long)cout * cin * 9 + cout;
  return sizeof(double) * (size_t)(dw_blocks(tiles(height, width) * n) * stride + 1) +
         sizeof(float) * (size_t)n * cout * height * width;
}

ep_tv_status ep_tv_conv3x3_backward(int32_t n, int32_t cin, int32_t cout, int32_t height,
                                    int32_t width, const float* x, const float* weight,
                                    const float* y, const float* dy, float* dx, float* dweight,
                                    float* dbias, void* work, size_t work_bytes, void* cuda_stream) {
  if (!conv_args_ok(n, cin, cout, height, width) || !x || !weight || !dy || !dweight || !dbias || !work)
    return EP_TV_ERR_ARG;
  if (n > 65535 || (dx && cin > kMaxOut)) return EP_TV_ERR_ARG;
  if (work_bytes < ep_tv_conv3x3_backward_work(n, cin, cout, height, width)) return EP_TV_ERR_ARG;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  // the partial gradients, in FP64 (the caller's scratch need only be 4-byte aligned)
  double* part = (double*)(((uintptr_t)work + 7) & ~(uintptr_t)7);
  const long long n_tiles = tiles(height, width) * n;
  const int nblk = dw_blocks(n_tiles);
  const long long stride = (long long)cout * cin * 9 + cout;
  // dx is formed last, after dweight and dbias are written and while other blocks write dx:
  // from a copy of the (masked) gradient, unless it is dy itself and no output lies on it,
  // and from a copy of the weights where dx lies on them
  const long long n_dy = (long long)n * cout * height * width, n_dx = (long long)n * cin * height * width;
  const long long n_w = (long long)cout * cin * 9;
  const bool copy_g =
      dx && (y || overlap(dx, n_dx, dy, n_dy) || overlap(dweight, n_w, dy, n_dy) || overlap(dbias, cout, dy, n_dy));
  float* g = copy_g ? (float*)(part + nblk * stride) : nullptr;
  if (!dw_smem_ok()) return EP_TV_ERR_CUDA;
  conv3x3_dw_kernel<<<dim3(nblk, (cin + 31) / 32), kDwThreads, kDwSmem, s>>>(
      cin, cout, height, width, (width + kT - 1) / kT, n_tiles, x, dy, y, g, part);
  reduce_parts_kernel<<<(unsigned)((stride + 31) / 32), 256, 0, s>>>(part, stride, nblk, dweight, dbias,
                                                                     (long long)cout * cin * 9);
  if (!dx) return launch_status();
  const float* w = weight;
  if (overlap(dx, n_dx, weight, n_w)) {
    // the partial gradients have been added up: their place holds the weights
    if (cudaMemcpyAsync(part, weight, sizeof(float) * n_w, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
      return EP_TV_ERR_CUDA;
    w = (const float*)part;
  }
  launch_conv<true>(n, cout, cin, height, width, g ? g : dy, w, nullptr, 0, dx, s);
  return launch_status();
}

ep_tv_status ep_tv_adam_step(int64_t count, float* param, const float* grad, float* m, float* v,
                             int32_t t, float lr, float beta1, float beta2, float eps,
                             void* cuda_stream) {
  if (count < 1 || !param || !grad || !m || !v || t < 1) return EP_TV_ERR_ARG;
  const float c1 = (float)(1.0 - pow((double)beta1, t)), c2 = (float)(1.0 - pow((double)beta2, t));
  adam_kernel<<<ew_grid(count), 256, 0, (cudaStream_t)cuda_stream>>>(count, param, grad, m, v, lr,
                                                                       beta1, beta2, eps, c1, c2);
  return launch_status();
}

ep_tv_status ep_tv_warmstart_loss(int32_t n, int32_t height, int32_t width, const float* out,
                                  const float* y, const float* mean, const float* tau,
                                  const float* log_xi, float w_mean, float* dout, double* loss,
                                  void* cuda_stream) {
  if (n < 1 || height < 1 || width < 1 || !out || !y || !mean || !tau || !log_xi || !dout || !loss)
    return EP_TV_ERR_ARG;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  if (cudaMemsetAsync(loss, 0, sizeof(double), s) != cudaSuccess) return EP_TV_ERR_CUDA;
  const long long hw = (long long)height * width;
  warmstart_loss_kernel<<<ew_grid(n * hw), 256, 0, s>>>(n, hw, out, y, mean, tau, log_xi, w_mean,
                                                        dout, loss);
  return launch_status();
}

}  // extern "C"
