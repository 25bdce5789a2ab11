// Training of the spatial EvSNet (stack of 3x3 convolutions + projection +
// BiLIF; the paper's temporal form is in train_temporal.cu and is dispatched
// from the entry points below) on the GPU: forward with membrane checkpoints, the paper's loss
// (Eq. 7-11) with its gradient, surrogate-gradient BPTT (Eq. 4), and Adam.
// FP32 throughout, or with BF16 weights the C -> C convolutions' forward, data
// and weight gradients on the tensor cores (train_tc.cu).
//
// Layout: B clips of K steps of H x W pixels.  Time is processed in segments of
// `ckpt_every` steps.  The forward keeps only the membrane potential V at the
// start of every segment (and the dense spikes the loss needs); the backward
// walks the segments in reverse, recomputes the segment's activations and
// membrane trajectory from the checkpoint, runs BiLIF backward through time
// inside the segment (carrying dL/dV to the previous segment), then the
// convolution backward for the segment's B x segment images.
//
// Surrogate (Eq. 4 reading): S_on = Theta(V' - Vth), S_off = Theta(-V' - Vth),
// dS_on/dV' = s(V' - Vth), dS_off/dV' = -s(-V' - Vth),
// s(x) = (alpha / 2) / (1 + (pi alpha x / 2)^2); reset V = V' - r (S_on - S_off)
// is differentiated (not detached).
#include <algorithm>
#include <mutex>
#include <cuda.h>
#include "et_internal.cuh"
#include "evsnet_common.h"
#include "f32x2.cuh"
#include "train_api.h"

namespace {

constexpr int TS = 16;          // spatial tile (TS x TS pixels per block)
constexpr int kMaxC = 16;       // channels (keeps each block's tiles under 48 KB)
constexpr float kPi = 3.14159265358979323846f;

struct Net {
  int L, C;
  float beta, vth, reset;
  const float* w;   // packed
  const float* b;
};

__host__ __device__ inline int64_t wofs(int l, int C) { return l == 0 ? 0 : 9LL * C + (int64_t)(l - 1) * 9 * C * C; }

// ------------------------------------------------------ forward conv, layer 0
// out[n][co][y][x] = ReLU(b[co] + sum_ky,kx w[co][ky][kx] X[n][y+ky-1][x+kx-1]), X read as
// l_{k+1} - l_k from the clip's log frames: image n is (clip b = n / nseg, step
// k = k0 + n % nseg).  A one-layer network also writes the projection I = bp + wp . a.
__global__ void __launch_bounds__(TS * TS)
conv_fwd(const float* __restrict__ logl, int K, int k0, int nseg, int C, int H, int W,
         const float* __restrict__ w, const float* __restrict__ b, float* __restrict__ out,
         const float* __restrict__ wp, const float* __restrict__ bp, float* __restrict__ I) {
  constexpr int Cin = 1;
  __shared__ float tin[kMaxC][TS + 2][TS + 2];
  __shared__ float tw[kMaxC * kMaxC * 9];
  const int n = blockIdx.z;
  const int tx = threadIdx.x % TS, ty = threadIdx.x / TS;
  const int x0 = blockIdx.x * TS, y0 = blockIdx.y * TS;
  const int64_t hw = (int64_t)H * W;
  for (int i = threadIdx.x; i < C * Cin * 9; i += TS * TS) tw[i] = w[i];
  for (int i = threadIdx.x; i < Cin * (TS + 2) * (TS + 2); i += TS * TS) {
    const int ci = i / ((TS + 2) * (TS + 2)), r = i % ((TS + 2) * (TS + 2));
    const int yy = y0 - 1 + r / (TS + 2), xx = x0 - 1 + r % (TS + 2);
    float v = 0.0f;
    if (yy >= 0 && yy < H && xx >= 0 && xx < W) {
      const int64_t g = (int64_t)yy * W + xx;
      const int bc = n / nseg, k = k0 + n % nseg;
      const float* lf = logl + (int64_t)bc * (K + 1) * hw;
      v = lf[(int64_t)(k + 1) * hw + g] - lf[(int64_t)k * hw + g];
    }
    tin[ci][r / (TS + 2)][r % (TS + 2)] = v;
  }
  __syncthreads();
  const int x = x0 + tx, y = y0 + ty;
  if (x >= W || y >= H) return;
  float Iv = bp ? bp[0] : 0.0f;
  for (int co = 0; co < C; ++co) {
    float acc = b[co];
    for (int ci = 0; ci < Cin; ++ci) {
      const float* wr = tw + (co * Cin + ci) * 9;
#pragma unroll
      for (int t = 0; t < 9; ++t) acc += wr[t] * tin[ci][ty + t / 3][tx + t % 3];
    }
    const float a = fmaxf(acc, 0.0f);
    out[((int64_t)n * C + co) * hw + (int64_t)y * W + x] = a;
    if (I) Iv += wp[co] * a;
  }
  if (I) I[(int64_t)n * hw + (int64_t)y * W + x] = Iv;
}

// ------------------------------------------------------------ BiLIF, forward
// One thread per (clip, pixel): walks the segment's steps.
__global__ void bilif_fwd(const float* __restrict__ I, int B, int K, int k0, int nseg, int64_t hw,
                          float beta, float vth, float reset, float* __restrict__ V,
                          float* __restrict__ V_ckpt, int seg, int n_ckpt, int8_t* __restrict__ spikes,
                          float* __restrict__ S_on, float* __restrict__ S_off, float* __restrict__ I_out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)B * hw) return;
  const int bc = (int)(i / hw);
  const int64_t p = i % hw;
  float v = V[i];
  V_ckpt[((int64_t)bc * n_ckpt + seg) * hw + p] = v;
  for (int s = 0; s < nseg; ++s) {
    const float Iv = I[((int64_t)bc * nseg + s) * hw + p];
    const float vp = beta * v + Iv;
    const float on = vp >= vth ? 1.0f : 0.0f, off = -vp >= vth ? 1.0f : 0.0f;
    v = vp - reset * (on - off);
    const int64_t o = ((int64_t)bc * K + k0 + s) * hw + p;
    spikes[o] = (int8_t)(on - off);
    if (S_on) { S_on[o] = on; S_off[o] = off; }
    if (I_out) I_out[o] = Iv;
  }
  V[i] = v;
}

// ----------------------------------------------------------- BiLIF, backward
__device__ __forceinline__ float sg(float x, float alpha) {
  const float u = 0.5f * kPi * alpha * x;
  return 0.5f * alpha / (1.0f + u * u);
}

// Recomputes V' over the segment from its checkpoint, then runs the reverse
// recursion; writes dL/dI per step and carries dL/dV to the previous segment.
__global__ void bilif_bwd(const float* __restrict__ I, int B, int K, int k0, int nseg, int64_t hw,
                          float beta, float vth, float reset, float alpha,
                          const float* __restrict__ V_ckpt, int seg, int n_ckpt,
                          const float* __restrict__ dSon, const float* __restrict__ dSoff,
                          float* __restrict__ gV, float* __restrict__ dI) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)B * hw) return;
  const int bc = (int)(i / hw);
  const int64_t p = i % hw;
  float vps[kMaxSeg];
  float v = V_ckpt[((int64_t)bc * n_ckpt + seg) * hw + p];
  for (int s = 0; s < nseg; ++s) {
    const float vp = beta * v + I[((int64_t)bc * nseg + s) * hw + p];
    const float on = vp >= vth ? 1.0f : 0.0f, off = -vp >= vth ? 1.0f : 0.0f;
    v = vp - reset * (on - off);
    vps[s] = vp;
  }
  float g = gV[i];
  for (int s = nseg - 1; s >= 0; --s) {
    const float vp = vps[s];
    const float a = sg(vp - vth, alpha), c = sg(-vp - vth, alpha);
    const int64_t o = ((int64_t)bc * K + k0 + s) * hw + p;
    const float gvp = g * (1.0f - reset * (a + c)) + dSon[o] * a - dSoff[o] * c;
    dI[((int64_t)bc * nseg + s) * hw + p] = gvp;
    g = gvp * beta;
  }
  gV[i] = g;
}

// ------------------------------------------------------ projection backward
// dz_{L-1}[c] = dI wp[c] 1(a > 0); grad wp[c] += sum dI a[c]; grad bp += sum dI.
__global__ void __launch_bounds__(256)
proj_bwd(const float* __restrict__ dI, const float* __restrict__ a, int N, int C, int64_t hw,
         const float* __restrict__ wp, float* __restrict__ dz, float* __restrict__ gwp,
         float* __restrict__ gbp) {
  __shared__ float red[kMaxC + 1][8];
  float accw[kMaxC + 1];
  for (int c = 0; c <= C; ++c) accw[c] = 0.0f;
  const int64_t total = (int64_t)N * hw;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t n = i / hw, p = i % hw;
    const float d = dI[i];
    accw[C] += d;
    for (int c = 0; c < C; ++c) {
      const int64_t o = (n * C + c) * hw + p;
      const float av = a[o];
      accw[c] += d * av;
      dz[o] = av > 0.0f ? d * wp[c] : 0.0f;
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int c = 0; c <= C; ++c) {
    float v = accw[c];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    if (lane == 0) red[c][warp] = v;
  }
  __syncthreads();
  if (threadIdx.x <= C) {
    float v = 0.0f;
    for (int wv = 0; wv < 8; ++wv) v += red[threadIdx.x][wv];
    if (threadIdx.x < C) atomicAdd(gwp + threadIdx.x, v);
    else atomicAdd(gbp, v);
  }
}

// ------------------------------------------------ conv weight backward, layer 0
// grad w[co][t] += sum_n,y,x dz[n][co][y][x] X[n][y+ky-1][x+kx-1] (X from the log
// frames as in the forward); grad b[co] += sum dz.  Persistent blocks
// accumulate over many tiles in registers, then one atomic per entry per block.
__global__ void __launch_bounds__(TS * TS)
conv_bwd_weight(const float* __restrict__ dz, const float* __restrict__ logl, int K, int k0,
                int nseg, int N, int C, int H, int W, float* __restrict__ gw, float* __restrict__ gb) {
  constexpr int Cin = 1;
  __shared__ float td[kMaxC][TS][TS];
  __shared__ float tin[kMaxC][TS + 2][TS + 2];
  constexpr int kPer = (kMaxC * kMaxC * 9 + kMaxC + TS * TS - 1) / (TS * TS);
  float acc[kPer];
#pragma unroll
  for (int j = 0; j < kPer; ++j) acc[j] = 0.0f;
  const int64_t hw = (int64_t)H * W;
  const int tiles_x = (W + TS - 1) / TS, tiles_y = (H + TS - 1) / TS;
  const int64_t ntiles = (int64_t)N * tiles_x * tiles_y;
  const int nent = C * Cin * 9 + C;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int n = (int)(tile / (tiles_x * tiles_y));
    const int tt = (int)(tile % (tiles_x * tiles_y));
    const int x0 = (tt % tiles_x) * TS, y0 = (tt / tiles_x) * TS;
    __syncthreads();
    for (int i = threadIdx.x; i < C * TS * TS; i += TS * TS) {
      const int co = i / (TS * TS), r = i % (TS * TS);
      const int yy = y0 + r / TS, xx = x0 + r % TS;
      td[co][r / TS][r % TS] = (yy < H && xx < W) ? dz[((int64_t)n * C + co) * hw + (int64_t)yy * W + xx] : 0.0f;
    }
    for (int i = threadIdx.x; i < Cin * (TS + 2) * (TS + 2); i += TS * TS) {
      const int ci = i / ((TS + 2) * (TS + 2)), r = i % ((TS + 2) * (TS + 2));
      const int yy = y0 - 1 + r / (TS + 2), xx = x0 - 1 + r % (TS + 2);
      float v = 0.0f;
      if (yy >= 0 && yy < H && xx >= 0 && xx < W) {
        const int64_t g = (int64_t)yy * W + xx;
        const int bc = n / nseg, k = k0 + n % nseg;
        const float* lf = logl + (int64_t)bc * (K + 1) * hw;
        v = lf[(int64_t)(k + 1) * hw + g] - lf[(int64_t)k * hw + g];
      }
      tin[ci][r / (TS + 2)][r % (TS + 2)] = v;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      const int e = threadIdx.x + j * TS * TS;
      if (e >= nent) break;
      float s = 0.0f;
      if (e < C * Cin * 9) {
        const int co = e / (Cin * 9), ci = (e / 9) % Cin, t = e % 9;
        const int ky = t / 3, kx = t % 3;
        for (int py = 0; py < TS; ++py)
          for (int px = 0; px < TS; ++px) s += td[co][py][px] * tin[ci][py + ky][px + kx];
      } else {
        const int co = e - C * Cin * 9;
        for (int py = 0; py < TS; ++py)
          for (int px = 0; px < TS; ++px) s += td[co][py][px];
      }
      acc[j] += s;
    }
  }
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const int e = threadIdx.x + j * TS * TS;
    if (e >= nent) break;
    if (e < C * Cin * 9) atomicAdd(gw + e, acc[j]);
    else atomicAdd(gb + (e - C * Cin * 9), acc[j]);
  }
}

// ------------------------------------------- C -> C layers, register-blocked
// FP32 convolutions with C input channels (all layers but the first), channels
// zero-padded to 16.  What bounds them is the FP32 pipe once shared memory is read
// rarely enough: a warp's 16-byte load takes 4 clk of the SM's 128 bytes per clk
// whatever its addresses, as long as 4 multiply-adds of the SM.
constexpr int CP = 16;
constexpr int CW = 32;             // columns of a tile: a warp's lanes
constexpr int kRows = 8;           // rows of one warp's forward tile
constexpr int kPitch = CW + 2;     // a staged row with its halo
constexpr int kWTap = CP * CP + 4; // words of a tap's staged weights (4 apart: fewer bank conflicts when staging)

// 4 bytes global -> shared without a register; zero when !ok
__device__ __forceinline__ void copy4(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(ok ? 4 : 0));
}

// Forward (out = ReLU(b + conv(in)); the last layer also I = bp + wp . out) or, kBwd,
// the data gradient: dzp[ci] = (sum_co,t w[co][ci][t] dz[co] at the mirrored tap)
// 1(mask > 0), i.e. the same sum with weights w'[t][co][ci] = w[co][ci][8 - t].
// A block of two warps owns 8 rows x 32 columns of an image; the input lies in
// shared memory by channel planes, a lane owns a column: 8 rows x 8 output
// channels (a half per warp) of sums as FP32 pairs, so that 8 four-byte loads and two
// 16-byte weight loads feed 64 multiply-adds (16 clk of shared memory for 16 of
// the FP32 pipe; 4 positions x 4 channels took 32).  Every sum runs over taps, then
// channels, in one chain of fused multiply-adds.  Up to seven blocks per SM hide each
// other's staging; 32 images of 93 x 67 are one wave of 864 blocks.  Average launch over
// a training pass on 50 steps of two such clips (segments of 32 and 4 images): forward
// 41 -> 25 us, data gradient 42 -> 31.  Single multiply-adds instead of pairs: 27 and 33;
// four warps on 16 rows (480 blocks, 3.2 per SM): 30 and 41.
template <bool kBwd>
__global__ void __launch_bounds__(64, 7)
conv16(const float* __restrict__ in, int C, int H, int W, const float* __restrict__ w,
       const float* __restrict__ b, float* __restrict__ out, const float* __restrict__ wp,
       const float* __restrict__ bp, float* __restrict__ I, const float* __restrict__ mask) {
  constexpr int kSR = kRows + 2, kPlane = kSR * kPitch;
  __shared__ __align__(16) float sw[9 * kWTap];     // [t][from][to]
  __shared__ float sx[CP * kPlane];                 // [channel][row][column]
  __shared__ uint32_t son[2][kBwd ? 64 : 1];
  const int n = blockIdx.z, tx = (W + CW - 1) / CW, x0 = blockIdx.x % tx * CW, y0 = blockIdx.x / tx * kRows;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t hw = (int64_t)H * W;
  const float* img = in + (int64_t)n * C * hw + (int64_t)(y0 - 1) * W + x0 - 1;
  {
    const bool okx = x0 - 1 + lane >= 0 && x0 - 1 + lane < W;
#pragma unroll 1
    for (int c = warp * 8; c < warp * 8 + 8; ++c) {
      const float* src = img + c * hw + lane;
      float* dst = sx + c * kPlane + lane;
#pragma unroll
      for (int r = 0; r < kSR; ++r) {
        const bool ok = okx && c < C && (unsigned)(y0 - 1 + r) < (unsigned)H;
        copy4(dst + r * kPitch, ok ? src + r * W : in, ok);
      }
    }
    // the two columns right of the lanes', lane = (row, column) of a channel
    const int r = tid >> 1 & 15, col = CW + (tid & 1);
    const bool ok = (unsigned)(y0 - 1 + r) < (unsigned)H && x0 - 1 + col < W;
    if (r < kSR)
#pragma unroll 4
      for (int c = tid >> 5; c < CP; c += 2)
        copy4(sx + c * kPlane + r * kPitch + col, ok && c < C ? img + c * hw + r * W + col : in, ok && c < C);
  }
  // weights [co][ci][t] -> [t][from][to], zero beyond C: a warp reads runs of 4 x 9 words
  {
    float v[4][9];
    int at[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int e = tid + 64 * k, co = (e & 7) + (e >> 2 & 8), ci = (e >> 3 & 3) + (e >> 4 & 12);
      const bool ok = co < C && ci < C;
      at[k] = kBwd ? co * CP + ci : ci * CP + co;
#pragma unroll
      for (int t = 0; t < 9; ++t) v[k][t] = ok ? w[(co * C + ci) * 9 + t] : 0.0f;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int t = 0; t < 9; ++t) sw[(kBwd ? 8 - t : t) * kWTap + at[k]] = v[k][t];
  }
  const int c0 = warp * 8, x = x0 + lane, y = y0;
  const int nr = x < W ? H - y : 0;                 // the lane's rows inside the image
  const int64_t o = ((int64_t)n * C + c0) * hw + (int64_t)y * W + x;
  if (kBwd)                                         // mask > 0, bit 8 (channel % 4) + row
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      float m[4][kRows];
      uint32_t bits = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int r = 0; r < kRows; ++r)
          m[j][r] = r < nr && c0 + 4 * q + j < C ? mask[o + (4 * q + j) * hw + r * W] : 0.0f;
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int r = 0; r < kRows; ++r) bits |= (m[j][r] > 0.0f ? 1u : 0u) << (8 * j + r);
      son[q][tid] = bits;
    }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();

  f32x2 acc[kRows / 2][8];                          // [row pair][channel]
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const float bc = !kBwd && c0 + c < C ? b[c0 + c] : 0.0f;
#pragma unroll
    for (int r = 0; r < kRows / 2; ++r) acc[r][c] = pack2f(bc, bc);
  }
#pragma unroll 1
  for (int t = 0; t < 9; ++t) {
    const float* xt = sx + t / 3 * kPitch + lane + t % 3;
    const float* wt = sw + t * kWTap + c0;
#pragma unroll
    for (int ci = 0; ci < CP; ++ci) {
      const float4 wa = *reinterpret_cast<const float4*>(wt + ci * CP);
      const float4 wb = *reinterpret_cast<const float4*>(wt + ci * CP + 4);
      const float wc[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
      f32x2 v[kRows / 2];
#pragma unroll
      for (int r = 0; r < kRows / 2; ++r)
        v[r] = pack2f(xt[ci * kPlane + 2 * r * kPitch], xt[ci * kPlane + (2 * r + 1) * kPitch]);
#pragma unroll
      for (int c = 0; c < 8; ++c)
#pragma unroll
        for (int r = 0; r < kRows / 2; ++r) acc[r][c] = fma2(pack2f(wc[c], wc[c]), v[r], acc[r][c]);
    }
  }
  float pI[kRows], p4[kRows];
#pragma unroll
  for (int q = 0; q < 2; ++q) {                     // four channels at a time
    float a[4][kRows];
    const uint32_t on = kBwd ? son[q][tid] : 0;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int r = 0; r < kRows / 2; ++r) unpack2f(acc[r][4 * q + j], a[j][2 * r], a[j][2 * r + 1]);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const bool okc = c0 + 4 * q + j < C;
      // Eq. 6 with sums of four channels, then (s0 + s1) + (s2 + s3)
      const float wq = !kBwd && I && okc ? wp[c0 + 4 * q + j] : 0.0f;
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        const float v = kBwd ? (on >> (8 * j + r) & 1u ? a[j][r] : 0.0f) : fmaxf(a[j][r], 0.0f);
        if (okc && r < nr) out[o + (4 * q + j) * hw + r * W] = v;
        if (!kBwd) p4[r] = j == 0 ? wq * v : fmaf(wq, v, p4[r]);
      }
    }
#pragma unroll
    for (int r = 0; r < kRows; ++r) pI[r] = q == 0 ? p4[r] : pI[r] + p4[r];
  }
  if (!kBwd && I) {
    __syncthreads();               // every warp is done with sx
    if (c0)
#pragma unroll
      for (int r = 0; r < kRows; ++r) sx[r * CW + lane] = pI[r];
    __syncthreads();
    if (!c0)
#pragma unroll
      for (int r = 0; r < kRows; ++r)
        if (r < nr)
          I[(int64_t)n * hw + (int64_t)(y + r) * W + x] = bp[0] + (pI[r] + sx[r * CW + lane]);
  }
}

dim3 conv16_grid(int H, int W, int N) {
  return dim3((unsigned)((int64_t)((W + CW - 1) / CW) * ((H + kRows - 1) / kRows)), 1, N);
}

// weight backward: grad w[co][ci][t] += sum_n,p dz[n][co][p] in[n][ci][p + off(t)],
// grad b[co] += sum dz.  Persistent blocks over tiles of 8 rows x 32 columns, staged
// channel-interleaved (16 floats per position, its four 16-byte groups permuted by
// the column so that staging stores and reads are free of bank conflicts).  Warp
// (ky, row pair), half-warp = one row, lane = (output quad, input quad): it walks the
// row's 32 positions with the last three input quads in registers and sums 4 x 4
// channels for the three taps of row ky: two 16-byte loads per 48 multiply-adds (8
// clk of shared memory for 12 of the FP32 pipe; a thread per tap and quads, without
// the window, had 8 for 4 and one block's 256 positions in one chain).  Sums stay
// in registers until the block's last tile; one atomic per entry and block then.
// Average launch over the pass above: 97 -> 31 us.  Staging by 4-byte cp.async into two
// buffers was slower (33 us; 38 with plain channel planes read 4 bytes at a time).
constexpr int kWRows = 8;
constexpr int kWThreads = 3 * (kWRows / 2) * 32;

__global__ void __launch_bounds__(kWThreads, 2)
conv16_bwd_weight(const float* __restrict__ dz, const float* __restrict__ in, int N, int C, int H,
                  int W, float* __restrict__ gw, float* __restrict__ gb) {
  constexpr int kWarps = kWThreads / 32, kXRows = kWRows + 2;
  constexpr int kPart = 9 * CP * CP;              // a row pair's sums
  __shared__ __align__(16) float sh[(kWRows * CW + kXRows * kPitch) * CP];
  __shared__ float sb[kWarps][4];
  static_assert(kWRows / 2 * kPart <= (kWRows * CW + kXRows * kPitch) * CP, "the sums fit the tiles' place");
  float* const sd = sh;
  float* const sx = sh + kWRows * CW * CP;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ky = warp % 3, row = warp / 3 * 2 + (lane >> 4), cq = lane & 3, iq = (lane >> 2) & 3;
  const int g = warp & 3;                         // the channel quad this warp stages (kWarps % 4 == 0)
  static_assert(kWarps % 4 == 0, "a warp stages one channel quad");
  const int64_t hw = (int64_t)H * W;
  const int tiles_x = (W + CW - 1) / CW, tiles_y = (H + kWRows - 1) / kWRows;
  const int64_t ntiles = (int64_t)N * tiles_x * tiles_y;
  const auto slot = [](int col, int q) { return col * CP + 4 * (q ^ ((col >> 1) & 3)); };
  f32x2 acc[3][4][2] = {};                        // [kx][output channel][input channel pair]
  float bs[4] = {};
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int n = (int)(tile / (tiles_x * tiles_y));
    const int tt = (int)(tile % (tiles_x * tiles_y));
    const int x0 = (tt % tiles_x) * CW, y0 = (tt / tiles_x) * kWRows;
    const float* dn = dz + ((int64_t)n * C + 4 * g) * hw;
    const float* xn = in + ((int64_t)n * C + 4 * g) * hw;
    float vd[kWRows * 4 / kWarps + 1][4];
#pragma unroll
    for (int k = 0; k < kWRows * 4 / kWarps + 1; ++k) {
      const int r = (warp + k * kWarps) >> 2, yy = y0 + r, xx = x0 + lane;
      const bool ok = r < kWRows && yy < H && xx < W;
#pragma unroll
      for (int j = 0; j < 4; ++j) vd[k][j] = ok && 4 * g + j < C ? dn[j * hw + (int64_t)yy * W + xx] : 0.0f;
    }
    __syncthreads();                              // the last tile's reads
#pragma unroll
    for (int k = 0; k < kWRows * 4 / kWarps + 1; ++k) {
      const int r = (warp + k * kWarps) >> 2;
      if (r < kWRows)
        *reinterpret_cast<float4*>(sd + r * CW * CP + slot(lane, g)) =
            make_float4(vd[k][0], vd[k][1], vd[k][2], vd[k][3]);
#pragma unroll
      for (int j = 0; j < 4; ++j) bs[j] += vd[k][j];
    }
    float vx[kXRows * 4 / kWarps + 1][4];
#pragma unroll
    for (int k = 0; k < kXRows * 4 / kWarps + 1; ++k) {
      const int r = (warp + k * kWarps) >> 2, yy = y0 - 1 + r, xx = x0 - 1 + lane;
      const bool ok = r < kXRows && yy >= 0 && yy < H && xx >= 0 && xx < W;
#pragma unroll
      for (int j = 0; j < 4; ++j) vx[k][j] = ok && 4 * g + j < C ? xn[j * hw + (int64_t)yy * W + xx] : 0.0f;
    }
#pragma unroll
    for (int k = 0; k < kXRows * 4 / kWarps + 1; ++k) {
      const int r = (warp + k * kWarps) >> 2;
      if (r < kXRows)
        *reinterpret_cast<float4*>(sx + r * kPitch * CP + slot(lane, g)) =
            make_float4(vx[k][0], vx[k][1], vx[k][2], vx[k][3]);
    }
    if (tid < kXRows * 8) {                       // the two columns right of the lanes'
      const int q = tid & 3, col = CW + ((tid >> 2) & 1), r = tid >> 3, yy = y0 - 1 + r, xx = x0 - 1 + col;
      const bool ok = yy >= 0 && yy < H && xx < W;
      const float* src = in + ((int64_t)n * C + 4 * q) * hw + (int64_t)yy * W + xx;
      float v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = ok && 4 * q + j < C ? src[j * hw] : 0.0f;
      *reinterpret_cast<float4*>(sx + r * kPitch * CP + slot(col, q)) = make_float4(v[0], v[1], v[2], v[3]);
    }
    __syncthreads();
    if (y0 + row < H) {
      const float* dr = sd + row * CW * CP;
      const float* xr = sx + (row + ky) * kPitch * CP;
      ulonglong2 win[3];
      win[0] = *reinterpret_cast<const ulonglong2*>(xr + slot(0, iq));
      win[1] = *reinterpret_cast<const ulonglong2*>(xr + slot(1, iq));
      // no position right of the image: its zero times an infinity in the image's
      // last column would be NaN
      const int np = W - x0;
#pragma unroll
      for (int p = 0; p < CW; ++p) {
        if (p >= np) break;
        win[(p + 2) % 3] = *reinterpret_cast<const ulonglong2*>(xr + slot(p + 2, iq));
        const float4 d = *reinterpret_cast<const float4*>(dr + slot(p, cq));
        const f32x2 d2[4] = {pack2f(d.x, d.x), pack2f(d.y, d.y), pack2f(d.z, d.z), pack2f(d.w, d.w)};
#pragma unroll
        for (int kx = 0; kx < 3; ++kx)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            acc[kx][j][0] = fma2(d2[j], win[(p + kx) % 3].x, acc[kx][j][0]);
            acc[kx][j][1] = fma2(d2[j], win[(p + kx) % 3].y, acc[kx][j][1]);
          }
      }
    }
  }
  // the block's sums: a warp's two rows by shuffle, the four row pairs in shared memory
  __syncthreads();
#pragma unroll
  for (int kx = 0; kx < 3; ++kx)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float v[4];
      unpack2f(acc[kx][j][0], v[0], v[1]);
      unpack2f(acc[kx][j][1], v[2], v[3]);
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] += __shfl_xor_sync(0xFFFFFFFFu, v[e], 16);
      if (lane < 16)
        *reinterpret_cast<float4*>(sh + (((warp / 3 * 3 + kx) * 4 + j) * 48 + ky * 16 + lane) * 4) =
            make_float4(v[0], v[1], v[2], v[3]);
    }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) bs[j] += __shfl_xor_sync(0xFFFFFFFFu, bs[j], o);
    if (lane == 0) sb[warp][j] = bs[j];
  }
  __syncthreads();
  for (int i = tid; i < 9 * C * C; i += kWThreads) {
    const int t = i % 9, ci = i / 9 % C, co = i / 9 / C;
    const float* s = sh + (((t % 3) * 4 + (co & 3)) * 48 + t / 3 * 16 + (ci >> 2) * 4 + (co >> 2)) * 4 + (ci & 3);
    atomicAdd(gw + i, (s[0] + s[kPart]) + (s[2 * kPart] + s[3 * kPart]));
  }
  if (tid < C) atomicAdd(gb + tid, (sb[tid >> 2][tid & 3] + sb[(tid >> 2) + 4][tid & 3]) + sb[(tid >> 2) + 8][tid & 3]);
}

// ------------------------------------------------------------ loss (Eq. 7-11)
// One thread per (clip, pixel) over the K steps:
//   L = sum over polarities of 1/2 [EMD(E, S) + EMD(E_rev, S_rev)] + lambda |sum|S| - sum|E||,
//   EMD(E, S) = (1/K) sum_i |c_i|, c_i = sum_{j<=i} (S_j - E_j),
// averaged over the B H W pixels.  The reversed EMD uses c'_i = T - c_{i-1}.
// Gradients: dEMD/dS_j = (1/K) sum_{i>=j} sgn c_i, dEMD_rev/dS_j = (1/K) sum_{i<=j} sgn c'_i.
__device__ __forceinline__ float sgnf(float x) { return x > 0.0f ? 1.0f : (x < 0.0f ? -1.0f : 0.0f); }

__global__ void __launch_bounds__(256)
emd_count_loss(const int8_t* __restrict__ spikes, const float* __restrict__ E, int B, int K,
               int64_t hw, float lambda, float* __restrict__ loss, float* __restrict__ dSon,
               float* __restrict__ dSoff) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t npx = (int64_t)B * hw;
  float l_emd = 0.0f, l_cnt = 0.0f;
  if (i < npx) {
    const int bc = (int)(i / hw);
    const int64_t p = i % hw;
    const int64_t base = (int64_t)bc * K * hw + p;
    // pass 1: totals
    float Ton = 0.0f, Toff = 0.0f, nS = 0.0f, nE = 0.0f;
    for (int k = 0; k < K; ++k) {
      const int s = spikes[base + k * hw];
      const float e = E[base + k * hw];
      const float son = s > 0 ? 1.0f : 0.0f, soff = s < 0 ? 1.0f : 0.0f;
      Ton += son - fmaxf(e, 0.0f);
      Toff += soff - fmaxf(-e, 0.0f);
      nS += son + soff;
      nE += fabsf(e);
    }
    // pass 2: losses and the totals of sgn c
    float con = 0.0f, coff = 0.0f, Son = 0.0f, Soff = 0.0f, lon = 0.0f, loff = 0.0f;
    for (int k = 0; k < K; ++k) {
      const int s = spikes[base + k * hw];
      const float e = E[base + k * hw];
      const float rpon = Ton - con, rpoff = Toff - coff;          // c'_k = T - c_{k-1}
      con += (s > 0 ? 1.0f : 0.0f) - fmaxf(e, 0.0f);
      coff += (s < 0 ? 1.0f : 0.0f) - fmaxf(-e, 0.0f);
      lon += fabsf(con) + fabsf(rpon);
      loff += fabsf(coff) + fabsf(rpoff);
      Son += sgnf(con);
      Soff += sgnf(coff);
    }
    const float invK = 1.0f / (float)K, inv = 1.0f / (float)npx;
    l_emd = 0.5f * invK * (lon + loff);
    l_cnt = fabsf(nS - nE);
    const float gc = lambda * sgnf(nS - nE);
    // pass 3: gradients
    con = coff = 0.0f;
    float pre_on = 0.0f, pre_off = 0.0f, rev_on = 0.0f, rev_off = 0.0f;
    for (int k = 0; k < K; ++k) {
      const int s = spikes[base + k * hw];
      const float e = E[base + k * hw];
      const float rpon = Ton - con, rpoff = Toff - coff;
      rev_on += sgnf(rpon);
      rev_off += sgnf(rpoff);
      const float g_on = 0.5f * invK * ((Son - pre_on) + rev_on) + gc;
      const float g_off = 0.5f * invK * ((Soff - pre_off) + rev_off) + gc;
      dSon[base + k * hw] = g_on * inv;
      dSoff[base + k * hw] = g_off * inv;
      con += (s > 0 ? 1.0f : 0.0f) - fmaxf(e, 0.0f);
      coff += (s < 0 ? 1.0f : 0.0f) - fmaxf(-e, 0.0f);
      pre_on += sgnf(con);
      pre_off += sgnf(coff);
    }
    l_emd *= inv;
    l_cnt *= inv;
  }
  // block reduction, one atomic per block and term
  __shared__ float r1[8], r2[8];
  for (int o = 16; o > 0; o >>= 1) {
    l_emd += __shfl_xor_sync(0xFFFFFFFFu, l_emd, o);
    l_cnt += __shfl_xor_sync(0xFFFFFFFFu, l_cnt, o);
  }
  if ((threadIdx.x & 31) == 0) { r1[threadIdx.x >> 5] = l_emd; r2[threadIdx.x >> 5] = l_cnt; }
  __syncthreads();
  if (threadIdx.x == 0) {
    float a = 0.0f, c = 0.0f;
    for (int wv = 0; wv < (int)(blockDim.x >> 5); ++wv) { a += r1[wv]; c += r2[wv]; }
    atomicAdd(loss + 1, a);
    atomicAdd(loss + 2, c);
    atomicAdd(loss, a + lambda * c);
  }
}

// ------------------------------------------------------------------- Adam
__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int64_t n, float lr, float b1, float b2,
                            float eps, float bc1, float bc2) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.0f - b1) * gi;
  const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
}

struct Workspace {
  float* act[kMaxLayers];   // [nseg B][C][H][W] per layer
  float* I;                 // [nseg B][H][W]
  float* dI;                // [nseg B][H][W]
  float* dz[2];             // [nseg B][C][H][W]
  float* V;                 // [B][H][W] running membrane / carried gradient
  size_t bytes;
};

bool layout(const et_evsnet_weights* net, const et_train_shape* sh, char* base, Workspace* ws) {
  const int64_t hw = (int64_t)sh->H * sh->W;
  const int64_t img = (int64_t)sh->ckpt_every * sh->B;
  size_t off = 0;
  auto take = [&](size_t bytes) -> float* {
    float* p = base ? reinterpret_cast<float*>(base + off) : nullptr;
    off += (bytes + 255) & ~(size_t)255;
    return p;
  };
  for (int l = 0; l < net->n_layers; ++l) ws->act[l] = take(sizeof(float) * img * net->C * hw);
  ws->I = take(sizeof(float) * img * hw);
  ws->dI = take(sizeof(float) * img * hw);
  ws->dz[0] = take(sizeof(float) * img * net->C * hw);
  ws->dz[1] = take(sizeof(float) * img * net->C * hw);
  ws->V = take(sizeof(float) * sh->B * hw);
  ws->bytes = off;
  return true;
}

int check(const et_evsnet_weights* net, const et_train_shape* sh) {
  if (!net || !sh || !net->w || !net->b) return ET_ERR_ARG;
  if (sh->B < 1 || sh->K < 1 || sh->H < 1 || sh->W < 1 || sh->ckpt_every < 1) return ET_ERR_ARG;
  if (net->n_layers < 1 || net->n_layers > kMaxLayers || net->C < 1) return ET_ERR_UNIMPLEMENTED;
  const bool spatial = net->kind == ET_NET_STACK && net->ks == 3 && net->kt == 1 && net->C <= kMaxC &&
                       net->ks0 == 0;
  if (!spatial && !et_train_is_temporal(net)) return ET_ERR_UNIMPLEMENTED;
  // BF16: the C -> C convolutions of the spatial form, or of the temporal form
  // (kt <= 7), on the tensor cores
  if (net->dtype != ET_F32 &&
      !(net->dtype == ET_BF16 && (spatial || (!spatial && et_train_tct_supported(net)))))
    return ET_ERR_UNIMPLEMENTED;
  if (sh->ckpt_every > kMaxSeg) return ET_ERR_UNIMPLEMENTED;
  return ET_OK;
}

// forward of one segment's convolutions: activations and I for the B x nseg images
int seg_forward(const float* logl, const et_train_shape* sh, const et_evsnet_weights* net,
                const Workspace& ws, int k0, int nseg, cudaStream_t st) {
  const int H = sh->H, W = sh->W, C = net->C, L = net->n_layers;
  const int N = sh->B * nseg;
  const dim3 grid((W + TS - 1) / TS, (H + TS - 1) / TS, N), grid16 = conv16_grid(H, W, N);
  const float* wproj = net->w + wofs(L, C);
  const float* bproj = net->b + (int64_t)L * C;
  for (int l = 0; l < L; ++l) {
    const bool last = l == L - 1;
    if (l == 0)
      conv_fwd<<<grid, TS * TS, 0, st>>>(logl, sh->K, k0, nseg, C, H, W, net->w, net->b, ws.act[0],
                                         wproj, bproj, last ? ws.I : nullptr);
    else if (net->dtype == ET_BF16) {
      const int rc = et_train_tc_conv(ws.act[l - 1], N, C, H, W, net->w + wofs(l, C),
                                      net->b + (int64_t)l * C, ws.act[l], wproj, bproj,
                                      last ? ws.I : nullptr, nullptr, false, st);
      if (rc != ET_OK) return rc;
    } else
      conv16<false><<<grid16, 64, 0, st>>>(ws.act[l - 1], C, H, W, net->w + wofs(l, C),
                                            net->b + (int64_t)l * C, ws.act[l], wproj, bproj,
                                            last ? ws.I : nullptr, nullptr);
    ET_CHECK_LAUNCH();
  }
  return ET_OK;
}

}  // namespace

extern "C" int et_train_workspace_bytes(const et_evsnet_weights* net, const et_train_shape* sh,
                                        size_t* bytes) {
  const int rc = check(net, sh);
  if (rc != ET_OK) return rc;
  if (!bytes) return ET_ERR_ARG;
  if (et_train_is_temporal(net)) {
    *bytes = et_train_temporal_bytes(net, sh);
    return ET_OK;
  }
  Workspace ws{};
  layout(net, sh, nullptr, &ws);
  *bytes = ws.bytes;
  return ET_OK;
}

extern "C" int et_evsnet_train_forward(const float* logl, const et_train_shape* sh,
                                       const et_evsnet_weights* net, int8_t* spikes, float* S_on,
                                       float* S_off, float* V_ckpt, float* I_out, void* workspace,
                                       size_t ws_bytes, void* stream_) {
  int rc = check(net, sh);
  if (rc != ET_OK) return rc;
  if (!logl || !spikes || !V_ckpt || !workspace || ((S_on == nullptr) != (S_off == nullptr)))
    return ET_ERR_ARG;
  if (reinterpret_cast<uintptr_t>(workspace) % sizeof(float) != 0) return ET_ERR_ARG;
  if (et_train_is_temporal(net)) {
    if (ws_bytes < et_train_temporal_bytes(net, sh)) return ET_ERR_ARG;
    return et_train_temporal_forward(logl, sh, net, spikes, S_on, S_off, V_ckpt, I_out, workspace,
                                     (cudaStream_t)stream_);
  }
  Workspace ws{};
  layout(net, sh, nullptr, &ws);
  if (ws_bytes < ws.bytes) return ET_ERR_ARG;
  layout(net, sh, static_cast<char*>(workspace), &ws);
  cudaStream_t st = (cudaStream_t)stream_;
  const int64_t hw = (int64_t)sh->H * sh->W;
  const int n_ckpt = (sh->K + sh->ckpt_every - 1) / sh->ckpt_every;
  ET_CHECK_CUDA(cudaMemsetAsync(ws.V, 0, sizeof(float) * sh->B * hw, st));
  for (int s = 0; s < n_ckpt; ++s) {
    const int k0 = s * sh->ckpt_every, nseg = std::min(sh->ckpt_every, sh->K - k0);
    rc = seg_forward(logl, sh, net, ws, k0, nseg, st);
    if (rc != ET_OK) return rc;
    const int64_t n = (int64_t)sh->B * hw;
    bilif_fwd<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(ws.I, sh->B, sh->K, k0, nseg, hw, net->beta,
                                                           net->vth, net->reset, ws.V, V_ckpt, s, n_ckpt,
                                                           spikes, S_on, S_off, I_out);
    ET_CHECK_LAUNCH();
  }
  return ET_OK;
}

extern "C" int et_emd_count_loss(const int8_t* spikes, const float* E, const et_train_shape* sh,
                                 float lambda, float* loss, float* dS_on, float* dS_off,
                                 void* stream_) {
  if (!sh || !spikes || !E || !loss || !dS_on || !dS_off) return ET_ERR_ARG;
  if (sh->B < 1 || sh->K < 1 || sh->H < 1 || sh->W < 1) return ET_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream_;
  const int64_t hw = (int64_t)sh->H * sh->W, n = (int64_t)sh->B * hw;
  ET_CHECK_CUDA(cudaMemsetAsync(loss, 0, 3 * sizeof(float), st));
  emd_count_loss<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(spikes, E, sh->B, sh->K, hw, lambda,
                                                                loss, dS_on, dS_off);
  ET_CHECK_LAUNCH();
  return ET_OK;
}

extern "C" int et_evsnet_train_backward(const float* logl, const et_train_shape* sh,
                                        const et_evsnet_weights* net, const float* V_ckpt,
                                        const float* dS_on, const float* dS_off, float alpha,
                                        float* grad_w, float* grad_b, void* workspace,
                                        size_t ws_bytes, void* stream_) {
  int rc = check(net, sh);
  if (rc != ET_OK) return rc;
  if (!logl || !V_ckpt || !dS_on || !dS_off || !grad_w || !grad_b || !workspace) return ET_ERR_ARG;
  if (reinterpret_cast<uintptr_t>(workspace) % sizeof(float) != 0) return ET_ERR_ARG;
  if (et_train_is_temporal(net)) {
    if (ws_bytes < et_train_temporal_bytes(net, sh)) return ET_ERR_ARG;
    return et_train_temporal_backward(logl, sh, net, V_ckpt, dS_on, dS_off, alpha, grad_w, grad_b,
                                      workspace, (cudaStream_t)stream_);
  }
  Workspace ws{};
  layout(net, sh, nullptr, &ws);
  if (ws_bytes < ws.bytes) return ET_ERR_ARG;
  layout(net, sh, static_cast<char*>(workspace), &ws);
  cudaStream_t st = (cudaStream_t)stream_;
  const int H = sh->H, W = sh->W, C = net->C, L = net->n_layers;
  const int64_t hw = (int64_t)H * W;
  const int n_ckpt = (sh->K + sh->ckpt_every - 1) / sh->ckpt_every;
  int dev = 0, nsm = 0;
  ET_CHECK_CUDA(cudaGetDevice(&dev));
  ET_CHECK_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  int wblocks = 0;   // resident weight-gradient blocks per SM: one wave of persistent blocks
  ET_CHECK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&wblocks, conv16_bwd_weight, kWThreads, 0));
  wblocks = std::max(wblocks, 1);
  ET_CHECK_CUDA(cudaMemsetAsync(ws.V, 0, sizeof(float) * sh->B * hw, st));   // dL/dV after the last step
  float* gwp = grad_w + wofs(L, C);
  float* gbp = grad_b + (int64_t)L * C;
  for (int s = n_ckpt - 1; s >= 0; --s) {
    const int k0 = s * sh->ckpt_every, nseg = std::min(sh->ckpt_every, sh->K - k0);
    const int N = sh->B * nseg;
    rc = seg_forward(logl, sh, net, ws, k0, nseg, st);
    if (rc != ET_OK) return rc;
    const int64_t n = (int64_t)sh->B * hw;
    bilif_bwd<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(ws.I, sh->B, sh->K, k0, nseg, hw, net->beta,
                                                           net->vth, net->reset, alpha, V_ckpt, s,
                                                           n_ckpt, dS_on, dS_off, ws.V, ws.dI);
    ET_CHECK_LAUNCH();
    proj_bwd<<<nsm * 4, 256, 0, st>>>(ws.dI, ws.act[L - 1], N, C, hw, net->w + wofs(L, C), ws.dz[0],
                                      gwp, gbp);
    ET_CHECK_LAUNCH();
    const dim3 grid16 = conv16_grid(H, W, N);
    int cur = 0;
    for (int l = L - 1; l >= 0; --l) {
      if (l == 0)
        conv_bwd_weight<<<nsm * 2, TS * TS, 0, st>>>(ws.dz[cur], logl, sh->K, k0, nseg, N, C, H, W,
                                                     grad_w + wofs(0, C), grad_b);
      else if (net->dtype == ET_BF16) {
        rc = et_train_tc_wgrad(ws.dz[cur], ws.act[l - 1], N, C, H, W, grad_w + wofs(l, C),
                               grad_b + (int64_t)l * C, st);
        if (rc != ET_OK) return rc;
      } else
        conv16_bwd_weight<<<nsm * wblocks, kWThreads, 0, st>>>(ws.dz[cur], ws.act[l - 1], N, C, H, W,
                                                               grad_w + wofs(l, C), grad_b + (int64_t)l * C);
      ET_CHECK_LAUNCH();
      if (l > 0) {
        if (net->dtype == ET_BF16) {
          rc = et_train_tc_conv(ws.dz[cur], N, C, H, W, net->w + wofs(l, C), nullptr, ws.dz[cur ^ 1],
                                nullptr, nullptr, nullptr, ws.act[l - 1], true, st);
          if (rc != ET_OK) return rc;
        } else {
          conv16<true><<<grid16, 64, 0, st>>>(ws.dz[cur], C, H, W, net->w + wofs(l, C), nullptr, ws.dz[cur ^ 1],
                                               nullptr, nullptr, nullptr, ws.act[l - 1]);
          ET_CHECK_LAUNCH();
        }
        cur ^= 1;
      }
    }
  }
  return ET_OK;
}

extern "C" int et_adam_step(float* p, const float* g, float* m, float* v, int64_t n, float lr,
                            float b1, float b2, float eps, int32_t step, void* stream_) {
  if (!p || !g || !m || !v || n < 0 || step < 1) return ET_ERR_ARG;
  if (n == 0) return ET_OK;
  const float bc1 = 1.0f - powf(b1, (float)step), bc2 = 1.0f - powf(b2, (float)step);
  adam_kernel<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream_>>>(p, g, m, v, n, lr, b1, b2,
                                                                             eps, bc1, bc2);
  ET_CHECK_LAUNCH();
  return ET_OK;
}

// ---------------------------------------------------------------------------
// Backward without a caller workspace.
//
// Some callers cannot hand the library a device workspace: a plugin that lives
// inside a host framework whose caching allocator owns all device memory and
// forbids side allocations, or a loop that must not call cudaMalloc / cudaFree
// because those calls may synchronise the whole device.  For them this entry
// point runs the same backward with its scratch in a fixed array compiled into
// the library.  The array exists once per device that loads the library and is
// kept until the process exits.
namespace {
constexpr size_t kStaticWorkspaceBytes = (size_t)32 << 20;   // 32 MiB
constexpr int kMaxDevices = 64;
std::mutex g_static_ws_mutex;
// Per device: the array's device address and the unique id of the context it
// was looked up in.  A module's __device__ arrays live in one context; after
// cudaDeviceReset (or any teardown of the primary context) the next context
// loads the module again and the array may sit elsewhere, so the address is
// looked up again whenever the current context's id differs.
struct StaticWs {
  void* ptr;
  unsigned long long ctx_id;
};
StaticWs g_static_ws[kMaxDevices] = {};
// Driver calls reached through the runtime's entry-point query (the library
// links only the runtime).
typedef CUresult (*CtxGetCurrentFn)(CUcontext*);
typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long*);
CtxGetCurrentFn g_ctx_get_current = nullptr;
CtxGetIdFn g_ctx_get_id = nullptr;

// Id of the calling thread's current context; 0 if none is current yet.
int current_context_id(unsigned long long* id) {
  *id = 0;
  if (!g_ctx_get_current || !g_ctx_get_id) {
    cudaDriverEntryPointQueryResult q1, q2;
    void* f1 = nullptr;
    void* f2 = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 12000, cudaEnableDefault, &q1) != cudaSuccess ||
        cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2) != cudaSuccess ||
        q1 != cudaDriverEntryPointSuccess || q2 != cudaDriverEntryPointSuccess || !f1 || !f2)
      return ET_ERR_CUDA;
    g_ctx_get_current = (CtxGetCurrentFn)f1;
    g_ctx_get_id = (CtxGetIdFn)f2;
  }
  CUcontext ctx = nullptr;
  if (g_ctx_get_current(&ctx) != CUDA_SUCCESS) return ET_ERR_CUDA;
  if (ctx && g_ctx_get_id(ctx, id) != CUDA_SUCCESS) return ET_ERR_CUDA;
  return ET_OK;
}
}  // namespace

// Device memory; host code must not use this name as an address (on the host it
// only stands for the symbol).  Its device address comes from cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_static_workspace[kStaticWorkspaceBytes];

extern "C" size_t et_train_static_workspace_capacity(void) { return kStaticWorkspaceBytes; }

extern "C" int et_evsnet_train_backward_static(const float* logl, const et_train_shape* sh,
                                               const et_evsnet_weights* net, const float* V_ckpt,
                                               const float* dS_on, const float* dS_off, float alpha,
                                               float* grad_w, float* grad_b, void* stream) {
  int rc = check(net, sh);
  if (rc != ET_OK) return rc;
  // scratch of either form (the temporal one keeps whole-clip activations)
  size_t need = 0;
  if (et_train_is_temporal(net)) {
    need = et_train_temporal_bytes(net, sh);
  } else {
    Workspace ws{};
    layout(net, sh, nullptr, &ws);
    need = ws.bytes;
  }
  if (need > kStaticWorkspaceBytes) return ET_ERR_CAPACITY;   // shape too large for the array
  int dev = 0;
  ET_CHECK_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return ET_ERR_ARG;
  void* base = nullptr;
  {
    // first call on this device (with it current), or first call in a new
    // context of it: look up the array's device address
    std::lock_guard<std::mutex> lock(g_static_ws_mutex);
    unsigned long long id = 0;
    rc = current_context_id(&id);
    if (rc != ET_OK) return rc;
    if (!g_static_ws[dev].ptr || id == 0 || g_static_ws[dev].ctx_id != id) {
      void* p = nullptr;
      ET_CHECK_CUDA(cudaGetSymbolAddress(&p, g_static_workspace));
      // the lookup makes the device's primary context current if none was
      rc = current_context_id(&id);
      if (rc != ET_OK) return rc;
      g_static_ws[dev].ptr = p;
      g_static_ws[dev].ctx_id = id;
    }
    base = g_static_ws[dev].ptr;
  }
  // the backward clears the part of the scratch that must start at zero (the
  // carried membrane gradient of the spatial form) and overwrites the rest
  // before reading it
  return et_evsnet_train_backward(logl, sh, net, V_ckpt, dS_on, dS_off, alpha, grad_w, grad_b, base,
                                  kStaticWorkspaceBytes, stream);
}
