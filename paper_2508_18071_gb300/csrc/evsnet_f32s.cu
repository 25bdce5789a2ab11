// EvSNet forward in FP32 for the spatial form of the workloads: a plain stack
// of 3x3 convolutions with ReLU (Eq. 5 with a spatial kernel, kt = 1) of up to
// 16 channels, the point-wise projection (Eq. 6) and BiLIF (Eq. 2-3).
//
// Each CTA owns a 32 x 16 pixel tile for the whole call and walks the frames;
// the membrane potentials of its pixels stay in registers.  Per step the
// log frame tile with an L-pixel halo is loaded (X = l_k - l_{k-1}, Eq. 1) and
// the layers run one after the other on shrinking regions of the padded tile
// (layer l is computed L - 1 - l pixels beyond the tile), with zero padding
// outside the image.
//
// What bounds it is shared memory: a warp's 16-byte load takes 4 clk of the SM's
// 128 bytes per clk whatever its addresses.  In layers 1.. a lane computes 8 output
// channels for 4 to 8 positions, as many as spread the layer's region over the CTA's
// eight warps: 8 weight loads and one per position feed 32 multiply-adds per position
// (48 to 64 clk of shared memory for 32 to 64 of the FP32 pipe; 4 positions x 4
// channels, 32 clk for 16, spent 68 k of a tile-step's 70 k clk on loads by this
// count).  Multiply-adds run as FP32 pairs over channels, rounded like fmaf, in one
// chain over taps, then input channels.
// Activations lie by groups of four channels, [group][position]: consecutive positions
// are consecutive 16-byte words.  A layer's outputs stay in registers until every warp
// has read its inputs and then replace them, so that one activation buffer serves all
// layers and two CTAs fit an SM at four layers.  In the last layer the two channel
// lanes of a position add their parts of the projection and each takes two rows of one
// column for BiLIF; events are gathered per warp.  641 x 363, four layers, 15 steps:
// 2.35 -> 1.66 ms (2.10 with 8 positions everywhere: six, five and four of the warps
// then have work).
#include "et_internal.cuh"
#include "event_emit.cuh"
#include "evsnet_common.h"
#include "f32x2.cuh"
#include <type_traits>

namespace {

constexpr int TW = 32, TH = 16;
constexpr int CP = 16;            // channels as stored (C <= 16, zero padded)

struct SParams {
  int L;
  float beta, vth, reset;
  int H, W, F, f0, t0;
  int Wp, Hp;
  int plane;                      // floats of one channel group's activations
  int off_b, off_w0, off_wl, off_wp, off_cur, off_prev;
};

constexpr int kWarps = 8;         // of a CTA; a warp's 16 position lanes x 2 channel lanes
constexpr int kThreads = kWarps * 32;
constexpr int kLastPos = TW * TH / (kWarps * 16);   // a lane's positions in the last layer
constexpr int kLastRows = kLastPos / 2;
static_assert(TW == 32 && kLastPos == 2 * kLastRows, "a lane of the last layer owns rows of one column");
constexpr int kStageCap = 64;    // events a warp holds before it appends them

__device__ __forceinline__ float4 relu4(float a, float b, float c, float d) {
  return make_float4(fmaxf(a, 0.0f), fmaxf(b, 0.0f), fmaxf(c, 0.0f), fmaxf(d, 0.0f));
}

// one 3x3 layer: sums of kP positions (words at[k] of act's first group) x the channels
// 8 cg .. whose weights start at wt, from the biases b
template <int kP>
__device__ __forceinline__ void conv_layer(const float* act, int plane, int Wp, const float* wt, const float* b,
                                           const int (&at)[kP], f32x2 (&acc)[kP][4]) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const f32x2 b2 = *reinterpret_cast<const f32x2*>(b + 2 * c);
#pragma unroll
    for (int k = 0; k < kP; ++k) acc[k][c] = b2;
  }
#pragma unroll 1
  for (int t = 0; t < 9; ++t) {
    const float* xt = act + 4 * ((t / 3 - 1) * Wp + t % 3 - 1);
#pragma unroll
    for (int g = 0; g < CP / 4; ++g, wt += 4 * CP, xt += plane) {
      ulonglong2 w[4][2];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        w[c][0] = *reinterpret_cast<const ulonglong2*>(wt + c * CP);
        w[c][1] = *reinterpret_cast<const ulonglong2*>(wt + c * CP + 4);
      }
#pragma unroll
      for (int k = 0; k < kP; ++k) {
        const float4 x = *reinterpret_cast<const float4*>(xt + at[k]);
        const float xc[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const f32x2 x2 = pack2f(xc[c], xc[c]);
          acc[k][0] = fma2(w[c][0].x, x2, acc[k][0]);
          acc[k][1] = fma2(w[c][0].y, x2, acc[k][1]);
          acc[k][2] = fma2(w[c][1].x, x2, acc[k][2]);
          acc[k][3] = fma2(w[c][1].y, x2, acc[k][3]);
        }
      }
    }
  }
}

template <int kBlocks>
__global__ void __launch_bounds__(kThreads, kBlocks)
evsnet_f32s_kernel(SParams P, int C, const float* __restrict__ logl, const float* __restrict__ wg,
                   const float* __restrict__ bg, float* __restrict__ Vg,
                   const float* __restrict__ last_l, et_event* events, int64_t cap,
                   unsigned long long* n_events, float* __restrict__ I_out,
                   int8_t* __restrict__ spikes) {
  extern __shared__ __align__(16) float sm[];
  __shared__ uint32_t staged[kWarps][kStageCap];
  const int L = P.L, Wp = P.Wp, Hp = P.Hp, tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31, pg = lane >> 1, cg = lane & 1;
  float* const act = sm;                          // [CP / 4][Hp Wp][4]
  float* const sb = sm + P.off_b;                 // [L][CP] biases, then the projection bias
  float* const w0 = sm + P.off_w0;                // [9][CP]
  float* const wl = sm + P.off_wl;                // [L-1][9][CP (ci)][CP (co)]
  float* const wp = sm + P.off_wp;                // [CP]
  float* cur = sm + P.off_cur;                    // log frame over the padded tile
  float* prev = sm + P.off_prev;
  const int tiles_x = (P.W + TW - 1) / TW;
  const int ox = (blockIdx.x % tiles_x) * TW, oy = (blockIdx.x / tiles_x) * TH;
  const int64_t npix = (int64_t)P.H * P.W;

  // packed FP32 weights: layer 0 [C][1][3][3], layers 1.. [C][C][3][3], projection [C]
  for (int i = tid; i < 9 * CP; i += kThreads) {
    const int t = i / CP, co = i % CP;
    w0[i] = co < C ? wg[co * 9 + t] : 0.0f;
  }
  for (int i = tid; i < (L - 1) * 9 * CP * CP; i += kThreads) {
    const int co = i % CP, ci = (i / CP) % CP, t = (i / (CP * CP)) % 9, l = 1 + i / (CP * CP * 9);
    wl[i] = (co < C && ci < C) ? wg[9 * C + (l - 1) * C * C * 9 + (co * C + ci) * 9 + t] : 0.0f;
  }
  for (int i = tid; i < L * CP; i += kThreads) {
    const int l = i / CP, c = i % CP;
    sb[i] = c < C ? bg[l * C + c] : 0.0f;
  }
  for (int i = tid; i < CP; i += kThreads) wp[i] = i < C ? wg[9 * C + (L - 1) * C * C * 9 + i] : 0.0f;
  if (tid == 0) sb[L * CP] = bg[L * C];
  // the lane's pixels in the last layer: column vx, rows vy ..
  const int vx = ox + 16 * cg + pg, vy = oy + kLastRows * warp;
  float V[kLastRows];
#pragma unroll
  for (int j = 0; j < kLastRows; ++j)
    V[j] = vx < P.W && vy + j < P.H ? Vg[(int64_t)(vy + j) * P.W + vx] : 0.0f;
  EventStage<kStageCap> stage(staged[warp], events, cap, n_events, (uint32_t)vx, (uint32_t)vy, (uint32_t)P.t0);
  // the frame before the first step: the caller's last frame, or frame 0 when
  // the state is fresh (the first step is then frame 1)
  for (int i = tid; i < Hp * Wp; i += kThreads) {
    const int gx = ox - L + i % Wp, gy = oy - L + i / Wp;
    float v = 0.0f;
    if (gx >= 0 && gx < P.W && gy >= 0 && gy < P.H)
      v = P.f0 == 0 ? last_l[(int64_t)gy * P.W + gx] : __ldg(logl + (int64_t)gy * P.W + gx);
    prev[i] = v;
  }

  for (int f = P.f0; f < P.F; ++f) {
    for (int i = tid; i < Hp * Wp; i += kThreads) {
      const int gx = ox - L + i % Wp, gy = oy - L + i / Wp;
      cur[i] = (gx >= 0 && gx < P.W && gy >= 0 && gy < P.H)
                   ? __ldg(logl + (int64_t)f * npix + (int64_t)gy * P.W + gx) : 0.0f;
    }
    __syncthreads();
    // layer 0 (one input channel) on rows / columns [1, Hp - 1) x [1, Wp - 1):
    // two positions per thread, all channels
    {
      const int rw = Wp - 2, n = (Hp - 2) * rw;
      for (int i = tid; i < n; i += 2 * kThreads) {
        int m[2];
        bool in[2];
        f32x2 acc[2][CP / 2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int ic = min(i + k * kThreads, n - 1), py = 1 + ic / rw, px = 1 + ic % rw;
          const int gx = ox - L + px, gy = oy - L + py;
          m[k] = py * Wp + px;
          in[k] = gx >= 0 && gx < P.W && gy >= 0 && gy < P.H;
#pragma unroll
          for (int c = 0; c < CP / 2; ++c) acc[k][c] = *reinterpret_cast<const f32x2*>(sb + 2 * c);
        }
#pragma unroll
        for (int t = 0; t < 9; ++t) {
          f32x2 x[2];
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const int q = m[k] + (t / 3 - 1) * Wp + (t % 3 - 1);
            const float v = cur[q] - prev[q];                   // Eq. 1
            x[k] = pack2f(v, v);
          }
#pragma unroll
          for (int c = 0; c < CP / 2; c += 2) {
            const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(w0 + t * CP + 2 * c);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              acc[k][c] = fma2(w.x, x[k], acc[k][c]);
              acc[k][c + 1] = fma2(w.y, x[k], acc[k][c + 1]);
            }
          }
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          if (i + k * kThreads >= n) break;
#pragma unroll
          for (int g = 0; g < CP / 4; ++g) {
            float a[4];
            unpack2f(acc[k][2 * g], a[0], a[1]);
            unpack2f(acc[k][2 * g + 1], a[2], a[3]);
            *reinterpret_cast<float4*>(act + g * P.plane + 4 * m[k]) =
                in[k] ? relu4(a[0], a[1], a[2], a[3]) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          }
        }
      }
    }
    __syncthreads();
    // layers 1 .. L-2, each on rows / columns [l + 1, ..): position k of lane (pg, cg)
    // is (k * kWarps + warp) * 16 + pg
    auto hidden = [&](auto pos, int l) {
      constexpr int kP = decltype(pos)::value;
      const int rw = TW + 2 * (L - 1 - l), n = (TH + 2 * (L - 1 - l)) * rw;
      int at[kP];
      uint32_t in = 0;                            // positions of the image
#pragma unroll
      for (int k = 0; k < kP; ++k) {
        const int ic = min((k * kWarps + warp) * 16 + pg, n - 1);
        const int py = l + 1 + ic / rw, px = l + 1 + ic % rw;
        const int gx = ox - L + px, gy = oy - L + py;
        at[k] = 4 * (py * Wp + px);
        in |= (gx >= 0 && gx < P.W && gy >= 0 && gy < P.H ? 1u : 0u) << k;
      }
      f32x2 acc[kP][4];
      conv_layer(act, P.plane, Wp, wl + (l - 1) * 9 * CP * CP + 8 * cg, sb + l * CP + 8 * cg, at, acc);
      __syncthreads();                            // every warp has read this layer's inputs
#pragma unroll
      for (int k = 0; k < kP; ++k) {
        if ((k * kWarps + warp) * 16 + pg >= n) break;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float a[4];
          unpack2f(acc[k][2 * h], a[0], a[1]);
          unpack2f(acc[k][2 * h + 1], a[2], a[3]);
          *reinterpret_cast<float4*>(act + (2 * cg + h) * P.plane + at[k]) =
              (in >> k & 1u) ? relu4(a[0], a[1], a[2], a[3]) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
      }
      __syncthreads();
    };
#pragma unroll 1
    for (int l = 1; l < L - 1; ++l) {
      const int per = L - 1 - l;                  // 5, 6, 7, 8 positions of a lane cover its region
      if (per == 1) hidden(std::integral_constant<int, 5>{}, l);
      else if (per == 2 || kBlocks == 2) hidden(std::integral_constant<int, 6>{}, l);
      else if (per == 3) hidden(std::integral_constant<int, 7>{}, l);
      else hidden(std::integral_constant<int, 8>{}, l);
    }
    // the last layer on the tile, into projection + BiLIF: a warp owns kLastRows rows
    {
      int at[kLastPos];
#pragma unroll
      for (int k = 0; k < kLastPos; ++k)
        at[k] = 4 * ((L + kLastRows * warp + k / 2) * Wp + L + 16 * (k % 2) + pg);
      f32x2 acc[kLastPos][4];
      conv_layer(act, P.plane, Wp, wl + (L - 2) * 9 * CP * CP + 8 * cg, sb + (L - 1) * CP + 8 * cg, at, acc);
      // Eq. 6: sums of four channels, the lane's two, then the other lane's
      float I[kLastPos];
#pragma unroll
      for (int k = 0; k < kLastPos; ++k) {
        float s[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float4 wpv = *reinterpret_cast<const float4*>(wp + 8 * cg + 4 * h);
          float a[4];
          unpack2f(acc[k][2 * h], a[0], a[1]);
          unpack2f(acc[k][2 * h + 1], a[2], a[3]);
          s[h] = wpv.x * fmaxf(a[0], 0.0f);
          s[h] = fmaf(wpv.y, fmaxf(a[1], 0.0f), s[h]);
          s[h] = fmaf(wpv.z, fmaxf(a[2], 0.0f), s[h]);
          s[h] = fmaf(wpv.w, fmaxf(a[3], 0.0f), s[h]);
        }
        I[k] = s[0] + s[1];
        I[k] += __shfl_xor_sync(0xffffffffu, I[k], 1);
        I[k] = sb[L * CP] + I[k];
      }
      // lane cg takes the positions of its column
      uint32_t fired = 0, neg = 0;
#pragma unroll
      for (int j = 0; j < kLastRows; ++j) {
        const float Ij = cg ? I[2 * j + 1] : I[2 * j];
        const float vp = P.beta * V[j] + Ij;                    // Eq. 2-3
        const int S = vp >= P.vth ? 1 : (vp <= -P.vth ? -1 : 0);
        V[j] = vp - P.reset * (float)S;
        if (vx >= P.W || vy + j >= P.H) continue;
        fired |= (S != 0 ? 1u : 0u) << j;
        neg |= (S < 0 ? 1u : 0u) << j;
        const int64_t o = (int64_t)(f - P.f0) * npix + (int64_t)(vy + j) * P.W + vx;
        if (I_out) I_out[o] = Ij;
        if (spikes) spikes[o] = (int8_t)S;
      }
      if (P.t0 + f < 0) fired = 0;                              // delayed labels below 0: none
      stage.add_rows<kLastRows>(fired, neg, (uint32_t)f, 0);
    }
    // the frame loop's barrier after the next frame's load covers the last layer's reads
    float* t = cur; cur = prev; prev = t;
  }
  stage.flush();
#pragma unroll
  for (int j = 0; j < kLastRows; ++j)
    if (vx < P.W && vy + j < P.H) Vg[(int64_t)(vy + j) * P.W + vx] = V[j];
}

}  // namespace

int et_evsnet_forward_f32s(const float* logl, int32_t F, const et_evsnet_weights* net,
                           et_evsnet_state* st, int32_t t0, et_event* events, int64_t cap,
                           int64_t* n_events, float* I_out, int8_t* spikes, cudaStream_t stream) {
  if (net->kind != ET_NET_STACK || net->ks != 3 || net->kt != 1 || net->n_layers < 2 || net->C > CP)
    return ET_ERR_UNIMPLEMENTED;
  SParams P{};
  P.L = net->n_layers;
  P.beta = net->beta; P.vth = net->vth; P.reset = net->reset;
  P.H = st->H; P.W = st->W; P.F = F; P.f0 = st->initialized ? 0 : 1; P.t0 = t0;
  P.Wp = TW + 2 * P.L; P.Hp = TH + 2 * P.L;
  auto al4 = [](int x) { return (x + 3) & ~3; };           // 16-byte alignment in floats
  // a channel group's activations, an odd multiple of 64 bytes: the two channel lanes
  // of a position store to different banks
  P.plane = (P.Hp * P.Wp + 7) / 8 * 32 + 16;
  int off = CP / 4 * P.plane;
  P.off_b = off; off += al4(P.L * CP + 1);
  P.off_w0 = off; off += 9 * CP;
  P.off_wl = off; off += (P.L - 1) * 9 * CP * CP;
  P.off_wp = off; off += CP;
  P.off_cur = off; off += al4(P.Hp * P.Wp);
  P.off_prev = off; off += al4(P.Hp * P.Wp);
  const size_t smem = sizeof(float) * (size_t)off;
  int dev = 0, max_smem = 0;
  ET_CHECK_CUDA(cudaGetDevice(&dev));
  ET_CHECK_CUDA(cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  // from seven layers on the halo is most of the work: the general kernel takes the call
  if (P.L > 6) return ET_ERR_UNIMPLEMENTED;
  // Up to four layers (98 KB, at most 6 positions per lane) two CTAs fit an SM and share
  // its registers; from five on one has them alone
  auto kern = P.L <= 4 ? evsnet_f32s_kernel<2> : evsnet_f32s_kernel<1>;
  cudaFuncAttributes fa;
  ET_CHECK_CUDA(cudaFuncGetAttributes(&fa, kern));
  if (smem + fa.sharedSizeBytes > (size_t)max_smem) return ET_ERR_UNIMPLEMENTED;
  const int tiles = ((P.W + TW - 1) / TW) * ((P.H + TH - 1) / TH);
  const int rc = et_allow_shared(kern);
  if (rc != ET_OK) return rc;
  kern<<<tiles, kThreads, smem, stream>>>(
      P, net->C, logl, net->w, net->b, st->V, st->last_l, events, cap,
      reinterpret_cast<unsigned long long*>(n_events), I_out, spikes);
  ET_CHECK_LAUNCH();
  return ET_OK;
}
