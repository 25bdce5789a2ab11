// EvSNet forward in FP32 for the pixel-wise form (Eq. 5 with kernel kt along
// time, plain stack or residual blocks, optionally a one-step spatial stem;
// Eq. 6; BiLIF of Eq. 2-3) at kt = 7 and 13 to 16 channels, with the input
// history of every layer in shared memory.  Same sums in the same order as evsnet_pix.cu.
//
// The history is 2.3 KB per pixel (6 layers x 6 steps x 16 channels) and every
// step reads all of it; from L2 that bounds the kernel.  Here a CTA keeps 32
// pixels' rings (kt - 1 + 8 steps per layer) in shared memory for the whole call,
// next to all layers' weights, one CTA per SM walking tiles of 32 pixels.
// Steps are taken eight at a time: layer by layer, with one barrier between
// layers, a thread computes two output channels (its warp's) of one pixel (its
// lane) for all eight.  What bounds this is the FP32 pipes, next the shared
// memory's 128 bytes per clock into registers (a 16-byte read by a warp takes
// four clocks whatever the addresses): with the eight steps' input rows in
// registers a tap needs 8 weight reads and one new row (4 reads) for 256
// multiply-adds, 48 of 64 clocks.  Rows are 64 bytes per pixel, their 16-byte
// pieces permuted by (pixel >> 1) & 3 so that eight pixels meet 32 different
// banks.  A residual block's input is read back from its inner layer's ring.
//
// The paper's form, 640 x 360: 16 steps 4.04 -> 2.38 ms, 8 steps 2.36 -> 1.39, 1
// step 0.85 -> 0.75; 77 x 61, 8 steps 0.51 -> 0.042 (32-pixel tiles reach 147 SMs
// where 256-thread blocks reached 19).  On the way: two steps x 4 channels per
// thread, 20 reads per 64 pair multiply-adds, 3.55 ms; eight steps x 4 channels
// on 4 warps, every pair instruction behind a register copy, 3.15 ms.
#include "et_internal.cuh"
#include "event_emit.cuh"
#include "evsnet_common.h"
#include <algorithm>
#include <type_traits>

namespace {

constexpr int kP = 32;           // pixels per tile
constexpr int kT = 8;            // steps per chunk
constexpr int kThreads = 256;    // 8 warps x 2 channels
constexpr int CP = 16;
constexpr int kKt = 7;
constexpr int kRow = kP * CP;    // floats of one ring slot
constexpr int kStageCap = 128;

struct Pix16Params {
  int kind, L, C, kt, ks0, R;
  float beta, vth, reset;
  int H, W, F, f0, t0;
  int tiles;
  int woff[kMaxLayers + 1];
  int off_s;              // scratch slots of the last layer's output, -1: in layer 1's ring
  int off_w, off_b, off_x, off_I;   // float offsets in shared memory (rings first)
};

__device__ __forceinline__ int piece(int px, int j) { return px * CP + 4 * (j ^ ((px >> 1) & 3)); }

__global__ void __launch_bounds__(kThreads, 1)
evsnet_pix16_kernel(Pix16Params P, const float* __restrict__ logl, const float* __restrict__ wg,
                    const float* __restrict__ bg, float* __restrict__ Vg, float* __restrict__ hist,
                    const float* __restrict__ last_l, et_event* events, int64_t cap,
                    unsigned long long* n_events, float* __restrict__ I_out, int8_t* __restrict__ spikes) {
  extern __shared__ __align__(16) float sm[];
  __shared__ uint32_t staged[kStageCap];
  const int L = P.L, C = P.C, kt = kKt, hk = kt - 1, ks0 = P.ks0, R = P.R;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int c0 = 2 * warp;         // this thread's output channels c0, c0 + 1 of pixel `lane`
  float* sw = sm + P.off_w;        // [L-1][kt][CP / 2 (co / 2)][CP (ci)][2], then layer 0 [taps][CP], projection [CP]
  float* sb = sm + P.off_b;        // [L][CP], then the projection's bias
  float* xr = sm + P.off_x;        // [R][kP]: X of a temporal layer 0
  float* sI = sm + P.off_I;        // [kT][kP]
  const int taps0 = ks0 > 0 ? ks0 * ks0 : kt;
  float* w0 = sw + (L - 1) * kt * CP * CP;
  float* swp = w0 + taps0 * CP;
  for (int i = tid; i < (L - 1) * kt * CP * CP; i += kThreads) {
    const int co = (i / (2 * CP)) % (CP / 2) * 2 + i % 2, ci = (i / 2) % CP;
    const int tau = (i / (CP * CP)) % kt, l = 1 + i / (CP * CP * kt);
    sw[i] = co < C && ci < C ? __ldg(wg + P.woff[l] + (co * C + ci) * kt + tau) : 0.0f;
  }
  for (int i = tid; i < taps0 * CP; i += kThreads) w0[i] = i % CP < C ? wg[(i % CP) * taps0 + i / CP] : 0.0f;
  for (int i = tid; i < CP; i += kThreads) swp[i] = i < C ? wg[P.woff[L] + i] : 0.0f;
  for (int i = tid; i < L * CP; i += kThreads) sb[i] = i % CP < C ? bg[(i / CP) * C + i % CP] : 0.0f;
  if (tid == 0) sb[L * CP] = bg[L * C];
  const int64_t npix = (int64_t)P.H * P.W;
  const int S = P.F - P.f0;        // steps of the call; step s is frame f0 + s
  auto ring = [&](int l, int pos) { return sm + ((l - 1) * R + pos) * kRow; };
  auto wrap = [&](int pos) { return pos >= R ? pos - R : pos; };
  auto frame = [&](int f, int64_t q) { return f < 0 ? last_l[q] : __ldg(logl + (int64_t)f * npix + q); };

  for (int tile = blockIdx.x; tile < P.tiles; tile += gridDim.x) {
    const int64_t q0 = (int64_t)tile * kP;
    const int np = (int)min((int64_t)kP, npix - q0);
    const int64_t ql = q0 + min(lane, np - 1);       // loads of a pixel past the end: the last one's, unused
    __syncthreads();                                  // the previous tile's rings have been read
    // history: step -hk + j at ring position j, all copies in flight at once
    for (int i = warp; i < (L - 1) * hk * CP; i += kThreads / 32) {
      const int c = i % CP, j = (i / CP) % hk, l = 1 + i / (CP * hk);
      float* dst = ring(l, j) + piece(lane, c >> 2) + (c & 3);
      if (lane < np && c < C)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                     "l"(hist + (((int64_t)l * hk + j) * C + c) * npix + ql)
                     : "memory");
      else
        *dst = 0.0f;
    }
    if (ks0 == 0)
      for (int j = warp; j < hk; j += kThreads / 32)
        xr[j * kP + lane] = lane < np ? hist[(int64_t)j * C * npix + ql] : 0.0f;
    float V = (warp == 0 && lane < np) ? Vg[ql] : 0.0f;
    EventStage<kStageCap> stage(staged, events, cap, n_events, (uint32_t)(ql % P.W), (uint32_t)(ql / P.W),
                                (uint32_t)P.t0);
    // X of the chunk's steps (temporal layer 0): warp j the chunk's step j,
    // loaded a chunk ahead
    float xnext = 0.0f;
    auto load_x = [&](int s0) {
      const int s = s0 + warp;
      if (ks0 == 0 && s < S) xnext = frame(P.f0 + s, ql) - frame(P.f0 + s - 1, ql);   // Eq. 1
    };
    load_x(0);
    asm volatile("cp.async.wait_all;" ::: "memory");   // the first step's barrier shows every thread's copies
    int base = hk < R ? hk : 0;    // ring position of the chunk's first step (step s at (s + hk) mod R)
    for (int s0 = 0; s0 < S; s0 += kT) {
      const int tc = min(kT, S - s0);
      // the chunk's network for up to NS steps
      auto steps = [&](auto ns) {
      constexpr int NS = decltype(ns)::value;
      const int old = wrap(base + R - hk);        // ring position of the first step's oldest tap
      // where the last layer's output goes: eight slots of layer 1's ring that
      // are no later chunk's history (its oldest hk and this chunk's first 8 - hk),
      // or, in networks whose last layer still reads that ring, slots of their own
      float* scratch = P.off_s >= 0 ? sm + P.off_s : ring(1, 0);
      const int sc0 = P.off_s >= 0 ? 0 : old;
      // ---- layer 0
      if (ks0 == 0) {
        if (warp < tc) xr[wrap(base + warp) * kP + lane] = xnext;
        load_x(s0 + kT);
      }
      __syncthreads();
      float acc[NS][2];
      auto start = [&](int l) {
#pragma unroll
        for (int s = 0; s < NS; ++s) { acc[s][0] = sb[l * CP + c0]; acc[s][1] = sb[l * CP + c0 + 1]; }
      };
      // ReLU (after adding the block input h, if given) of the chunk's steps into
      // slots of `out`, the first at ring position `pos`
      auto put = [&](float* out, int pos, const float* h) {
        int hp = base;
#pragma unroll
        for (int s = 0; s < NS; ++s) {
          if (s < tc) {
            const int o = piece(lane, warp >> 1) + (c0 & 3);
            float2 v = make_float2(acc[s][0], acc[s][1]);
            if (h) {
              const float2 hv = *reinterpret_cast<const float2*>(h + hp * kRow + o);
              v.x = hv.x + v.x;
              v.y = hv.y + v.y;
            }
            *reinterpret_cast<float2*>(out + pos * kRow + o) = make_float2(fmaxf(v.x, 0.0f), fmaxf(v.y, 0.0f));
          }
          pos = wrap(pos + 1);
          hp = wrap(hp + 1);
        }
      };
      start(0);
      if (ks0 == 0) {
        // one new X per tap, as below
        float xs[NS];
        int pos = old;
#pragma unroll
        for (int s = 0; s < NS; ++s) {
          xs[s] = xr[pos * kP + lane];
          pos = wrap(pos + 1);
        }
        for (int t = 0; t < kt; ++t) {
          const float2 w = *reinterpret_cast<const float2*>(w0 + t * CP + c0);
#pragma unroll
          for (int s = 0; s < NS; ++s) {
            acc[s][0] = fmaf(w.x, xs[s], acc[s][0]);
            acc[s][1] = fmaf(w.y, xs[s], acc[s][1]);
          }
#pragma unroll
          for (int s = 0; s + 1 < NS; ++s) xs[s] = xs[s + 1];
          xs[NS - 1] = xr[pos * kP + lane];
          pos = wrap(pos + 1);
        }
      } else {
        // spatial stem, taps in row-major order, zero outside the image
        const int y = (int)(ql / P.W), x = (int)(ql - (int64_t)y * P.W), r0 = ks0 >> 1;
        const int f = P.f0 + s0;
        for (int dy = 0; dy < ks0; ++dy) {
          const int yy = y + dy - r0;
          if (yy < 0 || yy >= P.H) continue;
          for (int dx = 0; dx < ks0; ++dx) {
            const int xx = x + dx - r0;
            if (xx < 0 || xx >= P.W) continue;
            const int64_t qq = (int64_t)yy * P.W + xx;
            const float2 w = *reinterpret_cast<const float2*>(w0 + (dy * ks0 + dx) * CP + c0);
            float fr[NS + 1];
#pragma unroll
            for (int s = 0; s <= NS; ++s) fr[s] = frame(f - 1 + min(s, tc), qq);
#pragma unroll
            for (int s = 0; s < NS; ++s) {
              acc[s][0] = fmaf(w.x, fr[s + 1] - fr[s], acc[s][0]);
              acc[s][1] = fmaf(w.y, fr[s + 1] - fr[s], acc[s][1]);
            }
          }
        }
      }
      put(ring(1, 0), base, nullptr);
      __syncthreads();
      // ---- layers 1 .. L - 1
      for (int l = 1; l < L; ++l) {
        const float* rl = ring(l, 0);
        const float* wl = sw + ((l - 1) * kt * (CP / 2) + warp) * 2 * CP;
        start(l);
        int pos = old;
        // the steps' rows of the current tap
        float4 x[NS][4];
        auto row = [&](float4 (&r)[4]) {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            r[j] = *reinterpret_cast<const float4*>(rl + pos * kRow + piece(lane, j));
          pos = wrap(pos + 1);
        };
#pragma unroll
        for (int s = 0; s < NS; ++s) row(x[s]);
        // tap t, the rows of step s at x[(s + o) % NS]
        auto tap = [&](int t, int o) {
          const float4* w4 = reinterpret_cast<const float4*>(wl + t * CP * CP);   // two input channels each
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float4 wa = w4[2 * j], wb = w4[2 * j + 1];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float wx = e == 0 ? wa.x : e == 1 ? wa.z : e == 2 ? wb.x : wb.z;
              const float wy = e == 0 ? wa.y : e == 1 ? wa.w : e == 2 ? wb.y : wb.w;
#pragma unroll
              for (int s = 0; s < NS; ++s) {
                const float4 xv = x[(s + o) % NS][j];
                const float xe = e == 0 ? xv.x : e == 1 ? xv.y : e == 2 ? xv.z : xv.w;
                acc[s][0] = fmaf(wx, xe, acc[s][0]);
                acc[s][1] = fmaf(wy, xe, acc[s][1]);
              }
            }
          }
        };
#pragma unroll
        for (int t = 0; t < kKt; ++t) {
          tap(t, t);
          if (t + 1 < kKt) row(x[t % NS]);
        }
        // a closing layer adds the block's input, which is its inner layer's;
        // the last layer's output goes to the scratch slots
        const bool last = l + 1 == L;
        put(last ? scratch : ring(l + 1, 0), last ? sc0 : base,
            P.kind == ET_NET_RESIDUAL && l >= 2 && l % 2 == 0 ? ring(l - 1, 0) : nullptr);
        __syncthreads();
      }
      // ---- Eq. 6 projection, warp j the chunk's step j
      if (warp < tc) {
        const float* r = scratch + wrap(sc0 + warp) * kRow;
        float Iv = sb[L * CP];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 v = *reinterpret_cast<const float4*>(r + piece(lane, j));
          Iv = fmaf(swp[4 * j], v.x, Iv);
          Iv = fmaf(swp[4 * j + 1], v.y, Iv);
          Iv = fmaf(swp[4 * j + 2], v.z, Iv);
          Iv = fmaf(swp[4 * j + 3], v.w, Iv);
        }
        sI[warp * kP + lane] = Iv;
      }
      __syncthreads();
      };
      // a call's few or last steps don't pay for eight
      if (tc > 4) steps(std::integral_constant<int, 8>());
      else if (tc > 2) steps(std::integral_constant<int, 4>());
      else steps(std::integral_constant<int, 2>());
      // ---- BiLIF (Eq. 2-3) by warp 0 while the others go on to the next chunk
      if (warp == 0) {
        for (int j = 0; j < tc; ++j) {
          const int f = P.f0 + s0 + j;
          const float I = sI[j * kP + lane];
          const float vp = P.beta * V + I;
          const int sp = vp >= P.vth ? 1 : (vp <= -P.vth ? -1 : 0);
          V = vp - P.reset * (float)sp;
          if (lane < np) {
            const int64_t o = (int64_t)(s0 + j) * npix + ql;
            if (I_out) I_out[o] = I;
            if (spikes) spikes[o] = (int8_t)sp;
          }
          // delayed labels below 0: none
          stage.add(lane < np && sp != 0 && P.t0 + f >= 0 ? 1u : 0u, (uint32_t)f, (uint32_t)f, sp);
        }
      }
      base = wrap(base + kT);
    }
    if (warp == 0) {
      stage.flush();
      if (lane < np) Vg[ql] = V;
    }
    // the last hk inputs of every layer back to the state, oldest first: step
    // S - hk + j at ring position (S + j) mod R
    const int first = S % R;
    for (int i = warp; i < (L - 1) * hk * 4; i += kThreads / 32) {
      const int c4 = (i & 3) * 4, j = (i >> 2) % hk, l = 1 + (i >> 2) / hk;
      const float4 v = *reinterpret_cast<const float4*>(ring(l, (first + j) % R) + piece(lane, i & 3));
      float* h = hist + (((int64_t)l * hk + j) * C + c4) * npix + ql;
      if (lane < np) {
        if (c4 < C) h[0] = v.x;
        if (c4 + 1 < C) h[npix] = v.y;
        if (c4 + 2 < C) h[2 * npix] = v.z;
        if (c4 + 3 < C) h[3 * npix] = v.w;
      }
    }
    if (ks0 == 0)
      for (int j = warp; j < hk; j += kThreads / 32)
        if (lane < np) hist[(int64_t)j * C * npix + ql] = xr[((first + j) % R) * kP + lane];
  }
}

// Whether evsnet_pix.cu takes less time for S steps.  This kernel pays for set-up
// and history once per tile and for up to eight steps at a time, and its stem reads
// the frames once per warp; the other one pays per step, and fills the device from
// 256 pixels per SM on instead of 32.  Both sides are sums fitted to 300 calls of
// each (C = 13 and 16, 2 to 7 layers, ks0 0 to 7, 1 to 32 steps, 187 x 253 to 720 x
// 1280; ns per 1000 pixels of full waves, within 15 and 28 %): the slower side is
// taken in few of them, by 14 % at most.  640 x 360, C = 16, here / there: 3 layers,
// 1 step 0.35 / 0.24 ms, 8 steps 0.65 / 0.81, behind a 5 x 5 stem 1.07 / 0.79; 7
// layers, 1 step 0.78 / 0.87, 16 steps 2.43 / 4.08.
bool pix_is_faster(const Pix16Params& P, int S, int64_t npix, int nsm) {
  auto waves = [&](int per) { return (npix + (int64_t)per * nsm - 1) / ((int64_t)per * nsm) * per; };
  const int64_t l = P.L - 1, rest = S % kT;
  const int64_t s8 = S - rest + (rest == 0 ? 0 : rest <= 2 ? 2 : rest <= 4 ? 4 : kT);   // steps as chunks run them
  const int64_t there = 23 * l * P.C + S * (43 + (19 * l * P.C + 1) / 2);
  const int64_t here = 520 + 295 * l + s8 * (80 + 71 * l) + P.ks0 * P.ks0 * (17 + 7 * (int64_t)S);
  return waves(256) * there < waves(kP) * here;
}

}  // namespace

int et_evsnet_forward_pix16(const float* logl, int32_t F, const et_evsnet_weights* net,
                            et_evsnet_state* st, int32_t t0, et_event* events, int64_t cap,
                            int64_t* n_events, float* I_out, int8_t* spikes, cudaStream_t stream) {
  if (net->ks != 1 || net->kt != kKt || net->C > CP || net->C <= CP - 4 || net->n_layers < 2)
    return ET_ERR_UNIMPLEMENTED;
  Pix16Params P{};
  P.kind = net->kind; P.L = net->n_layers; P.C = net->C; P.kt = net->kt; P.ks0 = net->ks0;
  P.R = P.kt - 1 + kT;
  P.beta = net->beta; P.vth = net->vth; P.reset = net->reset;
  P.H = st->H; P.W = st->W; P.F = F; P.f0 = st->initialized ? 0 : 1; P.t0 = t0;
  // a fresh state's first frame alone is no step: membrane and history stay as
  // they are.  The kernel counts on a step: its copies of the history become
  // visible to the warps that write it back at a step's barrier.
  if (P.F <= P.f0) return ET_OK;
  int wo = 0;
  const int taps0 = P.ks0 > 0 ? P.ks0 * P.ks0 : P.kt;
  for (int l = 0; l < P.L; ++l) {
    P.woff[l] = wo;
    wo += l == 0 ? P.C * taps0 : P.C * P.C * P.kt;
  }
  P.woff[P.L] = wo;
  P.off_w = (P.L - 1) * P.R * kRow;
  P.off_b = P.off_w + (P.L - 1) * P.kt * CP * CP + taps0 * CP + CP;
  P.off_x = P.off_b + P.L * CP + 4;
  P.off_I = P.off_x + (P.ks0 > 0 ? 0 : P.R * kP);
  P.off_s = P.L < 4 ? P.off_I + kT * kP : -1;
  const size_t smem = sizeof(float) * ((size_t)P.off_I + kT * kP + (P.L < 4 ? P.R * kRow : 0));
  const int64_t tiles = ((int64_t)P.H * P.W + kP - 1) / kP;
  P.tiles = (int)tiles;
  int dev = 0, max_smem = 0, nsm = 0;
  ET_CHECK_CUDA(cudaGetDevice(&dev));
  ET_CHECK_CUDA(cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  ET_CHECK_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  if (pix_is_faster(P, P.F - P.f0, (int64_t)P.H * P.W, nsm)) return ET_ERR_UNIMPLEMENTED;
  auto kern = evsnet_pix16_kernel;
  if (smem + sizeof(uint32_t) * kStageCap > (size_t)max_smem) return ET_ERR_UNIMPLEMENTED;
  const int rc = et_allow_shared(kern);
  if (rc != ET_OK) return rc;
  kern<<<(unsigned)std::min<int64_t>(tiles, nsm), kThreads, smem, stream>>>(
      P, logl, net->w, net->b, st->V, st->hist, st->last_l, events, cap,
      reinterpret_cast<unsigned long long*>(n_events), I_out, spikes);
  ET_CHECK_LAUNCH();
  return ET_OK;
}
