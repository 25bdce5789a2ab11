// Training of the paper's pixel-wise temporal EvSNet (Sec. 3.3, Eq. 5-6:
// convolutions along time only, kernel kt, optional residual blocks, a
// point-wise projection and BiLIF) on the GPU, FP32.
//
// With a 1x1 spatial extent every pixel is an independent 1-D network over the
// clip, so the activations are kept for the whole clip (no segment recompute
// of the convolutions is needed for the temporal coupling): layout
// [B][K][H W][C], one pixel-step's channels contiguous.  BiLIF keeps V at the
// start of every ckpt_every steps and runs its reverse recursion per segment,
// as the spatial form does.
//
// Convolution along time, causal: out[k][co] = b[co] + sum_ci,tau
// w[co][ci][tau] in[k - (kt - 1) + tau][ci]; steps before the clip are zero.
// Residual blocks (Eq. 5): a_i = ReLU(conv_{2i-1}(h_{i-1})),
// h_i = ReLU(h_{i-1} + conv_{2i}(a_i)).
#include <algorithm>
#include "et_internal.cuh"
#include "evsnet_common.h"
#include "train_api.h"
#include "train_tma.cuh"
#include "f32x2.cuh"

#define ET_TRY(expr)                 \
  do {                               \
    const int rc_ = (expr);          \
    if (rc_ != ET_OK) return rc_;    \
  } while (0)

namespace {

constexpr int kMaxC = 16;
constexpr int kMaxKt = 9;
constexpr float kPi = 3.14159265358979323846f;

// packed weight offset of layer l; n0 = weights per output channel of layer 0
// (kt, or ks0 * ks0 for a spatial stem)
inline int64_t twofs(int l, int C, int kt, int n0) {
  return l == 0 ? 0 : (int64_t)C * n0 + (int64_t)(l - 1) * C * C * kt;
}
inline int layer0_taps(const et_evsnet_weights* net) {
  return net->ks0 > 0 ? net->ks0 * net->ks0 : net->kt;
}

// ------------------------------------------------------- forward conv, layer 0
// 64 bytes written per pixel-step.  One thread per pixel computes
// all channels; a warp's 32 rows then go through shared memory (16-byte pieces
// permuted so that neither side meets a bank twice) and leave as whole 512-byte
// lines.  X is read as l_{k+1} - l_k from the clip's log frames.
constexpr int kMaxStem = 7;

// ReLU of a warp's 32 rows (lane = pixel idx0 + lane, `n` of them in the image)
// to out; a one-layer network also writes the projection I = bp + wp . out.
// stage: the warp's 2 KB.  vec: 16 channels and 16-byte aligned rows (here and
// below; otherwise rows are read and written a word at a time).
__device__ __forceinline__ void store_rows(float (&acc)[kMaxC], int64_t idx0, int n, int C, bool vec, float* stage,
                                           float* __restrict__ out, const float* __restrict__ wp,
                                           const float* __restrict__ bp, float* __restrict__ I) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int c = 0; c < kMaxC; ++c) acc[c] = fmaxf(acc[c], 0.0f);
  if (I && lane < n) {
    float Iv = bp[0];
#pragma unroll
    for (int c = 0; c < kMaxC; ++c)
      if (c < C) Iv = fmaf(wp[c], acc[c], Iv);
    I[idx0 + lane] = Iv;
  }
  if (vec) {
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 4; ++j)
      *reinterpret_cast<float4*>(stage + lane * kMaxC + 4 * (j ^ ((lane >> 1) & 3))) =
          make_float4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int pix = r * 8 + (lane >> 2), j = lane & 3;
      const float4 v = *reinterpret_cast<const float4*>(stage + pix * kMaxC + 4 * (j ^ ((pix >> 1) & 3)));
      if (pix < n) *reinterpret_cast<float4*>(out + (idx0 + pix) * kMaxC + 4 * j) = v;
    }
  } else if (lane < n) {
#pragma unroll
    for (int c = 0; c < kMaxC; ++c)
      if (c < C) out[(idx0 + lane) * C + c] = acc[c];
  }
}

__device__ __forceinline__ void fma_tap(const float* __restrict__ w, float x, float (&acc)[kMaxC]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float4 v = reinterpret_cast<const float4*>(w)[j];
    acc[4 * j] = fmaf(v.x, x, acc[4 * j]);
    acc[4 * j + 1] = fmaf(v.y, x, acc[4 * j + 1]);
    acc[4 * j + 2] = fmaf(v.z, x, acc[4 * j + 2]);
    acc[4 * j + 3] = fmaf(v.w, x, acc[4 * j + 3]);
  }
}

// [tap][channel] and biases, zero beyond C
__device__ __forceinline__ void stage_taps(float (*sw)[kMaxC], float* sb, const float* __restrict__ w,
                                           const float* __restrict__ b, int taps, int C) {
  for (int i = threadIdx.x; i < kMaxC * taps; i += blockDim.x) {
    const int t = i / kMaxC, c = i % kMaxC;
    sw[t][c] = c < C ? w[c * taps + t] : 0.0f;
  }
  if (threadIdx.x < kMaxC) sb[threadIdx.x] = threadIdx.x < C ? b[threadIdx.x] : 0.0f;
  __syncthreads();
}

// The layer-0 kernels walk along steps or rows with their neighbours in registers:
// long walks where there are 16 per SM, shorter ones in small calls, whose time is
// one walk's chain of loads (the longest throughout against these, 3 x 3 stem, 1 clip
// of 9 x 20 x 24: forward 29 -> 5.5 us, weight gradient 23 -> 9; a thread per
// pixel-step 6.2 and 10).
inline int walk_length(int longest, int shortest, int64_t want, int64_t others, int n) {
  int len = longest;
  while (len > shortest && others * ((n + len - 1) / len) < want) len /= 2;
  return len;
}

// Temporal layer 0, taps over the last kt steps: a thread walks up to kWalk steps
// of its pixel with the last T = 7 or 9 X in registers (T >= kt), one new log
// value per step (4 clips x 64 x 128 x 128: 0.30 -> 0.062 ms; HBM floor 0.042).
constexpr int kWalk = 16, kWalkMin = 4;
template <int T>
__global__ void __launch_bounds__(128)
tconv_fwd(const float* __restrict__ logl, int B, int K, int64_t hw, int C, bool vec, int kt, int walk,
          const float* __restrict__ w, const float* __restrict__ b, float* __restrict__ out,
          const float* __restrict__ wp, const float* __restrict__ bp, float* __restrict__ I) {
  __shared__ __align__(16) float sw[kMaxKt][kMaxC], sb[kMaxC], stage[4][32 * kMaxC];
  stage_taps(sw, sb, w, b, kt, C);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t groups = (uint32_t)((hw + 31) / 32), segs = (uint32_t)(K + walk - 1) / walk;
  const uint32_t it = blockIdx.x * 4 + warp;
  if (it >= (uint32_t)B * segs * groups) return;
  const int64_t p0 = (int64_t)(it % groups) * 32, p = min(p0 + lane, hw - 1);
  const int n = (int)min((int64_t)32, hw - p0);
  const int k0 = (int)(it / groups % segs) * walk, bc = (int)(it / groups / segs);
  const float* lf = logl + (int64_t)bc * (K + 1) * hw + p;
  float xs[T];                            // X of steps k - T + 1 .. k
#pragma unroll
  for (int t = 1; t < T; ++t) {
    const int k = k0 - T + t;
    xs[t] = k >= 0 ? lf[(int64_t)(k + 1) * hw] - lf[(int64_t)k * hw] : 0.0f;
  }
  float prev = lf[(int64_t)k0 * hw];
  const int ns = min(walk, K - k0);
  float nxt = lf[(int64_t)(k0 + 1) * hw];
  for (int j = 0; j < ns; ++j) {
    const int k = k0 + j;
#pragma unroll
    for (int t = 0; t + 1 < T; ++t) xs[t] = xs[t + 1];
    xs[T - 1] = nxt - prev;
    prev = nxt;
    nxt = lf[(int64_t)min(k + 2, K) * hw];
    float acc[kMaxC];
#pragma unroll
    for (int c = 0; c < kMaxC; ++c) acc[c] = sb[c];
    const int tau0 = max(0, kt - 1 - k) + T - kt;   // steps before the clip are zero: no product
#pragma unroll
    for (int t = 0; t < T; ++t)
      if (t >= tau0) fma_tap(sw[t - (T - kt)], xs[t], acc);
    store_rows(acc, ((int64_t)bc * K + k) * hw + p0, n, C, vec, stage[warp], out, wp, bp, I);
  }
}

// 3 x 3 spatial stem (one step, zero outside the image, taps in row-major
// order): a thread walks up to kRows rows of one column of one step with the X of
// three rows x three columns in registers (8 clips x 64 steps x 128 x 128: 0.50
// ms with 4-byte pieces written 64 bytes apart, now 0.167; HBM floor 0.084).
constexpr int kRows = 16;
struct Rows3 {
  const float* l1;                        // the step's frame and the one before, at the thread's column
  const float* l0;
  int H, W;
  bool lft, rgt;
  // X of row y, columns x - 1 .. x + 1, zero outside the image (loads always
  // inside it, so that the next rows' loads need no branch)
  __device__ __forceinline__ void load(int y, float (&r)[3]) const {
    const bool in = y >= 0 && y < H;
    const int64_t o = (int64_t)min(max(y, 0), H - 1) * W, ol = o - (lft ? 1 : 0), og = o + (rgt ? 1 : 0);
    const float a = l1[ol] - l0[ol], b = l1[o] - l0[o], c = l1[og] - l0[og];
    r[0] = in && lft ? a : 0.0f;
    r[1] = in ? b : 0.0f;
    r[2] = in && rgt ? c : 0.0f;
  }
};

__global__ void __launch_bounds__(128)
tstem3_fwd(const float* __restrict__ logl, int B, int K, int H, int W, int C, bool vec, int rows,
           const float* __restrict__ w, const float* __restrict__ b, float* __restrict__ out,
           const float* __restrict__ wp, const float* __restrict__ bp, float* __restrict__ I) {
  __shared__ __align__(16) float sw[9][kMaxC], sb[kMaxC], stage[4][32 * kMaxC];
  stage_taps(sw, sb, w, b, 9, C);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t hw = (int64_t)H * W;
  const uint32_t groups = (uint32_t)(W + 31) / 32, strips = (uint32_t)(H + rows - 1) / rows;
  const uint32_t it = blockIdx.x * 4 + warp;
  if (it >= (uint32_t)B * K * strips * groups) return;
  const int x0 = (int)(it % groups) * 32, x = min(x0 + lane, W - 1), y0 = (int)(it / groups % strips) * rows;
  const uint32_t bk = it / groups / strips;
  const float* l1 = logl + ((int64_t)(bk / K) * (K + 1) + bk % K + 1) * hw + x;
  const Rows3 R{l1, l1 - hw, H, W, x > 0, x + 1 < W};
  float r0[3], r1[3], r2[3];
  R.load(y0 - 1, r0);
  R.load(y0, r1);
  const int ny = min(rows, H - y0);
  R.load(y0 + 1, r2);
  for (int j = 0; j < ny; ++j) {
    const int y = y0 + j;
    float nx[3];
    R.load(y + 2, nx);
    float acc[kMaxC];
#pragma unroll
    for (int c = 0; c < kMaxC; ++c) acc[c] = sb[c];
    const bool up = y > 0, dn = y + 1 < H;
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      const float v = t < 3 ? r0[t % 3] : t < 6 ? r1[t % 3] : r2[t % 3];
      // taps outside the image: no product
      if ((t >= 3 || up) && (t < 6 || dn) && (t % 3 != 0 || R.lft) && (t % 3 != 2 || R.rgt)) fma_tap(sw[t], v, acc);
    }
    store_rows(acc, (int64_t)bk * hw + (int64_t)y * W + x0, min(32, W - x0), C, vec, stage[warp], out,
               wp, bp, I);
#pragma unroll
    for (int t = 0; t < 3; ++t) { r0[t] = r1[t]; r1[t] = r2[t]; r2[t] = nx[t]; }
  }
}

// the other stem sizes, one thread per pixel-step
__global__ void __launch_bounds__(128)
tstem_fwd(const float* __restrict__ logl, int B, int K, int H, int W, int C, bool vec, int ks0,
          const float* __restrict__ w, const float* __restrict__ b, float* __restrict__ out,
          const float* __restrict__ wp, const float* __restrict__ bp, float* __restrict__ I) {
  __shared__ __align__(16) float sw[kMaxStem * kMaxStem][kMaxC], sb[kMaxC], stage[4][32 * kMaxC];
  stage_taps(sw, sb, w, b, ks0 * ks0, C);
  const int64_t hw = (int64_t)H * W;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, r0 = ks0 >> 1;
  const int64_t p0 = ((int64_t)blockIdx.x * 4 + warp) * 32, p = min(p0 + lane, hw - 1);
  if (p0 >= hw) return;
  const int y = (int)(p / W), x = (int)(p - (int64_t)y * W);
  for (int bk = blockIdx.y; bk < B * K; bk += gridDim.y) {
    const float* l1 = logl + ((int64_t)(bk / K) * (K + 1) + bk % K + 1) * hw;
    const float* l0 = l1 - hw;
    float acc[kMaxC];
#pragma unroll
    for (int c = 0; c < kMaxC; ++c) acc[c] = sb[c];
    for (int dy = 0; dy < ks0; ++dy) {
      const int yy = y + dy - r0;
      if (yy < 0 || yy >= H) continue;
      for (int dx = 0; dx < ks0; ++dx) {
        const int xx = x + dx - r0;
        if (xx < 0 || xx >= W) continue;
        const int64_t q = (int64_t)yy * W + xx;
        fma_tap(sw[dy * ks0 + dx], l1[q] - l0[q], acc);
      }
    }
    __syncwarp();
    store_rows(acc, (int64_t)bk * hw + p0, (int)min((int64_t)32, hw - p0), C, vec, stage[warp], out, wp, bp, I);
  }
}

// --------------------------------------------------------------------- BiLIF
__device__ __forceinline__ float sg(float x, float alpha) {
  const float u = 0.5f * kPi * alpha * x;
  return 0.5f * alpha / (1.0f + u * u);
}

// One thread per (clip, pixel) over the whole clip; V at the start of every
// segment goes to V_ckpt [B][n_ckpt][hw].
__global__ void tbilif_fwd(const float* __restrict__ I, int B, int K, int64_t hw, int ck, int n_ckpt,
                           float beta, float vth, float reset, float* __restrict__ V_ckpt,
                           int8_t* __restrict__ spikes, float* __restrict__ S_on,
                           float* __restrict__ S_off, float* __restrict__ I_out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)B * hw) return;
  const int bc = (int)(i / hw);
  const int64_t p = i % hw;
  float v = 0.0f;
  for (int k = 0; k < K; ++k) {
    if (k % ck == 0) V_ckpt[((int64_t)bc * n_ckpt + k / ck) * hw + p] = v;
    const int64_t o = ((int64_t)bc * K + k) * hw + p;
    const float Iv = I[o];
    const float vp = beta * v + Iv;
    const float on = vp >= vth ? 1.0f : 0.0f, off = -vp >= vth ? 1.0f : 0.0f;
    v = vp - reset * (on - off);
    spikes[o] = (int8_t)(on - off);
    if (S_on) { S_on[o] = on; S_off[o] = off; }
    if (I_out) I_out[o] = Iv;
  }
}

// Reverse recursion per segment (V' recomputed from the segment's checkpoint).
__global__ void tbilif_bwd(const float* __restrict__ I, int B, int K, int64_t hw, int ck, int n_ckpt,
                           float beta, float vth, float reset, float alpha,
                           const float* __restrict__ V_ckpt, const float* __restrict__ dSon,
                           const float* __restrict__ dSoff, float* __restrict__ dI) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)B * hw) return;
  const int bc = (int)(i / hw);
  const int64_t p = i % hw;
  float g = 0.0f;
  for (int s = n_ckpt - 1; s >= 0; --s) {
    const int k0 = s * ck, nseg = min(ck, K - k0);
    float vps[kMaxSeg];
    float v = V_ckpt[((int64_t)bc * n_ckpt + s) * hw + p];
    for (int j = 0; j < nseg; ++j) {
      const float vp = beta * v + I[((int64_t)bc * K + k0 + j) * hw + p];
      const float on = vp >= vth ? 1.0f : 0.0f, off = -vp >= vth ? 1.0f : 0.0f;
      v = vp - reset * (on - off);
      vps[j] = vp;
    }
    for (int j = nseg - 1; j >= 0; --j) {
      const float vp = vps[j];
      const float a = sg(vp - vth, alpha), c = sg(-vp - vth, alpha);
      const int64_t o = ((int64_t)bc * K + k0 + j) * hw + p;
      const float gvp = g * (1.0f - reset * (a + c)) + dSon[o] * a - dSoff[o] * c;
      dI[o] = gvp;
      g = gvp * beta;
    }
  }
}

// ------------------------------------------------------ projection backward
// dz[c] = dI wp[c] 1(h > 0); grad wp[c] += sum dI h[c]; grad bp += sum dI.
// Bound by HBM (132 bytes per pixel-step): four lanes per pixel-step, 16-byte
// accesses (8 clips x 64 steps x 128 x 128: 0.57 -> 0.19 ms).
// a quad's channels 4 g .. of row idx (zero beyond C)
__device__ __forceinline__ float4 load_quad(const float* __restrict__ src, int64_t idx, int g, int C, bool vec) {
  if (vec) return __ldg(reinterpret_cast<const float4*>(src + idx * kMaxC) + g);
  const float* r = src + idx * C + 4 * g;
  return make_float4(4 * g < C ? r[0] : 0.0f, 4 * g + 1 < C ? r[1] : 0.0f, 4 * g + 2 < C ? r[2] : 0.0f,
                     4 * g + 3 < C ? r[3] : 0.0f);
}

__global__ void __launch_bounds__(256)
tproj_bwd(const float* __restrict__ dI, const float* __restrict__ h, int64_t n, int C, bool vec,
          const float* __restrict__ wp, float* __restrict__ dz, float* __restrict__ gwp,
          float* __restrict__ gbp) {
  __shared__ float red[8][kMaxC + 1];
  const int g = threadIdx.x & 3, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float wv[4], acc[4] = {}, accd = 0.0f;
#pragma unroll
  for (int j = 0; j < 4; ++j) wv[j] = 4 * g + j < C ? wp[4 * g + j] : 0.0f;
#pragma unroll 4
  for (int64_t i = (int64_t)blockIdx.x * 64 + (threadIdx.x >> 2); i < n; i += (int64_t)gridDim.x * 64) {
    const float d = dI[i];
    const float4 a = load_quad(h, i, g, C, vec);
    const float av[4] = {a.x, a.y, a.z, a.w};
    float z[4];
    accd += d;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      acc[j] += d * av[j];
      z[j] = av[j] > 0.0f ? d * wv[j] : 0.0f;
    }
    if (vec) {
      *reinterpret_cast<float4*>(dz + i * kMaxC + 4 * g) = make_float4(z[0], z[1], z[2], z[3]);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (4 * g + j < C) dz[i * C + 4 * g + j] = z[j];
    }
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[j] += __shfl_xor_sync(0xFFFFFFFFu, acc[j], o);
    accd += __shfl_xor_sync(0xFFFFFFFFu, accd, o);
  }
  if (lane < 4)
#pragma unroll
    for (int j = 0; j < 4; ++j) red[warp][4 * g + j] = acc[j];
  if (lane == 0) red[warp][kMaxC] = accd;
  __syncthreads();
  if (threadIdx.x < C || threadIdx.x == kMaxC) {
    float v = 0.0f;
    for (int wr = 0; wr < 8; ++wr) v += red[wr][threadIdx.x];
    atomicAdd(threadIdx.x < C ? gwp + threadIdx.x : gbp, v);
  }
}

// ------------------------------------------------- weight backward, layer 0
// Four lanes per pixel (lane g = output channels 4 g ..), the taps' sums in
// registers; one atomic per entry per block at the end.
// sums over the 8 pixels of a warp and the warps of a block, added to
// gw[co * taps + t] and gb[co]
template <int T>
__device__ __forceinline__ void quad_grads(float (&acc)[T][4], float (&bias)[4], int g, int C, int taps, int t0,
                                           float* __restrict__ gw, float* __restrict__ gb) {
  __shared__ float red[T + 1][kMaxC];
  for (int i = threadIdx.x; i < (T + 1) * kMaxC; i += blockDim.x) (&red[0][0])[i] = 0.0f;
  __syncthreads();
#pragma unroll
  for (int t = 0; t <= T; ++t)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float v = t < T ? acc[t < T ? t : 0][j] : bias[j];
      for (int o = 4; o < 32; o <<= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
      if ((threadIdx.x & 31) < 4) atomicAdd(&red[t][4 * g + j], v);
    }
  __syncthreads();
  for (int i = threadIdx.x; i < (T + 1) * kMaxC; i += blockDim.x) {
    const int t = i / kMaxC, co = i % kMaxC;
    if (co >= C) continue;
    if (t == T) atomicAdd(gb + co, red[t][co]);
    else if (t >= t0) atomicAdd(gw + co * taps + t - t0, red[t][co]);
  }
}

// Rows of dz on their way to one lane (its own 16 bytes of each): kAhead rows in
// flight by cp.async, since the taps' sums leave registers for 16 warps per SM
// only and a warp's 512 bytes per row are far from covering the HBM latency.
constexpr int kAhead = 8;
struct QuadRing {
  float4* slot;                            // this lane's first slot; the next one is 256 float4 on
  const float* src;
  int64_t idx0, step;                      // row of step j: idx0 + j step
  int g, C, n;
  bool vec;
  __device__ __forceinline__ void request(int j) {
    if (vec && j < n)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                       (uint32_t)__cvta_generic_to_shared(slot + (j & (kAhead - 1)) * 256)),
                   "l"(src + (idx0 + j * step) * kMaxC + 4 * g)
                   : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  __device__ __forceinline__ void start() {
#pragma unroll
    for (int j = 0; j < kAhead - 1; ++j) request(j);
  }
  // row j (in order), requesting row j + kAhead - 1
  __device__ __forceinline__ float4 take(int j) {
    request(j + kAhead - 1);
    if (!vec) return load_quad(src, idx0 + j * step, g, C, false);
    asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory");
    return slot[(j & (kAhead - 1)) * 256];
  }
};

// Temporal layer 0: grad w[co][tau] += sum dz[k][co] X[k - kt + 1 + tau];
// grad b[co] += sum dz[k][co].  A thread walks up to kWalkB steps of one pixel with
// the last T = 7 or 9 X in registers (T >= kt; the taps before are dropped):
// one new log value and one 16-byte row piece per step.  68 bytes per pixel-step
// (4 clips x 64 x 128 x 128: 0.41 ms with staged pixel-steps, 0.21 without the
// row ring, now 0.101; HBM floor 0.042).
constexpr int kWalkB = 32, kWalkBMin = 4;
template <int T>
__global__ void __launch_bounds__(256, 2)
tconv_bwd_weight(const float* __restrict__ dz, const float* __restrict__ logl, int B, int K,
                 int64_t hw, int C, bool vec, int kt, int walk, float* __restrict__ gw, float* __restrict__ gb) {
  __shared__ float4 ring[kAhead * 256];
  const int g = threadIdx.x & 3, pl = (threadIdx.x & 31) >> 2;
  float acc[T][4] = {}, bias[4] = {};
  // (a clip batch that fits the device has fewer than 2^32 rows: 32-bit item numbers)
  const uint32_t groups = (uint32_t)((hw + 7) / 8), segs = (uint32_t)(K + walk - 1) / walk;
  const uint32_t items = (uint32_t)B * segs * groups;
  for (uint32_t it = blockIdx.x * 8 + (threadIdx.x >> 5); it < items; it += gridDim.x * 8) {
    const int64_t p = (int64_t)(it % groups) * 8 + pl;
    const int k0 = (int)(it / groups % segs) * walk, bc = (int)(it / groups / segs);
    if (p >= hw) continue;
    const int n = min(walk, K - k0);
    QuadRing rows{ring + threadIdx.x, dz, ((int64_t)bc * K + k0) * hw + p, hw, g, C, n, vec};
    rows.start();
    const float* lf = logl + (int64_t)bc * (K + 1) * hw + p;
    float xs[T];                          // X of steps k - T + 1 .. k
#pragma unroll
    for (int t = 1; t < T; ++t) {
      const int k = k0 - T + t;
      xs[t] = k >= 0 ? lf[(int64_t)(k + 1) * hw] - lf[(int64_t)k * hw] : 0.0f;
    }
    float prev = lf[(int64_t)k0 * hw], nxt[4];   // log values of the next four steps
#pragma unroll
    for (int t = 0; t < 4; ++t) nxt[t] = lf[(int64_t)min(k0 + 1 + t, K) * hw];
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
#pragma unroll
      for (int t = 0; t + 1 < T; ++t) xs[t] = xs[t + 1];
      xs[T - 1] = nxt[0] - prev;
      prev = nxt[0];
#pragma unroll
      for (int t = 0; t < 3; ++t) nxt[t] = nxt[t + 1];
      nxt[3] = lf[(int64_t)min(k0 + j + 5, K) * hw];
      const float4 d = rows.take(j);
      bias[0] += d.x; bias[1] += d.y; bias[2] += d.z; bias[3] += d.w;
#pragma unroll
      for (int t = 0; t < T; ++t) {
        acc[t][0] = fmaf(d.x, xs[t], acc[t][0]);
        acc[t][1] = fmaf(d.y, xs[t], acc[t][1]);
        acc[t][2] = fmaf(d.z, xs[t], acc[t][2]);
        acc[t][3] = fmaf(d.w, xs[t], acc[t][3]);
      }
    }
  }
  quad_grads<T>(acc, bias, g, C, kt, T - kt, gw, gb);
}

// 3 x 3 stem: grad w[co][tap] += sum dz[k][co] X_nbr(tap)[k]; grad b[co] += sum
// dz[k][co].  A thread walks up to kRowsB rows of one column of one step with the X of
// three rows x three columns in registers: three new X (six log values) and one
// 16-byte row piece per pixel.  68 bytes per pixel-step (8 clips x 64 x 128 x
// 128: 1.25 ms with staged pixel-steps, 0.40 without the row ring, now 0.255;
// HBM floor 0.084).
constexpr int kRowsB = 32;
__global__ void __launch_bounds__(256, 2)
tstem3_bwd_weight(const float* __restrict__ dz, const float* __restrict__ logl, int B, int K, int H,
                  int W, int C, bool vec, int walk, float* __restrict__ gw, float* __restrict__ gb) {
  __shared__ float4 ring[kAhead * 256];
  const int g = threadIdx.x & 3, pl = (threadIdx.x & 31) >> 2;
  float acc[9][4] = {}, bias[4] = {};
  const int64_t hw = (int64_t)H * W;
  const uint32_t groups = (uint32_t)(W + 7) / 8, strips = (uint32_t)(H + walk - 1) / walk;
  const uint32_t items = (uint32_t)B * K * strips * groups;
  for (uint32_t it = blockIdx.x * 8 + (threadIdx.x >> 5); it < items; it += gridDim.x * 8) {
    const int x = (int)(it % groups) * 8 + pl, y0 = (int)(it / groups % strips) * walk;
    const uint32_t bk = it / groups / strips;
    if (x >= W) continue;
    const float* l1 = logl + ((int64_t)(bk / K) * (K + 1) + bk % K + 1) * hw + x;
    const Rows3 R{l1, l1 - hw, H, W, x > 0, x + 1 < W};
    const int n = min(walk, H - y0);
    QuadRing rows{ring + threadIdx.x, dz, bk * hw + (int64_t)y0 * W + x, W, g, C, n, vec};
    rows.start();
    float r0[3], r1[3], r2[3], r3[3];
    R.load(y0 - 1, r0);
    R.load(y0, r1);
    R.load(y0 + 1, r2);
    R.load(y0 + 2, r3);
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
      float nx[3];
      R.load(y0 + j + 3, nx);
      const float4 d = rows.take(j);
      bias[0] += d.x; bias[1] += d.y; bias[2] += d.z; bias[3] += d.w;
#pragma unroll
      for (int t = 0; t < 9; ++t) {
        const float v = t < 3 ? r0[t % 3] : t < 6 ? r1[t % 3] : r2[t % 3];
        acc[t][0] = fmaf(d.x, v, acc[t][0]);
        acc[t][1] = fmaf(d.y, v, acc[t][1]);
        acc[t][2] = fmaf(d.z, v, acc[t][2]);
        acc[t][3] = fmaf(d.w, v, acc[t][3]);
      }
#pragma unroll
      for (int t = 0; t < 3; ++t) { r0[t] = r1[t]; r1[t] = r2[t]; r2[t] = r3[t]; r3[t] = nx[t]; }
    }
  }
  quad_grads<9>(acc, bias, g, C, 9, 0, gw, gb);
}

// -------------------------------------- weight backward, spatial stem
// The other stem sizes (1, 5, 7): persistent blocks stage 128 pixel-steps at a
// time in shared memory; each thread owns (co, tap) entries, one atomic per
// entry per block.
constexpr int kPts = 128;
__global__ void __launch_bounds__(256)
tstem_bwd_weight(const float* __restrict__ dz, const float* __restrict__ logl, int B, int K, int H,
                 int W, int C, int ks0, float* __restrict__ gw, float* __restrict__ gb) {
  constexpr int kTaps = kMaxStem * kMaxStem;
  __shared__ float sd[kPts][kMaxC];
  __shared__ float sx[kPts][kTaps + 1];
  constexpr int kPer = (kMaxC * kTaps + kMaxC + 255) / 256;
  float acc[kPer];
#pragma unroll
  for (int j = 0; j < kPer; ++j) acc[j] = 0.0f;
  const int nt = ks0 * ks0, r0 = ks0 >> 1;
  const int nent = C * nt + C;
  const int64_t hw = (int64_t)H * W;
  const int64_t npts = (int64_t)B * K * hw;
  for (int64_t c0 = (int64_t)blockIdx.x * kPts; c0 < npts; c0 += (int64_t)gridDim.x * kPts) {
    __syncthreads();
    for (int i = threadIdx.x; i < kPts * C; i += blockDim.x) {
      const int pt = i / C, co = i % C;
      const int64_t idx = c0 + pt;
      sd[pt][co] = idx < npts ? dz[idx * C + co] : 0.0f;
    }
    for (int i = threadIdx.x; i < kPts * nt; i += blockDim.x) {
      const int pt = i / nt, tap = i % nt;
      const int64_t idx = c0 + pt;
      float v = 0.0f;
      if (idx < npts) {
        const int64_t p = idx % hw;
        const int k = (int)((idx / hw) % K), bc = (int)(idx / (hw * K));
        const int yy = (int)(p / W) + tap / ks0 - r0, xx = (int)(p % W) + tap % ks0 - r0;
        if (yy >= 0 && yy < H && xx >= 0 && xx < W) {
          const float* l1 = logl + ((int64_t)bc * (K + 1) + k + 1) * hw;
          const int64_t q = (int64_t)yy * W + xx;
          v = l1[q] - l1[q - hw];
        }
      }
      sx[pt][tap] = v;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      const int e = threadIdx.x + j * 256;
      if (e >= nent) break;
      float s = 0.0f;
      if (e < C * nt) {
        const int co = e / nt, tap = e % nt;
        for (int pt = 0; pt < kPts; ++pt) s += sd[pt][co] * sx[pt][tap];
      } else {
        const int co = e - C * nt;
        for (int pt = 0; pt < kPts; ++pt) s += sd[pt][co];
      }
      acc[j] += s;
    }
  }
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const int e = threadIdx.x + j * 256;
    if (e >= nent) break;
    if (e < C * nt) atomicAdd(gw + e, acc[j]);
    else atomicAdd(gb + (e - C * nt), acc[j]);
  }
}

// ------------------------------------------- C -> C layers, vectorised weights
// The layers with C < 16 input channels, or whose rows lie off 16-byte
// boundaries: weights staged as [tau][input][output],
// zero-padded to 16 x 16 per tap, so that one 16-byte shared load (the same
// address for the whole warp) feeds four FMAs.  (C = 16 otherwise: the kernels below.)
constexpr int CP = 16;

__device__ __forceinline__ void load_ch(const float* __restrict__ src, int C, float (&x)[CP]) {
#pragma unroll
  for (int c = 0; c < CP; ++c) x[c] = c < C ? __ldg(src + c) : 0.0f;
}

// acc0[o] += sum_i w[i][o] x0[i] and acc1[o] += sum_i w[i][o] x1[i] for one tap's
// 16 x 16 block of shared weights: two steps per weight load
__device__ __forceinline__ void fma_block2(const float* __restrict__ w, const float (&x0)[CP],
                                           const float (&x1)[CP], int C, float (&acc0)[CP],
                                           float (&acc1)[CP]) {
#pragma unroll
  for (int i = 0; i < CP; ++i) {
    if (i >= C) break;
    const float4* w4 = reinterpret_cast<const float4*>(w + i * CP);
#pragma unroll
    for (int j = 0; j < CP / 4; ++j) {
      const float4 v = w4[j];
      acc0[4 * j] = fmaf(v.x, x0[i], acc0[4 * j]);
      acc0[4 * j + 1] = fmaf(v.y, x0[i], acc0[4 * j + 1]);
      acc0[4 * j + 2] = fmaf(v.z, x0[i], acc0[4 * j + 2]);
      acc0[4 * j + 3] = fmaf(v.w, x0[i], acc0[4 * j + 3]);
      acc1[4 * j] = fmaf(v.x, x1[i], acc1[4 * j]);
      acc1[4 * j + 1] = fmaf(v.y, x1[i], acc1[4 * j + 1]);
      acc1[4 * j + 2] = fmaf(v.z, x1[i], acc1[4 * j + 2]);
      acc1[4 * j + 3] = fmaf(v.w, x1[i], acc1[4 * j + 3]);
    }
  }
}

// a pixel-step's channels, zero outside the clip's steps [0, K)
__device__ __forceinline__ void load_step(const float* __restrict__ base, int k, int K, int64_t step,
                                          int C, float (&x)[CP]) {
  if (k < 0 || k >= K) {
#pragma unroll
    for (int c = 0; c < CP; ++c) x[c] = 0.0f;
  } else {
    load_ch(base + k * step, C, x);
  }
}

// forward of a C -> C layer: out = ReLU(b + conv(in) [+ res]), the last layer
// also I = bp + wp . out.  One thread per (clip, pair of steps 2j and 2j + 1,
// pixel): each tap's weights serve both steps, the input of step k - kt + 2 + tau
// serving the second step at tap tau and the first at tau + 1.
__global__ void __launch_bounds__(256, 3)
tconv16_fwd(const float* __restrict__ in, int B, int K, int64_t hw, int C, int kt,
            const float* __restrict__ w, const float* __restrict__ b, const float* __restrict__ res,
            float* __restrict__ out, const float* __restrict__ wp, const float* __restrict__ bp,
            float* __restrict__ I) {
  __shared__ __align__(16) float sw[kMaxKt * CP * CP];   // [tau][ci][co]
  for (int i = threadIdx.x; i < kt * CP * CP; i += blockDim.x) {
    const int co = i % CP, ci = (i / CP) % CP, tau = i / (CP * CP);
    sw[i] = (co < C && ci < C) ? w[(co * C + ci) * kt + tau] : 0.0f;
  }
  __syncthreads();
  const int KP = (K + 1) / 2;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)B * KP * hw) return;
  const int64_t p = t % hw;
  const int k = 2 * (int)((t / hw) % KP), bc = (int)(t / (hw * KP));
  const int64_t step = hw * C;
  const float* base = in + ((int64_t)bc * K * hw + p) * C;
  float acc0[CP], acc1[CP];
#pragma unroll
  for (int co = 0; co < CP; ++co) acc0[co] = acc1[co] = co < C ? b[co] : 0.0f;
  float xa[CP];
  load_step(base, k - (kt - 1), K, step, C, xa);
  for (int tau = 0; tau < kt; ++tau) {
    float xb[CP];
    load_step(base, k - (kt - 1) + tau + 1, K, step, C, xb);
    fma_block2(sw + tau * CP * CP, xa, xb, C, acc0, acc1);
#pragma unroll
    for (int c = 0; c < CP; ++c) xa[c] = xb[c];
  }
  auto finish = [&](float (&acc)[CP], int h) {
    const int64_t idx = ((int64_t)bc * K + k + h) * hw + p;
    float Iv = bp ? bp[0] : 0.0f;
#pragma unroll
    for (int co = 0; co < CP; ++co) {
      if (co >= C) break;
      const float z = res ? acc[co] + res[idx * C + co] : acc[co];
      acc[co] = fmaxf(z, 0.0f);
      if (I) Iv += wp[co] * acc[co];
    }
#pragma unroll
    for (int co = 0; co < CP; ++co)
      if (co < C) out[idx * C + co] = acc[co];
    if (I) I[idx] = Iv;
  };
  finish(acc0, 0);
  if (k + 1 < K) finish(acc1, 1);
}

// data backward: out[s][ci] = (add[s][ci] + sum_tau,co w[co][ci][tau] dz[s + kt - 1 - tau][co])
// 1(mask[s][ci] > 0); weights staged [tau][co][ci]; two steps per thread as above
__global__ void __launch_bounds__(256, 3)
tconv16_bwd_data(const float* __restrict__ dz, int B, int K, int64_t hw, int C, int kt,
                 const float* __restrict__ w, const float* __restrict__ add,
                 const float* __restrict__ mask, float* __restrict__ out) {
  __shared__ __align__(16) float sw[kMaxKt * CP * CP];   // [tau][co][ci]
  for (int i = threadIdx.x; i < kt * CP * CP; i += blockDim.x) {
    const int ci = i % CP, co = (i / CP) % CP, tau = i / (CP * CP);
    sw[i] = (co < C && ci < C) ? w[(co * C + ci) * kt + tau] : 0.0f;
  }
  __syncthreads();
  const int KP = (K + 1) / 2;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)B * KP * hw) return;
  const int64_t p = t % hw;
  const int s = 2 * (int)((t / hw) % KP), bc = (int)(t / (hw * KP));
  const int64_t step = hw * C;
  const float* base = dz + ((int64_t)bc * K * hw + p) * C;
  float acc0[CP], acc1[CP];
#pragma unroll
  for (int ci = 0; ci < CP; ++ci) acc0[ci] = acc1[ci] = 0.0f;
  float gb[CP];   // dz[s + kt - tau] for the second step
  load_step(base, s + kt, K, step, C, gb);
  for (int tau = 0; tau < kt; ++tau) {
    float ga[CP];
    load_step(base, s + kt - 1 - tau, K, step, C, ga);
    fma_block2(sw + tau * CP * CP, ga, gb, C, acc0, acc1);
#pragma unroll
    for (int c = 0; c < CP; ++c) gb[c] = ga[c];
  }
  auto finish = [&](const float (&acc)[CP], int h) {
    const int64_t idx = ((int64_t)bc * K + s + h) * hw + p;
#pragma unroll
    for (int ci = 0; ci < CP; ++ci) {
      if (ci >= C) break;
      const int64_t o = idx * C + ci;
      const float v = add ? add[o] + acc[ci] : acc[ci];
      out[o] = mask[o] > 0.0f ? v : 0.0f;
    }
  };
  finish(acc0, 0);
  if (s + 1 < K) finish(acc1, 1);
}

// weight backward of a C -> C layer: grad w[co][ci][tau] += sum dz[k][co] in[k - kt + 1 + tau][ci],
// grad b[co] += sum dz[k][co].  Persistent blocks stage kPts16 pixel-steps:
// dz as [pt][16], the shifted inputs as [pt][tau][16].  Thread e < 16 kt owns
// (tap tau = e / 16, output quad e % 4, input quad (e / 4) % 4), 16 sums with
// two 16-byte shared loads per 16 FMAs; the next 16 threads own the bias sums.
constexpr int kPts16 = 64;
inline int twgrad_threads(int kt) { return (16 * kt + 16 + 31) / 32 * 32; }

__global__ void __launch_bounds__(320)
tconv16_bwd_weight(const float* __restrict__ dz, const float* __restrict__ in, int B, int K,
                   int64_t hw, int C, int kt, float* __restrict__ gw, float* __restrict__ gb) {
  extern __shared__ __align__(16) float tsm[];
  float* sd = tsm;                      // [kPts16][CP]
  float* sx = tsm + kPts16 * CP;        // [kPts16][kt][CP]
  __shared__ int64_t s_row0[kPts16];    // offset of the point's pixel at step 0 of its clip
  __shared__ int s_k[kPts16];           // the point's step, -1 past the end
  const int e = threadIdx.x;
  const int tau = e / 16, cq = e % 4, iq = (e / 4) % 4;
  float acc[4][4] = {};
  float bsum = 0.0f;
  const int64_t npts = (int64_t)B * K * hw, step = hw * C;
  for (int64_t c0 = (int64_t)blockIdx.x * kPts16; c0 < npts; c0 += (int64_t)gridDim.x * kPts16) {
    __syncthreads();
    for (int pt = threadIdx.x; pt < kPts16; pt += blockDim.x) {
      const int64_t idx = c0 + pt;
      if (idx < npts) {
        const int64_t p = idx % hw;
        const int k = (int)((idx / hw) % K), bc = (int)(idx / (hw * K));
        s_row0[pt] = ((int64_t)bc * K * hw + p) * C;
        s_k[pt] = k;
      } else {
        s_row0[pt] = 0;
        s_k[pt] = -1;
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kPts16 * CP; i += blockDim.x) {
      const int pt = i / CP, co = i % CP;
      sd[i] = (s_k[pt] >= 0 && co < C) ? dz[(c0 + pt) * C + co] : 0.0f;
    }
    for (int i = threadIdx.x; i < kPts16 * kt * CP; i += blockDim.x) {
      const int pt = i / (kt * CP), r = i % (kt * CP), tt = r / CP, ci = r % CP;
      const int kk = s_k[pt] - (kt - 1) + tt;
      sx[i] = (s_k[pt] >= 0 && kk >= 0 && ci < C) ? in[s_row0[pt] + kk * step + ci] : 0.0f;
    }
    __syncthreads();
    if (e < 16 * kt) {
#pragma unroll 4
      for (int pt = 0; pt < kPts16; ++pt) {
        const float4 d = *reinterpret_cast<const float4*>(sd + pt * CP + 4 * cq);
        const float4 x = *reinterpret_cast<const float4*>(sx + (pt * kt + tau) * CP + 4 * iq);
        const float dv[4] = {d.x, d.y, d.z, d.w}, xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[a][c] = fmaf(dv[a], xv[c], acc[a][c]);
      }
    } else if (e < 16 * kt + CP) {
      const int co = e - 16 * kt;
      for (int pt = 0; pt < kPts16; ++pt) bsum += sd[pt * CP + co];
    }
  }
  if (e < 16 * kt) {
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int co = 4 * cq + a, ci = 4 * iq + c;
        if (co < C && ci < C) atomicAdd(gw + (co * C + ci) * kt + tau, acc[a][c]);
      }
  } else if (e < 16 * kt + C) {
    atomicAdd(gb + (e - 16 * kt), bsum);
  }
}

// ------------------------------------------------- C -> C layers of 16 channels
// Forward (out = ReLU(b + conv(in) [+ extra]), the last layer also I = bp + wp .
// out) and data gradient (out = ([extra +] conv^T(in)) 1(mask > 0); in reversed
// time the same causal convolution) of a layer: each output sums its taps oldest
// first and, within a tap, channels in order, like tconv16_fwd / _bwd_data.
// A CTA owns 128 pixels and walks chunks of 8 steps, numbered with time innermost
// and split evenly over one CTA per SM.  Steps arrive as TMA boxes (64-byte rows,
// read by each pixel's thread without bank conflicts) in three groups of 8: the
// previous chunk's (its last kt - 1 steps are this chunk's past), this one's and
// the next one's.  A thread computes 4 steps of a pixel: four input channels of a tap
// are 16 weight loads (the same address for the whole warp) and 4 input ones for 128
// pair multiply-adds, 80 clk of shared memory (4 per 16-byte load of a warp) for 64 of
// the FP32 pipe: shared memory bounds it (4 clips x 64 x 128 x 128: 0.35 ms forward, 0.38
// data gradient).
constexpr int kStepChunk = 8;
constexpr int kRing = 3 * kStepChunk;
constexpr uint32_t kDrainIters = 1u << 22;   // bound of the waits for boxes in flight after a wait gave up

struct F32ConvArgs {
  int K, kt;
  int64_t hw;
  int tiles, nch;
  int64_t total;           // B * tiles * nch chunks
  const float* w;
  const float* b;
  const float* extra;
  const float* mask;
  float* out;
  const float* wp;
  const float* bp;
  float* I;
  uint32_t wait_iters;
};

template <bool kBwd>
__global__ void __launch_bounds__(256, 1)
tconv16_tma(const __grid_constant__ CUtensorMap m_in, F32ConvArgs A) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint64_t bar[3];
  const int tid = threadIdx.x, px = tid & (kBoxPix - 1), half = tid >> 7;
  const int K = A.K, kt = A.kt, nch = A.nch;
  float* sw = reinterpret_cast<float*>(sm + kRing * kBox);     // [tau][input][output]
  for (int i = tid; i < kt * 256; i += 256) {
    const int tau = i % kt, r = i / kt, lo = r % 16, hi = r / 16;   // w[hi = co][lo = ci][tau]
    sw[(tau * 16 + (kBwd ? hi : lo)) * 16 + (kBwd ? lo : hi)] = A.w[i];
  }
  if (tid == 0)
    for (int i = 0; i < 3; ++i) mbar_init(&bar[i], 1);
  __syncthreads();
  const int64_t t0 = A.total * blockIdx.x / gridDim.x, t1 = A.total * (blockIdx.x + 1) / gridDim.x;
  // processing order u = 0 .. K-1 is time s = u (forward) or s = K-1-u (data gradient)
  auto step_of = [&](int u) { return kBwd ? K - 1 - u : u; };
  // chunk t lives in group (t - t0 + 1) mod 3; thread 0 requests its boxes
  uint32_t asked = 0, asked_odd = 0;     // thread 0: groups requested, and those requested an odd number of times
  auto load_chunk = [&](int64_t t) {
    const int64_t sg = t / nch;
    const int c = (int)(t - sg * nch), tile = (int)(sg % A.tiles), bc = (int)(sg / A.tiles);
    const int g = (int)((t - t0 + 1) % 3), n = min(kStepChunk, K - kStepChunk * c);
    asked |= 1u << g;
    asked_odd ^= 1u << g;
    mbar_arrive_expect_tx(&bar[g], (uint32_t)(n * kBox));
    for (int j = 0; j < n; ++j)
      tma_load_3d(sm + (g * kStepChunk + j) * kBox, &m_in, 0, tile * kBoxPix, bc * K + step_of(kStepChunk * c + j),
                  &bar[g]);
  };
  const bool mid = t0 % nch != 0;        // the range starts inside a clip: its past is the chunk before
  if (tid == 0) {
    if (mid) load_chunk(t0 - 1);
    if (t0 < t1) load_chunk(t0);
    if (t0 + 1 < t1) load_chunk(t0 + 1);
  }
  uint32_t phase = 0;
  bool ok = true, bail = false;
  if (mid) { ok = mbar_wait(&bar[0], 0, A.wait_iters); phase ^= 1u; }
  int64_t seg = t0 / nch;
  int c = (int)(t0 - seg * nch), tile = (int)(seg % A.tiles), bc = (int)(seg / A.tiles);
  int g = 1;
  int64_t t = t0;
  while (t < t1) {
    const int gp = g == 0 ? 2 : g - 1;   // the previous chunk's group
    if (c == 0) {                        // steps before the clip are zero
      uint4* z = reinterpret_cast<uint4*>(sm + (gp * kStepChunk + kStepChunk - (kt - 1)) * kBox);
      for (int i = tid; i < (kt - 1) * kBox / 16; i += 256) z[i] = make_uint4(0, 0, 0, 0);
      __syncthreads();
    }
    ok &= mbar_wait(&bar[g], (phase >> g) & 1u, A.wait_iters);
    phase ^= 1u << g;
    const int u0 = kStepChunk * c + 4 * half;
    const int64_t p = (int64_t)tile * kBoxPix + px;
    if (u0 < K) {
      f32x2 acc[4][8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const f32x2 b0 = kBwd ? 0ull : pack2f(__ldg(A.b + 2 * i), __ldg(A.b + 2 * i + 1));
#pragma unroll
        for (int s = 0; s < 4; ++s) acc[s][i] = b0;
      }
      int pos = g * kStepChunk + 4 * half - (kt - 1);   // ring position of the first step's oldest tap
      if (pos < 0) pos += kRing;
#pragma unroll 1
      for (int tau = 0; tau < kt; ++tau) {
        const unsigned char* row[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) row[s] = sm + (pos + s >= kRing ? pos + s - kRing : pos + s) * kBox;
        const float* wt = sw + tau * 256;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float4 x[4];
#pragma unroll
          for (int s = 0; s < 4; ++s) x[s] = *box_row(row[s], px, q);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            ulonglong2 wv[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) wv[j] = reinterpret_cast<const ulonglong2*>(wt + (4 * q + e) * 16)[j];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
              const float xe = e == 0 ? x[s].x : e == 1 ? x[s].y : e == 2 ? x[s].z : x[s].w;
              const f32x2 xx = pack2f(xe, xe);
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                acc[s][2 * j] = fma2(wv[j].x, xx, acc[s][2 * j]);
                acc[s][2 * j + 1] = fma2(wv[j].y, xx, acc[s][2 * j + 1]);
              }
            }
          }
        }
        pos = pos + 1 == kRing ? 0 : pos + 1;
      }
      if (p < A.hw) {
        float4 ex[4][4], mk[4][4];
        int64_t idx[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          idx[s] = ((int64_t)bc * K + step_of(min(u0 + s, K - 1))) * A.hw + p;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (A.extra) ex[s][j] = __ldg(reinterpret_cast<const float4*>(A.extra + idx[s] * 16) + j);
            if (kBwd) mk[s][j] = __ldg(reinterpret_cast<const float4*>(A.mask + idx[s] * 16) + j);
          }
        }
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          if (u0 + s >= K) break;
          float Iv = (!kBwd && A.I) ? A.bp[0] : 0.0f;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            float v[4];
            unpack2f(acc[s][2 * j], v[0], v[1]);
            unpack2f(acc[s][2 * j + 1], v[2], v[3]);
            const float e4[4] = {ex[s][j].x, ex[s][j].y, ex[s][j].z, ex[s][j].w};
            const float m4[4] = {mk[s][j].x, mk[s][j].y, mk[s][j].z, mk[s][j].w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if (A.extra) v[i] = v[i] + e4[i];
              if (kBwd) {
                v[i] = m4[i] > 0.0f ? v[i] : 0.0f;
              } else {
                v[i] = fmaxf(v[i], 0.0f);
                if (A.I) Iv = fmaf(__ldg(A.wp + 4 * j + i), v[i], Iv);
              }
            }
            reinterpret_cast<float4*>(A.out + idx[s] * 16)[j] = make_float4(v[0], v[1], v[2], v[3]);
          }
          if (!kBwd && A.I) A.I[idx[s]] = Iv;
        }
      }
    }
    fence_proxy_async_smem();
    bail = __syncthreads_or(!ok) != 0;
    if (bail) break;
    // the previous chunk's group is free for the chunk after the next
    if (tid == 0 && t + 2 < t1) load_chunk(t + 2);
    g = g == 2 ? 0 : g + 1;
    if (++c == nch) {
      c = 0;
      if (++tile == A.tiles) { tile = 0; ++bc; }
    }
    ++t;
  }
  if (!bail) return;
  // a box did not come within the bound: this chunk and those left become NaN, so
  // that the loss shows the failure, and the boxes in flight are waited for
  // (bounded) before the shared memory is given back
  const float nan = __int_as_float(0x7fc00000);
  for (; t < t1; ++t) {
    seg = t / nch;
    c = (int)(t - seg * nch); tile = (int)(seg % A.tiles); bc = (int)(seg / A.tiles);
    const int64_t p = (int64_t)tile * kBoxPix + px;
    for (int u = kStepChunk * c + 4 * half; p < A.hw && u < min(K, kStepChunk * c + 4 * half + 4); ++u) {
      const int64_t idx = ((int64_t)bc * K + step_of(u)) * A.hw + p;
      for (int j = 0; j < 4; ++j) reinterpret_cast<float4*>(A.out + idx * 16)[j] = make_float4(nan, nan, nan, nan);
      if (!kBwd && A.I) A.I[idx] = nan;
    }
  }
  if (tid == 0)
    for (int i = 0; i < 3; ++i)
      if ((asked >> i) & 1u) mbar_wait(&bar[i], ((asked_odd >> i) & 1u) ^ 1u, kDrainIters);
}

// Weight gradient: grad w[co][ci][tau] += sum dz[k][co] in[k - kt + 1 + tau][ci],
// grad b[co] += sum dz[k][co].  A warp walks two neighbouring pixels through
// time, lane = (pixel, 4 output channels, 4 input channels): the last T >= kt
// input rows stay in registers, so a step's two 16-byte reads serve T x 16
// multiply-adds (T = 7: 56 pair instructions of 66 issued).  The rows come
// through a ring of kWDepth steps per warp, filled by cp.async (128 bytes of
// either tensor per step).
constexpr int kWDepth = 16;
constexpr int kWWarps = 8;
template <int T>
__global__ void __launch_bounds__(32 * kWWarps, 1)
tconv16_wgrad_walk(const float* __restrict__ dz, const float* __restrict__ in, int B, int K, int64_t hw, int kt,
                   int seg, float* __restrict__ gw, float* __restrict__ gb) {
  __shared__ __align__(16) float ring[kWWarps][kWDepth][2][2][16];   // [step][dz, in][pixel][channel]
  __shared__ float sum[T * 256 + 16];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int pix = lane >> 4, cq = lane & 3, iq = (lane >> 2) & 3;
  f32x2 acc[T][4][2];
#pragma unroll
  for (int t = 0; t < T; ++t)
#pragma unroll
    for (int a = 0; a < 4; ++a) acc[t][a][0] = acc[t][a][1] = 0ull;
  float bias[4] = {};
  const uint32_t pairs = (uint32_t)((hw + 1) / 2), segs = (uint32_t)(K + seg - 1) / seg;
  const uint32_t items = (uint32_t)B * segs * pairs;   // rows that fit the device: below 2^32
  for (uint32_t it = blockIdx.x * kWWarps + warp; it < items; it += gridDim.x * kWWarps) {
    const int64_t p0 = (int64_t)(it % pairs) * 2;
    const int k0 = (int)(it / pairs % segs) * seg, bc = (int)(it / pairs / segs);
    const int k1 = min(K, k0 + seg), kb = max(0, k0 - (kt - 1));   // steps kb .. k0 - 1 only fill the registers
    const bool live = p0 + pix < hw;
    // lanes 0-15 copy 16 bytes each of a step's rows
    const int lt = (lane >> 3) & 1, lp = (lane >> 2) & 1, lc = lane & 3;
    const bool copy = lane < 16 && p0 + lp < hw;
    const float* src = (lt ? in : dz) + (((int64_t)bc * K) * hw + p0 + lp) * 16 + 4 * lc;
    auto request = [&](int k) {
      if (copy && k < k1)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         smem_u32(&ring[warp][k & (kWDepth - 1)][lt][lp][4 * lc])),
                     "l"(src + (int64_t)k * hw * 16)
                     : "memory");
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    __syncwarp();                        // the ring of the previous item has been read
#pragma unroll
    for (int j = 0; j < kWDepth - 1; ++j) request(kb + j);
    f32x2 xr[T][2];                      // input rows of the last T steps, row of step kb + j at j mod T
#pragma unroll
    for (int t = 0; t < T; ++t) xr[t][0] = xr[t][1] = 0ull;
    for (int kk = kb; kk < k1; kk += T) {
#pragma unroll
      for (int r = 0; r < T; ++r) {
        const int k = kk + r;
        if (k < k1) {
          asm volatile("cp.async.wait_group %0;" ::"n"(kWDepth - 2) : "memory");
          __syncwarp();                  // every lane's copies of step k have landed; step k - 1 has been read
          request(k + kWDepth - 1);
          const float(*row)[2][16] = ring[warp][k & (kWDepth - 1)];
          float4 d = *reinterpret_cast<const float4*>(&row[0][pix][4 * cq]);
          ulonglong2 x = *reinterpret_cast<const ulonglong2*>(&row[1][pix][4 * iq]);
          if (!live) x.x = x.y = 0ull;
          if (!live || k < k0) d = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          xr[r][0] = x.x;
          xr[r][1] = x.y;
          const float dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            bias[a] += dv[a];
            const f32x2 dd = pack2f(dv[a], dv[a]);
#pragma unroll
            for (int t = 0; t < T; ++t) {   // tap t of T meets the row of step k - (T - 1) + t
              const f32x2(&xt)[2] = xr[(r + 1 + t) % T];
              acc[t][a][0] = fma2(dd, xt[0], acc[t][a][0]);
              acc[t][a][1] = fma2(dd, xt[1], acc[t][a][1]);
            }
          }
        }
      }
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  for (int i = threadIdx.x; i < T * 256 + 16; i += blockDim.x) sum[i] = 0.0f;
  __syncthreads();
#pragma unroll
  for (int t = 0; t < T; ++t)
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float lo, hi;
        unpack2f(acc[t][a][h], lo, hi);
        lo += __shfl_xor_sync(0xFFFFFFFFu, lo, 16);
        hi += __shfl_xor_sync(0xFFFFFFFFu, hi, 16);
        if (lane < 16) {
          float* e = &sum[(t * 16 + 4 * cq + a) * 16 + 4 * iq + 2 * h];
          atomicAdd(e, lo);
          atomicAdd(e + 1, hi);
        }
      }
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    float v = bias[a] + __shfl_xor_sync(0xFFFFFFFFu, bias[a], 16);
    if (lane < 4) atomicAdd(&sum[T * 256 + 4 * cq + a], v);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kt * 256; i += blockDim.x) {   // gw[co][ci][tau]
    const int tau = i % kt, ci = i / kt % 16, co = i / (kt * 16);
    atomicAdd(gw + i, sum[((tau + T - kt) * 16 + co) * 16 + ci]);
  }
  if (threadIdx.x < 16) atomicAdd(gb + threadIdx.x, sum[T * 256 + threadIdx.x]);
}

int sm_count(int* n) {
  int dev = 0;
  ET_CHECK_CUDA(cudaGetDevice(&dev));
  ET_CHECK_CUDA(cudaDeviceGetAttribute(n, cudaDevAttrMultiProcessorCount, dev));
  return ET_OK;
}

int launch_conv_tma(bool data_grad, const float* in, int B, int K, int64_t hw, int kt, const float* w,
                    const float* b, const float* extra, const float* mask, float* out, const float* wp,
                    const float* bp, float* I, cudaStream_t st) {
  const int64_t tiles = (hw + kBoxPix - 1) / kBoxPix, nch = (K + kStepChunk - 1) / kStepChunk;
  F32ConvArgs A{K, kt, hw, (int)tiles, (int)nch, B * tiles * nch, w, b, extra, mask, out, wp, bp, I,
                et_tc_wait_iters()};
  CUtensorMap m_in;
  ET_TRY(map_rows(&m_in, in, (int64_t)B * K, hw));
  int nsm = 0;
  ET_TRY(sm_count(&nsm));
  const int smem = kRing * kBox + kt * 256 * (int)sizeof(float);
  auto kern = data_grad ? tconv16_tma<true> : tconv16_tma<false>;
  ET_TRY(et_allow_shared(kern));
  kern<<<(unsigned)std::min<int64_t>(A.total, nsm), 256, smem, st>>>(m_in, A);
  ET_CHECK_LAUNCH();
  return ET_OK;
}

int launch_wgrad_walk(const float* dz, const float* in, int B, int K, int64_t hw, int kt, float* gw, float* gb,
                      cudaStream_t st) {
  int nsm = 0;
  ET_TRY(sm_count(&nsm));
  // whole clips per warp, or segments of at least 16 steps (each rereads the
  // kt - 1 steps before it) when there are fewer than two pixel pairs per warp
  const int64_t pairs = (hw + 1) / 2 * B, want = 2ll * nsm * kWWarps;
  int seg = K;
  if (pairs < want) seg = (int)std::max<int64_t>(16, K / std::max<int64_t>(1, want / pairs));
  auto kern = kt <= 3 ? tconv16_wgrad_walk<3> : kt <= 5 ? tconv16_wgrad_walk<5>
              : kt <= 7 ? tconv16_wgrad_walk<7> : tconv16_wgrad_walk<9>;
  const int64_t items = pairs * ((K + seg - 1) / seg);
  kern<<<(unsigned)std::min<int64_t>((items + kWWarps - 1) / kWWarps, nsm), 32 * kWWarps, 0, st>>>(
      dz, in, B, K, hw, kt, seg, gw, gb);
  ET_CHECK_LAUNCH();
  return ET_OK;
}

struct TWorkspace {
  float* act[kMaxLayers];   // [B][K][hw][C] per layer (post-activation)
  float* I;                 // [B][K][hw]
  float* dI;
  float* g[3];              // [B][K][hw][C] gradient buffers
  size_t bytes;
  bool vec;                 // 16 channels and rows on 16-byte boundaries
};

void tlayout(const et_evsnet_weights* net, const et_train_shape* sh, char* base, TWorkspace* ws) {
  const int64_t n = (int64_t)sh->B * sh->K * sh->H * sh->W;
  size_t off = 0;
  auto take = [&](size_t bytes) -> float* {
    float* p = base ? reinterpret_cast<float*>(base + off) : nullptr;
    off += (bytes + 255) & ~(size_t)255;
    return p;
  };
  for (int l = 0; l < net->n_layers; ++l) ws->act[l] = take(sizeof(float) * n * net->C);
  ws->I = take(sizeof(float) * n);
  ws->dI = take(sizeof(float) * n);
  for (int j = 0; j < 3; ++j) ws->g[j] = take(sizeof(float) * n * net->C);
  ws->bytes = off;
  ws->vec = net->C == kMaxC && (reinterpret_cast<uintptr_t>(base) & 15) == 0;
}

// all layers over the whole clip: activations and I
int tforward(const float* logl, const et_train_shape* sh, const et_evsnet_weights* net,
             const TWorkspace& ws, cudaStream_t st) {
  const int C = net->C, L = net->n_layers, kt = net->kt;
  const int64_t hw = (int64_t)sh->H * sh->W;
  const unsigned grid2 = (unsigned)(((int64_t)sh->B * ((sh->K + 1) / 2) * hw + 255) / 256);   // step pairs
  const int n0 = layer0_taps(net);
  const float* wp = net->w + twofs(L, C, kt, n0);
  const float* bp = net->b + (int64_t)L * C;
  float* I0 = L == 1 ? ws.I : nullptr;
  int nsm = 0;
  ET_TRY(sm_count(&nsm));
  const int64_t warps = 16ll * nsm;
  if (net->ks0 == 3) {
    const int64_t others = (int64_t)sh->B * sh->K * ((sh->W + 31) / 32);
    const int rows = walk_length(kRows, 1, warps, others, sh->H);
    const int64_t items = others * ((sh->H + rows - 1) / rows);
    tstem3_fwd<<<(unsigned)((items + 3) / 4), 128, 0, st>>>(logl, sh->B, sh->K, sh->H, sh->W, C, ws.vec, rows, net->w,
                                                           net->b, ws.act[0], wp, bp, I0);
  } else if (net->ks0 > 0) {
    const dim3 grid((unsigned)((hw + 127) / 128), (unsigned)std::min<int64_t>((int64_t)sh->B * sh->K, 65535));
    tstem_fwd<<<grid, 128, 0, st>>>(logl, sh->B, sh->K, sh->H, sh->W, C, ws.vec, net->ks0, net->w, net->b,
                                    ws.act[0], wp, bp, I0);
  } else {
    const int64_t others = (int64_t)sh->B * ((hw + 31) / 32);
    const int walk = walk_length(kWalk, kWalkMin, warps, others, sh->K);
    const int64_t items = others * ((sh->K + walk - 1) / walk);
    (kt <= 7 ? tconv_fwd<7> : tconv_fwd<9>)<<<(unsigned)((items + 3) / 4), 128, 0, st>>>(
        logl, sh->B, sh->K, hw, C, ws.vec, kt, walk, net->w, net->b, ws.act[0], wp, bp, I0);
  }
  ET_CHECK_LAUNCH();
  for (int l = 1; l < L; ++l) {
    // residual form: even layers close a block and add its input
    const float* res = (net->kind == ET_NET_RESIDUAL && l % 2 == 0) ? ws.act[l - 2] : nullptr;
    if (net->dtype == ET_BF16) {
      const int rc = et_train_tct_conv(ws.act[l - 1], sh->B, sh->K, hw, C, kt, net->w + twofs(l, C, kt, n0),
                                       net->b + (int64_t)l * C, res, nullptr, ws.act[l], wp, bp,
                                       l == L - 1 ? ws.I : nullptr, false, st);
      if (rc != ET_OK) return rc;
      continue;
    }
    if (use_tma(sh->B, sh->K, hw, C, ws.act[l - 1], ws.act[l])) {
      ET_TRY(launch_conv_tma(false, ws.act[l - 1], sh->B, sh->K, hw, kt, net->w + twofs(l, C, kt, n0),
                             net->b + (int64_t)l * C, res, nullptr, ws.act[l], wp, bp, l == L - 1 ? ws.I : nullptr,
                             st));
      continue;
    }
    tconv16_fwd<<<grid2, 256, 0, st>>>(ws.act[l - 1], sh->B, sh->K, hw, C, kt, net->w + twofs(l, C, kt, n0),
                               net->b + (int64_t)l * C, res, ws.act[l], wp, bp,
                               l == L - 1 ? ws.I : nullptr);
    ET_CHECK_LAUNCH();
  }
  return ET_OK;
}

}  // namespace

bool et_train_is_temporal(const et_evsnet_weights* net) {
  const bool stem_ok = net->ks0 == 0 || (net->ks0 > 0 && net->ks0 <= kMaxStem && net->ks0 % 2 == 1);
  return net->ks == 1 && net->kt >= 1 && net->kt <= kMaxKt && net->C <= kMaxC && stem_ok &&
         (net->kind == ET_NET_STACK || (net->kind == ET_NET_RESIDUAL && net->n_layers % 2 == 1));
}

size_t et_train_temporal_bytes(const et_evsnet_weights* net, const et_train_shape* sh) {
  TWorkspace ws{};
  tlayout(net, sh, nullptr, &ws);
  return ws.bytes;
}

int et_train_temporal_forward(const float* logl, const et_train_shape* sh,
                              const et_evsnet_weights* net, int8_t* spikes, float* S_on,
                              float* S_off, float* V_ckpt, float* I_out, void* workspace,
                              cudaStream_t st) {
  TWorkspace ws{};
  tlayout(net, sh, static_cast<char*>(workspace), &ws);
  int rc = tforward(logl, sh, net, ws, st);
  if (rc != ET_OK) return rc;
  const int64_t hw = (int64_t)sh->H * sh->W, npx = (int64_t)sh->B * hw;
  const int n_ckpt = (sh->K + sh->ckpt_every - 1) / sh->ckpt_every;
  tbilif_fwd<<<(unsigned)((npx + 255) / 256), 256, 0, st>>>(
      ws.I, sh->B, sh->K, hw, sh->ckpt_every, n_ckpt, net->beta, net->vth, net->reset, V_ckpt,
      spikes, S_on, S_off, I_out);
  ET_CHECK_LAUNCH();
  return ET_OK;
}

int et_train_temporal_backward(const float* logl, const et_train_shape* sh,
                               const et_evsnet_weights* net, const float* V_ckpt,
                               const float* dS_on, const float* dS_off, float alpha,
                               float* grad_w, float* grad_b, void* workspace, cudaStream_t st) {
  TWorkspace ws{};
  tlayout(net, sh, static_cast<char*>(workspace), &ws);
  int rc = tforward(logl, sh, net, ws, st);
  if (rc != ET_OK) return rc;
  const int C = net->C, L = net->n_layers, kt = net->kt, B = sh->B, K = sh->K;
  const int64_t hw = (int64_t)sh->H * sh->W, npx = (int64_t)B * hw, n = (int64_t)B * K * hw;
  const int n_ckpt = (K + sh->ckpt_every - 1) / sh->ckpt_every;
  int dev = 0, nsm = 0;
  ET_CHECK_CUDA(cudaGetDevice(&dev));
  ET_CHECK_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  tbilif_bwd<<<(unsigned)((npx + 255) / 256), 256, 0, st>>>(
      ws.I, B, K, hw, sh->ckpt_every, n_ckpt, net->beta, net->vth, net->reset, alpha, V_ckpt, dS_on,
      dS_off, ws.dI);
  ET_CHECK_LAUNCH();
  const unsigned grid2 = (unsigned)((npx * ((K + 1) / 2) + 255) / 256);   // step pairs
  const unsigned wgrid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(nsm * 8, (n + kPts - 1) / kPts));
  float* dz = ws.g[0];
  const int n0 = layer0_taps(net);
  tproj_bwd<<<nsm * 8, 256, 0, st>>>(ws.dI, ws.act[L - 1], n, C, ws.vec, net->w + twofs(L, C, kt, n0), dz,
                                     grad_w + twofs(L, C, kt, n0), grad_b + (int64_t)L * C);
  ET_CHECK_LAUNCH();
  const int wthr = twgrad_threads(kt);
  const size_t wsmem = sizeof(float) * kPts16 * CP * (1 + kt);
  int wblocks = 0;   // resident weight-gradient blocks per SM: one wave of persistent blocks
  ET_CHECK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&wblocks, tconv16_bwd_weight, wthr, wsmem));
  const unsigned wgrid16 = (unsigned)std::max<int64_t>(
      1, std::min<int64_t>((int64_t)nsm * std::max(wblocks, 1), (n + kPts16 - 1) / kPts16));
  auto wgrad = [&](const float* d, int l) -> int {
    // layer 0: a walk per warp, the resident two blocks of 8 warps per SM (four per
    // SM: 2 clips of 33 x 37 x 45 26 us instead of 18, as each block ends with its
    // share of the atomics; 8 clips of 64 x 128 x 128 0.262 ms instead of 0.255)
    const int64_t warps = 16ll * nsm;
    auto blocks = [&](int64_t items) { return (unsigned)std::min<int64_t>((items + 7) / 8, nsm * 2); };
    if (l == 0 && net->ks0 == 3) {
      const int64_t others = (int64_t)B * K * ((sh->W + 7) / 8);
      const int walk = walk_length(kRowsB, 1, warps, others, sh->H);
      tstem3_bwd_weight<<<blocks(others * ((sh->H + walk - 1) / walk)), 256, 0, st>>>(
          d, logl, B, K, sh->H, sh->W, C, ws.vec, walk, grad_w, grad_b);
    }
    else if (l == 0 && net->ks0 > 0)
      tstem_bwd_weight<<<wgrid, 256, 0, st>>>(d, logl, B, K, sh->H, sh->W, C, net->ks0, grad_w, grad_b);
    else if (l == 0) {
      const int64_t others = (int64_t)B * ((hw + 7) / 8);
      const int walk = walk_length(kWalkB, kWalkBMin, warps, others, K);
      (kt <= 7 ? tconv_bwd_weight<7> : tconv_bwd_weight<9>)<<<blocks(others * ((K + walk - 1) / walk)), 256, 0, st>>>(
          d, logl, B, K, hw, C, ws.vec, kt, walk, grad_w, grad_b);
    }
    else if (net->dtype == ET_BF16)
      return et_train_tct_wgrad(d, ws.act[l - 1], B, K, hw, C, kt, grad_w + twofs(l, C, kt, n0),
                                grad_b + (int64_t)l * C, st);
    else if (use_tma(B, K, hw, C, d, ws.act[l - 1]))
      return launch_wgrad_walk(d, ws.act[l - 1], B, K, hw, kt, grad_w + twofs(l, C, kt, n0),
                               grad_b + (int64_t)l * C, st);
    else
      tconv16_bwd_weight<<<wgrid16, wthr, wsmem, st>>>(d, ws.act[l - 1], B, K, hw, C, kt, grad_w + twofs(l, C, kt, n0),
                                          grad_b + (int64_t)l * C);
    return ET_OK;
  };
  // data gradient through layer l: out = (add + conv_l^T(d)) * 1(mask > 0)
  auto dgrad = [&](const float* d, int l, const float* add, const float* mask, float* out) -> int {
    if (net->dtype == ET_BF16)
      return et_train_tct_conv(d, B, K, hw, C, kt, net->w + twofs(l, C, kt, n0), nullptr, add, mask, out,
                               nullptr, nullptr, nullptr, true, st);
    if (use_tma(B, K, hw, C, d, out))
      return launch_conv_tma(true, d, B, K, hw, kt, net->w + twofs(l, C, kt, n0), nullptr, add, mask, out, nullptr,
                             nullptr, nullptr, st);
    tconv16_bwd_data<<<grid2, 256, 0, st>>>(d, B, K, hw, C, kt, net->w + twofs(l, C, kt, n0), add, mask, out);
    return ET_OK;
  };
  if (net->kind == ET_NET_STACK) {
    int cur = 0;
    for (int l = L - 1; l >= 0; --l) {
      ET_TRY(wgrad(ws.g[cur], l));
      ET_CHECK_LAUNCH();
      if (l > 0) {
        ET_TRY(dgrad(ws.g[cur], l, nullptr, ws.act[l - 1], ws.g[cur ^ 1]));
        ET_CHECK_LAUNCH();
        cur ^= 1;
      }
    }
    return ET_OK;
  }
  // residual: blocks i = M..1 own layers 2i - 1 (inner) and 2i (closing)
  int cz = 0;   // buffer holding dL/dz of the current block's output
  for (int i = (L - 1) / 2; i >= 1; --i) {
    const int la = 2 * i - 1, lc = 2 * i;
    const int cy = (cz + 1) % 3, cn = (cz + 2) % 3;
    ET_TRY(wgrad(ws.g[cz], lc));
    ET_CHECK_LAUNCH();
    // dy = conv_lc^T(dz) masked by a > 0
    ET_TRY(dgrad(ws.g[cz], lc, nullptr, ws.act[la], ws.g[cy]));
    ET_CHECK_LAUNCH();
    ET_TRY(wgrad(ws.g[cy], la));
    ET_CHECK_LAUNCH();
    // dz_prev = (dz + conv_la^T(dy)) masked by h_{i-1} > 0
    ET_TRY(dgrad(ws.g[cy], la, ws.g[cz], ws.act[la - 1], ws.g[cn]));
    ET_CHECK_LAUNCH();
    cz = cn;
  }
  ET_TRY(wgrad(ws.g[cz], 0));
  ET_CHECK_LAUNCH();
  return ET_OK;
}
