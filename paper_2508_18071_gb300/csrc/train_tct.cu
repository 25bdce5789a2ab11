// BF16 tensor-core convolutions for training the paper's pixel-wise temporal
// EvSNet (Eq. 5: causal convolutions of kernel kt along time between C <= 16
// channels; Sec. 3.3 training): the forward of a C -> C layer, the data
// gradient through it, and its weight gradient, on tcgen05 with BF16 operands
// and FP32 accumulation in TMEM.  Layer 0 (one input channel or a spatial
// stem), the projection, BiLIF and the loss stay FP32 on the CUDA cores
// (train_temporal.cu); activations and gradients stay FP32 in global memory
// ([B][K][H W][C], a pixel-step's channels contiguous), rounded to BF16 where
// they enter an MMA.
//
// Forward and data gradient (tct_conv): a CTA owns 128 consecutive pixels of
// one clip and walks its K steps two at a time -- forward in time for the
// forward, backward in time for the data gradient, which in reversed time is
// the same causal convolution with each tap's weights transposed.  The inputs
// of the last kt + 1 steps sit in a ring of shared-memory slots (128 pixels x
// 16 channels, K-major no-swizzle: two 2 KB planes of 8 channels); slot i of a
// chunk feeds its first step through tap i and its second through tap i - 1,
// so one MMA per slot (M = 128 pixels, K = 16 channels, N = 32: the window
// [W_i ; W_(i-1)] of the layer's taps stored in descending order) covers both
// steps, N = 16 for the first and last slot.  The next chunk's inputs are
// loaded into registers while the MMAs run.
//
// Weight gradient (tct_wgrad): the reduction over pixel-steps is the MMA's K
// dimension, so the operands are staged transposed: for every step, the input
// (channels as rows, pixels along K) into a doubled ring (each step written at
// slots j and j + 8 of 16, so the 8 consecutive slots of steps k - 7 .. k are
// always contiguous) and dL/dz the same way.  D[(tau', ci), co] =
// sum_p in[k - 7 + tau'][p][ci] dz[k][p][co] with M = 128 rows (8 slots x 16
// channels), N = 16, K = 16 pixels per MMA, accumulated in TMEM over the
// CTA's steps and pixels; window slot tau' holds tap tau = tau' - 8 + kt of
// the layer (slots below 8 - kt are not taps).  The bias gradient is summed
// on the CUDA cores while staging.
//
// MMA waits are bounded (et_set_wait_budget); on expiry the kernel writes NaN
// to the outputs it has not finished (the loss then reports it), waits a
// second bounded time for its MMAs in flight and frees its TMEM.
//
// With C = 16 channels a pixel-step is one 64-byte row, and both kernels have a
// second form (tct_conv16, tct_wgrad16) that moves whole tiles by TMA and keeps
// its CTAs resident over many tiles; the forms above serve C < 16 and tensors
// that don't start on a 16-byte boundary, which TMA can't address.
#include "et_internal.cuh"
#include "evsnet_common.h"
#include "tc_ptx.cuh"
#include "train_api.h"
#include "train_tma.cuh"
#include <cuda_bf16.h>
#include <algorithm>
#include <cstring>

namespace {

constexpr int TP = kBoxPix;              // pixels per CTA = MMA M (forward) = TMEM lanes
constexpr int CP = 16;                   // channels, zero-padded
constexpr int kMaxKtTc = 7;              // ring of kt + 1 <= 8 slots
constexpr int kSlot = TP * CP * 2;       // bytes of one ring slot
constexpr int kPlane = TP * 16;          // bytes of 8 channels of 128 rows
constexpr uint32_t kDrainIters = 1u << 22;

// two floats as one 32-bit word of BF16 (round to nearest even), low half first
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// a pixel-step's CP channels (zero beyond C) from FP32 global memory
__device__ __forceinline__ void load16(const float* __restrict__ src, int C, bool ok, float (&x)[CP]) {
#pragma unroll
  for (int c = 0; c < CP; ++c) x[c] = ok && c < C ? __ldg(src + c) : 0.0f;
}

// row m of a ring slot: channels 0-7 in plane 0, 8-15 in plane 1
__device__ __forceinline__ void store_slot(unsigned char* slot, int m, const float (&v)[CP]) {
  *reinterpret_cast<uint4*>(slot + m * 16) =
      make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
  *reinterpret_cast<uint4*>(slot + kPlane + m * 16) =
      make_uint4(pack2(v[8], v[9]), pack2(v[10], v[11]), pack2(v[12], v[13]), pack2(v[14], v[15]));
}

// ---------------------------------------------------------------- conv
// kBwd = false: out[s] = ReLU(b + sum_tau W_tau in[s - (kt-1) + tau] (+ res[s])),
//               and I[s] = bp + wp . out[s] when I is not null;
// kBwd = true:  out[s] = (add[s] + sum_tau W_tau^T in[s + (kt-1) - tau]) * 1(mask[s] > 0),
//               in = dL/dz of the layer's output, out = dL/dz of its input.
struct ConvArgs {
  const float* in;
  int B, K, C, kt;
  int64_t hw;
  const float* w;       // [co][ci][tau]
  const float* b;       // bias (forward)
  const float* extra;   // res (forward) or add (data gradient), may be null
  const float* mask;    // data gradient: the layer input's activation
  float* out;
  const float* wp;      // forward, last layer: projection
  const float* bp;
  float* I;
  uint32_t wait_iters;
};

template <bool kBwd>
__global__ void __launch_bounds__(TP)
tct_conv(ConvArgs A) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint64_t mma_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int bail;
  __shared__ float sb[CP], swp[CP];
  const int tid = threadIdx.x, warp = tid >> 5;
  const int C = A.C, K = A.K, kt = A.kt, R = kt + 1;
  const int64_t hw = A.hw;
  const int64_t tiles = (hw + TP - 1) / TP;
  const int bc = (int)(blockIdx.x / tiles);
  const int64_t p = (blockIdx.x % tiles) * TP + tid;
  const bool live = p < hw;
  unsigned char* ring = sm;                                    // [R] slots
  unsigned char* wB = sm + (size_t)R * kSlot;                  // kt blocks x 2 planes
  // B strip: block b holds tap kt - 1 - b; row n, K index k:
  //   forward: n = output channel, k = input channel: w[n][k][tau]
  //   data gradient: n = input channel, k = output channel: w[k][n][tau]
  for (int i = tid; i < kt * CP * CP; i += TP) {
    const int k = i % CP, n = (i / CP) % CP, tau = i / (CP * CP);
    float v = 0.0f;
    if (n < C && k < C) v = kBwd ? A.w[((int64_t)k * C + n) * kt + tau] : A.w[((int64_t)n * C + k) * kt + tau];
    unsigned char* dst = wB + (k >> 3) * (kt * CP * 16) + ((kt - 1 - tau) * CP + n) * 16 + (k & 7) * 2;
    *reinterpret_cast<__nv_bfloat16*>(dst) = __float2bfloat16_rn(v);
  }
  for (int i = tid; i < R * kSlot / 16; i += TP) reinterpret_cast<uint4*>(ring)[i] = make_uint4(0, 0, 0, 0);
  if (tid < CP) {
    sb[tid] = (!kBwd && A.b && tid < C) ? A.b[tid] : 0.0f;
    swp[tid] = (!kBwd && A.wp && tid < C) ? A.wp[tid] : 0.0f;
  }
  if (warp == 0) tmem_alloc(&tmem_slot, 32);
  if (tid == 0) { mbar_init(&mma_bar, 1); bail = 0; }
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
  const uint32_t idesc16 = umma_idesc_bf16(TP, CP), idesc32 = umma_idesc_bf16(TP, 2 * CP);
  const uint64_t a_desc0 = umma_desc(smem_u32(ring), kPlane, 128);
  const uint64_t b_desc0 = umma_desc(smem_u32(wB), kt * CP * 16, 128);
  constexpr uint64_t kBlock = (CP * 16) >> 4;
  const float bpv = (!kBwd && A.bp) ? A.bp[0] : 0.0f;
  // processing order u = 0 .. K-1 is time s = u (forward) or s = K-1-u (data gradient)
  auto step_of = [&](int u) { return kBwd ? K - 1 - u : u; };
  auto row = [&](int s) -> int64_t { return ((int64_t)bc * K + s) * hw + p; };
  const int nch = (K + 1) / 2;
  float nx[2][CP];                       // the next chunk's inputs
  auto load_chunk = [&](int c) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int u = 2 * c + j;
      load16(A.in + (live && u < K ? row(step_of(u)) : 0) * C, C, live && u < K, nx[j]);
    }
  };
  load_chunk(0);
  uint32_t phase = 0;
  int c = 0;
  for (; c < nch; ++c) {
    const int u0 = 2 * c, tc = min(2, K - u0);
#pragma unroll
    for (int j = 0; j < 2; ++j)
      if (j < tc) store_slot(ring + (size_t)((u0 + j) % R) * kSlot, tid, nx[j]);
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0) {
      const int p0 = ((u0 - (kt - 1)) % R + R) % R;
      auto a_of = [&](int i) {
        const int pos = p0 + i >= R ? p0 + i - R : p0 + i;
        return a_desc0 + (uint64_t)pos * (kSlot >> 4);
      };
      umma_bf16(tmem, a_of(0), b_desc0 + (uint64_t)(kt - 1) * kBlock, idesc16, 0);
      if (tc > 1) umma_bf16(tmem + CP, a_of(kt), b_desc0, idesc16, 0);
      for (int i = 1; i < kt; ++i) umma_bf16(tmem, a_of(i), b_desc0 + (uint64_t)(kt - 1 - i) * kBlock, idesc32, 1);
      umma_commit(&mma_bar);
    }
    if (c + 1 < nch) load_chunk(c + 1);
    const bool ok = mbar_wait(&mma_bar, phase, A.wait_iters);
    phase ^= 1;
    if (!ok) bail = 1;
    tc_fence_after();
    __syncthreads();
    if (bail) break;
    float acc[2][CP];
    tmem_ld16(tmem + lane_base, acc[0]);
    tmem_ld16(tmem + lane_base + CP, acc[1]);
    for (int j = 0; j < tc; ++j) {
      if (!live) break;
      const int s = step_of(u0 + j);
      float* o = A.out + row(s) * C;
      float v[CP];
      float Iv = bpv;
#pragma unroll
      for (int co = 0; co < CP; ++co) {
        if (!kBwd) {
          float z = acc[j][co] + sb[co];
          if (A.extra && co < C) z += A.extra[row(s) * C + co];
          v[co] = fmaxf(z, 0.0f);
          Iv = fmaf(swp[co], v[co], Iv);
        } else {
          float z = acc[j][co];
          if (co < C) {
            if (A.extra) z += A.extra[row(s) * C + co];
            z = A.mask[row(s) * C + co] > 0.0f ? z : 0.0f;
          }
          v[co] = z;
        }
      }
#pragma unroll
      for (int co = 0; co < CP; ++co)
        if (co < C) o[co] = v[co];
      if (!kBwd && A.I) A.I[row(s)] = Iv;
    }
    tc_fence_before();
  }
  if (bail) {
    // unfinished steps: NaN, so that the loss shows the failure
    if (live)
      for (int u = 2 * c; u < K; ++u) {
        const int s = step_of(u);
        for (int co = 0; co < C; ++co) A.out[row(s) * C + co] = __int_as_float(0x7fc00000);
        if (!kBwd && A.I) A.I[row(s)] = __int_as_float(0x7fc00000);
      }
    mbar_wait(&mma_bar, phase ^ 1u, kDrainIters);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, 32);
}

// ---------------------------------------------------------------- weight gradient
// grad w[co][ci][tau] += sum_{k,p} dz[k][p][co] in[k - (kt-1) + tau][p][ci],
// grad b[co] += sum_{k,p} dz[k][p][co]; one CTA per 128 pixels of a clip.
constexpr int kWSlots = 16;                       // doubled ring of 8 steps
constexpr int kWRows = kWSlots * CP;              // 256 rows (slot, ci) of 16 B per 8-pixel chunk
constexpr int kWChunk = kWRows * 16;              // bytes per 8-pixel chunk of the input ring
constexpr int kWABytes = (TP / 8) * kWChunk;      // 64 KB
constexpr int kWBBytes = (TP / 8) * CP * 16;      // 4 KB: dz^T, [chunk][co][8 pixels]

__device__ __forceinline__ void st_bf16(unsigned char* p, float v) {
  *reinterpret_cast<__nv_bfloat16*>(p) = __float2bfloat16_rn(v);
}

__global__ void __launch_bounds__(TP)
tct_wgrad(const float* __restrict__ dz, const float* __restrict__ in, int B, int K, int64_t hw, int C,
          int kt, float* __restrict__ gw, float* __restrict__ gb, uint32_t wait_iters) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint64_t mma_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int bail;
  __shared__ float red[TP / 32][CP];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t tiles = (hw + TP - 1) / TP;
  const int bc = (int)(blockIdx.x / tiles);
  const int64_t p = (blockIdx.x % tiles) * TP + tid;
  const bool live = p < hw;
  unsigned char* Abuf = sm;
  unsigned char* Bbuf = sm + kWABytes;
  for (int i = tid; i < (kWABytes + kWBBytes) / 16; i += TP) reinterpret_cast<uint4*>(sm)[i] = make_uint4(0, 0, 0, 0);
  if (warp == 0) tmem_alloc(&tmem_slot, 32);
  if (tid == 0) { mbar_init(&mma_bar, 1); bail = 0; }
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const uint32_t idesc = umma_idesc_bf16(TP, CP);
  // this thread's column in the transposed buffers: chunk tid / 8, element tid % 8
  unsigned char* acol = Abuf + (tid >> 3) * kWChunk + (tid & 7) * 2;
  unsigned char* bcol = Bbuf + (tid >> 3) * (CP * 16) + (tid & 7) * 2;
  auto row = [&](int s) -> int64_t { return ((int64_t)bc * K + s) * hw + p; };
  float gbp[CP];
#pragma unroll
  for (int c = 0; c < CP; ++c) gbp[c] = 0.0f;
  float nx[CP], nd[CP];
  load16(in + (live ? row(0) : 0) * C, C, live, nx);
  load16(dz + (live ? row(0) : 0) * C, C, live, nd);
  uint32_t phase = 0;
  for (int k = 0; k < K; ++k) {
    // stage step k: input at slots k % 8 and k % 8 + 8, dz^T
    const int q = k & 7;
#pragma unroll
    for (int c = 0; c < CP; ++c) {
      st_bf16(acol + (q * CP + c) * 16, nx[c]);
      st_bf16(acol + ((q + 8) * CP + c) * 16, nx[c]);
      st_bf16(bcol + c * 16, nd[c]);
      gbp[c] += nd[c];
    }
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0) {
      // window: the 8 slots of steps k - 7 .. k, rows base * 16 ..
      const int base = (k + 1) & 7;
      const uint64_t a0 = umma_desc(smem_u32(Abuf) + base * CP * 16, kWChunk, 128);
      const uint64_t b0 = umma_desc(smem_u32(Bbuf), CP * 16, 128);
      for (int j = 0; j < TP / 16; ++j)
        umma_bf16(tmem, a0 + (uint64_t)(2 * j) * (kWChunk >> 4), b0 + (uint64_t)(2 * j) * ((CP * 16) >> 4), idesc,
                  (k > 0 || j > 0) ? 1u : 0u);
      umma_commit(&mma_bar);
    }
    if (k + 1 < K) {
      load16(in + (live ? row(k + 1) : 0) * C, C, live, nx);
      load16(dz + (live ? row(k + 1) : 0) * C, C, live, nd);
    }
    const bool ok = mbar_wait(&mma_bar, phase, wait_iters);
    phase ^= 1;
    if (!ok) bail = 1;
    tc_fence_after();
    __syncthreads();
    if (bail) break;
  }
  if (bail) {
    mbar_wait(&mma_bar, phase ^ 1u, kDrainIters);
    if (tid == 0) atomicAdd(gw, __int_as_float(0x7fc00000));   // the gradient reports the failure
  } else {
    // lane tid = row (slot offset tau', input channel ci): tap tau = tau' - 8 + kt
    float d[CP];
    tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16), d);
    const int tp = tid / CP, ci = tid % CP, tau = tp - 8 + kt;
    if (tau >= 0 && ci < C)
      for (int co = 0; co < C; ++co) atomicAdd(gw + ((int64_t)co * C + ci) * kt + tau, d[co]);
#pragma unroll
    for (int c = 0; c < CP; ++c) {
      float v = live ? gbp[c] : 0.0f;
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
      if (lane == 0) red[warp][c] = v;
    }
    __syncthreads();
    if (tid < C) {
      float v = 0.0f;
      for (int wv = 0; wv < TP / 32; ++wv) v += red[wv][tid];
      atomicAdd(gb + tid, v);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, 32);
}


// ================================================================ C = 16, by TMA
// (boxes of one step of 128 pixels: train_tma.cuh)
struct Conv16Args {
  int K, kt;
  int64_t hw;
  int tiles, nch;        // 128-pixel tiles per step; chunks of two steps per clip
  int64_t total;         // B * tiles * nch chunks
  const float* w;
  const float* b;
  int has_extra;
  const float* wp;
  const float* bp;
  float* I;
  uint32_t wait_iters;
};

// Same arithmetic as tct_conv, bit for bit.  Bound by HBM: per pixel-step 64
// bytes of input and output each, plus the residual (forward) or the mask and
// the added gradient (data gradient).  The B tiles nch chunks (a chunk = two
// steps of a tile) are numbered with time innermost and split evenly over the
// resident CTAs (2 per SM), so no last wave is half empty; a CTA that starts in
// the middle of a clip first refills the ring with the kt - 1 steps before.
// Shared memory per CTA: the ring (32 KB), the weights, and boxes: input x 2
// (forward; 1 for the data gradient), O x 2 -- the residual or the mask, which
// each thread overwrites with its own output row, stored from there by TMA --
// and E, the data gradient's added term.  Thread 0 issues copies and MMAs: the
// input box is requested again as soon as it is converted, an O box a whole
// chunk ahead, once the store before has read it.
template <bool kBwd>
__global__ void __launch_bounds__(TP, 2)
tct_conv16(const __grid_constant__ CUtensorMap m_in, const __grid_constant__ CUtensorMap m_extra,
           const __grid_constant__ CUtensorMap m_mask, const __grid_constant__ CUtensorMap m_out, Conv16Args A) {
  constexpr int kIn = kBwd ? 1 : 2;      // input chunk buffers
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint64_t in_bar[kIn], o_bar[2], e_bar, mma_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ float sb[CP], swp[CP];
  const int tid = threadIdx.x, warp = tid >> 5;
  const int K = A.K, kt = A.kt, R = kt + 1, nch = A.nch;
  unsigned char* in_box = sm;                                  // [kIn][2 steps]
  unsigned char* o_box = in_box + kIn * 2 * kBox;              // [2][2 steps]
  unsigned char* e_box = o_box + 2 * 2 * kBox;                 // [2 steps], data gradient only
  unsigned char* ring = e_box + (kBwd ? 2 * kBox : 0);         // [R] slots
  unsigned char* wB = ring + (size_t)R * kSlot;
  // B strip as in tct_conv; the weights are read in their own order
  for (int i = tid; i < kt * CP * CP; i += TP) {
    const int tau = i % kt, r = i / kt, lo = r % CP, hi = r / CP;   // w[hi][lo][tau]
    const int n = kBwd ? lo : hi, k = kBwd ? hi : lo;
    unsigned char* dst = wB + (k >> 3) * (kt * CP * 16) + ((kt - 1 - tau) * CP + n) * 16 + (k & 7) * 2;
    *reinterpret_cast<__nv_bfloat16*>(dst) = __float2bfloat16_rn(A.w[i]);
  }
  if (tid < CP) {
    sb[tid] = (!kBwd && A.b) ? A.b[tid] : 0.0f;
    swp[tid] = (!kBwd && A.wp) ? A.wp[tid] : 0.0f;
  }
  if (warp == 0) tmem_alloc(&tmem_slot, 32);
  if (tid == 0) {
    for (int i = 0; i < kIn; ++i) mbar_init(&in_bar[i], 1);
    mbar_init(&o_bar[0], 1);
    mbar_init(&o_bar[1], 1);
    mbar_init(&e_bar, 1);
    mbar_init(&mma_bar, 1);
  }
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
  const uint32_t idesc16 = umma_idesc_bf16(TP, CP), idesc32 = umma_idesc_bf16(TP, 2 * CP);
  const uint64_t a_desc0 = umma_desc(smem_u32(ring), kPlane, 128);
  const uint64_t b_desc0 = umma_desc(smem_u32(wB), kt * CP * 16, 128);
  constexpr uint64_t kBlock = (CP * 16) >> 4;
  const float bpv = (!kBwd && A.bp) ? A.bp[0] : 0.0f;
  const bool has_o = kBwd || A.has_extra != 0, has_e = kBwd && A.has_extra != 0;

  // this CTA's chunks [t0, t1), preceded by the chunks that only refill the ring
  const int64_t t0 = A.total * blockIdx.x / gridDim.x, t1 = A.total * (blockIdx.x + 1) / gridDim.x;
  const int64_t ts = t0 - min((int64_t)(kt / 2), t0 % nch);
  // processing order u = 0 .. K-1 is time s = u (forward) or s = K-1-u (data gradient)
  auto step_of = [&](int u) { return kBwd ? K - 1 - u : u; };
  // boxes of chunk t of a tensor (thread 0): coordinates (channel, pixel, clip step)
  auto load_boxes = [&](const CUtensorMap* m, int64_t t, unsigned char* dst, uint64_t* bar) {
    const int64_t seg = t / nch;
    const int c = (int)(t - seg * nch), tile = (int)(seg % A.tiles), bc = (int)(seg / A.tiles);
    const int n = min(2, K - 2 * c);
    mbar_arrive_expect_tx(bar, (uint32_t)(n * kBox));
    for (int j = 0; j < n; ++j)
      tma_load_3d(dst + j * kBox, m, 0, tile * TP, bc * K + step_of(2 * c + j), bar);
  };
  uint32_t n_in[2] = {0, 0}, n_o[2] = {0, 0}, n_e = 0;   // thread 0: boxes requested per buffer
  if (tid == 0 && ts < t1) {
    for (int i = 0; i < kIn; ++i)
      if (ts + i < t1) { load_boxes(&m_in, ts + i, in_box + i * 2 * kBox, &in_bar[i]); ++n_in[i]; }
    if (has_o) { load_boxes(kBwd ? &m_mask : &m_extra, t0, o_box, &o_bar[0]); ++n_o[0]; }
    if (has_e) { load_boxes(&m_extra, t0, e_box, &e_bar); ++n_e; }
  }
  uint32_t in_phase = 0, o_phase = 0, e_phase = 0, mma_phase = 0;   // next parities, one bit per buffer
  int64_t seg = ts / nch;
  int c = (int)(ts - seg * nch), tile = (int)(seg % A.tiles), bc = (int)(seg / A.tiles);
  bool fresh = true;                     // the ring must be zero before this chunk
  bool bail = false;
  int n_mma = 0;
  int64_t t = ts;
  for (; t < t1; ++t) {
    const int u0 = 2 * c, tc = min(2, K - u0);
    const int64_t p = (int64_t)tile * TP + tid;
    const bool live = p < A.hw;
    bool fail = false;
    if (fresh || c == 0) {
      for (int i = tid; i < R * kSlot / 16; i += TP) reinterpret_cast<uint4*>(ring)[i] = make_uint4(0, 0, 0, 0);
      __syncthreads();                   // a row of the ring is zeroed by one thread and filled by another
      fresh = false;
    }
    // ---- the chunk's input, rounded to BF16, into the ring
    {
      const int bi = kIn == 1 ? 0 : (int)((t - ts) & 1);
      fail |= !mbar_wait(&in_bar[bi], (in_phase >> bi) & 1u, A.wait_iters);
      in_phase ^= 1u << bi;
      for (int j = 0; j < tc; ++j) {
        float v[CP];
        box_load(in_box + (bi * 2 + j) * kBox, tid, v);
        store_slot(ring + (size_t)((u0 + j) % R) * kSlot, tid, v);
      }
      fence_proxy_async_smem();
      tc_fence_before();
      bail = __syncthreads_or(fail) != 0;
      if (bail) break;
      tc_fence_after();
      if (tid == 0 && t + kIn < t1) {
        load_boxes(&m_in, t + kIn, in_box + bi * 2 * kBox, &in_bar[bi]);
        ++n_in[bi];
      }
    }
    if (t >= t0) {
      const int oi = (int)((t - t0) & 1);
      if (tid == 0) {
        const int p0 = ((u0 - (kt - 1)) % R + R) % R;
        auto a_of = [&](int i) {
          const int pos = p0 + i >= R ? p0 + i - R : p0 + i;
          return a_desc0 + (uint64_t)pos * (kSlot >> 4);
        };
        umma_bf16(tmem, a_of(0), b_desc0 + (uint64_t)(kt - 1) * kBlock, idesc16, 0);
        if (tc > 1) umma_bf16(tmem + CP, a_of(kt), b_desc0, idesc16, 0);
        for (int i = 1; i < kt; ++i)
          umma_bf16(tmem, a_of(i), b_desc0 + (uint64_t)(kt - 1 - i) * kBlock, idesc32, 1);
        umma_commit(&mma_bar);
        // the other O buffer is free once the previous chunk's store has read it
        bulk_wait_read();
        if (has_o && t + 1 < t1) {
          load_boxes(kBwd ? &m_mask : &m_extra, t + 1, o_box + (oi ^ 1) * 2 * kBox, &o_bar[oi ^ 1]);
          ++n_o[oi ^ 1];
        }
      }
      ++n_mma;
      if (has_o) {
        fail |= !mbar_wait(&o_bar[oi], (o_phase >> oi) & 1u, A.wait_iters);
        o_phase ^= 1u << oi;
      }
      if (has_e) {
        fail |= !mbar_wait(&e_bar, e_phase, A.wait_iters);
        e_phase ^= 1u;
      }
      fail |= !mbar_wait(&mma_bar, mma_phase, A.wait_iters);
      mma_phase ^= 1u;
      // without a load into O, the store of two chunks ago must have read it
      // (thread 0 waited for every store before it issued this chunk's MMAs,
      // whose commit this thread has just seen)
      tc_fence_after();
      float acc[2][CP];
      tmem_ld32(tmem + lane_base, &acc[0][0]);
      for (int j = 0; j < tc; ++j) {
        float ex[CP], mk[CP];
        if (has_o) box_load(o_box + (oi * 2 + j) * kBox, tid, kBwd ? mk : ex);
        if (has_e) box_load(e_box + j * kBox, tid, ex);
        float v[CP];
        float Iv = bpv;
#pragma unroll
        for (int co = 0; co < CP; ++co) {
          if (!kBwd) {
            float z = acc[j][co] + sb[co];
            if (has_o) z += ex[co];
            v[co] = fmaxf(z, 0.0f);
            Iv = fmaf(swp[co], v[co], Iv);
          } else {
            float z = acc[j][co];
            if (has_e) z += ex[co];
            v[co] = mk[co] > 0.0f ? z : 0.0f;
          }
        }
        box_store(o_box + (oi * 2 + j) * kBox, tid, v);
        if (!kBwd && A.I && live) A.I[((int64_t)bc * K + step_of(u0 + j)) * A.hw + p] = Iv;
      }
      fence_proxy_async_smem();
      tc_fence_before();
      bail = __syncthreads_or(fail) != 0;
      if (bail) break;
      if (tid == 0) {
        for (int j = 0; j < tc; ++j)
          tma_store_3d(&m_out, 0, tile * TP, bc * K + step_of(u0 + j), o_box + (oi * 2 + j) * kBox);
        bulk_commit();
        if (has_e && t + 1 < t1) { load_boxes(&m_extra, t + 1, e_box, &e_bar); ++n_e; }
      }
    }
    if (++c == nch) {
      c = 0;
      if (++tile == A.tiles) { tile = 0; ++bc; }
    }
  }
  if (tid == 0) bulk_wait_all();
  if (bail) {
    // unfinished chunks: NaN (through the output's tensor map, like every
    // store), so that the loss shows the failure; then the copies and MMAs in
    // flight are waited for (bounded)
    __syncthreads();
    if (tid == 0) {
      for (int i = 0; i < kIn; ++i)
        if (n_in[i]) mbar_wait(&in_bar[i], (n_in[i] - 1) & 1u, kDrainIters);
      for (int i = 0; i < 2; ++i)
        if (n_o[i]) mbar_wait(&o_bar[i], (n_o[i] - 1) & 1u, kDrainIters);
      if (n_e) mbar_wait(&e_bar, (n_e - 1) & 1u, kDrainIters);
    }
    if (n_mma) mbar_wait(&mma_bar, (uint32_t)(n_mma - 1) & 1u, kDrainIters);
    __syncthreads();
    float nan[CP];
#pragma unroll
    for (int i = 0; i < CP; ++i) nan[i] = __int_as_float(0x7fc00000);
    box_store(o_box, tid, nan);
    fence_proxy_async_smem();
    __syncthreads();
    for (t = max(t, t0); t < t1; ++t) {
      const int64_t sg = t / nch;
      const int ct = (int)(t - sg * nch), tl = (int)(sg % A.tiles), b = (int)(sg / A.tiles);
      for (int u = 2 * ct; u < min(K, 2 * ct + 2); ++u) {
        const int64_t row = (int64_t)b * K + step_of(u);
        if (tid == 0) tma_store_3d(&m_out, 0, tl * TP, (int)row, o_box);
        const int64_t p = (int64_t)tl * TP + tid;
        if (!kBwd && A.I && p < A.hw) A.I[row * A.hw + p] = nan[0];
      }
    }
    if (tid == 0) { bulk_commit(); bulk_wait_all(); }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, 32);
}

// Weight gradient, as tct_wgrad but without transposing: both operands are
// MN-major, so a ring slot is the BF16 rows as they come (8-channel planes of
// 128 pixels, 16-byte rows: a core matrix is 8 pixels of 8 channels), two
// 16-byte stores per pixel and step instead of 32 two-byte ones.  A chunk of
// two steps k, k + 1 meets the whole ring of 8 slots (steps k - 6 .. k + 1) in
// 8 MMAs of M = 128 (slot, input channel), N = 32 (step, output channel),
// K = 16 pixels; slot r and step j pair at tap (r - k - j + kt - 1) mod 8, no
// tap where that is >= kt.  k mod 8 takes four values, so four accumulators of
// 32 TMEM columns, each always for one of them, leave the tap of every entry
// fixed while the ring turns.  The chunks are split evenly over the resident
// CTAs (2 per SM) as in tct_conv16; an accumulator sums a quarter of its CTA's
// chunks, one atomic per entry and CTA follows.  The MMAs' additions round
// towards zero, so an accumulator's error grows with the length of its sum (about
// 2^-26 per addition: at 32 clips of 64 x 256 x 256 on the resident CTAs alone 6.7e-5 of
// the gradient's norm, tct_wgrad 7.8e-6): a CTA takes at most 2 K chunks, half of
// tct_wgrad's sum of K steps, and larger calls whole waves of CTAs (2.64 -> 2.81 ms,
// 6.7e-5 -> 3.2e-6).  24 chunks where K is small: the atomics' rounding, one per CTA
// and entry, is as large there.
// Bound by HBM: 128 bytes per pixel-step (8 clips x 64 x 128 x 128: 0.50 ms
// transposed, 0.27 with one step and N = 16 per 8 MMAs on a doubled ring, now
// 0.182; floor 0.158).
constexpr int kWStage = 2;               // chunks in flight
constexpr int kWAcc = 4;

struct Wgrad16Args {
  int K, kt;
  int64_t hw;
  int tiles, nch;
  int64_t total;        // B * tiles * nch chunks
  float* gw;
  float* gb;
  uint32_t wait_iters;
};

// kind::f16 instruction descriptor with both operands MN-major
__host__ __device__ constexpr uint32_t umma_idesc_bf16_mn(int M, int N) {
  return umma_idesc_bf16(M, N) | (1u << 15) | (1u << 16);
}

__global__ void __launch_bounds__(TP, 2)
tct_wgrad16(const __grid_constant__ CUtensorMap m_dz, const __grid_constant__ CUtensorMap m_in, Wgrad16Args A) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint64_t bar[kWStage], mma_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ float red[TP / 32][CP];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int K = A.K, kt = A.kt, nch = A.nch;
  unsigned char* stage = sm;                                    // [kWStage][input x 2, dz x 2]
  unsigned char* ring = stage + kWStage * 4 * kBox;             // [8] slots, step s at s mod 8
  unsigned char* dslot = ring + 8 * kSlot;                      // [2]
  if (warp == 0) tmem_alloc(&tmem_slot, kWAcc * 2 * CP);
  if (tid == 0) {
    for (int i = 0; i < kWStage; ++i) mbar_init(&bar[i], 1);
    mbar_init(&mma_bar, 1);
  }
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
  // a clip's odd last step meets the ring alone (N = 16): products with the step
  // after it would be 0 times the ring, NaN where that holds infinities
  constexpr uint32_t idesc2 = umma_idesc_bf16_mn(TP, 2 * CP), idesc1 = umma_idesc_bf16_mn(TP, CP);
  for (int i = 0; i < kWAcc * 2; ++i) tmem_zero16(tmem + lane_base + (uint32_t)(i * CP));
  tmem_wait_st();
  // MN-major, no swizzle: leading offset = next 8 pixels (K), stride offset =
  // next 8 channels (the planes of consecutive slots are 2 KB apart)
  const uint64_t a_desc = umma_desc(smem_u32(ring), 128, kPlane), b_desc = umma_desc(smem_u32(dslot), 128, kPlane);
  const int64_t t0 = A.total * blockIdx.x / gridDim.x, t1 = A.total * (blockIdx.x + 1) / gridDim.x;
  const int64_t ts = t0 - min((int64_t)(kt / 2), t0 % nch);
  auto load_chunk = [&](int64_t t) {
    const int64_t sg = t / nch;
    const int k = 2 * (int)(t - sg * nch), tl = (int)(sg % A.tiles), b = (int)(sg / A.tiles), n = min(2, K - k);
    const int i = (int)((t - ts) % kWStage);
    unsigned char* dst = stage + i * 4 * kBox;
    mbar_arrive_expect_tx(&bar[i], (uint32_t)(2 * n * kBox));
    for (int j = 0; j < n; ++j) {
      tma_load_3d(dst + j * kBox, &m_in, 0, tl * TP, b * K + k + j, &bar[i]);
      tma_load_3d(dst + (2 + j) * kBox, &m_dz, 0, tl * TP, b * K + k + j, &bar[i]);
    }
  };
  int64_t loaded = 0;                    // thread 0: chunks requested
  if (tid == 0)
    for (int i = 0; i < kWStage && ts + i < t1; ++i) { load_chunk(ts + i); ++loaded; }
  float gbr[CP];
#pragma unroll
  for (int i = 0; i < CP; ++i) gbr[i] = 0.0f;
  uint32_t phase = 0, mma_phase = 0;
  uint32_t used = 0;                     // accumulators that hold something
  int c = (int)(ts % nch);
  bool fresh = true, bail = false;
  int n_mma = 0;
  for (int64_t t = ts; t < t1; ++t) {
    const int si = (int)((t - ts) % kWStage), k = 2 * c, n = min(2, K - k);
    bool fail = !mbar_wait(&bar[si], (phase >> si) & 1u, A.wait_iters);
    phase ^= 1u << si;
    // the previous chunk's MMAs have read the ring and the dz slots
    if (n_mma) {
      fail |= !mbar_wait(&mma_bar, mma_phase ^ 1u, A.wait_iters);
      tc_fence_after();
    }
    if (fresh || c == 0) {
      for (int i = tid; i < 8 * kSlot / 16; i += TP) reinterpret_cast<uint4*>(ring)[i] = make_uint4(0, 0, 0, 0);
      __syncthreads();                   // a row of the ring is zeroed by one thread and filled by another
      fresh = false;
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      if (j >= n) break;
      float x[CP], d[CP];
      box_load(stage + (si * 4 + j) * kBox, tid, x);
      box_load(stage + (si * 4 + 2 + j) * kBox, tid, d);
      store_slot(ring + ((k + j) & 7) * kSlot, tid, x);
      store_slot(dslot + j * kSlot, tid, d);
      if (t >= t0)
#pragma unroll
        for (int i = 0; i < CP; ++i) gbr[i] += d[i];
    }
    fence_proxy_async_smem();
    tc_fence_before();
    bail = __syncthreads_or(fail) != 0;
    if (bail) break;
    tc_fence_after();
    if (tid == 0 && t + kWStage < t1) { load_chunk(t + kWStage); ++loaded; }
    if (t >= t0) {
      const int q = c & (kWAcc - 1);
      if (tid == 0) {
        for (int j = 0; j < TP / 16; ++j)
          umma_bf16(tmem + (uint32_t)(q * 2 * CP), a_desc + (uint64_t)(j * 16), b_desc + (uint64_t)(j * 16),
                    n == 2 ? idesc2 : idesc1, 1u);
        umma_commit(&mma_bar);
      }
      used |= 1u << q;
      ++n_mma;
      mma_phase ^= 1u;
    }
    if (++c == nch) c = 0;
  }
  if (!bail && n_mma) {
    const bool fail = !mbar_wait(&mma_bar, mma_phase ^ 1u, A.wait_iters);
    bail = __syncthreads_or(fail) != 0;
    tc_fence_after();
  }
  if (bail) {
    if (tid == 0) {
      for (int i = 0; i < kWStage; ++i) {
        // requests so far into stage i: those numbered i, i + kWStage, ...
        const int64_t m = (loaded - i + kWStage - 1) / kWStage;
        if (m > 0) mbar_wait(&bar[i], (uint32_t)((m - 1) & 1), kDrainIters);
      }
      atomicAdd(A.gw, __int_as_float(0x7fc00000));   // the gradient reports the failure
    }
    if (n_mma) mbar_wait(&mma_bar, mma_phase ^ 1u, kDrainIters);
  } else {
    // the accumulators' entries summed per (tap, output, input channel) in the
    // staging area (free: every chunk has been read)
    float* sum = reinterpret_cast<float*>(stage);
    for (int i = tid; i < kt * CP * CP; i += TP) sum[i] = 0.0f;
    __syncthreads();
    const int r = tid / CP, ci = tid % CP;   // lane = row (slot r, input channel ci)
    for (int q = 0; q < kWAcc; ++q) {
      if (!((used >> q) & 1u)) continue;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        float v[CP];
        tmem_ld16(tmem + lane_base + (uint32_t)((2 * q + j) * CP), v);
        const int tau = (r - 2 * q - j + kt - 1) & 7;
        if (tau < kt)
#pragma unroll
          for (int co = 0; co < CP; ++co) atomicAdd(&sum[(tau * CP + co) * CP + ci], v[co]);
      }
    }
#pragma unroll
    for (int i = 0; i < CP; ++i) {
      float v = gbr[i];                  // rows beyond hw are zero
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
      if (lane == 0) red[warp][i] = v;
    }
    __syncthreads();
    for (int i = tid; i < kt * CP * CP; i += TP) {   // gw[co][ci][tau]
      const int tau = i % kt, cc = i / kt % CP, co = i / (kt * CP);
      atomicAdd(A.gw + i, sum[(tau * CP + co) * CP + cc]);
    }
    if (tid < CP) {
      float v = 0.0f;
      for (int wv = 0; wv < TP / 32; ++wv) v += red[wv][tid];
      atomicAdd(A.gb + tid, v);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, kWAcc * 2 * CP);
}

}  // namespace

// ---------------------------------------------------------------- host
namespace {

int resident_ctas(int64_t work, int* out) {
  int dev = 0, nsm = 0;
  ET_CHECK_CUDA(cudaGetDevice(&dev));
  ET_CHECK_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  *out = (int)std::max<int64_t>(1, std::min<int64_t>(work, 2 * nsm));
  return ET_OK;
}

}  // namespace

bool et_train_tct_supported(const et_evsnet_weights* net) {
  return net->kt >= 1 && net->kt <= kMaxKtTc && net->C >= 1 && net->C <= CP;
}

int et_train_tct_conv(const float* in, int B, int K, int64_t hw, int C, int kt, const float* w, const float* b,
                      const float* extra, const float* mask, float* out, const float* wp, const float* bp,
                      float* I, bool data_grad, cudaStream_t st) {
  if (kt < 1 || kt > kMaxKtTc || C < 1 || C > CP || B < 1 || K < 1 || hw < 1) return ET_ERR_UNIMPLEMENTED;
  if (use_tma(B, K, hw, C, in, out) && use_tma(B, K, hw, C, extra, mask)) {
    const int64_t tiles = (hw + TP - 1) / TP, nch = (K + 1) / 2;
    Conv16Args A{K, kt, hw, (int)tiles, (int)nch, B * tiles * nch, w, b, extra != nullptr, wp, bp, I,
                 et_tc_wait_iters()};
    CUtensorMap m_in, m_extra, m_mask, m_out;
    std::memset(&m_extra, 0, sizeof(m_extra));
    std::memset(&m_mask, 0, sizeof(m_mask));
    int rc = map_rows(&m_in, in, (int64_t)B * K, hw);
    if (rc == ET_OK) rc = map_rows(&m_out, out, (int64_t)B * K, hw);
    if (rc == ET_OK && extra) rc = map_rows(&m_extra, extra, (int64_t)B * K, hw);
    if (rc == ET_OK && data_grad) rc = map_rows(&m_mask, mask, (int64_t)B * K, hw);
    int grid = 0;
    if (rc == ET_OK) rc = resident_ctas(A.total, &grid);
    if (rc != ET_OK) return rc;
    // input x 2 and O x 2 (forward), or input, O x 2 and E: four or four chunks
    const size_t smem = (size_t)(data_grad ? 1 + 2 + 1 : 2 + 2) * 2 * kBox + (size_t)(kt + 1) * kSlot +
                        (size_t)kt * CP * CP * 2;
    auto kern = data_grad ? tct_conv16<true> : tct_conv16<false>;
    if ((rc = et_allow_shared(kern)) != ET_OK) return rc;
    kern<<<grid, TP, smem, st>>>(m_in, m_extra, m_mask, m_out, A);
    ET_CHECK_LAUNCH();
    return ET_OK;
  }
  ConvArgs A{in, B, K, C, kt, hw, w, b, extra, mask, out, wp, bp, I, et_tc_wait_iters()};
  const size_t smem = (size_t)(kt + 1) * kSlot + (size_t)kt * CP * CP * 2;
  const int64_t blocks = (int64_t)B * ((hw + TP - 1) / TP);
  if (blocks > 0x7FFFFFFF) return ET_ERR_ARG;
  auto launch = [&](auto kern) -> int {
    const int rc = et_allow_shared(kern);
    if (rc != ET_OK) return rc;
    kern<<<(unsigned)blocks, TP, smem, st>>>(A);
    ET_CHECK_LAUNCH();
    return ET_OK;
  };
  return data_grad ? launch(tct_conv<true>) : launch(tct_conv<false>);
}

int et_train_tct_wgrad(const float* dz, const float* in, int B, int K, int64_t hw, int C, int kt, float* gw,
                       float* gb, cudaStream_t st) {
  if (kt < 1 || kt > kMaxKtTc || C < 1 || C > CP || B < 1 || K < 1 || hw < 1) return ET_ERR_UNIMPLEMENTED;
  if (use_tma(B, K, hw, C, dz, in)) {
    const int64_t tiles = (hw + TP - 1) / TP, nch = (K + 1) / 2;
    Wgrad16Args A{K, kt, hw, (int)tiles, (int)nch, B * tiles * nch, gw, gb, et_tc_wait_iters()};
    CUtensorMap m_dz, m_in;
    int rc = map_rows(&m_dz, dz, (int64_t)B * K, hw);
    if (rc == ET_OK) rc = map_rows(&m_in, in, (int64_t)B * K, hw);
    int ctas = 0;
    if (rc == ET_OK) rc = resident_ctas(A.total, &ctas);
    if (rc != ET_OK) return rc;
    const int64_t wave = (int64_t)ctas * std::max(2 * K, 24), grid = (A.total + wave - 1) / wave * ctas;
    if (grid > 0x7FFFFFFF) return ET_ERR_ARG;
    const size_t smem = (size_t)kWStage * 4 * kBox + 10 * kSlot;
    ET_CHECK_CUDA(cudaFuncSetAttribute(tct_wgrad16, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    tct_wgrad16<<<(unsigned)grid, TP, smem, st>>>(m_dz, m_in, A);
    ET_CHECK_LAUNCH();
    return ET_OK;
  }
  const size_t smem = (size_t)kWABytes + kWBBytes;
  const int64_t blocks = (int64_t)B * ((hw + TP - 1) / TP);
  if (blocks > 0x7FFFFFFF) return ET_ERR_ARG;
  auto kern = tct_wgrad;
  ET_CHECK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  kern<<<(unsigned)blocks, TP, smem, st>>>(dz, in, B, K, hw, C, kt, gw, gb, et_tc_wait_iters());
  ET_CHECK_LAUNCH();
  return ET_OK;
}
