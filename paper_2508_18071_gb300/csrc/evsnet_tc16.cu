// EvSNet forward on the tcgen05 tensor cores for stacks of 3x3 convolutions of
// at most 16 channels with BF16 operands (evsnet_tc.cu has the other widths and
// FP8): Eq. 5 with kernel extent in space, the projection (Eq. 6) and BiLIF (Eq.
// 2-3).  Weights and inputs of layers 1.. rounded to BF16, FP32 accumulation;
// layer 0, the projection and BiLIF FP32 on the CUDA cores.  Same sums in the
// same order as evsnet_tc.cu.
//
// With 16 output channels an MMA of M = 128 positions, N = 16, K = 16 uses a
// small part of the tensor core and costs what N = 48 costs (57 to 75 clocks);
// nine of them per 128 positions and layer bounded evsnet_tc.cu.  Here one MMA
// applies a column of three taps: its input rows feed the output rows above, at
// and below them, whose accumulators lie in neighbouring TMEM columns.  For that
// a step of one image row has to be a step of one M block, so a CTA's tile, 32
// columns by 4 S rows, is stored with row j + S q (q = 0..3) as the q-th quarter
// of block j: block j + 1 is one row further down in all four quarters.  The rows
// that wrap (S q - 1 above block 0, S q + S below block S - 1) are stored a second
// time in blocks -1 and S.  Input block i is three MMAs (one per column shift),
//   D[:, columns of blocks i - 1 .. i + 1] += A_i [W(ky = 2) | W(1) | W(0)],
// 3 (S + 2) per layer instead of 9 S, and every output still sums its taps in
// row-major order (the accumulators start at zero: the epilogue clears what it
// has read).
//
// A column shift moves the operand's start by one 16-byte row, so the tile's
// outermost columns, like its outermost rows, become invalid by one per layer:
// 32 x 4 S positions give (32 - 2 (L - 1)) x (4 S - 2 (L - 1)) pixels.  Warp w
// reads TMEM quarter w % 4 of the first (w < 4) or second half of the blocks: its lane is the
// column, quarter and block are the row, and a thread keeps the membrane of its
// pixels in registers for the whole call.  The next frame is copied (cp.async) while
// the current one's tensor-core layers run.
//
// Trained 4-layer network, 1280 x 720: 95 -> 42.5 us per frame plus 30 us per call;
// 253 x 187: 25 -> 6.5 us per frame.  Alone on its SM a tile of S = 8 takes 16 k
// clocks per step, of them 4.9 k for 90 MMAs (53 each, the rate of their issue), 2.7
// k layer 0 and 1.2 to 1.6 k per epilogue; with three CTAs per SM it is 9.5 k per
// tile-step, bound by instruction issue beside the MMAs.
#include "et_internal.cuh"
#include "event_emit.cuh"
#include "evsnet_common.h"
#include "f32x2.cuh"
#include "tc_ptx.cuh"
#include <cuda_bf16.h>
#include <algorithm>

namespace {

constexpr int kThreads = 256;
constexpr int TW = 32;                 // columns of a tile
constexpr int CP = 16;
constexpr int kMaxS = 8;               // M blocks of a tile
constexpr int kXP = TW + 2;            // pitch of the X tile
constexpr int kStageCap = 192;         // events a warp holds before it appends them
constexpr int kLayerB = 3 * 3 * CP * CP * 2;   // bytes of a layer's B operands: 3 column shifts x 48 rows x 32 B
constexpr uint32_t kDrainIters = 1u << 22;
constexpr unsigned long long kTimeoutBit = 1ull << 62;

struct Tc16Params {
  int H, W, F, f0, t0, L, C;
  float beta, vth, reset;
  int tiles_x;
  int plane;                             // bytes of one 8-channel plane of the activations
  int off_wB, off_f32, off_x;            // shared-memory byte offsets
  uint32_t tmem_cols, wait_iters;
};

__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}

__device__ __forceinline__ uint32_t pack2x(f32x2 v) {
  float lo, hi;
  unpack2f(v, lo, hi);
  return pack2(lo, hi);
}

// ReLU of two BF16 values (a NaN becomes 0, as in fmaxf)
__device__ __forceinline__ uint32_t relu2(uint32_t v) {
  const __nv_bfloat162 z = __floats2bfloat162_rn(0.0f, 0.0f);
  const __nv_bfloat162 h = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&v), z);
  return *reinterpret_cast<const uint32_t*>(&h);
}

template <int S>                       // M blocks of a tile: 4, 6 or 8
__global__ void __launch_bounds__(kThreads, 3)
evsnet_tc16_kernel(Tc16Params P, const float* __restrict__ logl, const float* __restrict__ wg,
                   const float* __restrict__ bg, float* __restrict__ Vg, const float* __restrict__ last_l,
                   et_event* events, int64_t cap, unsigned long long* n_events, float* __restrict__ I_out,
                   int8_t* __restrict__ spikes) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint64_t mma_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ uint32_t staged[kThreads / 32][kStageCap];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int L = P.L, C = P.C, halo = L - 1, quarter = warp & 3;
  const int ox = (blockIdx.x % P.tiles_x) * (TW - 2 * halo) - halo;        // image column of tile column 0
  const int oy = (blockIdx.x / P.tiles_x) * (4 * S - 2 * halo) - halo;
  const int64_t npix = (int64_t)P.H * P.W;
  unsigned char* act = sm + 128;         // block i at (i + 1) * 128 rows of 16 bytes, two planes
  unsigned char* wB = sm + P.off_wB;
  float* w0 = reinterpret_cast<float*>(sm + P.off_f32);   // [9][CP]
  float* bs = w0 + 9 * CP;               // [L][CP]
  float* wp = bs + L * CP;               // [CP], then the projection's bias
  // log frames over rows -1 .. 4 S, columns -1 .. 32 of the tile, zero outside the
  // image: frame f in one buffer, f - 1 in the other
  constexpr int nx = (4 * S + 2) * kXP;
  float* frames = reinterpret_cast<float*>(sm + P.off_x);

  // ---- set-up: zero operands, weights, the previous frame, membranes
  for (int i = tid; i < P.off_wB / 16; i += kThreads) reinterpret_cast<uint4*>(sm)[i] = make_uint4(0, 0, 0, 0);
  for (int i = tid; i < 9 * CP; i += kThreads) w0[i] = i % CP < C ? wg[(i % CP) * 9 + i / CP] : 0.0f;
  for (int i = tid; i < L * CP; i += kThreads) bs[i] = i % CP < C ? bg[(i / CP) * C + i % CP] : 0.0f;
  const int wproj = 9 * C + (L - 1) * C * C * 9;
  for (int i = tid; i <= CP; i += kThreads) wp[i] = i == CP ? bg[L * C] : (i < C ? wg[wproj + i] : 0.0f);
  // B operands: per layer l >= 1 and column shift kx, rows n = 16 (2 - ky) + co
  // in two 16-byte columns of 8 input channels
  for (int i = tid; i < (L - 1) * 9 * CP * CP; i += kThreads) {
    const int ci = i % CP, n = (i / CP) % 48, kx = (i / (CP * 48)) % 3, l = i / (CP * 144);
    const int co = n % CP, ky = 2 - n / CP;
    const float v = co < C && ci < C ? wg[9 * C + l * C * C * 9 + (co * C + ci) * 9 + ky * 3 + kx] : 0.0f;
    *reinterpret_cast<__nv_bfloat16*>(wB + l * kLayerB + kx * (48 * 32) + (ci >> 3) * (48 * 16) + n * 16 +
                                      (ci & 7) * 2) = __float2bfloat16_rn(v);
  }
  // starts the copy of a frame into its buffer (f & 1); this thread's positions
  // are tid, tid + 256, ... (kept as numbers: a register spilled here is read back
  // from L2 every step, the L1 being what the shared memory leaves)
  auto load_frame = [&](const float* src, int f) {
    int col = tid % kXP, row = tid / kXP;
#pragma unroll 1
    for (int i = tid; i < nx; i += kThreads) {
      const int gx = ox - 1 + col, gy = oy - 1 + row;
      const bool in = gx >= 0 && gx < P.W && gy >= 0 && gy < P.H;
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(frames + (f & 1) * nx + i)),
                   "l"(src + (in ? (int64_t)gy * P.W + gx : 0)), "r"(in ? 4 : 0)
                   : "memory");
      col += kThreads % kXP;
      row += kThreads / kXP;
      if (col >= kXP) { col -= kXP; ++row; }
    }
  };
  load_frame(P.f0 == 0 ? last_l : logl, P.f0 + 1);        // the frame before the first step
  if (P.f0 < P.F) load_frame(logl + (int64_t)P.f0 * npix, P.f0);
  // this thread's pixels: column `lane`, row b + S quarter of its S / 2 blocks b
  const int b_first = (warp >> 2) * (S / 2);
  const int gx = ox + lane;
  const bool col_ok = lane >= halo && lane < TW - halo && gx < P.W;
  float V[S / 2];
#pragma unroll
  for (int k = 0; k < S / 2; ++k) {
    const int b = b_first + k, r = b + S * quarter, gy = oy + r;
    const bool own = col_ok && r >= halo && r < 4 * S - halo && gy < P.H;
    V[k] = own ? Vg[(int64_t)gy * P.W + gx] : 0.0f;
  }
  EventStage<kStageCap> stage(staged[warp], events, cap, n_events, (uint32_t)gx, (uint32_t)(oy + S * quarter),
                              (uint32_t)P.t0);
  if (warp == 0) tmem_alloc(&tmem_slot, P.tmem_cols);
  if (tid == 0) mbar_init(&mma_bar, 1);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
  for (int b = b_first; b < b_first + S / 2; ++b) tmem_zero16(tmem + lane_base + (uint32_t)(b * CP));
  tmem_wait_st();
  uint32_t phase = 0;
  bool bail = false;
  // eight channels w (plane h) of a position's BF16 row, ReLU applied here, zero
  // outside the image: block b, quarter q, column `lane`; also into block -1 or S
  // where the row wraps
  auto put = [&](int b, int q, int h, uint4 w, bool in) {
    w = in ? make_uint4(relu2(w.x), relu2(w.y), relu2(w.z), relu2(w.w)) : make_uint4(0u, 0u, 0u, 0u);
    unsigned char* a = act + h * P.plane + (q * TW + lane) * 16;
    *reinterpret_cast<uint4*>(a + (b + 1) * (128 * 16)) = w;
    if (b == S - 1 && q < 3) *reinterpret_cast<uint4*>(a + TW * 16) = w;
    if (b == 0 && q > 0) *reinterpret_cast<uint4*>(a + (S + 1) * (128 * 16) - TW * 16) = w;
  };

  for (int f = P.f0; f < P.F; ++f) {
    // ---- the frame, requested while the previous one's layers ran
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // ---- layer 0: column `lane` of S / 2 consecutive rows per warp (two warps
    // share a quarter), eight channels of all of them at a time: a tap's weights,
    // 32 bytes per lane, then serve four rows
    {
      const int r = warp * (S / 2), rb = (warp & 1) * (S / 2), rq = warp >> 1;
      const float* cur = frames + (f & 1) * nx + r * kXP + lane;
      const float* old = frames + (~f & 1) * nx + r * kXP + lane;
      float x[S / 2 + 2][3];             // X (Eq. 1)
#pragma unroll
      for (int j = 0; j < S / 2 + 2; ++j)
#pragma unroll
        for (int i = 0; i < 3; ++i) x[j][i] = cur[j * kXP + i] - old[j * kXP + i];
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        f32x2 acc[S / 2][4];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const ulonglong2 b2 = *reinterpret_cast<const ulonglong2*>(bs + 8 * h + 4 * c);
#pragma unroll
          for (int k = 0; k < S / 2; ++k) { acc[k][2 * c] = b2.x; acc[k][2 * c + 1] = b2.y; }
        }
#pragma unroll
        for (int t = 0; t < 9; ++t) {
          const ulonglong2 wa = *reinterpret_cast<const ulonglong2*>(w0 + t * CP + 8 * h);
          const ulonglong2 wb = *reinterpret_cast<const ulonglong2*>(w0 + t * CP + 8 * h + 4);
#pragma unroll
          for (int k = 0; k < S / 2; ++k) {
            const f32x2 d = pack2f(x[k + t / 3][t % 3], x[k + t / 3][t % 3]);
            acc[k][0] = fma2(wa.x, d, acc[k][0]);
            acc[k][1] = fma2(wa.y, d, acc[k][1]);
            acc[k][2] = fma2(wb.x, d, acc[k][2]);
            acc[k][3] = fma2(wb.y, d, acc[k][3]);
          }
        }
#pragma unroll
        for (int k = 0; k < S / 2; ++k) {
          const int gy = oy + r + k;
          put(rb + k, rq, h, make_uint4(pack2x(acc[k][0]), pack2x(acc[k][1]), pack2x(acc[k][2]), pack2x(acc[k][3])),
              gx >= 0 && gx < P.W && gy >= 0 && gy < P.H);
        }
      }
    }
    // ---- tensor-core layers
    for (int l = 1; l < L; ++l) {
      fence_proxy_async_smem();
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      if (tid == 0) {
        // operand descriptors differ only in their start address (16-byte units): a
        // block is 128 rows on, a column shift one row (A) or 96 rows (B), an output
        // row 16 rows of B
        const uint64_t a_desc = umma_desc(smem_u32(act) - 16, (uint32_t)P.plane, 128);
        const uint64_t bl = umma_desc(smem_u32(wB) + (uint32_t)((l - 1) * kLayerB), 48 * 16, 128);
        // input block i into the output blocks from `lo` on, B from row 16 `skip`
        auto block = [&](int i, int lo, int skip, uint32_t idesc) {
          const uint64_t a = a_desc + (uint64_t)((i + 1) * 128), w = bl + (uint64_t)(skip * CP);
          const uint32_t d = tmem + (uint32_t)(lo * CP);
#pragma unroll
          for (int kx = 0; kx < 3; ++kx) umma_bf16(d, a + (uint64_t)kx, w + (uint64_t)(kx * 96), idesc, 1u);
        };
        constexpr uint32_t id16 = umma_idesc_bf16(128, 16), id32 = umma_idesc_bf16(128, 32),
                           id48 = umma_idesc_bf16(128, 48);
        block(-1, 0, 2, id16);
        block(0, 0, 1, id32);
#pragma unroll
        for (int i = 1; i < S - 1; ++i) block(i, i - 1, 0, id48);
        block(S - 1, S - 2, 0, id32);
        block(S, S - 1, 0, id16);
        umma_commit(&mma_bar);
      }
      __syncwarp();
      // layer 0 has read the previous frame: its buffer takes the next one
      if (l == 1 && f + 1 < P.F) load_frame(logl + (int64_t)(f + 1) * npix, f + 1);
      const bool ok = mbar_wait(&mma_bar, phase, P.wait_iters);
      phase ^= 1u;
      if (!ok && lane == 0) atomicOr(n_events, kTimeoutBit);
      bail = __syncthreads_or(!ok) != 0;
      if (bail) break;
      tc_fence_after();
      const ulonglong2* bl = reinterpret_cast<const ulonglong2*>(bs + l * CP);
      // block k's accumulators (cleared for the next layer) plus the bias
      auto take = [&](int k, f32x2 (&acc)[CP / 2]) {
        const uint32_t t = tmem + lane_base + (uint32_t)((b_first + k) * CP);
        float raw[CP];
        tmem_ld16(t, raw);
        tmem_zero16(t);
#pragma unroll
        for (int c = 0; c < CP / 4; ++c) {
          const ulonglong2 b2 = bl[c];
          acc[2 * c] = add2(pack2f(raw[4 * c], raw[4 * c + 1]), b2.x);
          acc[2 * c + 1] = add2(pack2f(raw[4 * c + 2], raw[4 * c + 3]), b2.y);
        }
      };
      // (the loops over blocks stay rolled where they can: the kernel's code has to
      // stay in the instruction cache from step to step)
      if (l < L - 1) {
#pragma unroll 1
        for (int k = 0; k < S / 2; ++k) {
          const int b = b_first + k, r = b + S * quarter, gy = oy + r;
          f32x2 acc[CP / 2];
          take(k, acc);
          if (lane >= l && lane < TW - l && r >= l && r < 4 * S - l)
#pragma unroll
            for (int h = 0; h < 2; ++h)
              put(b, quarter, h, make_uint4(pack2x(acc[4 * h]), pack2x(acc[4 * h + 1]), pack2x(acc[4 * h + 2]),
                                            pack2x(acc[4 * h + 3])), gx >= 0 && gx < P.W && gy >= 0 && gy < P.H);
        }
      } else {
        uint32_t fired = 0, neg = 0;     // spikes and negative ones by block
        const int64_t q0 = (int64_t)(f - P.f0) * npix + (int64_t)(oy + b_first + S * quarter) * P.W + gx;
#pragma unroll
        for (int k = 0; k < S / 2; ++k) {
          const int r = b_first + k + S * quarter, gy = oy + r;
          f32x2 acc[CP / 2];
          take(k, acc);
          float I = wp[CP];
#pragma unroll
          for (int c = 0; c < CP / 2; ++c) {
            float lo, hi;
            unpack2f(acc[c], lo, hi);
            I = fmaf(wp[2 * c], fmaxf(lo, 0.0f), I);
            I = fmaf(wp[2 * c + 1], fmaxf(hi, 0.0f), I);
          }
          const float vp = P.beta * V[k] + I;
          const int sp = vp >= P.vth ? 1 : (vp <= -P.vth ? -1 : 0);
          if (col_ok && r >= halo && r < 4 * S - halo && gy < P.H) {
            V[k] = vp - P.reset * (float)sp;
            if (I_out) I_out[q0 + k * P.W] = I;
            if (spikes) spikes[q0 + k * P.W] = (int8_t)sp;
            fired |= sp != 0 ? 1u << k : 0u;
            neg |= sp < 0 ? 1u << k : 0u;
          }
        }
        if (P.t0 + f >= 0)               // delayed labels below 0: none
          stage.template add_rows<S / 2>(fired, neg, (uint32_t)f, (uint32_t)b_first);
      }
      tmem_wait_st();
      tc_fence_before();
    }
    if (bail) break;
  }
  if (bail) {
    // a bounded wait gave up: the MMAs still in flight get a second bounded wait
    // before the TMEM is released; membranes stay as they were
    mbar_wait(&mma_bar, phase ^ 1u, kDrainIters);
  } else {
    stage.flush();
#pragma unroll
    for (int k = 0; k < S / 2; ++k) {
      const int b = b_first + k, r = b + S * quarter, gy = oy + r;
      if (col_ok && r >= halo && r < 4 * S - halo && gy < P.H) Vg[(int64_t)gy * P.W + gx] = V[k];
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, P.tmem_cols);
}

}  // namespace

int et_evsnet_forward_tc16(const float* logl, int32_t F, const et_evsnet_weights* net,
                           et_evsnet_state* st, int32_t t0, et_event* events, int64_t cap,
                           int64_t* n_events, float* I_out, int8_t* spikes, cudaStream_t stream) {
  Tc16Params P{};
  P.H = st->H; P.W = st->W; P.F = F; P.f0 = st->initialized ? 0 : 1; P.t0 = t0;
  P.L = net->n_layers; P.C = net->C;
  P.beta = net->beta; P.vth = net->vth; P.reset = net->reset;
  int dev = 0, nsm = 0;
  ET_CHECK_CUDA(cudaGetDevice(&dev));
  ET_CHECK_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  // the tile height (even S) that leaves the busiest SM the least work: its tiles
  // times the MMAs of one, 3 (S + 2) per layer (us per frame at S = 4 / 6 / 8:
  // 1280 x 720 59.5 / 46.6 / 42.5; 641 x 363 32.6 / 26.5 / 23.0; 253 x 187 6.3 /
  // 6.5 / 7.9)
  const int halo = P.L - 1, tw = TW - 2 * halo;
  P.tiles_x = (P.W + tw - 1) / tw;
  int S = 0;
  int64_t tiles = 0, best = -1;
  for (int s = 4; s <= kMaxS; s += 2) {
    const int th = 4 * s - 2 * halo;
    const int64_t n = (int64_t)P.tiles_x * ((P.H + th - 1) / th), cost = (n + nsm - 1) / nsm * (s + 2);
    if (best < 0 || cost <= best) { best = cost; tiles = n; S = s; }
  }
  P.plane = ((S + 2) * 128 + 16) * 16;
  auto al = [](int x) { return (x + 127) & ~127; };
  P.off_wB = al(128 + 2 * P.plane);
  P.off_f32 = P.off_wB + al((P.L - 1) * kLayerB);
  P.off_x = P.off_f32 + al(4 * (9 * CP + P.L * CP + CP + 4));
  const int smem = P.off_x + 2 * 4 * (4 * S + 2) * kXP;
  P.tmem_cols = S * CP <= 64 ? 64 : 128;
  P.wait_iters = et_tc_wait_iters();
  auto kern = S == 4 ? evsnet_tc16_kernel<4> : S == 6 ? evsnet_tc16_kernel<6> : evsnet_tc16_kernel<8>;
  const int rc = et_allow_shared(kern);
  if (rc != ET_OK) return rc;
  kern<<<(unsigned)tiles, kThreads, smem, stream>>>(
      P, logl, net->w, net->b, st->V, st->last_l, events, cap, reinterpret_cast<unsigned long long*>(n_events),
      I_out, spikes);
  ET_CHECK_LAUNCH();
  return ET_OK;
}
