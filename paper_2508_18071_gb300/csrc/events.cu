// Contrast-threshold event generator (paper Sec. 3.1).
//
// One thread per pixel walks the frames in order.  The decision is FP64 with
// explicitly rounded operations (no contraction), reproducible bit for bit by
// any IEEE FP64 implementation fed the same float32 log frames; this device
// does two FP64 operations per SM and clock, so almost every step is decided by
// an FP32 estimate whose error bound leaves no doubt about the FP64 result:
//   e = |l - float(r)| differs from |d| by at most 2^-23 (|r| + e);
//   no event when e plus that bound stays below C;
//   n = floor(e / C) when e / C is farther than the bound from a whole number;
// anything else (and NaN, infinities, huge n) takes the exact path.  An event
// then costs one FP64 addition (n = 1) and one conversion.  Lanes reach their
// next undecided step on their own (frames wait in shared memory, 16 at a time)
// and take events together.
#include "et_internal.cuh"
#include "event_emit.cuh"

namespace {

constexpr int kThr = 256;
constexpr int kFrames = 16;      // frames a thread loads at once
constexpr int kStageCap = 128;   // events a warp holds before it appends them

__global__ void __launch_bounds__(kThr)
threshold_kernel(const float* __restrict__ logl, int F, int H, int W, double C, int t0,
                 double* __restrict__ ref, int initialized, et_event* events, int64_t cap,
                 unsigned long long* n_events) {
  __shared__ float frames[kFrames][kThr];
  __shared__ uint32_t staged[kThr / 32][kStageCap];
  const int tid = threadIdx.x;
  const int64_t npix = (int64_t)H * W;
  const int64_t q = (int64_t)blockIdx.x * kThr + tid;
  const bool live = q < npix;
  double r = 0.0;
  if (live) r = initialized ? ref[q] : (double)__ldg(logl + q);
  float rf = (float)r;
  // C is a float widened; one whose reciprocal or products could leave the
  // normal range takes the exact path throughout
  const float Cf = (float)C;
  const bool normal = Cf > 1e-30f && Cf < 1e30f;
  const float lim = normal ? Cf : 0.0f, inv = normal ? 1.0f / Cf : __int_as_float(0x7fc00000);
  const uint32_t x = live ? (uint32_t)(q % W) : 0u, y = live ? (uint32_t)(q / W) : 0u;
  EventStage<kStageCap> stage(staged[tid >> 5], events, cap, n_events, x, y, (uint32_t)t0);
  constexpr float kUlp = 1.0f / 2097152.0f;        // 2^-21: four times the bound above
  for (int f0 = initialized ? 0 : 1; f0 < F; f0 += kFrames) {
    const int nf = min(kFrames, F - f0);
    // each thread reads only its own column back: no barrier
#pragma unroll
    for (int j = 0; j < kFrames; ++j)
      if (live && j < nf) frames[j][tid] = __ldg(logl + (int64_t)(f0 + j) * npix + q);
    int j = live ? 0 : nf;
    while (true) {
      // to the next step that may hold an event
      float l = 0.0f, e = 0.0f;
      bool hit = false;
      while (j < nf) {
        l = frames[j][tid];
        e = fabsf(l - rf);
        hit = !(e + kUlp * (fabsf(rf) + e) < lim);
        if (hit) break;
        ++j;
      }
      if (!__any_sync(0xFFFFFFFFu, hit)) break;
      uint32_t n = 0;
      int p = 0;
      if (hit) {
        const float qf = e * inv, k = floorf(qf), frac = qf - k;
        const float tol = kUlp * ((fabsf(rf) + e) * inv + qf + 1.0f);
        if (frac > tol && frac < 1.0f - tol && qf < 65536.0f) {
          if (k > 0.0f) {
            p = l > rf ? 1 : -1;
            n = (uint32_t)k;
            const double kC = n == 1 ? C : __dmul_rn((double)n, C);
            r = __dadd_rn(r, p > 0 ? kC : -kC);
            rf = (float)r;
          }
        } else {
          const double d = __dsub_rn((double)l, r);
          const double kd = floor(__ddiv_rn(fabs(d), C));
          if (kd > 0.0) {
            p = d > 0.0 ? 1 : -1;
            n = (uint32_t)kd;
            r = __dadd_rn(r, __dmul_rn(__dmul_rn((double)p, kd), C));
            rf = (float)r;
          }
        }
      }
      stage.add(n, (uint32_t)(f0 + j), (uint32_t)f0, p);
      if (hit) ++j;
    }
  }
  stage.flush();
  if (live && F > 0) ref[q] = r;
}

}  // namespace

extern "C" int et_threshold_events(const float* logl, int32_t F, int32_t H, int32_t W, float C,
                                   int32_t t0, double* ref, int32_t initialized, et_event* events,
                                   int64_t cap, int64_t* n_events, void* stream_) {
  if (F < 0 || H < 1 || W < 1 || H > 65535 || W > 65535 || !(C > 0.0f) || cap < 0) return ET_ERR_ARG;
  if (!ref || !n_events || (F > 0 && !logl) || (cap > 0 && !events)) return ET_ERR_ARG;
  cudaStream_t stream = (cudaStream_t)stream_;
  ET_CHECK_CUDA(cudaMemsetAsync(n_events, 0, sizeof(int64_t), stream));
  if (F == 0) return ET_OK;
  const int64_t npix = (int64_t)H * W;
  const int threads = 256;
  const int64_t blocks = (npix + threads - 1) / threads;
  threshold_kernel<<<(unsigned)blocks, threads, 0, stream>>>(
      logl, F, H, W, (double)C, t0, ref, initialized, events, cap,
      reinterpret_cast<unsigned long long*>(n_events));
  ET_CHECK_LAUNCH();
  return ET_OK;
}
