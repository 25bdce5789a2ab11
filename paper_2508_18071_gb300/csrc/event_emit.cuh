// Warp-aggregated event append shared by the event-producing kernels.
#pragma once
#include "et_internal.cuh"

// Every lane of the warp must call this (lanes without events pass n = 0).
// Lane i appends n_i copies of (x, y, t, p); one atomicAdd per warp reserves
// the slots.  Slots at or beyond `cap` are counted but not written.  Sum holds the
// warp's count: 64 bits where a lane's may be near 2^32 (an infinite step).
template <typename Sum = uint32_t>
__device__ __forceinline__ void emit_events_warp(et_event* events, int64_t cap,
                                                 unsigned long long* counter, uint32_t n,
                                                 uint32_t x, uint32_t y, uint32_t t, int p) {
  const unsigned lane = threadIdx.x & 31u;
  Sum incl = n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const Sum v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= (unsigned)o) incl += v;
  }
  const Sum total = __shfl_sync(0xFFFFFFFFu, incl, 31);
  if (total == 0) return;
  unsigned long long base = 0;
  if (lane == 31) base = atomicAdd(counter, (unsigned long long)total);
  base = __shfl_sync(0xFFFFFFFFu, base, 31);
  const unsigned long long start = base + (incl - n);
  uint32_t* out = reinterpret_cast<uint32_t*>(events);
  // slots at or beyond cap are counted only: the loop stops there
  for (uint32_t i = 0; i < n && start + i < (unsigned long long)cap; ++i) {
    const unsigned long long slot = start + i;
    out[3 * slot] = x | (y << 16);
    out[3 * slot + 1] = t;
    out[3 * slot + 2] = (uint32_t)(uint8_t)(int8_t)p;
  }
}

// A warp's events gathered in shared memory and appended kCap at a time: the
// appends of all warps meet on one counter, whose atomics the device serves one
// after the other (a 25-frame 720p call with an append per warp and step makes
// 720,000 of them), and an append's round trip holds its warp up.  An event is
// packed as (step - base) << 11 | dy << 6 | lane << 1 | (p > 0); x and y are the
// lane's, y plus dy rows (dy < 32).
template <int kCap>
struct EventStage {
  uint32_t* buf;        // the warp's kCap entries in shared memory
  int n = 0;            // entries held (the same in every lane)
  uint32_t base = 0;    // step of the packed entries' zero
  et_event* events;
  int64_t cap;
  unsigned long long* counter;
  uint32_t x, y, t0;    // the lane's pixel; label of step 0

  __device__ __forceinline__ EventStage(uint32_t* buf_, et_event* events_, int64_t cap_,
                                        unsigned long long* counter_, uint32_t x_, uint32_t y_, uint32_t t0_)
      : buf(buf_), events(events_), cap(cap_), counter(counter_), x(x_), y(y_), t0(t0_) {}

  __device__ __forceinline__ void flush() {
    if (n == 0) return;
    const unsigned lane = threadIdx.x & 31u;
    __syncwarp();
    unsigned long long at = 0;
    if (lane == 0) at = atomicAdd(counter, (unsigned long long)n);
    at = __shfl_sync(0xFFFFFFFFu, at, 0);
    uint32_t* out = reinterpret_cast<uint32_t*>(events);
    for (int i0 = 0; i0 < n; i0 += 32) {
      const int i = i0 + (int)lane;
      const uint32_t e = i < n ? buf[i] : 0u;
      const uint32_t xy = __shfl_sync(0xFFFFFFFFu, x | (y << 16), (e >> 1) & 31u);
      const unsigned long long slot = at + (unsigned long long)i;
      if (i < n && slot < (unsigned long long)cap) {
        out[3 * slot] = xy + (((e >> 6) & 31u) << 16);
        out[3 * slot + 1] = t0 + base + (e >> 11);
        out[3 * slot + 2] = (e & 1u) ? 1u : 0xFFu;
      }
    }
    __syncwarp();
    n = 0;
  }

  // every lane of the warp calls this: cnt events of polarity p at `step`, dy
  // rows below the lane's pixel (`first` = the smallest step any lane passes, at
  // most 2^15 below it; it never decreases from call to call)
  __device__ __forceinline__ void add(uint32_t cnt, uint32_t step, uint32_t first, int p, uint32_t dy = 0) {
    const unsigned lane = threadIdx.x & 31u;
    const unsigned any = __ballot_sync(0xFFFFFFFFu, cnt != 0);
    if (!any) return;
    int rank = __popc(any & ((1u << lane) - 1u)), total = __popc(any);
    if (__any_sync(0xFFFFFFFFu, cnt > 1)) {
      // more than the entries hold from one lane alone: counted in full, and
      // the append below then goes straight to the buffer
      const uint32_t c = min(cnt, (uint32_t)kCap + 1u);
      uint32_t incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= (unsigned)o) incl += v;
      }
      rank = (int)(incl - c);
      total = (int)__shfl_sync(0xFFFFFFFFu, incl, 31);
      if (total > kCap) {
        emit_events_warp<unsigned long long>(events, cap, counter, cnt, x, y + dy, t0 + step, p);
        return;
      }
    }
    if (n + total > kCap || first + (1u << 15) - base >= (1u << 20)) flush();
    if (n == 0) base = first;
    for (uint32_t i = 0; i < cnt; ++i)
      buf[n + rank + (int)i] = ((step - base) << 11) | (dy << 6) | (lane << 1) | (p > 0 ? 1u : 0u);
    n += total;
  }

  // every lane of the warp calls this: bit k of `fired` is an event at `step`,
  // dy0 + k rows below the lane's pixel (or, kSteps, at step + k and dy0 rows
  // below), negative where bit k of `neg` is set (32 kRows <= kCap)
  template <int kRows, bool kSteps = false>
  __device__ __forceinline__ void add_rows(uint32_t fired, uint32_t neg, uint32_t step, uint32_t dy0) {
    static_assert(32 * kRows <= kCap, "a call's events fit the entries");
    const unsigned lane = threadIdx.x & 31u, below = (1u << lane) - 1u;
    if (!__any_sync(0xFFFFFFFFu, fired != 0)) return;
    unsigned m[kRows];
    int total = 0;
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
      m[k] = __ballot_sync(0xFFFFFFFFu, (fired >> k) & 1u);
      total += __popc(m[k]);
    }
    if (n + total > kCap || step + (1u << 15) - base >= (1u << 20)) flush();
    if (n == 0) base = step;
    const uint32_t e = ((step - base) << 11) | (dy0 << 6) | (lane << 1);
    int at = n;
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
      if ((fired >> k) & 1u) buf[at + __popc(m[k] & below)] =
            e + ((uint32_t)k << (kSteps ? 11 : 6)) + (((neg >> k) & 1u) ^ 1u);
      at += __popc(m[k]);
    }
    n = at;
  }
};
