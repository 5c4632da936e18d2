// Compensated summation helpers shared by the mixed-precision and the
// compensated fp32 reductions and by the trees of the split-row gemv and of
// the combines of row partials: a (sum, compensation) pair updated with
// Knuth's TwoSum (the rounding error of every add is carried exactly in the
// compensation), merged pairwise across a warp and a CTA.
#pragma once
#include "lift_internal.cuh"

namespace lift {
namespace {

struct Comp {
  float s, c;
};

// s + v with the rounding error folded into c (TwoSum: 6 flops, no branch).
__device__ __forceinline__ void two_sum_add(Comp& a, float v) {
  const float t = __fadd_rn(a.s, v);
  const float bp = __fsub_rn(t, a.s);
  const float e = __fadd_rn(__fsub_rn(a.s, __fsub_rn(t, bp)), __fsub_rn(v, bp));
  a.c = __fadd_rn(a.c, e);
  a.s = t;
}

__device__ __forceinline__ Comp comp_merge(Comp a, const Comp& b) {
  a.c = __fadd_rn(a.c, b.c);
  two_sum_add(a, b.s);
  return a;
}

__device__ __forceinline__ double comp_value(const Comp& a) {
  return isfinite(a.s) ? __dadd_rn((double)a.s, (double)a.c) : (double)a.s;
}

// the pair's value in fp32, rounded once
__device__ __forceinline__ float comp_value32(const Comp& a) { return neumaier_value(a.s, a.c); }

__device__ __forceinline__ Comp warp_comp(Comp v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    Comp w;
    w.s = __shfl_down_sync(0xffffffffu, v.s, o);
    w.c = __shfl_down_sync(0xffffffffu, v.c, o);
    v = comp_merge(v, w);
  }
  return v;
}

// The same for R rows at once (R a power of two): at each of the first
// log2(R) levels a lane gives half of its rows to its partner and keeps the
// other half, so R rows take R - 1 merges and the rest of one tree instead of
// R trees.  Merges commute, so the bits are warp_comp's.  Row r's value ends
// in lane r * (32 / R).
template <int R>
__device__ __forceinline__ Comp warp_comp_rows(Comp (&v)[R]) {
  const int lane = threadIdx.x & (kWarp - 1);
#pragma unroll
  for (int n = R / 2, o = kWarp / 2; n > 0; n /= 2, o /= 2) {
    const bool up = lane & o;
#pragma unroll
    for (int k = 0; k < n; ++k) {
      const Comp keep = up ? v[k + n] : v[k], give = up ? v[k] : v[k + n];
      Comp w;
      w.s = __shfl_xor_sync(0xffffffffu, give.s, o);
      w.c = __shfl_xor_sync(0xffffffffu, give.c, o);
      v[k] = comp_merge(keep, w);
    }
  }
#pragma unroll
  for (int o = kWarp / 2 / R; o > 0; o >>= 1) {
    Comp w;
    w.s = __shfl_down_sync(0xffffffffu, v[0].s, o);
    w.c = __shfl_down_sync(0xffffffffu, v[0].c, o);
    v[0] = comp_merge(v[0], w);
  }
  return v[0];
}

// The last levels of the tree, over lanes 0 .. N-1 (zeros above them would
// change nothing).  Valid in lane 0.
template <int N>
__device__ __forceinline__ Comp warp_comp_first(Comp v) {
#pragma unroll
  for (int o = N / 2; o > 0; o >>= 1) {
    Comp w;
    w.s = __shfl_down_sync(0xffffffffu, v.s, o);
    w.c = __shfl_down_sync(0xffffffffu, v.c, o);
    v = comp_merge(v, w);
  }
  return v;
}

template <int THREADS>
__device__ __forceinline__ Comp block_comp(Comp v) {
  __shared__ float rs[kWarp], rc[kWarp];
  v = warp_comp(v);
  if constexpr (THREADS > kWarp) {
    const int lane = threadIdx.x & (kWarp - 1), warp = threadIdx.x / kWarp;
    if (lane == 0) {
      rs[warp] = v.s;
      rc[warp] = v.c;
    }
    __syncthreads();
    if (warp == 0) {
      v.s = lane < THREADS / kWarp ? rs[lane] : 0.f;
      v.c = lane < THREADS / kWarp ? rc[lane] : 0.f;
      v = warp_comp(v);
    }
  }
  return v;
}

// The end of a reduction whose CTAs leave one FP64 partial each.  One pass (a
// ticket): the last CTA to arrive adds them.  Two passes (no ticket): a second
// kernel, launched as a programmatic dependent, adds them in the same order --
// the same bits -- while the next call is already being scheduled; a last CTA
// that does so competes with the next call's first loads.  `value` is valid in
// thread 0.
template <int THREADS, bool ROOT = false>
__device__ __forceinline__ void finish64(double value, double* __restrict__ partials, unsigned* ticket,
                                         float* result, double* result64) {
  __shared__ bool is_last;
  __shared__ double red64[kWarp];
  const int t = threadIdx.x;
  const int64_t G = gridDim.x;
  if (ticket == nullptr) {
    if (t == 0) partials[blockIdx.x] = value;
    return;
  }
  if (t == 0) {
    partials[blockIdx.x] = value;
    __threadfence();
    is_last = atomicAdd(ticket, 1u) == static_cast<unsigned>(G - 1);
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  double s = 0.0;
  for (int64_t i = t; i < G; i += THREADS) s = __dadd_rn(s, __ldcg(partials + i));
  s = block_tree64<THREADS>(s, red64);
  if (t == 0) {
    if (ROOT) s = __dsqrt_rn(s);
    *result = static_cast<float>(s);
    if (result64) *result64 = s;
    *ticket = 0u;
  }
}

template <int THREADS, bool ROOT>
__global__ void __launch_bounds__(THREADS)
    combine64_kernel(const double* __restrict__ partials, int64_t G, float* result, double* result64) {
  pdl_trigger();   // the next call's first kernel may be scheduled (it waits for this one)
  pdl_wait();      // the first pass has finished
  __shared__ double red64[kWarp];
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < G; i += THREADS) s = __dadd_rn(s, __ldcg(partials + i));
  s = block_tree64<THREADS>(s, red64);
  if (threadIdx.x == 0) {
    if (ROOT) s = __dsqrt_rn(s);
    *result = static_cast<float>(s);
    if (result64) *result64 = s;
  }
}

// Two passes pay from about this many bytes read on: the host submits the
// second launch while the first kernel runs.
constexpr int64_t kTwoPassBytes = 16 << 20;

template <int THREADS, bool ROOT = false>
struct Combine64 {
  static const void* kernel() { return reinterpret_cast<const void*>(&combine64_kernel<THREADS, ROOT>); }
  static lift_status launch(const double* partials, int64_t G, float* result, double* result64,
                            cudaStream_t s) {
    void* args[] = {&partials, &G, &result, &result64};
    return launch_config(kernel(), dim3(1), dim3(THREADS), 0, 1, s, args, true);
  }
};

}  // namespace
}  // namespace lift
