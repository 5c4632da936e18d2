// Vector programs on unaligned inputs: asum, dot, nrm2, sum, the compensated
// asum and dot, scal and axpy of vectors that start 4, 8 or 12 bytes past a
// 16-byte boundary -- slices of larger arrays -- and, for the two-input
// programs, at different offsets.  The default entry points come here when
// the picked variant's vectors need an alignment that the pointers do not
// have; a variant asked for by id runs its 4-byte form instead.
//
// The program is that of the aligned kernels with the vector padded in
// front: element i of the call is element i + m of a vector that starts on
// the 16-byte boundary below x (m = 0 .. 3 elements; scal and axpy take the
// boundary below y), its tiles are split from there, and the elements
// before m and past n + m are the neutral zero.  Only elements of the call
// are read: the tiles at either end use guarded 4-byte loads.
//
// A second array at another offset is read in the aligned 16-byte blocks it
// lies in, and each vector is put together from a block and the next one:
// a warp's blocks are consecutive (lane l of vector j holds block 32 j + l),
// so the next block is one shuffle away, and lane 0 loads one block more per
// J for the last vector of lane 31.  4-byte loads, the alternative, cost 6 to
// 10 % of the bandwidth where they are coalesced and many are in flight, and
// the 4-byte forms with a few loads per thread much more.
//
// Bound by DRAM.  Measured, us per call, dot_comp + axpy + nrm2 + asum of
// 2^24 + 43 elements, offsets 1 and 3: 94.9 with the 4-byte forms, 80.6 with
// these and 75.3 with their prefetches and second kernel (69 at the copy
// bandwidth); alone in a graph: axpy 38.3 -> 30.5, scal 24.9
// -> 21.3, nrm2 17.3 -> 15.3, dot 25.6 -> 23.6, dot_comp 25.3 -> 24.2.
#include "comp_sum.cuh"

namespace lift {
namespace {

constexpr int kUnThreads = 256, kUnVecs = 4;                 // vectors per thread and tile (reductions)
constexpr int kUnTile = kUnThreads * 4 * kUnVecs;
constexpr int kUnTicket = 3;                                 // workspace counter of this family

// Vectors e + 4 * (32 j + lane), j < J, of an array that starts at the
// aligned address a (J + 1 blocks in lane 0 if the array is shifted).
template <int J>
__device__ __forceinline__ void ld_blocks(const float* a, int lane, bool shifted, Vec<4> (&v)[J + 1]) {
#pragma unroll
  for (int j = 0; j < J; ++j) ld_stream(a + 4 * (kWarp * j + lane), v[j]);
  if (shifted && lane == 0) ld_stream(a + 4 * kWarp * J, v[J]);
}

// Blocks -> vectors that start d = 1 .. 3 elements into them.
template <int J>
__device__ __forceinline__ void shift_blocks(int d, int lane, Vec<4> (&v)[J + 1]) {
#pragma unroll
  for (int j = 0; j < J; ++j) {
    float n[3];
#pragma unroll
    for (int l = 0; l < 3; ++l)
      n[l] = __shfl_sync(0xffffffffu, lane == 0 ? v[j + 1].v[l] : v[j].v[l], (lane + 1) & (kWarp - 1));
    const Vec<4> b = v[j];
    v[j].v[0] = d == 1 ? b.v[1] : d == 2 ? b.v[2] : b.v[3];
    v[j].v[1] = d == 1 ? b.v[2] : d == 2 ? b.v[3] : n[0];
    v[j].v[2] = d == 1 ? b.v[3] : d == 2 ? n[0] : n[1];
    v[j].v[3] = d == 1 ? n[0] : d == 2 ? n[1] : n[2];
  }
}

template <int J>
__device__ __forceinline__ void zero_last(Vec<4> (&v)[J + 1]) {
#pragma unroll
  for (int l = 0; l < 4; ++l) v[J].v[l] = 0.f;
}

// elements first .. first+3 of [lo, hi), zeros outside
__device__ __forceinline__ void ld_between(const float* base, int64_t first, int64_t lo, int64_t hi,
                                           Vec<4>& o) {
#pragma unroll
  for (int l = 0; l < 4; ++l)
    o.v[l] = first + l >= lo && first + l < hi ? __ldg(base + first + l) : 0.f;
}

// Whole tiles: every element, and every block a shifted array's vectors are
// put together from, lies inside the call's elements.
__device__ __forceinline__ bool whole_tile(int64_t tile, int64_t size, int64_t lo, int64_t hi, int d) {
  return tile * size >= lo + d && (tile + 1) * size + (d ? 4 : 0) <= hi;
}

// The folds.  One tile's vectors a (zipped with b) into the thread's sum.
template <int OP>
struct PlainFold {       // the fold of reduce_f32.cuh: lanes from zero, then Neumaier per tile
  static constexpr bool kTwo = OP == LIFT_OP_DOT;
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void tile(const Vec<4>* a, const Vec<4>* b) {
    float ts[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int j = 0; j < kUnVecs; ++j)
#pragma unroll
      for (int l = 0; l < 4; ++l) {
        const float v = a[j].v[l];
        const float t = OP == LIFT_OP_ASUM ? fabsf(v)
                        : OP == LIFT_OP_DOT ? __fmul_rn(v, b[j].v[l])
                        : OP == LIFT_OP_NRM2 ? __fmul_rn(v, v) : v;
        ts[l] = __fadd_rn(ts[l], t);
      }
    neumaier_add(s, c, __fadd_rn(__fadd_rn(__fadd_rn(ts[0], ts[1]), ts[2]), ts[3]));
  }
  __device__ __forceinline__ double cta_value(float* red) {
    return (double)block_tree<kUnThreads>(neumaier_value(s, c), red);
  }
};

template <int OP>
struct CompFold {        // the fold of compensated.cu: TwoSum (and TwoProduct) per element
  static constexpr bool kTwo = OP == LIFT_OP_DOT;
  Comp acc[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
  __device__ __forceinline__ void tile(const Vec<4>* a, const Vec<4>* b) {
#pragma unroll
    for (int j = 0; j < kUnVecs; ++j)
#pragma unroll
      for (int l = 0; l < 4; ++l) {
        if constexpr (OP == LIFT_OP_ASUM) {
          two_sum_add(acc[l], fabsf(a[j].v[l]));
        } else {
          const float p = __fmul_rn(a[j].v[l], b[j].v[l]);
          const float e = __fmaf_rn(a[j].v[l], b[j].v[l], -p);
          two_sum_add(acc[l], p);
          acc[l].c = __fadd_rn(acc[l].c, e);
        }
      }
  }
  __device__ __forceinline__ double cta_value(float*) {
    Comp v = acc[0];
#pragma unroll
    for (int l = 1; l < 4; ++l) v = comp_merge(v, acc[l]);
    return comp_value(block_comp<kUnThreads>(v));
  }
};

// x and y are aligned; the call's elements are x[lo .. hi) and y[lo + d .. hi + d).
template <class F, bool ROOT>
__global__ void __launch_bounds__(kUnThreads)
    unaligned_reduce(const float* __restrict__ x, const float* __restrict__ y, int64_t lo, int64_t hi,
                     int d, double* __restrict__ partials, unsigned* ticket, float* result,
                     double* result64) {
  constexpr int J = kUnVecs;
  __shared__ float red[kWarp];
  const int t = threadIdx.x, lane = t & (kWarp - 1);
  const int64_t G = gridDim.x, T = (hi + kUnTile - 1) / kUnTile;
  if (t < 2 && whole_tile(blockIdx.x + t * G, kUnTile, lo, hi, d)) {    // the CTA's first two tiles
    const int64_t e = (blockIdx.x + t * G) * kUnTile;
    prefetch_l2(x + e, kUnTile * sizeof(float));
    if constexpr (F::kTwo) prefetch_l2(y + e, kUnTile * sizeof(float));
  }
  pdl_wait();      // the previous kernel on the stream has completed
  const int64_t off = (int64_t)(t / kWarp) * (kWarp * 4 * J);     // the warp's part of a tile
  F f;
  Vec<4> cx[J + 1], cy[J + 1];
  zero_last<J>(cx);
  zero_last<J>(cy);
  auto load = [&](int64_t tile, Vec<4> (&a)[J + 1], Vec<4> (&b)[J + 1]) {
    const int64_t e = tile * kUnTile + off;
    if (whole_tile(tile, kUnTile, lo, hi, d)) {
      ld_blocks<J>(x + e, lane, false, a);
      if constexpr (F::kTwo) ld_blocks<J>(y + e, lane, d != 0, b);
    } else if (tile < T) {
#pragma unroll
      for (int j = 0; j < J; ++j) {
        const int64_t first = e + 4 * (kWarp * j + lane);
        ld_between(x, first, lo, hi, a[j]);
        if constexpr (F::kTwo) ld_between(y + d, first, lo, hi, b[j]);
      }
    }
  };
  int64_t tile = blockIdx.x;
  if constexpr (F::kTwo) {
    // two arrays have eight loads per thread in flight as it is, and a second
    // set of registers would halve the CTAs per SM (dot of 2^24 elements, offsets
    // 1 and 3: 25.5 us with it, 23.6 without)
    for (; tile < T; tile += G) {
      load(tile, cx, cy);
      if (d != 0 && whole_tile(tile, kUnTile, lo, hi, d)) shift_blocks<J>(d, lane, cy);
      f.tile(cx, cy);
    }
  } else {
    load(tile, cx, cy);
    while (tile < T) {               // the next tile's loads are in flight during the fold
      Vec<4> nx[J + 1];
      const int64_t nxt = tile + G;
      load(nxt, nx, cy);
      f.tile(cx, cy);
#pragma unroll
      for (int j = 0; j < J; ++j) cx[j] = nx[j];
      tile = nxt;
    }
  }
  pdl_trigger();   // streaming done: the next call's first kernel may be scheduled
  finish64<kUnThreads, ROOT>(f.cta_value(red), partials, ticket, result, result64);
}

constexpr int kMapVecs = 2, kMapTile = kUnThreads * 4 * kMapVecs;

// y[i] <- alpha * x[i] (scal) or alpha * x[i] + y[i] (axpy), one CTA per
// tile; y is aligned, the call's elements are y[lo .. hi) and x[lo + d ..).
template <bool AXPY>
__global__ void __launch_bounds__(kUnThreads)
    unaligned_map(const float* x, float* y, int64_t lo, int64_t hi, int d, float alpha) {
  constexpr int J = kMapVecs;
  const int lane = threadIdx.x & (kWarp - 1);
  const int64_t tile = gridDim.x - 1 - blockIdx.x;          // last tile first
  if (threadIdx.x < (AXPY ? 2 : 1) && blockIdx.x < kPrefetchCtas && whole_tile(tile, kMapTile, lo, hi, d))
    prefetch_l2((threadIdx.x == 0 ? x : y) + tile * kMapTile, kMapTile * sizeof(float));
  pdl_trigger();   // the next call's first kernel may be scheduled (it waits for this one)
  pdl_wait();      // the previous kernel on the stream has completed
  const int64_t e = tile * kMapTile + (int64_t)(threadIdx.x / kWarp) * (kWarp * 4 * J);
  const bool whole = whole_tile(tile, kMapTile, lo, hi, d);
  Vec<4> a[J + 1], b[J];
  zero_last<J>(a);
  if (whole) {
    ld_blocks<J>(x + e, lane, d != 0, a);
    if constexpr (AXPY) {
#pragma unroll
      for (int j = 0; j < J; ++j) ld_stream(y + e + 4 * (kWarp * j + lane), b[j]);
    }
    if (d != 0) shift_blocks<J>(d, lane, a);
  } else {
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int64_t first = e + 4 * (kWarp * j + lane);
      ld_between(x + d, first, lo, hi, a[j]);
      if constexpr (AXPY) ld_between(y, first, lo, hi, b[j]);
    }
  }
#pragma unroll
  for (int j = 0; j < J; ++j) {
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const float z = __fmul_rn(alpha, a[j].v[l]);
      if constexpr (AXPY) a[j].v[l] = __fadd_rn(z, b[j].v[l]);
      else a[j].v[l] = z;
    }
    const int64_t first = e + 4 * (kWarp * j + lane);
    if (whole) {
      st_stream(y + first, a[j]);
    } else {
#pragma unroll
      for (int l = 0; l < 4; ++l)
        if (first + l >= lo && first + l < hi) y[first + l] = a[j].v[l];
    }
  }
}

// elements past the 16-byte boundary below p
int phase(const void* p) { return (int)(reinterpret_cast<uintptr_t>(p) / 4 % 4); }
// The address `back` elements before p: the aligned start of the block p
// lies in, so never read below p itself.
const float* before(const void* p, int back) {
  return reinterpret_cast<const float*>(reinterpret_cast<uintptr_t>(p) - 4 * (uintptr_t)back);
}

template <class F, bool ROOT>
struct UnalignedReduce {
  static const void* kernel() { return reinterpret_cast<const void*>(&unaligned_reduce<F, ROOT>); }
  static lift_status launch(const Variant& v, const Args& a, cudaStream_t s) {
    const int m = phase(a.x);
    int64_t lo = m, hi = a.n + m;
    int d = F::kTwo ? (phase(a.y) - m + 4) % 4 : 0;
    const float* x = before(a.x, m);
    const float* y = F::kTwo ? before(a.y, m + d) : nullptr;
    const int64_t T = hi > 0 ? (hi + kUnTile - 1) / kUnTile : 1;
    int64_t g = persistent_grid(kernel(), kUnThreads, 0, 1);
    if (g <= 0) return set_error(LIFT_ERR_CUDA, std::string("no resident CTA for ") + v.info.name);
    if (g > a.ws->capacity64) return set_error(LIFT_ERR_UNSUPPORTED, "grid exceeds workspace");
    const int64_t per = (T + g - 1) / g;
    g = (T + per - 1) / per;
    double* partials = a.ws->partials64;
    const bool two = (F::kTwo ? 8 : 4) * a.n >= kTwoPassBytes;
    unsigned* ticket = two ? nullptr : a.ws->tickets + kUnTicket;
    float* result = a.result;
    double* result64 = a.result64;
    void* args[] = {&x, &y, &lo, &hi, &d, &partials, &ticket, &result, &result64};
    const lift_status rc =
        launch_config(kernel(), dim3((unsigned)g), dim3(kUnThreads), 0, 1, s, args, true);
    return rc != LIFT_OK || !two ? rc
                                 : Combine64<kUnThreads, ROOT>::launch(partials, g, result, result64, s);
  }
};

template <bool AXPY>
struct UnalignedMap {
  static const void* kernel() { return reinterpret_cast<const void*>(&unaligned_map<AXPY>); }
  static lift_status launch(const Variant&, const Args& a, cudaStream_t s) {
    const int m = phase(a.out);
    int64_t lo = m, hi = a.n + m;
    int d = (phase(a.x) - m + 4) % 4;
    const float* x = before(a.x, m + d);
    float* y = const_cast<float*>(before(a.out, m));
    float alpha = a.alpha;
    const int64_t T = (hi + kMapTile - 1) / kMapTile;
    if (T > INT32_MAX) return set_error(LIFT_ERR_UNSUPPORTED, "more tiles than CTAs in a grid");
    void* args[] = {&x, &y, &lo, &hi, &d, &alpha};
    return launch_config(kernel(), dim3((unsigned)T), dim3(kUnThreads), 0, 1, s, args, true);
  }
};

template <class K>
Variant unaligned_variant(int op, const char* name) {
  Variant v{};
  v.info.op = op;
  v.info.id = -1;          // not a registered variant: the default entry points' own
  v.info.vw = 4;
  v.info.threads = kUnThreads;
  snprintf(v.info.name, sizeof(v.info.name), "%s_unaligned", name);
  v.launch = &K::launch;
  v.align_bytes = 4;
  v.fallback = -1;
  return v;
}

}  // namespace

// The form of op for unaligned pointers, or nullptr.
const Variant* unaligned_form(int op) {
  static const Variant asum = unaligned_variant<UnalignedReduce<PlainFold<LIFT_OP_ASUM>, false>>(LIFT_OP_ASUM, "asum");
  static const Variant dot = unaligned_variant<UnalignedReduce<PlainFold<LIFT_OP_DOT>, false>>(LIFT_OP_DOT, "dot");
  static const Variant nrm2 = unaligned_variant<UnalignedReduce<PlainFold<LIFT_OP_NRM2>, true>>(LIFT_OP_NRM2, "nrm2");
  static const Variant sum = unaligned_variant<UnalignedReduce<PlainFold<LIFT_OP_SUM>, false>>(LIFT_OP_SUM, "sum");
  static const Variant asum_comp =
      unaligned_variant<UnalignedReduce<CompFold<LIFT_OP_ASUM>, false>>(LIFT_OP_ASUM_COMP, "asum_comp");
  static const Variant dot_comp =
      unaligned_variant<UnalignedReduce<CompFold<LIFT_OP_DOT>, false>>(LIFT_OP_DOT_COMP, "dot_comp");
  static const Variant scal = unaligned_variant<UnalignedMap<false>>(LIFT_OP_SCAL, "scal");
  static const Variant axpy = unaligned_variant<UnalignedMap<true>>(LIFT_OP_AXPY, "axpy");
  switch (op) {
    case LIFT_OP_ASUM: return &asum;
    case LIFT_OP_DOT: return &dot;
    case LIFT_OP_NRM2: return &nrm2;
    case LIFT_OP_SUM: return &sum;
    case LIFT_OP_ASUM_COMP: return &asum_comp;
    case LIFT_OP_DOT_COMP: return &dot_comp;
    case LIFT_OP_SCAL: return &scal;
    case LIFT_OP_AXPY: return &axpy;
  }
  return nullptr;
}

}  // namespace lift
