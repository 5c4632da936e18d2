// gemv kernels that fold R rows at a time (arXiv 1502.02389, Fig. 5 gemv;
// the same per-row expressions as the warp-per-row kernel of scal_gemv.cu
// and the split-row kernel of gemv_split.cu).
//
// A row's sum is spread over more threads than the 32 lanes of a warp, so the
// trees over them keep the compensations: the error of a row is no larger
// than the warp-per-row kernel's.
//
// Both older forms load one vector of x for every vector of A, and give a
// row to one warp or CTA at a time.  Here a warp (WARPS form) or a CTA
// (split form) folds R consecutive rows together: a vector of x is loaded
// once for R rows, and U vectors of each of the R rows are in flight before
// the first is folded.  That matters where a row cannot be read with
// 128-bit loads -- lda or N not a multiple of 4, or A or x off a 16-byte
// boundary -- and every request moves only 4 bytes per lane: a 4-byte
// request that straddles a 128-byte line takes two L1 passes, and R rows
// per load of x keep those passes on A.
//
// What bounds it: DRAM for large matrices; for a matrix with few rows, the
// number of CTAs in flight (hence the split over segments).  Measured (us,
// graph of back-to-back calls on cold data, against the warp-per-row 4-byte
// kernel that such calls ran before): 32 x 1000003: 23.5 (6841; 18.8 at the
// copy bandwidth); 4097 x 3001: 11.6 (24.1); 8191 x 8191: 43.8 (64.2);
// 65536 x 1023: 47.5 (59.6).  Rows of 16-byte granules: 32 x 1000000: 22.1
// (432 for the bulk-copy ring, 23.5 for the one-row split form).
//
// The last, partial step of a row is read with guarded loads of all U
// vectors at once (zeros past the end, which change nothing), so a ragged
// row costs one more step instead of up to U dependent ones.
#include "comp_sum.cuh"

namespace lift {

// second pass shared with gemv-T (gemv_t.cu): out_j from per[j*per .. +per)
lift_status launch_rows_combine(int64_t n, int64_t per, float alpha, float beta,
                                const float* partials, float* y, cudaStream_t s);
// y <- fl(0 + fl(beta * y)) (0 when beta == 0): the N == 0 case (gemv_t.cu)
lift_status gemv_t_empty_rows(int64_t N, float beta, float* y, cudaStream_t s);

namespace {

template <int VW>
__device__ __forceinline__ void ld_x_rows(const float* p, Vec<VW>& o) {
  if constexpr (VW == 1) {
    o.v[0] = __ldg(p);
  } else {
#pragma unroll
    for (int q = 0; q < VW / 4; ++q) {
      const float4 t = __ldg(reinterpret_cast<const float4*>(p) + q);
      o.v[4 * q] = t.x;
      o.v[4 * q + 1] = t.y;
      o.v[4 * q + 2] = t.z;
      o.v[4 * q + 3] = t.w;
    }
  }
}

// Fold columns c, c + STEP, ... below c_end of R rows (row pointers a) into
// one GroupedDot per row: the vectors of one lane or thread, in order.
template <int VW, int R, int U, int STEP>
__device__ __forceinline__ void fold_r_rows(const float* const (&a)[R], const float* x, int64_t c,
                                            int64_t c_end, GroupedDot<VW> (&acc)[R]) {
  static_assert(kGemvGroup % U == 0, "an unrolled step stays inside one group");
  int k = 0;                           // vectors folded (mod the group)
  for (; c + (int64_t)(U - 1) * STEP + VW <= c_end; c += (int64_t)U * STEP) {
    Vec<VW> v[R][U], b[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
      for (int r = 0; r < R; ++r) ld_stream(a[r] + c + u * STEP, v[r][u]);
      ld_x_rows<VW>(x + c + u * STEP, b[u]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r].add(v[r][u], b[u]);
    k = (k + U) & (kGemvGroup - 1);
    if (k == 0) {
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r].flush();
    }
  }
  if (c < c_end) {
    Vec<VW> v[R][U], b[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t e = c + u * STEP;
      if (e + VW <= c_end) {
#pragma unroll
        for (int r = 0; r < R; ++r) ld_stream(a[r] + e, v[r][u]);
        ld_x_rows<VW>(x + e, b[u]);
      } else {                         // the ragged last vector, or none (zeros)
#pragma unroll
        for (int r = 0; r < R; ++r) ld_guarded<VW>(a[r], e, c_end, v[r][u]);
        ld_guarded<VW>(x, e, c_end, b[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r].add(v[r][u], b[u]);
  }
}

template <int R>
__device__ __forceinline__ void row_pointers(const float* A, int64_t lda, int64_t r0, int64_t M,
                                             const float* (&a)[R]) {
#pragma unroll
  for (int r = 0; r < R; ++r) a[r] = A + (r0 + r < M ? r0 + r : M - 1) * lda;   // past M: unused
}

// R rows split into S segments of L columns: one CTA per (row group,
// segment), threads of the CTA along the columns.
template <int THREADS, int VW, int R, int U>
__global__ void __launch_bounds__(THREADS)
    gemv_split_rows(int64_t M, int64_t N, float alpha, const float* __restrict__ A, int64_t lda,
                    const float* __restrict__ x, float beta, float* __restrict__ y, int64_t L,
                    int64_t S, float* __restrict__ partials) {
  constexpr int W = THREADS / kWarp;
  static_assert(R <= W, "one warp per row in the last stage of the tree");
  __shared__ Comp red[R][kWarp];
  const int lane = threadIdx.x & (kWarp - 1), warp = threadIdx.x / kWarp;
  const int64_t r0 = blockIdx.x / S * R, seg = blockIdx.x % S;
  const int64_t c_end = (seg + 1) * L < N ? (seg + 1) * L : N;
  if (threadIdx.x < R && blockIdx.x < kPrefetchCtas && r0 + threadIdx.x < M) {   // two steps of every row
    const int64_t c = seg * L, len = c_end - c < 2 * U * THREADS * VW ? c_end - c : 2 * U * THREADS * VW;
    prefetch_l2(A + (r0 + threadIdx.x) * lda + c, 4 * len);
  }
  pdl_wait();      // the previous kernel on the stream has completed
  const float* a[R];
  row_pointers<R>(A, lda, r0, M, a);
  GroupedDot<VW> acc[R];
#pragma unroll
  for (int r = 0; r < R; ++r) acc[r].init();
  fold_r_rows<VW, R, U, THREADS * VW>(a, x, seg * L + (int64_t)threadIdx.x * VW, c_end, acc);
  pdl_trigger();   // streaming done: the combine kernel (or the next call's) may be scheduled
  Comp v[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    acc[r].close();
    v[r] = {acc[r].s, acc[r].c};
  }
  const Comp mine = warp_comp_rows<R>(v);
  if (lane % (kWarp / R) == 0) red[lane / (kWarp / R)][warp] = mine;
  __syncthreads();
  if (warp >= R || r0 + warp >= M) return;
  const float d = comp_value32(warp_comp_first<W>(red[warp][lane % W]));
  if (lane != 0) return;
  if (S > 1) {
    partials[(r0 + warp) * S + seg] = d;
  } else {
    const float z = __fmul_rn(alpha, d);
    y[r0 + warp] = beta == 0.f ? z : __fadd_rn(z, __fmul_rn(beta, y[r0 + warp]));
  }
}

// R rows per warp, the 32 lanes along the columns (no split of a row).
template <int WARPS, int VW, int R, int U>
__global__ void __launch_bounds__(WARPS * kWarp)
    gemv_warp_rows(int64_t M, int64_t N, float alpha, const float* __restrict__ A, int64_t lda,
                   const float* __restrict__ x, float beta, float* __restrict__ y) {
  const int lane = threadIdx.x & (kWarp - 1);
  const int64_t total = (int64_t)gridDim.x * WARPS * R;
  const int64_t first = ((int64_t)blockIdx.x * WARPS + threadIdx.x / kWarp) * R + lane;
  if (lane < R && blockIdx.x < kPrefetchCtas && first < M)
    prefetch_l2(A + first * lda, 4 * (N < 2048 ? N : 2048));
  pdl_trigger();   // the next call's first kernel may be scheduled (it waits for this one)
  pdl_wait();      // the previous kernel on the stream has completed
  for (int64_t r0 = ((int64_t)blockIdx.x * WARPS + threadIdx.x / kWarp) * R; r0 < M; r0 += total) {
    const float* a[R];
    row_pointers<R>(A, lda, r0, M, a);
    GroupedDot<VW> acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r].init();
    fold_r_rows<VW, R, U, kWarp * VW>(a, x, lane * VW, N, acc);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float d = warp_tree(acc[r].value());
      if (lane == 0 && r0 + r < M) {
        const float z = __fmul_rn(alpha, d);
        y[r0 + r] = beta == 0.f ? z : __fadd_rn(z, __fmul_rn(beta, y[r0 + r]));
      }
    }
  }
}

template <int THREADS, int VW, int R, int U>
struct GemvSplitRows {
  static constexpr int64_t kStep = (int64_t)THREADS * VW;
  static const void* kernel() {
    return reinterpret_cast<const void*>(&gemv_split_rows<THREADS, VW, R, U>);
  }
  // Segments per row S so that the row groups times S fill one wave of
  // resident CTAs and no more (a second, nearly empty wave would cost a
  // whole segment's time); L a multiple of THREADS * VW.
  static void shape(const Args& a, int64_t& L, int64_t& S) {
    const int64_t g = persistent_grid(kernel(), THREADS, 0, 1);
    const int64_t groups = a.M > 0 ? (a.M + R - 1) / R : 1;
    int64_t want = g / groups;
    DeviceState* st = current_state();
    const int64_t cap = st && a.M > 0 ? st->ws.capacity / a.M : 1;
    if (want > cap) want = cap;
    if (want < 1) want = 1;
    const int64_t per = (a.N + want - 1) / want;
    L = (per + kStep - 1) / kStep * kStep;
    if (L < kStep) L = kStep;
    S = (a.N + L - 1) / L;
    if (S < 1) S = 1;
  }
  static int64_t grid(const Variant&, const Args& a) {
    int64_t L, S;
    shape(a, L, S);
    return (a.M + R - 1) / R * S;
  }
  static lift_status launch(const Variant& v, const Args& a, cudaStream_t s) {
    if (a.M == 0) return LIFT_OK;
    if (a.N == 0) return gemv_t_empty_rows(a.M, a.beta, a.out, s);
    int64_t L, S;
    shape(a, L, S);
    const int64_t g = (a.M + R - 1) / R * S;
    if (g > 0x7fffffffLL) return set_error(LIFT_ERR_UNSUPPORTED, "gemv split: grid too large");
    if (S > 1 && a.M * S > a.ws->capacity)
      return set_error(LIFT_ERR_UNSUPPORTED, "gemv split: partials exceed the workspace");
    int64_t M = a.M, N = a.N, lda = a.lda;
    float alpha = a.alpha, beta = a.beta;
    const float* A = a.A;
    const float* x = static_cast<const float*>(a.x);
    float* y = a.out;
    float* partials = partials_for(a, M * S);
    void* args[] = {&M, &N, &alpha, &A, &lda, &x, &beta, &y, &L, &S, &partials};
    const lift_status r =
        launch_config(kernel(), dim3((unsigned)g), dim3(THREADS), 0, 1, s, args, true);
    if (r != LIFT_OK || S == 1) return r;
    return launch_rows_combine(M, S, alpha, beta, partials, y, s);
  }
};

template <int WARPS, int VW, int R, int U>
struct GemvWarpRows {
  static const void* kernel() {
    return reinterpret_cast<const void*>(&gemv_warp_rows<WARPS, VW, R, U>);
  }
  // one CTA per WARPS * R rows (capped at 2^31 - 1 CTAs; the row loop still
  // covers every row), dealt to the SMs by the hardware
  static int64_t grid(const Variant&, const Args& a) {
    const int64_t need = (a.M + WARPS * R - 1) / (WARPS * R);
    return need < 1 ? 1 : need < INT32_MAX ? need : INT32_MAX;
  }
  static lift_status launch(const Variant& v, const Args& a, cudaStream_t s) {
    if (a.M == 0) return LIFT_OK;
    if (a.N == 0) return gemv_t_empty_rows(a.M, a.beta, a.out, s);
    int64_t M = a.M, N = a.N, lda = a.lda;
    float alpha = a.alpha, beta = a.beta;
    const float* A = a.A;
    const float* x = static_cast<const float*>(a.x);
    float* y = a.out;
    void* args[] = {&M, &N, &alpha, &A, &lda, &x, &beta, &y};
    return launch_config(kernel(), dim3((unsigned)grid(v, a)), dim3(WARPS * kWarp), 0, 1, s, args,
                         true);
  }
};

template <class K>
Variant rows_variant(const char* name, int threads, int vw) {
  Variant v{};
  v.info.op = LIFT_OP_GEMV;
  v.info.vw = vw;
  v.info.threads = threads;
  v.info.stride = 1;
  v.info.cluster = 1;
  snprintf(v.info.name, sizeof(v.info.name), "gemv_%s", name);
  v.launch = &K::launch;
  v.grid = &K::grid;
  v.align_bytes = vw * 4;
  v.fallback = 0;
  return v;
}

template <int THREADS, int VW, int R, int U>
Variant split_rows_variant(const char* name) {
  Variant v = rows_variant<GemvSplitRows<THREADS, VW, R, U>>(name, THREADS, VW);
  v.info.tile = THREADS * VW;
  v.info.passes = 2;
  v.info.rows = 1;
  v.info.lanes = THREADS;
  v.info.final_threads = kWarp;
  return v;
}

template <int WARPS, int VW, int R, int U>
Variant warp_rows_variant(const char* name) {
  Variant v = rows_variant<GemvWarpRows<WARPS, VW, R, U>>(name, WARPS * kWarp, VW);
  v.info.passes = 1;
  v.info.rows = WARPS;
  v.info.lanes = kWarp;
  v.info.grid = 1;
  return v;
}

}  // namespace

// (threads, vector width, rows, vectors of a row in flight)
#define LIFT_GEMV_SPLIT_ROWS_VARIANTS(X)   \
  X(256, 1, 4, 8, "split_t256_v1_r4_u8")   \
  X(128, 1, 4, 8, "split_t128_v1_r4_u8")   \
  X(256, 1, 2, 8, "split_t256_v1_r2_u8")   \
  X(128, 4, 2, 4, "split_t128_v4_r2_u4")

void gemv_split_rows_shape(const char* name, const Args& a, int64_t* L, int64_t* S) {
  int64_t l = 0, s = 0;
#define X(T, V, R, U, NAME) \
  if (std::string("gemv_") + NAME == name) GemvSplitRows<T, V, R, U>::shape(a, l, s);
  LIFT_GEMV_SPLIT_ROWS_VARIANTS(X)
#undef X
  *L = l;
  *S = s;
}

// registered after every other gemv family (earlier ids are stable)
void register_gemv_rows(std::vector<Variant>& L) {
  const size_t first = L.size();
#define X(T, V, R, U, NAME) L.push_back(split_rows_variant<T, V, R, U>(NAME));
  LIFT_GEMV_SPLIT_ROWS_VARIANTS(X)
#undef X
  L.push_back(warp_rows_variant<4, 1, 2, 8>("w4_v1_r2_u8"));
  for (size_t i = first; i < L.size(); ++i) L[i].info.id = static_cast<int>(i);
}

}  // namespace lift
