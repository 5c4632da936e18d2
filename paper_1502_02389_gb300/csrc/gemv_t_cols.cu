// gemv-T (y <- alpha * A^T x + beta * y) with several strided columns per
// thread: the two-pass expression of gemv_t.cu, loaded differently.
//
// Per column, the row block's rows are folded in groups (kFineBlock below) in
// row order from zero and the group sums added with Neumaier's compensated
// step; the RB block values are added as the 32 lanes of a warp add them (lane
// l takes blocks l, l+32, ..., then a halving tree of (sum, compensation)
// pairs) -- the program of gemv_t_kernel's and gemv_t_staged's two-pass forms
// with shorter groups.  A thread here owns Q column vectors THREADS * VW apart,
// so that
//  * with VW == 1 a matrix whose rows are not whole 16-byte granules is
//    still read with coalesced 128-byte requests, Q * U of them in flight
//    per thread, and one load of x_i serves Q columns;
//  * a row block that covers every row (RB == 1: a matrix with more columns
//    than one wave of CTAs) has no second pass: the epilogue is applied in
//    registers, where the other forms write one partial per column and
//    combine it with a warp per column;
//  * with RB <= 32 the partials are row-major and the second pass gives a
//    thread to a column (the halving tree in registers, coalesced loads)
//    instead of a warp.
//
// Bound by DRAM for large matrices.  Measured (us, graph of back-to-back
// calls on cold data, against what such calls ran before): 32 x 1000003:
// 22.5 (37.9; 18.8 at the copy bandwidth); 4097 x 3001: 11.5 (31.5);
// 8191 x 8191: 44.8 (59.0); 65536 x 1023: 47.8 (110); 20000 x 333: 9.5
// (113); 32 x 1000000: 24.2 (144); 1000 x 777: 5.4 (52).  Two columns per
// thread with every CTA that fits lead four columns on 4 CTAs per SM (8191 x
// 8191: 54.1) and 64- or 32-thread CTAs (65.5, 59.9).
#include "comp_sum.cuh"

namespace lift {

lift_status launch_rows_combine(int64_t n, int64_t per, float alpha, float beta,
                                const float* partials, float* y, cudaStream_t s);

namespace {

// Rows that a thread folds plainly before it adds their sum to a column's
// compensated sum: 16, where the forms that such calls ran before have 32 but
// fewer or shorter row blocks (400 x 86988: relative l2 error 1.16e-7 with 32,
// 1.14e-7 for one staged block of 400 rows).  In the 4-byte forms pairs where
// row blocks are short: as one group, the rows of a block of 20 gave 9534 x
// 120 9.2e-8, the one-pass form with its blocks of 8 rows 7.1e-8; with pairs
// it is 5.8e-8.  In long blocks pairs would cost 4 to 9 % (4097 x 3001: 11.5
// -> 12.7 us).  40: a block is at most 2.4 times the one-pass form's (512 row
// blocks against 1216 CTAs), whose error is that of groups of 16 from 20 rows
// on; blocks of 4 rows, the least, are the one-pass form's own.
constexpr int64_t kFineBlock = 40;
constexpr int kFineGroup = 2, kGroup = 16;
constexpr int kColsTree = 32;           // row blocks the thread-per-column combine takes
constexpr int64_t kColsMaxBlocks = 512; // row blocks of a call
constexpr int kColsCombineThreads = 64;

// U rows of the thread's Q column vectors folded into gs; the groups of G rows
// that end before the last of them are closed.
template <int VW, int Q, int U, int G>
__device__ __forceinline__ void fold_rows_of(const Vec<VW> (&a)[U][Q], const float (&xv)[U],
                                             float (&gs)[Q][VW], float (&acc)[Q][VW],
                                             float (&cmp)[Q][VW]) {
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
      for (int l = 0; l < VW; ++l) {
        gs[q][l] = __fadd_rn(gs[q][l], __fmul_rn(a[u][q].v[l], xv[u]));
        if ((u + 1) % G == 0 && u + 1 < U) {
          neumaier_add(acc[q][l], cmp[q][l], gs[q][l]);
          gs[q][l] = 0.f;
        }
      }
}

// U rows i .. i+U-1 of the thread's Q column vectors.  FULL: every column of
// the CTA and every row exists; otherwise guarded (zeros, which change no sum).
template <int VW, int Q, int U, int G, bool FULL>
__device__ __forceinline__ void fold_step(const float* __restrict__ A, int64_t lda, int64_t N,
                                          const float* __restrict__ x, int64_t c0, int cstep,
                                          int64_t i, int64_t iend, float (&gs)[Q][VW],
                                          float (&acc)[Q][VW], float (&cmp)[Q][VW]) {
  Vec<VW> a[U][Q];
  float xv[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const float* row = A + (i + u) * lda;
    const bool have = FULL || i + u < iend;
    xv[u] = have ? __ldg(x + i + u) : 0.f;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int64_t c = c0 + (int64_t)q * cstep;
      if (FULL || (have && c + VW <= N)) ld_stream(row + c, a[u][q]);
      else ld_guarded<VW>(row, c, have ? N : 0, a[u][q]);
    }
  }
  fold_rows_of<VW, Q, U, G>(a, xv, gs, acc, cmp);
}

// The same where columns end inside the CTA and every row exists, 4-byte forms:
// a column past N is the last one again (its sum is never stored), so that the
// loads need no guards.
template <int Q, int U, int G>
__device__ __forceinline__ void fold_step_clamped(const float* __restrict__ A, int64_t lda, int64_t N,
                                                  const float* __restrict__ x, int64_t c0, int cstep,
                                                  int64_t i, float (&gs)[Q][1], float (&acc)[Q][1],
                                                  float (&cmp)[Q][1]) {
  Vec<1> a[U][Q];
  float xv[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const float* row = A + (i + u) * lda;
    xv[u] = __ldg(x + i + u);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int64_t c = c0 + (int64_t)q * cstep;
      ld_stream(row + (c < N ? c : N - 1), a[u][q]);
    }
  }
  fold_rows_of<1, Q, U, G>(a, xv, gs, acc, cmp);
}

// How a CTA whose columns end inside it (N not a multiple of CB) reads them:
// with guards, or clamped -- beside the whole-CTA loop, or instead of it.  The
// whole-CTA loop overlaps most loads where it stands alone (8191 x 8191: 45.2
// us, 48.8 with a second loop beside it), so the clamped loop replaces it where
// one of at most two column blocks ends early (80000 x 65: 17.0 us, guarded
// 19.9; 65536 x 255: 16.6, 18.5) and stands beside it in the short blocks'
// kernel (20000 x 333: 9.9, guarded 13.2, instead of it 10.2).
enum Edge { kGuard, kClamp, kClampAll };

// AHEAD: two steps of rows are asked for before the previous call has ended,
// where there are row blocks (4097 x 3001: 13.1 -> 11.9 us); a matrix with more
// columns than a wave of CTAs gains nothing, and the kernel without it has one
// CTA per SM less (32 x 1000003: 22.0 us, 22.6 with eight).
template <int THREADS, int VW, int Q, int U, bool AHEAD, int G, int EDGE>
__global__ void __launch_bounds__(THREADS)
    gemv_t_cols(int64_t M, int64_t N, float alpha, const float* __restrict__ A, int64_t lda,
                const float* __restrict__ x, float beta, float* __restrict__ y, int64_t B,
                float* __restrict__ partials) {
  constexpr int CB = THREADS * VW * Q, kStep = THREADS * VW;
  constexpr int kRows = G < U ? U : G;      // rows between two checks
  static_assert(kRows % U == 0 && (U % G == 0 || G % U == 0), "steps and groups nest");
  const int64_t cb = blockIdx.x, rb = blockIdx.y, RB = gridDim.y;
  const int64_t c0 = cb * CB + (int64_t)threadIdx.x * VW;
  const int64_t r0 = rb * B, r1 = r0 + B < M ? r0 + B : M;
  const bool full = (cb + 1) * CB <= N;
  if constexpr (AHEAD) {
    if (threadIdx.x < 2 * U && r0 + threadIdx.x < r1)
      prefetch_l2(A + (r0 + threadIdx.x) * lda + cb * CB, 4 * (full ? CB : N - cb * CB));
  }
  pdl_wait();      // the previous kernel on the stream has completed
  float acc[Q][VW], cmp[Q][VW];
#pragma unroll
  for (int q = 0; q < Q; ++q)
#pragma unroll
    for (int l = 0; l < VW; ++l) acc[q][l] = cmp[q][l] = 0.f;
  for (int64_t i = r0; i < r1;) {
    const int64_t ge = i + kRows < r1 ? i + kRows : r1;
    float gs[Q][VW];
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
      for (int l = 0; l < VW; ++l) gs[q][l] = 0.f;
    if (full && EDGE != kClampAll) {
      for (; i + U <= ge; i += U)
        fold_step<VW, Q, U, G, true>(A, lda, N, x, c0, kStep, i, ge, gs, acc, cmp);
    } else if constexpr (EDGE != kGuard) {
      for (; i + U <= ge; i += U)
        fold_step_clamped<Q, U, G>(A, lda, N, x, c0, kStep, i, gs, acc, cmp);
    }
    for (; i < ge; i += U)
      fold_step<VW, Q, U, G, false>(A, lda, N, x, c0, kStep, i, ge, gs, acc, cmp);
    i = ge;
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
      for (int l = 0; l < VW; ++l) neumaier_add(acc[q][l], cmp[q][l], gs[q][l]);
  }
  pdl_trigger();   // streaming done: the combine kernel (or the next call's) may be scheduled
#pragma unroll
  for (int q = 0; q < Q; ++q)
#pragma unroll
    for (int l = 0; l < VW; ++l) {
      const int64_t c = c0 + (int64_t)q * kStep + l;
      if (c >= N) continue;
      const float p = neumaier_value(acc[q][l], cmp[q][l]);
      if (RB == 1) {
        const float z = __fmul_rn(alpha, p);
        y[c] = beta == 0.f ? z : __fadd_rn(z, __fmul_rn(beta, y[c]));
      } else {
        partials[RB <= kColsTree ? rb * N + c : c * RB + rb] = p;
      }
    }
}

// Second pass for RB <= T <= 32 row-major partials: thread per column, the
// halving tree of a warp whose lane l holds block l (zeros past RB; the levels
// that would only add zeros left out: 100001 columns of two blocks are 0.7 us
// faster so).
template <int T>
__global__ void __launch_bounds__(kColsCombineThreads)
    gemv_t_combine_cols(int64_t N, int RB, float alpha, float beta,
                        const float* __restrict__ partials, float* __restrict__ y) {
  pdl_trigger();   // the next call's first kernel may be scheduled (it waits for this one)
  pdl_wait();      // the first pass has finished
  const int64_t j = (int64_t)blockIdx.x * kColsCombineThreads + threadIdx.x;
  if (j >= N) return;
  Comp v[T];
#pragma unroll
  for (int b = 0; b < T; ++b) v[b] = {b < RB ? __ldcg(partials + b * N + j) : 0.f, 0.f};
#pragma unroll
  for (int o = T / 2; o > 0; o >>= 1)
#pragma unroll
    for (int b = 0; b < o; ++b) v[b] = comp_merge(v[b], v[b + o]);
  const float z = __fmul_rn(alpha, comp_value32(v[0]));
  y[j] = beta == 0.f ? z : __fadd_rn(z, __fmul_rn(beta, y[j]));
}

lift_status launch_combine_cols(int64_t N, int RB, float alpha, float beta, const float* partials,
                                float* y, cudaStream_t s) {
  const unsigned g = (unsigned)((N + kColsCombineThreads - 1) / kColsCombineThreads);
  const void* k = RB <= 2   ? reinterpret_cast<const void*>(&gemv_t_combine_cols<2>)
                  : RB <= 8 ? reinterpret_cast<const void*>(&gemv_t_combine_cols<8>)
                            : reinterpret_cast<const void*>(&gemv_t_combine_cols<kColsTree>);
  void* args[] = {&N, &RB, &alpha, &beta, &partials, &y};
  return launch_config(k, dim3(g), dim3(kColsCombineThreads), 0, 1, s, args, true);
}

template <int THREADS, int VW, int Q, int U, int PER_SM, int G = kGroup,
          int EDGE = kGuard>
struct GemvTCols {
  static constexpr int CB = THREADS * VW * Q;
  static const void* kernel() {
    return reinterpret_cast<const void*>(&gemv_t_cols<THREADS, VW, Q, U, false, G, EDGE>);
  }
  // the form of long blocks and guarded edges: the shape is taken from its occupancy
  using Base = GemvTCols<THREADS, VW, Q, U, PER_SM>;
  // (column blocks, row blocks, rows per block): at most one wave of PER_SM
  // CTAs per SM, within the partials workspace and kColsMaxBlocks row blocks
  static void shape(const Args& a, int64_t& ncb, int64_t& RB, int64_t& B) {
    ncb = (a.N + CB - 1) / CB;
    int64_t g = persistent_grid(Base::kernel(), THREADS, 0, 1);
    DeviceState* st = current_state();
    if (st && g > (int64_t)PER_SM * st->sm_count) g = (int64_t)PER_SM * st->sm_count;
    int64_t want = g > ncb ? g / ncb : 1;
    const int64_t cap = st ? st->ws.capacity / (a.N > 0 ? a.N : 1) : 1;
    if (want > cap) want = cap;
    if (want > kColsMaxBlocks) want = kColsMaxBlocks;
    if (want > a.M) want = a.M;
    if (want < 1) want = 1;
    B = (a.M + want - 1) / want;
    B = (B + 3) / 4 * 4;
    RB = (a.M + B - 1) / B;
  }
  static int64_t grid(const Variant&, const Args& a) {
    int64_t ncb, RB, B;
    shape(a, ncb, RB, B);
    return ncb * RB;
  }
  static lift_status launch(const Variant& v, const Args& a, cudaStream_t s) {
    if (a.N == 0) return LIFT_OK;
    if (a.M == 0) return set_error(LIFT_ERR_UNSUPPORTED, "gemv_t with M == 0 goes through gemv_t_scale");
    int64_t ncb, RB, B;
    shape(a, ncb, RB, B);
    if constexpr (VW == 1 && G == kGroup && EDGE == kGuard) {
      if (B > 4 && B <= kFineBlock)
        return GemvTCols<THREADS, VW, Q, U, PER_SM, kFineGroup, kClamp>::launch(v, a, s);
      if (ncb <= 2 && a.N % CB != 0)
        return GemvTCols<THREADS, VW, Q, U, PER_SM, kGroup, kClampAll>::launch(v, a, s);
    }
    if (RB * a.N > a.ws->capacity)     // the bound of the other forms, also where RB == 1
      return set_error(LIFT_ERR_UNSUPPORTED, "gemv_t: N exceeds the partials workspace");
    if (ncb > 0x7fffffffLL) return set_error(LIFT_ERR_UNSUPPORTED, "gemv_t: grid too large");
    int64_t M = a.M, N = a.N, lda = a.lda;
    float alpha = a.alpha, beta = a.beta;
    const float* A = a.A;
    const float* x = static_cast<const float*>(a.x);
    float* y = a.out;
    float* partials = a.ws->partials;
    void* args[] = {&M, &N, &alpha, &A, &lda, &x, &beta, &y, &B, &partials};
    if (RB == 1)
      return launch_config(kernel(), dim3((unsigned)ncb), dim3(THREADS), 0, 1, s, args, true);
    const void* ahead = reinterpret_cast<const void*>(&gemv_t_cols<THREADS, VW, Q, U, true, G, EDGE>);
    const lift_status r = launch_config(ahead, dim3((unsigned)ncb, (unsigned)RB), dim3(THREADS), 0, 1, s,
                                        args, true);
    if (r != LIFT_OK) return r;
    if (RB <= kColsTree) return launch_combine_cols(N, (int)RB, alpha, beta, partials, y, s);
    return launch_rows_combine(N, RB, alpha, beta, partials, y, s);
  }
};

template <int THREADS, int VW, int Q, int U, int PER_SM>
Variant cols_variant(const char* name) {
  using K = GemvTCols<THREADS, VW, Q, U, PER_SM>;
  Variant v{};
  v.info.op = LIFT_OP_GEMV_T;
  v.info.tile = THREADS * VW * Q;
  v.info.vw = VW;
  v.info.threads = THREADS;
  v.info.stride = 1;
  v.info.cluster = 1;
  v.info.passes = VW == 1 ? 4 : 3;
  v.info.rows = U;
  v.info.lanes = 1;
  v.info.final_threads = kWarp;
  snprintf(v.info.name, sizeof(v.info.name), "gemv_t_%s", name);
  v.launch = &K::launch;
  v.grid = &K::grid;
  v.align_bytes = VW * 4;
  v.fallback = 0;
  return v;
}

}  // namespace

// (threads, vector width, vectors per thread, rows in flight, CTAs per SM)
#define LIFT_GEMV_T_COLS_VARIANTS(X)          \
  X(128, 1, 2, 8, 8, "t128_v1_q2_u8_p2")      \
  X(128, 4, 1, 8, 6, "t128_v4_q1_u8_p2")

void gemv_t_cols_shape(const char* name, const Args& a, int64_t* B, int64_t* RB) {
  int64_t ncb = 0, rb = 0, b = 0;
#define X(T, V, Q, U, P, NAME) \
  if (std::string("gemv_t_") + NAME == name) GemvTCols<T, V, Q, U, P>::shape(a, ncb, rb, b);
  LIFT_GEMV_T_COLS_VARIANTS(X)
#undef X
  *B = b;
  *RB = rb;
}

// registered after the families of gemv_t.cu (earlier ids are stable)
void register_gemv_t_cols(std::vector<Variant>& L) {
  const size_t first = L.size();
#define X(T, V, Q, U, P, NAME) L.push_back(cols_variant<T, V, Q, U, P>(NAME));
  LIFT_GEMV_T_COLS_VARIANTS(X)
#undef X
  for (size_t i = first; i < L.size(); ++i) L[i].info.id = static_cast<int>(i);
}

}  // namespace lift
