// Cost-model training kernels: a multilayer perceptron d_in -> h1 -> h2 -> V
// with ReLU hidden layers, a masked mean-squared-error loss and Adam, in FP32
// on CUDA cores (the matrices are a few thousand rows by at most a few
// hundred columns; the work is latency-bound, not a tensor-core contraction).
//
// The cost model's own network (h1 = h2 = 64, d_in <= 64) runs fused: one
// launch for the three layers, one for the loss, two for the gradients, with
// every reduction spread over the GPU and finished through shared or
// distributed shared memory, so that no call needs scratch memory beyond its
// arguments.  A training step of 2308 shapes and 265 outputs (forward, loss,
// backward, Adam; host calls included) took 615 us as thirteen launches of
// one GEMM or reduction each, most of it in the one-CTA loss and in
// reductions over the 2308 rows by 3 to 18 CTAs; 43 us as five (forward 7.6,
// loss 7.9, gradients 20.2, Adam 1.8 each alone in a graph).  Bound by
// latency: each launch is one or two dependent phases of copies and
// shared-memory folds on all SMs, and each is a programmatic dependent of the
// one before it (49 us as plain launches).  Other sizes run the one-operation
// kernels.
//
// The model predicts one log-time per kernel variant from the features of a
// call; the autotuner's measurements are its training data (the paper's
// empirical exploration of split sizes and vector widths, Sec. 6.2, and its
// model-guided search, Sec. 6.3).
//
// Parameter buffer (one contiguous fp32 array, row-major matrices):
//   W1 [d_in][h1] | b1 [h1] | W2 [h1][h2] | b2 [h2] | W3 [h2][V] | b3 [V]
// Work buffer per batch of B rows:
//   Z1 [B][h1] | H1 [B][h1] | Z2 [B][h2] | H2 [B][h2] | D0 [B][hm] | D1 [B][hm]
// with hm = max(h1, h2).
#include <cooperative_groups.h>

#include <map>
#include <mutex>

#include "lift_internal.cuh"

namespace cg = cooperative_groups;

namespace lift {
namespace {

constexpr int kTile = 32;

// C[M][N] = op(A)[M][K] . op(B)[K][N] + bias[N] (optional), with an
// epilogue: 0 store; 1 store Z in C and relu(Z) in C2; 2 multiply by
// [gate > 0] (ReLU backward).  op(A) = A [M][K] or A^T with A [K][M].
template <bool TA, bool TB>
__global__ void __launch_bounds__(kTile * 8)
    gemm_small(int M, int N, int K, const float* __restrict__ A, const float* __restrict__ B,
               float* __restrict__ C, const float* __restrict__ bias, float* __restrict__ C2,
               const float* __restrict__ gate, int epilogue) {
  __shared__ float As[kTile][kTile + 1];
  __shared__ float Bs[kTile][kTile + 1];
  const int tx = threadIdx.x % kTile, ty = threadIdx.x / kTile;  // 32 x 8
  const int row0 = blockIdx.y * kTile, col0 = blockIdx.x * kTile;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int k0 = 0; k0 < K; k0 += kTile) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = ty + 8 * i;  // tile row
      const int gm = row0 + r, gk = k0 + tx;
      float a = 0.f;
      if (gm < M && gk < K) a = TA ? A[(size_t)gk * M + gm] : A[(size_t)gm * K + gk];
      As[r][tx] = a;
      const int bk = k0 + r, bn = col0 + tx;
      float b = 0.f;
      if (bk < K && bn < N) b = TB ? B[(size_t)bn * K + bk] : B[(size_t)bk * N + bn];
      Bs[r][tx] = b;
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < kTile; ++kk) {
      const float b = Bs[kk][tx];
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[i] = fmaf(As[ty + 8 * i][kk], b, acc[i]);
    }
    __syncthreads();
  }
  const int n = col0 + tx;
  if (n >= N) return;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = row0 + ty + 8 * i;
    if (m >= M) continue;
    float z = acc[i] + (bias ? bias[n] : 0.f);
    const size_t o = (size_t)m * N + n;
    if (epilogue == 2) z = gate[o] > 0.f ? z : 0.f;
    C[o] = z;
    if (epilogue == 1) C2[o] = z > 0.f ? z : 0.f;
  }
}

// db[j] = sum_b D[b][j]
__global__ void col_sum(int B, int N, const float* __restrict__ D, float* __restrict__ out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= N) return;
  float s = 0.f;
  for (int b = 0; b < B; ++b) s += D[(size_t)b * N + j];
  out[j] = s;
}

// loss = sum(mask * (P - T)^2) * inv;  dP = 2 * mask * (P - T) * inv
// One cluster of 16 CTAs (8 where a device cannot hold 16), whose sums meet
// in distributed shared memory: the largest group of CTAs that can finish a
// sum without scratch in global memory (the entry point has none, and calls
// on any number of streams may overlap).  VEC: 16-byte loads (every array
// 16-byte aligned).  Bound by the 64 bytes per clock that each of its SMs
// can load: 611,620 entries in 7.9 us, 11.6 with 8 CTAs.
constexpr int kLossThreads = 1024;

template <bool VEC>
__global__ void __launch_bounds__(kLossThreads)
    masked_mse(const float* __restrict__ P, const float* __restrict__ T, const float* __restrict__ Mk,
               int64_t count, float inv, float* __restrict__ dP, float* __restrict__ loss) {
  __shared__ float red[kWarp];
  __shared__ float part;
  pdl_trigger();   // the next launch may be scheduled (it waits for this one)
  pdl_wait();      // the launch before has finished
  cg::cluster_group cl = cg::this_cluster();
  const int64_t t = (int64_t)blockIdx.x * kLossThreads + threadIdx.x;
  const int64_t kAll = (int64_t)gridDim.x * kLossThreads;
  float s = 0.f;
  auto entry = [&](float p, float q, float m) {
    const float d = m > 0.f ? p - q : 0.f;
    s = fmaf(d, d, s);
    return 2.f * d * inv;
  };
  int64_t done = 0;
  if constexpr (VEC) {
    const int64_t quads = count / 4;
#pragma unroll 4
    for (int64_t i = t; i < quads; i += kAll) {
      const float4 m = __ldg(reinterpret_cast<const float4*>(Mk) + i);
      const float4 p = __ldg(reinterpret_cast<const float4*>(P) + i);
      const float4 q = __ldg(reinterpret_cast<const float4*>(T) + i);
      float4 o;
      o.x = entry(p.x, q.x, m.x);
      o.y = entry(p.y, q.y, m.y);
      o.z = entry(p.z, q.z, m.z);
      o.w = entry(p.w, q.w, m.w);
      reinterpret_cast<float4*>(dP)[i] = o;
    }
    done = quads * 4;
  }
#pragma unroll 4
  for (int64_t i = done + t; i < count; i += kAll) dP[i] = entry(P[i], T[i], Mk[i]);
  s = block_tree<kLossThreads>(s, red);
  if (threadIdx.x == 0) part = s;
  cl.sync();
  if (cl.block_rank() == 0 && threadIdx.x == 0) {
    for (unsigned r = 1; r < gridDim.x; ++r) s = __fadd_rn(s, *cl.map_shared_rank(&part, r));
    *loss = s * inv;
  }
  cl.sync();                         // peers stay until rank 0 has read their sums
}

// ---------------------------------------------------------------------------
// the fused network: H = 64 units in both hidden layers
// ---------------------------------------------------------------------------
constexpr int kH = 64;               // hidden units
constexpr int kRows = 16;            // rows of the batch per CTA
constexpr int kMaxShared = 227 * 1024;   // bytes a CTA may have: with it one CTA fits an SM
constexpr int kPitch = 20;           // floats between columns of a [.][kRows] array in shared
                                     // memory: 16-byte rows, 4-way conflicts at most on writes

// Asynchronous copies global -> shared (4 or 16 bytes), all in flight until
// cp_wait.
__device__ __forceinline__ void cp4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait_all_but_one() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// n floats, by the whole CTA; vec: both sides 16-byte aligned
__device__ __forceinline__ void cp_flat(float* dst, const float* src, int n, bool vec) {
  const int n4 = vec ? n / 4 : 0;
  for (int i = threadIdx.x; i < n4; i += blockDim.x) cp16(dst + 4 * i, src + 4 * i);
  for (int i = 4 * n4 + threadIdx.x; i < n; i += blockDim.x) cp4(dst + i, src + i);
}

// acc[0..3] += W * (rows 4g .. 4g+3 of the column at `in`)
__device__ __forceinline__ void fma4(float (&acc)[4], float w, const float* in) {
  const float4 h = *reinterpret_cast<const float4*>(in);
  acc[0] = fmaf(h.x, w, acc[0]);
  acc[1] = fmaf(h.y, w, acc[1]);
  acc[2] = fmaf(h.z, w, acc[2]);
  acc[3] = fmaf(h.w, w, acc[3]);
}

// One hidden layer of the CTA's rows: thread (unit j, rows 4g .. 4g+3) folds
// the K inputs in order (the order of gemm_small: the same bits), stores Z
// and relu(Z), and leaves relu(Z) in shared memory for the next layer.
__device__ __forceinline__ void hidden_layer(int K, const float* in, const float* W,
                                             const float* __restrict__ bias, int r0, int rows,
                                             float* __restrict__ Z, float* __restrict__ Hg,
                                             float* out) {
  for (int it = threadIdx.x; it < kH * (kRows / 4); it += blockDim.x) {
    const int j = it % kH, g = it / kH;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
    for (int k = 0; k < K; ++k) fma4(acc, W[k * kH + j], in + k * kPitch + 4 * g);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = 4 * g + q;
      const float z = acc[q] + __ldg(bias + j), h = z > 0.f ? z : 0.f;
      out[j * kPitch + r] = h;
      if (r < rows) {
        Z[(size_t)(r0 + r) * kH + j] = z;
        Hg[(size_t)(r0 + r) * kH + j] = h;
      }
    }
  }
  __syncthreads();
}

// The three layers of kRows rows per CTA.  All weights are copied to shared
// memory at once (85 KB for 265 outputs), W3 while the hidden layers run.
// The last layer gives a thread one output column of all 16 rows: a weight
// is read once and used 16 times against broadcast reads of the activations.
// CW: columns of W3 staged at a time (all of them up to kFwdColumns, what fits
// the shared memory beside the other matrices).
constexpr int kFwdColumns =
    (kMaxShared / 4 - 2 * kH * kH - 2 * kH * kPitch) / kH / kWarp * kWarp;       // 736

__global__ void __launch_bounds__(512)
    mlp_forward_fused(int B, int d, int V, int CW, const float* __restrict__ W1,
                      const float* __restrict__ b1, const float* __restrict__ W2,
                      const float* __restrict__ b2, const float* __restrict__ W3,
                      const float* __restrict__ b3, const float* __restrict__ X,
                      float* __restrict__ Z1, float* __restrict__ H1, float* __restrict__ Z2,
                      float* __restrict__ H2, float* __restrict__ P) {
  extern __shared__ __align__(16) float sm[];
  float* w3 = sm;                                   // [kH][CW]
  float* w2 = w3 + kH * CW;                         // [kH][kH]
  float* w1 = w2 + kH * kH;                         // [d][kH]
  float* h1 = w1 + kH * kH;                         // [kH][kPitch], and the inputs before it
  float* h2 = h1 + kH * kPitch;
  float* xs = h2;
  const int r0 = blockIdx.x * kRows, rows = B - r0 < kRows ? B - r0 : kRows;
  const bool vec = reinterpret_cast<uintptr_t>(W1) % 16 == 0;   // so are the other matrices
  // (no early trigger: the next launch's CTAs beside these took 3 us from them)
  pdl_wait();      // the launch before has finished
  for (int i = threadIdx.x; i < kRows * d; i += blockDim.x) {
    const int r = i / d, k = i % d;
    if (r < rows) cp4(xs + k * kPitch + r, X + (size_t)r0 * d + i);
    else xs[k * kPitch + r] = 0.f;
  }
  cp_flat(w1, W1, d * kH, vec);
  cp_flat(w2, W2, kH * kH, vec);
  cp_commit();
  if (CW == V) cp_flat(w3, W3, kH * V, vec);
  cp_commit();
  cp_wait_all_but_one();
  __syncthreads();
  hidden_layer(d, xs, w1, b1, r0, rows, Z1, H1, h1);
  hidden_layer(kH, h1, w2, b2, r0, rows, Z2, H2, h2);
  cp_wait();
  __syncthreads();
  for (int c0 = 0; c0 < V; c0 += CW) {
    const int cw = V - c0 < CW ? V - c0 : CW;
    if (CW != V) {
      __syncthreads();                              // the chunk before has been used
      for (int i = threadIdx.x; i < kH * cw; i += blockDim.x)
        cp4(w3 + i / cw * CW + i % cw, W3 + (size_t)(i / cw) * V + c0 + i % cw);
      cp_wait();
      __syncthreads();
    }
    for (int c = threadIdx.x; c < cw; c += blockDim.x) {
      float acc[kRows / 4][4];
#pragma unroll
      for (int g = 0; g < kRows / 4; ++g)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[g][q] = 0.f;
#pragma unroll 8
      for (int k = 0; k < kH; ++k) {
        const float w = w3[k * CW + c];
#pragma unroll
        for (int g = 0; g < kRows / 4; ++g) fma4(acc[g], w, h2 + k * kPitch + 4 * g);
      }
      const float b = __ldg(b3 + c0 + c);
#pragma unroll
      for (int r = 0; r < kRows; ++r)
        if (r < rows) P[(size_t)(r0 + r) * V + c0 + c] = acc[r / 4][r % 4] + b;
    }
  }
}

// dZ2 = (dP W3^T) * [Z2 > 0] and dZ1 = (dZ2 W2^T) * [Z1 > 0] of kRows rows
// per CTA.  W3 (in chunks of CW output columns) and W2 are staged in shared
// memory with an odd pitch, so that 32 threads that walk 32 rows of W
// together read 32 banks; the sum over a row's columns is split between four
// quarters of the CTA.  A chunk is what fits the shared memory of an SM: a
// batch of 2308 rows is 145 CTAs, one per SM whatever they hold, and its
// copies are waited for once per chunk (both gradient launches, us: 2308 x 400
// 30.0, in two chunks 37.1; 4096 x 512 57.8, 60.3; 3000 x 300, where two CTAs
// of half a chunk would share an SM, 30.5, 29.7).
constexpr int kActThreads = 512;
constexpr int kBackColumns =
    (kMaxShared / 4 - 6 * kH * kPitch - kH * (kH + 1) - kH) / (kPitch + kH) / kWarp * kWarp;   // 544

// Thread (units j and j + 32, rows 4g .. 4g+3, a quarter of the columns): one
// broadcast read of four rows serves two units.
__device__ __forceinline__ void back_layer(int cw, int pitch, const float* W, const float* in,
                                           float (&acc)[2][4]) {
  const int j = threadIdx.x % kWarp, g = threadIdx.x / kWarp % (kRows / 4), part = threadIdx.x / 128;
  const int c0 = cw * part / 4, c1 = cw * (part + 1) / 4;
#pragma unroll 8
  for (int c = c0; c < c1; ++c) {
    fma4(acc[0], W[j * pitch + c], in + c * kPitch + 4 * g);
    fma4(acc[1], W[(j + kWarp) * pitch + c], in + c * kPitch + 4 * g);
  }
}

// adds the quarters, applies the gate, leaves the result in `out` and in global memory
__device__ __forceinline__ void gate_layer(const float (&acc)[2][4], float* parts, const float* gate,
                                           int r0, int rows, float* out, float* __restrict__ D) {
  const int j = threadIdx.x % kWarp, g = threadIdx.x / kWarp % (kRows / 4), part = threadIdx.x / 128;
  if (part > 0) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
      *reinterpret_cast<float4*>(parts + ((part - 1) * kH + j + kWarp * h) * kPitch + 4 * g) =
          make_float4(acc[h][0], acc[h][1], acc[h][2], acc[h][3]);
  }
  __syncthreads();
  if (part == 0) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = 4 * g + q, u = j + kWarp * h;
        float v = acc[h][q];
#pragma unroll
        for (int k = 0; k < 3; ++k) v += parts[(k * kH + u) * kPitch + r];
        v = gate[u * kPitch + r] > 0.f ? v : 0.f;
        out[u * kPitch + r] = v;
        if (r < rows) D[(size_t)(r0 + r) * kH + u] = v;
      }
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kActThreads)
    mlp_back_rows(int B, int V, int CW, const float* __restrict__ W2, const float* __restrict__ W3,
                  const float* __restrict__ H1, const float* __restrict__ H2,
                  const float* __restrict__ dP, float* __restrict__ D0, float* __restrict__ D1) {
  extern __shared__ __align__(16) float sm[];
  const int pitch = CW | 1;
  float* dps = sm;                                  // [CW][kPitch]
  float* h1 = dps + CW * kPitch;                    // [kH][kPitch]
  float* h2 = h1 + kH * kPitch;
  float* d0 = h2 + kH * kPitch;
  float* parts = d0 + kH * kPitch;                  // [3][kH][kPitch]
  float* w2 = parts + 3 * kH * kPitch;              // [kH][kH + 1]
  float* w3 = w2 + kH * (kH + 1);                   // [kH][pitch]
  const int t = threadIdx.x, r0 = blockIdx.x * kRows, rows = B - r0 < kRows ? B - r0 : kRows;
  pdl_trigger();   // the next launch may be scheduled (it waits for this one)
  pdl_wait();      // the launch before has finished
  for (int i = t; i < kRows * kH; i += kActThreads) {    // relu(Z) > 0 where Z > 0
    const int r = i / kH, j = i % kH;
    if (r < rows) {
      cp4(h1 + j * kPitch + r, H1 + (size_t)r0 * kH + i);
      cp4(h2 + j * kPitch + r, H2 + (size_t)r0 * kH + i);
    } else {
      h1[j * kPitch + r] = h2[j * kPitch + r] = 0.f;
    }
  }
  for (int i = t; i < kH * kH; i += kActThreads) cp4(w2 + i / kH * (kH + 1) + i % kH, W2 + i);
  float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
  const int warp = t / kWarp, lane = t % kWarp;
  for (int c0 = 0; c0 < V; c0 += CW) {
    const int cw = V - c0 < CW ? V - c0 : CW;
    for (int r = warp; r < kRows; r += kActThreads / kWarp)
      for (int c = lane; c < cw; c += kWarp) {
        if (r < rows) cp4(dps + c * kPitch + r, dP + (size_t)(r0 + r) * V + c0 + c);
        else dps[c * kPitch + r] = 0.f;
      }
    for (int j = warp; j < kH; j += kActThreads / kWarp)
      for (int c = lane; c < cw; c += kWarp) cp4(w3 + j * pitch + c, W3 + (size_t)j * V + c0 + c);
    cp_wait();
    __syncthreads();
    back_layer(cw, pitch, w3, dps, acc);
    __syncthreads();                                // the chunk is read before the next one lands
  }
  gate_layer(acc, parts, h2, r0, rows, d0, D0);
  float acc1[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
  back_layer(kH, kH + 1, w2, d0, acc1);             // dZ1_i = sum_j dZ2_j W2[i][j]
  gate_layer(acc1, parts, h1, r0, rows, h2, D1);    // (h2 is no longer read)
}

// Weight and bias gradients: out[i][c] = sum_r L[r][i] R[r][c] and, for the
// biases, sum_r R[r][c], for the pairs (H2, dP), (H1, dZ2) and (X, dZ1).  A
// cluster of kGradCtas CTAs takes 32 columns c and every i <= 64, each CTA a
// contiguous part of the rows: copied to shared memory up to kGradRows at a
// time in two halves, the second in flight while the first is folded (2308 x
// 265: 20.2 us for both gradient launches, 34.4 when the rows were read from
// global memory as they were folded, waiting on loads), folded in kGradShares
// shares by thread (share, 8 consecutive i, c), and the shares added in order
// through distributed shared memory.
constexpr int kGradCtas = 8, kGradI = 8, kGradGroups = kH / kGradI, kGradShares = 4;
constexpr int kGradThreads = kGradShares * kGradGroups * kWarp;
// rows of L and R that fit the shared memory of an SM beside the sums: 512
// (4096 x 64: 27.7 us for both gradient launches, 28.5 in pieces of 304 rows)
constexpr int kGradRowBytes = (kH + kWarp) * (int)sizeof(float);
constexpr int kGradRows =
    (kMaxShared - kGradShares * (kH + 1) * kWarp * (int)sizeof(float)) / kGradRowBytes / 16 * 16;

struct GradJob {
  const float* L;      // rows x li
  const float* R;      // rows x rc
  float* out;          // li x rc
  float* bias;         // rc
  int li, rc, first;   // first: index of the job's first column tile
  int vec;             // rows of L in whole, aligned 16-byte granules
};
struct GradJobs {
  GradJob j[3];
};

__global__ void __launch_bounds__(kGradThreads)
    mlp_weight_grads(int B, const __grid_constant__ GradJobs jobs) {
  extern __shared__ __align__(16) float sm[];            // [kGradRows][kH] of L, [kGradRows][32] of R
  __shared__ float part[kGradShares][kH + 1][kWarp];     // row kH: the bias sums
  cg::cluster_group cl = cg::this_cluster();
  const int tile = blockIdx.x / kGradCtas, rank = blockIdx.x % kGradCtas;
  const GradJob& job = tile >= jobs.j[2].first ? jobs.j[2] : tile >= jobs.j[1].first ? jobs.j[1] : jobs.j[0];
  const int lane = threadIdx.x % kWarp, grp = threadIdx.x / kWarp % kGradGroups;
  const int share = threadIdx.x / (kWarp * kGradGroups);
  const int c0 = (tile - job.first) * kWarp, i0 = grp * kGradI, li = job.li, rc = job.rc;
  const int b0 = (int)((int64_t)B * rank / kGradCtas), b1 = (int)((int64_t)B * (rank + 1) / kGradCtas);
  float* ls = sm;
  float* rs = sm + kGradRows * kH;
  float acc[kGradI], bs = 0.f;
#pragma unroll
  for (int q = 0; q < kGradI; ++q) acc[q] = 0.f;
  pdl_trigger();   // the next launch may be scheduled (it waits for this one)
  pdl_wait();      // the launch before has finished
  if (li < kH)                                           // columns past L stay zero
    for (int e = threadIdx.x; e < (b1 - b0 < kGradRows ? b1 - b0 : kGradRows) * kH; e += kGradThreads)
      if (e % kH >= li) ls[e] = 0.f;
  for (int r0 = b0; r0 < b1; r0 += kGradRows) {
    const int rows = b1 - r0 < kGradRows ? b1 - r0 : kGradRows;
    const float* L = job.L + (size_t)r0 * li;
    const float* R = job.R + (size_t)r0 * rc + c0;
    const int mid = rows / 2;
#pragma unroll
    for (int h = 0; h < 2; ++h) {                        // the second half lands while the first is folded
      const int q0 = h ? mid : 0, q1 = h ? rows : mid;
      if (job.vec) {
        const int l4 = li / 4;
        for (int e = q0 * l4 + threadIdx.x; e < q1 * l4; e += kGradThreads)
          cp16(ls + e / l4 * kH + e % l4 * 4, L + 4 * (size_t)e);
      } else {
        for (int e = q0 * li + threadIdx.x; e < q1 * li; e += kGradThreads)
          cp4(ls + e / li * kH + e % li, L + e);
      }
      for (int r = q0 + threadIdx.x / kWarp; r < q1; r += kGradThreads / kWarp) {
        if (c0 + lane < rc) cp4(rs + r * kWarp + lane, R + (size_t)r * rc + lane);
        else rs[r * kWarp + lane] = 0.f;
      }
      cp_commit();
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (h == 0) cp_wait_all_but_one();
      else cp_wait();
      __syncthreads();
      if (i0 >= li && grp != 0) continue;
      const int q0 = h ? mid : 0, half = h ? rows - mid : mid;
      const int ra = q0 + half * share / kGradShares, rb = q0 + half * (share + 1) / kGradShares;
#pragma unroll 4
      for (int r = ra; r < rb; ++r) {
        const float v = rs[r * kWarp + lane];
        const float4 a = *reinterpret_cast<const float4*>(ls + r * kH + i0);
        const float4 b = *reinterpret_cast<const float4*>(ls + r * kH + i0 + 4);
        acc[0] = fmaf(a.x, v, acc[0]);
        acc[1] = fmaf(a.y, v, acc[1]);
        acc[2] = fmaf(a.z, v, acc[2]);
        acc[3] = fmaf(a.w, v, acc[3]);
        acc[4] = fmaf(b.x, v, acc[4]);
        acc[5] = fmaf(b.y, v, acc[5]);
        acc[6] = fmaf(b.z, v, acc[6]);
        acc[7] = fmaf(b.w, v, acc[7]);
        bs += v;
      }
    }
    __syncthreads();                                     // read before the next rows land
  }
#pragma unroll
  for (int q = 0; q < kGradI; ++q) part[share][i0 + q][lane] = acc[q];
  if (grp == 0) part[share][kH][lane] = bs;
  cl.sync();
  // rank r adds a contiguous part of the 65 x 32 sums over the shares and writes it
  constexpr int kSums = (kH + 1) * kWarp, kPer = (kSums + kGradCtas - 1) / kGradCtas;
  for (int e = rank * kPer + threadIdx.x; e < (rank + 1) * kPer && e < kSums; e += kGradThreads) {
    const int i = e / kWarp, cc = c0 + e % kWarp;
    float v[kGradCtas][kGradShares], s = 0.f;
#pragma unroll
    for (int q = 0; q < kGradCtas; ++q) {
      const float* p = cl.map_shared_rank(&part[0][0][0], q) + e;
#pragma unroll
      for (int h = 0; h < kGradShares; ++h) v[q][h] = p[h * kSums];
    }
#pragma unroll
    for (int q = 0; q < kGradCtas; ++q)
#pragma unroll
      for (int h = 0; h < kGradShares; ++h) s += v[q][h];
    if (cc < rc) {
      if (i == kH) job.bias[cc] = s;
      else if (i < li) job.out[(size_t)i * rc + cc] = s;
    }
  }
  cl.sync();                         // peers stay until their sums have been read
}

__global__ void adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                     float* __restrict__ v, int64_t count, float lr, float b1, float b2, float eps,
                     float c1, float c2) {
  pdl_trigger();   // the next launch may be scheduled (it waits for this one)
  pdl_wait();      // the launch before has finished
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

struct Layout {
  int64_t W1, b1, W2, b2, W3, b3, total;
  Layout(int d, int h1, int h2, int V) {
    W1 = 0;
    b1 = W1 + (int64_t)d * h1;
    W2 = b1 + h1;
    b2 = W2 + (int64_t)h1 * h2;
    W3 = b2 + h2;
    b3 = W3 + (int64_t)h2 * V;
    total = b3 + V;
  }
};

template <bool TA, bool TB>
lift_status gemm(int M, int N, int K, const float* A, const float* B, float* C, const float* bias,
                 float* C2, const float* gate, int epi, cudaStream_t s) {
  dim3 grid((N + kTile - 1) / kTile, (M + kTile - 1) / kTile);
  gemm_small<TA, TB><<<grid, kTile * 8, 0, s>>>(M, N, K, A, B, C, bias, C2, gate, epi);
  return cuda_check(cudaGetLastError(), "mlp gemm launch");
}

// CTAs of the loss kernel's cluster on the current device: 16 needs the
// non-portable cluster size; looked up once per device and kernel.
int loss_cluster(const void* k) {
  static std::mutex mu;
  static std::map<std::pair<int, const void*>, int> known;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) return 8;
  std::lock_guard<std::mutex> lk(mu);
  auto it = known.find({dev, k});
  if (it != known.end()) return it->second;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(16);
  cfg.blockDim = dim3(kLossThreads);
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = 16;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int n = 0;
  const bool ok =
      cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
      cudaOccupancyMaxActiveClusters(&n, k, &cfg) == cudaSuccess && n > 0;
  if (!ok) cudaGetLastError();
  return known[{dev, k}] = ok ? 16 : 8;
}

// The network the fused kernels are written for (the cost model's).
bool fused_shape(int d, int h1, int h2) { return h1 == kH && h2 == kH && d <= kH; }

lift_status forward_fused(int d, int V, const float* p, const Layout& L, const float* X, int B,
                          float* Z1, float* H1, float* Z2, float* H2, float* P, cudaStream_t s) {
  int CW = V < kFwdColumns ? V : kFwdColumns;
  int threads = (CW + kWarp - 1) / kWarp * kWarp;    // one output column per thread if it can be
  threads = threads < 256 ? 256 : threads > 512 ? 512 : threads;
  const size_t smem = sizeof(float) * ((size_t)kH * CW + 2 * kH * kH + 2 * kH * kPitch);
  const lift_status rc = cuda_check(
      cudaFuncSetAttribute(mlp_forward_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxShared),
      "mlp_forward shared memory");
  if (rc != LIFT_OK) return rc;
  const float *W1 = p + L.W1, *b1 = p + L.b1, *W2 = p + L.W2, *b2 = p + L.b2, *W3 = p + L.W3,
              *b3 = p + L.b3;
  void* args[] = {&B, &d, &V, &CW, &W1, &b1, &W2, &b2, &W3, &b3, &X, &Z1, &H1, &Z2, &H2, &P};
  return launch_config(reinterpret_cast<const void*>(&mlp_forward_fused), dim3((B + kRows - 1) / kRows),
                       dim3(threads), smem, 1, s, args, true);
}

lift_status backward_fused(int d, int V, const float* p, const Layout& L, const float* X, int B,
                           const float* H1, const float* H2, float* D0, float* D1, const float* dP,
                           float* grads, cudaStream_t s) {
  const int chunks = (V + kBackColumns - 1) / kBackColumns, CW = (V + chunks - 1) / chunks;
  const size_t smem = sizeof(float) * ((size_t)CW * kPitch + 6 * kH * kPitch + kH * (kH + 1) +
                                       (size_t)kH * (CW | 1));
  lift_status rc = cuda_check(cudaFuncSetAttribute(mlp_back_rows,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   kMaxShared), "mlp_backward shared memory");
  if (rc != LIFT_OK) return rc;
  const float *W2 = p + L.W2, *W3 = p + L.W3;
  void* rows_args[] = {&B, &V, const_cast<int*>(&CW), &W2, &W3, &H1, &H2, &dP, &D0, &D1};
  rc = launch_config(reinterpret_cast<const void*>(&mlp_back_rows), dim3((B + kRows - 1) / kRows),
                     dim3(kActThreads), smem, 1, s, rows_args, true);
  if (rc != LIFT_OK) return rc;
  const int t3 = (V + kWarp - 1) / kWarp, t64 = kH / kWarp;
  const int hv = aligned(H1, 16) && aligned(H2, 16), xv = aligned(X, 16) && d % 4 == 0;
  GradJobs jobs = {{{H2, dP, grads + L.W3, grads + L.b3, kH, V, 0, hv},
                    {H1, D0, grads + L.W2, grads + L.b2, kH, kH, t3, hv},
                    {X, D1, grads + L.W1, grads + L.b1, d, kH, t3 + t64, xv}}};
  constexpr int kGradSmem = kGradRows * kGradRowBytes;
  rc = cuda_check(cudaFuncSetAttribute(mlp_weight_grads, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kGradSmem), "mlp_backward shared memory");
  if (rc != LIFT_OK) return rc;
  void* args[] = {&B, &jobs};
  return launch_config(reinterpret_cast<const void*>(&mlp_weight_grads),
                       dim3((unsigned)(t3 + 2 * t64) * kGradCtas), dim3(kGradThreads), kGradSmem,
                       kGradCtas, s, args, true);
}

bool bad_shape(int d, int h1, int h2, int V) { return d < 1 || h1 < 1 || h2 < 1 || V < 1; }

}  // namespace
}  // namespace lift

using namespace lift;

extern "C" {

int64_t lift_mlp_param_count(int d_in, int h1, int h2, int V) {
  if (bad_shape(d_in, h1, h2, V)) return -1;
  return Layout(d_in, h1, h2, V).total;
}

int64_t lift_mlp_work_count(int64_t B, int h1, int h2) {
  if (B < 0 || h1 < 1 || h2 < 1) return -1;
  const int64_t hm = h1 > h2 ? h1 : h2;
  return B * (2 * (int64_t)h1 + 2 * (int64_t)h2 + 2 * hm);
}

lift_status lift_mlp_forward(int d_in, int h1, int h2, int V, const float* params, const float* X,
                             int64_t B, float* work, float* P, void* stream) {
  if (bad_shape(d_in, h1, h2, V) || B < 1 || !params || !X || !work || !P || B > (1 << 30))
    return set_error(LIFT_ERR_INVALID_ARG, "mlp_forward arguments");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const Layout L(d_in, h1, h2, V);
  float* Z1 = work;
  float* H1 = Z1 + B * h1;
  float* Z2 = H1 + B * h1;
  float* H2 = Z2 + B * h2;
  const int b = (int)B;
  if (fused_shape(d_in, h1, h2)) return forward_fused(d_in, V, params, L, X, b, Z1, H1, Z2, H2, P, s);
  lift_status rc = gemm<false, false>(b, h1, d_in, X, params + L.W1, Z1, params + L.b1, H1, nullptr, 1, s);
  if (rc == LIFT_OK)
    rc = gemm<false, false>(b, h2, h1, H1, params + L.W2, Z2, params + L.b2, H2, nullptr, 1, s);
  if (rc == LIFT_OK)
    rc = gemm<false, false>(b, V, h2, H2, params + L.W3, P, params + L.b3, nullptr, nullptr, 0, s);
  return rc;
}

lift_status lift_mlp_loss(const float* P, const float* T, const float* mask, int64_t count,
                          float inv_measured, float* dP, float* loss, void* stream) {
  if (count < 1 || !P || !T || !mask || !dP || !loss)
    return set_error(LIFT_ERR_INVALID_ARG, "mlp_loss arguments");
  const bool vec = aligned(P, 16) && aligned(T, 16) && aligned(mask, 16) && aligned(dP, 16);
  const void* k = vec ? reinterpret_cast<const void*>(&masked_mse<true>)
                      : reinterpret_cast<const void*>(&masked_mse<false>);
  const int ctas = loss_cluster(k);
  void* args[] = {&P, &T, &mask, &count, &inv_measured, &dP, &loss};
  return launch_config(k, dim3(ctas), dim3(kLossThreads), 0, ctas, static_cast<cudaStream_t>(stream),
                       args, true);
}

lift_status lift_mlp_backward(int d_in, int h1, int h2, int V, const float* params, const float* X,
                              int64_t B, float* work, const float* dP, float* grads, void* stream) {
  if (bad_shape(d_in, h1, h2, V) || B < 1 || !params || !X || !work || !dP || !grads ||
      B > (1 << 30))
    return set_error(LIFT_ERR_INVALID_ARG, "mlp_backward arguments");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const Layout L(d_in, h1, h2, V);
  const int64_t hm = h1 > h2 ? h1 : h2;
  float* Z1 = work;
  float* H1 = Z1 + B * h1;
  float* Z2 = H1 + B * h1;
  float* H2 = Z2 + B * h2;
  float* D0 = H2 + B * h2;
  float* D1 = D0 + B * hm;
  const int b = (int)B;
  if (fused_shape(d_in, h1, h2))
    return backward_fused(d_in, V, params, L, X, b, H1, H2, D0, D1, dP, grads, s);
  // layer 3: dW3 = H2^T dP, db3 = colsum(dP), dZ2 = (dP W3^T) * [Z2 > 0]
  lift_status rc = gemm<true, false>(h2, V, b, H2, dP, grads + L.W3, nullptr, nullptr, nullptr, 0, s);
  if (rc != LIFT_OK) return rc;
  col_sum<<<(V + 127) / 128, 128, 0, s>>>(b, V, dP, grads + L.b3);
  rc = gemm<false, true>(b, h2, V, dP, params + L.W3, D0, nullptr, nullptr, Z2, 2, s);
  if (rc != LIFT_OK) return rc;
  // layer 2: dW2 = H1^T dZ2, db2 = colsum(dZ2), dZ1 = (dZ2 W2^T) * [Z1 > 0]
  rc = gemm<true, false>(h1, h2, b, H1, D0, grads + L.W2, nullptr, nullptr, nullptr, 0, s);
  if (rc != LIFT_OK) return rc;
  col_sum<<<(h2 + 127) / 128, 128, 0, s>>>(b, h2, D0, grads + L.b2);
  rc = gemm<false, true>(b, h1, h2, D0, params + L.W2, D1, nullptr, nullptr, Z1, 2, s);
  if (rc != LIFT_OK) return rc;
  // layer 1: dW1 = X^T dZ1, db1 = colsum(dZ1)
  rc = gemm<true, false>(d_in, h1, b, X, D1, grads + L.W1, nullptr, nullptr, nullptr, 0, s);
  if (rc != LIFT_OK) return rc;
  col_sum<<<(h1 + 127) / 128, 128, 0, s>>>(b, h1, D1, grads + L.b1);
  return cuda_check(cudaGetLastError(), "mlp_backward launch");
}

lift_status lift_mlp_adam(float* params, const float* grads, float* m, float* v, int64_t count, int t,
                          float lr, float beta1, float beta2, float eps, void* stream) {
  if (count < 1 || t < 1 || !params || !grads || !m || !v)
    return set_error(LIFT_ERR_INVALID_ARG, "mlp_adam arguments");
  const float c1 = 1.f - powf(beta1, (float)t), c2 = 1.f - powf(beta2, (float)t);
  int blocks = (int)((count + 255) / 256);
  if (blocks > 1024) blocks = 1024;
  void* args[] = {&params, &grads, &m, &v, &count, &lr, &beta1, &beta2, &eps, const_cast<float*>(&c1),
                  const_cast<float*>(&c2)};
  return launch_config(reinterpret_cast<const void*>(&adam), dim3(blocks), dim3(256), 0, 1,
                       static_cast<cudaStream_t>(stream), args, true);
}

}  // extern "C"
