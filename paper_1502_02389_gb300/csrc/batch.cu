// Batched persistent launch: many asum / dot / scal / gemv calls of uneven
// sizes in one graph-captured launch that pulls work items from a queue.
//
// Each op is split into work items (split^ITEM of its vector, or a block of
// gemv rows): map(op) over the batch becomes a map-workgroup over items
// handed out by an atomic queue head (largest items first, so the tail of
// the launch is made of small items).  A CTA processes an item exactly as
// the standalone kernels process their tiles (the item's tiles in order,
// thread t folding vectors t + THREADS*j of each tile, adding the tile's
// lanes, and adding the tile values with Neumaier's compensated step, then
// the block tree); for asum / dot
// each item leaves one fp32 partial, and the CTA that
// finishes an op's last item (an atomic per-op counter) adds that op's item
// partials in item order in FP64 (thread t takes partials t, t+256, ...,
// then an FP64 block tree) and writes the rounded result; an op of one item
// is written by the CTA that folds it.  Nothing waits: the queue and the
// counters are atomics, and the CTAs that use them last return them to zero,
// so that a run is one kernel and nothing else.  The other schedule of the
// same map-workgroup launches one CTA per queue position instead of popping
// the queue, and lets the hardware deal the CTAs to the SMs as earlier ones
// retire; the items, their order and the combine are the same.
//
// A batch of small ops is bound by what a CTA does between items, so the
// persistent kernel fetches ahead: while item i is folded, the first warp has
// the op of item i+1, the item of i+2 and the queue position of i+3 in flight
// (each CTA's first three positions are its own).  4000 ops of 2^8 to 2^14
// elements and 64 to 256 rows and columns took 81 us when every item began
// with the chain position -> item -> op -> data, ended with a fence and an
// atomic, and the run began with two memset nodes; 48 now (22 at the copy
// bandwidth).  Large batches are bound by DRAM: 2000 ops of 5.9 GB take
// 861 us, the copy bandwidth's time (959 with gemv rows one at a time).
//
// Per op, the policy's variant choice (batch_pick: FIXED, TABLE or MLP) is
// mapped to a processing mode: vector ops take the (tile, vector width) of
// the chosen variant when the batch kernel has that mode, gemv takes its
// vector width.  A pointer that is not aligned for the mode's vector width
// gets the 4-byte mode.
#include <algorithm>
#include <string>
#include <vector>

#include "lift_internal.cuh"

namespace lift {
namespace {

constexpr int kThreads = 256;
// Bytes moved per work item: about 1/16 of a CTA's share of the batch, so
// that the CTAs end together, but at least 64 KiB, so that an item is long
// enough to hide the fetch of the next (118 ops of up to 4M elements: 68 us
// with 64 KB items, 79 with 32 KB), and at most 256 KiB (2000 ops: 858 us
// with 128 KB, 861 with 256 KB).
constexpr int64_t kItemBytesMax = 256 * 1024, kItemBytesMin = 64 * 1024, kItemsPerCta = 16;

// vector-op processing modes: (VW, J) with TILE = kThreads * VW * J
struct VecMode {
  int vw, j;
};
constexpr VecMode kVecModes[] = {{1, 4}, {4, 1}, {4, 2}, {4, 4}, {8, 1}, {8, 2}};
constexpr int kNumVecModes = 6;
constexpr int kGemvVW[] = {1, 4, 8};

struct OpDev {
  int op;            // LIFT_OP_ASUM / DOT / SCAL / GEMV
  int mode;          // vector mode index, or gemv vw index
  int64_t n, M, N, lda;
  float alpha, beta;
  const float* x;
  const float* y;
  const float* A;
  float* out;
  int64_t first_item, num_items;
};

struct ItemDev {
  int op_index;         // -1: no item
  int reserved;
  int64_t index;        // of the item's partial: items of an op are consecutive
  int64_t begin, end;   // elements (vector ops) or rows (gemv)
};
constexpr int kOpChunks = sizeof(OpDev) / 16, kItemChunks = sizeof(ItemDev) / 16;
static_assert(sizeof(OpDev) % 16 == 0 && sizeof(ItemDev) % 16 == 0 && kOpChunks + kItemChunks <= kWarp,
              "a warp copies an op and an item in one go");

struct BatchDev {
  const OpDev* ops;
  const ItemDev* items;       // in queue order
  float* partials;            // per item index
  unsigned* op_done;          // per op: items finished (0 between runs)
  unsigned long long* head;   // queue positions dealt beyond the first, then CTAs that left (0 between runs)
  int64_t num_items;
};

template <int OP, int VW>
__device__ __forceinline__ void fold(float* acc, const Vec<VW>& a, const Vec<VW>& b) {
#pragma unroll
  for (int l = 0; l < VW; ++l)
    acc[l] = OP == LIFT_OP_ASUM ? __fadd_rn(acc[l], fabsf(a.v[l]))
                                : __fadd_rn(acc[l], __fmul_rn(a.v[l], b.v[l]));
}

// One reduction item: elements [begin, end) of op o, in tiles of
// kThreads*VW*J elements; returns the CTA's value in thread 0.
template <int OP, int VW, int J>
__device__ float reduce_item(const OpDev& o, int64_t begin, int64_t end, float* red) {
  constexpr int64_t TILE = (int64_t)kThreads * VW * J;
  const int t = threadIdx.x;
  const float* const x = o.x;
  const float* const y = o.y;
  float acc = 0.f, cmp = 0.f;  // sum of the tile values and its Neumaier compensation
  int64_t base = begin;
  for (; base + TILE <= end; base += TILE) {
    Vec<VW> a[J], b[J];
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int64_t e = base + (int64_t)(t + kThreads * j) * VW;
      ld_stream(x + e, a[j]);
      if constexpr (OP == LIFT_OP_DOT) ld_stream(y + e, b[j]);
    }
    float ts[VW];
#pragma unroll
    for (int l = 0; l < VW; ++l) ts[l] = 0.f;
#pragma unroll
    for (int j = 0; j < J; ++j) fold<OP, VW>(ts, a[j], b[j]);
    float tv = ts[0];
#pragma unroll
    for (int l = 1; l < VW; ++l) tv = __fadd_rn(tv, ts[l]);
    neumaier_add(acc, cmp, tv);
  }
  if (base < end) {
    float ts[VW];
#pragma unroll
    for (int l = 0; l < VW; ++l) ts[l] = 0.f;
    Vec<VW> a[J], b[J];                // all loads before the first fold
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int64_t e = base + (int64_t)(t + kThreads * j) * VW;
      if (e + VW <= end) {
        ld_stream(x + e, a[j]);
        if constexpr (OP == LIFT_OP_DOT) ld_stream(y + e, b[j]);
      } else {
        ld_guarded<VW>(x, e, end, a[j]);
        if constexpr (OP == LIFT_OP_DOT) ld_guarded<VW>(y, e, end, b[j]);
      }
    }
#pragma unroll
    for (int j = 0; j < J; ++j) fold<OP, VW>(ts, a[j], b[j]);
    float tv = ts[0];
#pragma unroll
    for (int l = 1; l < VW; ++l) tv = __fadd_rn(tv, ts[l]);
    neumaier_add(acc, cmp, tv);
  }
  return block_tree<kThreads>(neumaier_value(acc, cmp), red);
}

template <int VW, int J>
__device__ void scal_item(const OpDev& o, int64_t begin, int64_t end) {
  constexpr int64_t TILE = (int64_t)kThreads * VW * J;
  const int t = threadIdx.x;
  const float* const x = o.x;
  float* const y = o.out;
  const float alpha = o.alpha;
  int64_t base = begin;
  for (; base + TILE <= end; base += TILE) {
    Vec<VW> a[J];
#pragma unroll
    for (int j = 0; j < J; ++j) ld_stream(x + base + (int64_t)(t + kThreads * j) * VW, a[j]);
#pragma unroll
    for (int j = 0; j < J; ++j) {
#pragma unroll
      for (int l = 0; l < VW; ++l) a[j].v[l] = __fmul_rn(alpha, a[j].v[l]);
      st_stream(y + base + (int64_t)(t + kThreads * j) * VW, a[j]);
    }
  }
  if (base < end) {                    // the ragged tile: all loads before the first store
    Vec<VW> a[J];
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int64_t e = base + (int64_t)(t + kThreads * j) * VW;
      if (e + VW <= end) ld_stream(x + e, a[j]);
      else ld_guarded<VW>(x, e, end, a[j]);
    }
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int64_t e = base + (int64_t)(t + kThreads * j) * VW;
#pragma unroll
      for (int l = 0; l < VW; ++l) a[j].v[l] = __fmul_rn(alpha, a[j].v[l]);
      if (e + VW <= end) {
        st_stream(y + e, a[j]);
      } else {
#pragma unroll
        for (int l = 0; l < VW; ++l)
          if (e + l < end) y[e + l] = a[j].v[l];
      }
    }
  }
}

template <int VW>
__device__ __forceinline__ void ld_x(const float* p, Vec<VW>& o) {
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

// Rows [r0, r1) of op o, R consecutive rows per warp: a vector of x is loaded
// once for R rows, and R * U vectors of A are in flight per lane.  Per row,
// the arithmetic of the warp-per-row kernel.  Columns are counted in 32 bits
// within pieces of 2^28 (whole groups), which keeps the loop in registers.
template <int VW, int R, int U>
__device__ __forceinline__ void gemv_item(const OpDev& o, int64_t r0, int64_t r1) {
  constexpr int kStep = kWarp * VW, kPiece = 1 << 28;
  static_assert(kGemvGroup % U == 0 && kPiece % (kGemvGroup * kStep) == 0, "whole groups");
  const int lane = threadIdx.x & (kWarp - 1);
  for (int64_t row = r0 + threadIdx.x / kWarp * R; row < r1; row += kThreads / kWarp * R) {
    const int have = r1 - row < R ? (int)(r1 - row) : R;
    float y0 = 0.f;                    // of row + lane, loaded ahead of the fold
    if (o.beta != 0.f && lane < have) y0 = o.out[row + lane];
    const float* a0 = o.A + row * o.lda + lane * VW;
    const float* x = o.x + lane * VW;
    GroupedDot<VW> acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r].init();
    for (int64_t left = o.N; left > 0; left -= kPiece, a0 += kPiece, x += kPiece) {
      const int n = (left < kPiece ? (int)left : kPiece) - lane * VW;   // columns from the lane's first
      const float* a[R];
#pragma unroll
      for (int r = 0; r < R; ++r) a[r] = a0 + (r < have ? r : 0) * o.lda;
      int c = 0, k = 0;                // k: the lane's vectors of the row (mod the group)
      for (; c + (U - 1) * kStep + VW <= n; c += U * kStep) {
        Vec<VW> va[R][U], vx[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
          for (int r = 0; r < R; ++r) ld_stream(a[r] + c + u * kStep, va[r][u]);
          ld_x<VW>(x + c + u * kStep, vx[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int r = 0; r < R; ++r) acc[r].add(va[r][u], vx[u]);
        k = (k + U) & (kGemvGroup - 1);
        if (k == 0) {
#pragma unroll
          for (int r = 0; r < R; ++r) acc[r].flush();
        }
      }
      if (c < n) {                     // the last, partial step: all its loads at once
        Vec<VW> va[R][U], vx[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = c + u * kStep;
          if (e + VW <= n) {
#pragma unroll
            for (int r = 0; r < R; ++r) ld_stream(a[r] + e, va[r][u]);
            ld_x<VW>(x + e, vx[u]);
          } else {
#pragma unroll
            for (int r = 0; r < R; ++r) ld_guarded<VW>(a[r], e, n, va[r][u]);
            ld_guarded<VW>(x, e, n, vx[u]);
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int r = 0; r < R; ++r) acc[r].add(va[r][u], vx[u]);
      }
    }
    float d = 0.f;                     // row + lane's dot
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float v = __shfl_sync(0xffffffffu, warp_tree(acc[r].value()), 0);
      if (lane == r) d = v;
    }
    if (lane < have) {
      const float z = __fmul_rn(o.alpha, d);
      o.out[row + lane] = o.beta == 0.f ? z : __fadd_rn(z, __fmul_rn(o.beta, y0));
    }
  }
}

template <int OP>
__device__ float reduce_dispatch(const OpDev& o, int64_t b, int64_t e, float* red) {
  switch (o.mode) {
    case 0: return reduce_item<OP, 1, 4>(o, b, e, red);
    case 1: return reduce_item<OP, 4, 1>(o, b, e, red);
    case 2: return reduce_item<OP, 4, 2>(o, b, e, red);
    case 3: return reduce_item<OP, 4, 4>(o, b, e, red);
    case 4: return reduce_item<OP, 8, 1>(o, b, e, red);
    default: return reduce_item<OP, 8, 2>(o, b, e, red);
  }
}

// One work item; `last` and the reduction scratch are shared by the CTA.
__device__ __forceinline__ void run_item(const BatchDev& B, const ItemDev& item, const OpDev& o,
                                         float* red, double* red64, bool* last) {
  if (o.op == LIFT_OP_ASUM || o.op == LIFT_OP_DOT) {
    const float r = o.op == LIFT_OP_ASUM ? reduce_dispatch<LIFT_OP_ASUM>(o, item.begin, item.end, red)
                                         : reduce_dispatch<LIFT_OP_DOT>(o, item.begin, item.end, red);
    if (o.num_items == 1) {            // the FP64 sum of one partial is the partial
      if (threadIdx.x == 0) *o.out = __fadd_rn(0.f, r);
      return;
    }
    if (threadIdx.x == 0) {
      B.partials[item.index] = r;
      __threadfence();
      *last = atomicAdd(B.op_done + item.op_index, 1u) == (unsigned)(o.num_items - 1);
    }
    __syncthreads();
    if (*last) {
      __threadfence();
      const double s = combine_partials<kThreads>(B.partials + o.first_item, o.num_items, red64);
      if (threadIdx.x == 0) {
        *o.out = static_cast<float>(s);
        B.op_done[item.op_index] = 0u;   // ready for the next run
      }
    }
  } else if (o.op == LIFT_OP_SCAL) {
    switch (o.mode) {
      case 0: scal_item<1, 4>(o, item.begin, item.end); break;
      case 1: scal_item<4, 1>(o, item.begin, item.end); break;
      case 2: scal_item<4, 2>(o, item.begin, item.end); break;
      case 3: scal_item<4, 4>(o, item.begin, item.end); break;
      case 4: scal_item<8, 1>(o, item.begin, item.end); break;
      default: scal_item<8, 2>(o, item.begin, item.end); break;
    }
  } else {
    switch (o.mode) {
      case 0:
        if (o.N <= 8 * kWarp) gemv_item<1, 4, 4>(o, item.begin, item.end);
        else gemv_item<1, 2, 8>(o, item.begin, item.end);
        break;
      case 1:
        if (item.end - item.begin > 16) gemv_item<4, 4, 1>(o, item.begin, item.end);
        else gemv_item<4, 2, 2>(o, item.begin, item.end);
        break;
      default: gemv_item<8, 1, 2>(o, item.begin, item.end); break;
    }
  }
}

__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// QUEUE: a persistent grid whose CTAs pop queue positions with an atomic;
// otherwise one CTA per queue position (CTA q takes position q), dealt to
// the SMs by the hardware in launch order as earlier CTAs retire.
template <bool QUEUE>
__device__ __forceinline__ void batch_body(const BatchDev& B) {
  __shared__ float red[kWarp];
  __shared__ double red64[kWarp];
  __shared__ bool s_last;
  if constexpr (!QUEUE) {
    if ((int64_t)blockIdx.x >= B.num_items) return;
    const ItemDev item = B.items[blockIdx.x];
    run_item(B, item, B.ops[item.op_index], red, red64, &s_last);
  } else {
    __shared__ __align__(16) ItemDev s_item[3];     // items i, i + 1 and the slot of i + 2
    __shared__ __align__(16) OpDev s_op[2];         // their ops, i and i + 1
    const int lane = threadIdx.x & (kWarp - 1);
    const bool fetcher = threadIdx.x < kWarp;
    const unsigned long long G = gridDim.x;
    // start the copy of the item at queue position q (op_index -1 past the
    // end), and of an op; lanes 0.. and kOpChunks.. move 16 bytes each
    auto get_item = [&](int slot, unsigned long long q) {
      const int k = lane - kOpChunks;
      if (q >= (unsigned long long)B.num_items) {
        if (k == 0) s_item[slot].op_index = -1;
      } else if (k >= 0 && k < kItemChunks) {
        copy16(reinterpret_cast<char*>(s_item + slot) + 16 * k,
               reinterpret_cast<const char*>(B.items + q) + 16 * k);
      }
    };
    auto get_op = [&](int slot, int op) {
      if (op >= 0 && lane < kOpChunks)
        copy16(reinterpret_cast<char*>(s_op + slot) + 16 * lane,
               reinterpret_cast<const char*>(B.ops + op) + 16 * lane);
    };
    unsigned long long q = 0;                       // queue position of item i + 2 (lane 0's)
    if (fetcher) {
      get_item(0, blockIdx.x);
      get_item(1, blockIdx.x + G);
      q = blockIdx.x + 2 * G;
      copy_wait();
      __syncwarp();
      get_op(0, s_item[0].op_index);
      copy_wait();
    }
    __syncthreads();
    for (int i = 0, i3 = 0; s_item[i3].op_index >= 0; i ^= 1, i3 = i3 == 2 ? 0 : i3 + 1) {
      if (fetcher) {
        get_op(i ^ 1, s_item[i3 == 2 ? 0 : i3 + 1].op_index);
        get_item(i3 == 0 ? 2 : i3 - 1, __shfl_sync(0xffffffffu, q, 0));
        if (lane == 0) q = atomicAdd(B.head, 1ull) + 3 * G;
      }
      run_item(B, s_item[i3], s_op[i], red, red64, &s_last);
      if (fetcher) copy_wait();
      __syncthreads();   // shared state is reused by the next item
    }
    // the last CTA to leave returns the queue to its start
    if (threadIdx.x == 0) {
      __threadfence();
      if (atomicAdd(B.head + 1, 1ull) == G - 1) {
        __threadfence();
        B.head[0] = 0ull;
        B.head[1] = 0ull;
      }
    }
  }
}

// 4 CTAs per SM (64 registers).  With the rows of gemv items loaded one at a
// time a batch with gemv ops wanted 5 (48 registers); several rows per warp
// have more loads in flight on fewer warps, and spill at 48 (2000 ops: 887 us
// against 866).
template <bool QUEUE>
__global__ void __launch_bounds__(kThreads, 4) batch_kernel(BatchDev B) {
  batch_body<QUEUE>(B);
}

}  // namespace
}  // namespace lift

struct lift_batch {
  int device = -1;
  int64_t count = 0, num_items = 0, bytes = 0;
  std::vector<lift::OpDev> ops_host;
  std::vector<int> mode;      // per op: the mode used
  std::vector<int> variant;   // per op: the policy's variant choice
  std::vector<int64_t> item;  // per op: elements (or rows) per work item
  lift::OpDev* ops = nullptr;
  lift::ItemDev* items = nullptr;
  float* partials = nullptr;
  unsigned* op_done = nullptr;
  unsigned long long* head = nullptr;
  int64_t grid = 0;           // CTAs of the persistent (queue) grid
  int schedule = LIFT_BATCH_QUEUE;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
};

using namespace lift;

namespace lift {
namespace {

int vec_mode_for(const lift_variant_info& v) {
  for (int m = 0; m < kNumVecModes; ++m)
    if (kThreads * kVecModes[m].vw * kVecModes[m].j == v.tile && kVecModes[m].vw == v.vw) return m;
  if (v.vw == 1) return 0;
  if (v.vw == 4) return v.tile >= 4096 ? 3 : (v.tile >= 2048 ? 2 : 1);
  return v.tile >= 4096 ? 5 : 4;
}

void free_batch(lift_batch* b) {
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  cudaFree(b->ops);
  cudaFree(b->items);
  cudaFree(b->partials);
  cudaFree(b->op_done);
  cudaFree(b->head);
  delete b;
}

int64_t op_bytes(const lift_op_desc& d) {
  switch (d.op) {
    case LIFT_OP_ASUM: return 4 * d.n;
    case LIFT_OP_DOT: return 8 * d.n;
    case LIFT_OP_SCAL: return 8 * d.n;
    default: return 4 * d.M * d.N + 4 * d.N + (d.beta != 0.f ? 8 : 4) * d.M;
  }
}

}  // namespace
}  // namespace lift

extern "C" {

lift_status lift_batch_create(const lift_op_desc* descs, int64_t count, lift_batch** out) {
  if (!out || count < 0 || (count > 0 && !descs))
    return set_error(LIFT_ERR_INVALID_ARG, "batch_create arguments");
  *out = nullptr;
  // validate everything before touching the device
  for (int64_t i = 0; i < count; ++i) {
    const lift_op_desc& d = descs[i];
    const std::string at = "batch op " + std::to_string(i) + ": ";
    if (d.op != LIFT_OP_ASUM && d.op != LIFT_OP_DOT && d.op != LIFT_OP_SCAL && d.op != LIFT_OP_GEMV)
      return set_error(LIFT_ERR_INVALID_ARG, at + "op id out of range");
    if (d.variant < -1 || d.variant >= (int)registry(d.op).size())
      return set_error(LIFT_ERR_INVALID_ARG, at + "variant id out of range");
    if (!d.out) return set_error(LIFT_ERR_INVALID_ARG, at + "out is NULL");
    if (d.op == LIFT_OP_GEMV) {
      if (d.M < 0 || d.N < 0 || d.lda < d.N) return set_error(LIFT_ERR_INVALID_ARG, at + "gemv sizes");
      if (d.M > 0 && d.N > 0 && (!d.A || !d.x)) return set_error(LIFT_ERR_INVALID_ARG, at + "gemv A/x");
    } else {
      if (d.n < 0) return set_error(LIFT_ERR_INVALID_ARG, at + "n < 0");
      if (d.n > 0 && !d.x) return set_error(LIFT_ERR_INVALID_ARG, at + "x is NULL");
      if (d.op == LIFT_OP_DOT && d.n > 0 && !d.y) return set_error(LIFT_ERR_INVALID_ARG, at + "y is NULL");
    }
    const void* ptrs[] = {d.x, d.y, d.A, d.out};
    for (const void* p : ptrs)
      if (p && !aligned(p, 4)) return set_error(LIFT_ERR_INVALID_ARG, at + "pointer not 4-byte aligned");
  }
  DeviceState* st = current_state();
  if (!st) return set_error(LIFT_ERR_NOT_INITIALIZED, "lift_init was not called for this device");
  lift_batch* b = new lift_batch();
  cudaGetDevice(&b->device);
  b->count = count;
  b->ops_host.resize(count);
  b->mode.resize(count);
  b->variant.resize(count);
  b->item.resize(count);
  std::vector<ItemDev> items;
  std::vector<std::pair<int64_t, int64_t>> cost;   // (bytes, item) for the queue order
  int per_sm = 0;
  lift_status rc = cuda_check(
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_kernel<true>, kThreads, 0),
      "batch occupancy");
  if (rc != LIFT_OK) {
    delete b;
    return rc;
  }
  b->grid = (int64_t)per_sm * st->sm_count;
  int64_t total = 0;
  for (int64_t i = 0; i < count; ++i) total += op_bytes(descs[i]);
  const int64_t item_bytes = std::min(
      kItemBytesMax, std::max(kItemBytesMin, total / (std::max<int64_t>(1, b->grid) * kItemsPerCta)));
  for (int64_t i = 0; i < count; ++i) {
    const lift_op_desc& d = descs[i];
    OpDev o{};
    o.op = d.op;
    o.n = d.n;
    o.M = d.M;
    o.N = d.N;
    o.lda = d.lda;
    o.alpha = d.alpha;
    o.beta = d.beta;
    o.x = d.x;
    o.y = d.y;
    o.A = d.A;
    o.out = d.out;
    int v = d.variant;
    if (v < 0) v = batch_pick(d.op, d.n, d.M, d.N);
    b->variant[i] = v;
    const lift_variant_info& info = registry(d.op)[v].info;
    o.first_item = (int64_t)items.size();
    if (d.op == LIFT_OP_GEMV) {
      int m = info.vw == 8 ? 2 : (info.vw == 4 ? 1 : 0);
      const int vw = kGemvVW[m];
      if (!aligned(d.A, 4 * vw) || !aligned(d.x, 4 * vw) || (d.lda * 4) % (4 * vw) != 0) m = 0;
      o.mode = m;
      const int64_t row_bytes = 4 * (d.N > 0 ? d.N : 1);
      int64_t rows = std::max<int64_t>(16, item_bytes / row_bytes / 16 * 16);
      b->item[i] = rows;
      for (int64_t r = 0; r < d.M; r += rows) {
        const int64_t e = std::min(d.M, r + rows);
        cost.push_back({(e - r) * row_bytes, (int64_t)items.size()});
        items.push_back({(int)i, 0, (int64_t)items.size(), r, e});
      }
    } else {
      int m = vec_mode_for(info);
      const int vw = kVecModes[m].vw;
      const bool ok = aligned(d.x, 4 * vw) && (d.op != LIFT_OP_DOT || aligned(d.y, 4 * vw)) &&
                      (d.op != LIFT_OP_SCAL || aligned(d.out, 4 * vw));
      if (!ok) m = 0;
      o.mode = m;
      const int64_t tile = (int64_t)kThreads * kVecModes[m].vw * kVecModes[m].j;
      const int64_t esz = d.op == LIFT_OP_ASUM ? 4 : 8;
      const int64_t per = std::max<int64_t>(1, item_bytes / (tile * esz)) * tile;
      b->item[i] = per;
      if (d.n == 0 && d.op != LIFT_OP_SCAL) {
        cost.push_back({0, (int64_t)items.size()});
        items.push_back({(int)i, 0, (int64_t)items.size(), 0, 0});   // one empty item: the combine writes 0
      }
      for (int64_t s = 0; s < d.n; s += per) {
        const int64_t e = std::min(d.n, s + per);
        cost.push_back({(e - s) * esz, (int64_t)items.size()});
        items.push_back({(int)i, 0, (int64_t)items.size(), s, e});
      }
    }
    o.num_items = (int64_t)items.size() - o.first_item;
    b->mode[i] = o.mode;
    b->ops_host[i] = o;
    b->bytes += op_bytes(d);
  }
  b->num_items = (int64_t)items.size();
  std::stable_sort(cost.begin(), cost.end(),
                   [](const std::pair<int64_t, int64_t>& a, const std::pair<int64_t, int64_t>& c) {
                     return a.first > c.first;
                   });
  std::vector<ItemDev> queue(items.size());
  for (size_t k = 0; k < cost.size(); ++k) queue[k] = items[cost[k].second];
  if (b->grid > b->num_items) b->grid = std::max<int64_t>(1, b->num_items);

  const size_t ni = std::max<size_t>(1, items.size()), no = std::max<int64_t>(1, count);
  rc = cuda_check(cudaMalloc(&b->ops, no * sizeof(OpDev)), "batch alloc");
  if (rc == LIFT_OK) rc = cuda_check(cudaMalloc(&b->items, ni * sizeof(ItemDev)), "batch alloc");
  if (rc == LIFT_OK) rc = cuda_check(cudaMalloc(&b->partials, ni * sizeof(float)), "batch alloc");
  if (rc == LIFT_OK) rc = cuda_check(cudaMalloc(&b->op_done, no * sizeof(unsigned)), "batch alloc");
  if (rc == LIFT_OK) rc = cuda_check(cudaMalloc(&b->head, 2 * sizeof(unsigned long long)), "batch alloc");
  if (rc == LIFT_OK) rc = cuda_check(cudaMemset(b->op_done, 0, no * sizeof(unsigned)), "batch init");
  if (rc == LIFT_OK)
    rc = cuda_check(cudaMemset(b->head, 0, 2 * sizeof(unsigned long long)), "batch init");
  if (rc == LIFT_OK && count > 0)
    rc = cuda_check(cudaMemcpy(b->ops, b->ops_host.data(), count * sizeof(OpDev), cudaMemcpyHostToDevice),
                    "batch upload");
  if (rc == LIFT_OK && !items.empty())
    rc = cuda_check(cudaMemcpy(b->items, queue.data(), queue.size() * sizeof(ItemDev),
                               cudaMemcpyHostToDevice), "batch upload");
  if (rc != LIFT_OK) {
    free_batch(b);
    return rc;
  }
  *out = b;
  return LIFT_OK;
}

// The graph: batch_kernel, captured once on a private stream, then launched
// on the caller's stream.
lift_status lift_batch_run(lift_batch* b, void* stream) {
  if (!b) return set_error(LIFT_ERR_INVALID_ARG, "batch is NULL");
  if (b->num_items == 0) return LIFT_OK;
  if (!b->exec) {
    cudaStream_t cap;
    lift_status rc = cuda_check(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking), "stream");
    if (rc != LIFT_OK) return rc;
    rc = cuda_check(cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal), "capture");
    if (rc == LIFT_OK) {
      BatchDev B{b->ops, b->items, b->partials, b->op_done, b->head, b->num_items};
      const bool q = b->schedule == LIFT_BATCH_QUEUE;
      const unsigned g = (unsigned)(q ? b->grid : b->num_items);
      if (q) batch_kernel<true><<<g, kThreads, 0, cap>>>(B);
      else batch_kernel<false><<<g, kThreads, 0, cap>>>(B);
      rc = cuda_check(cudaStreamEndCapture(cap, &b->graph), "end capture");
    }
    if (rc == LIFT_OK) rc = cuda_check(cudaGraphInstantiate(&b->exec, b->graph, 0), "instantiate");
    cudaStreamDestroy(cap);
    if (rc != LIFT_OK) return rc;
  }
  return cuda_check(cudaGraphLaunch(b->exec, static_cast<cudaStream_t>(stream)), "graph launch");
}

lift_status lift_batch_set_schedule(lift_batch* b, int schedule) {
  if (!b) return set_error(LIFT_ERR_INVALID_ARG, "batch is NULL");
  if (schedule != LIFT_BATCH_QUEUE && schedule != LIFT_BATCH_PER_ITEM)
    return set_error(LIFT_ERR_INVALID_ARG, "batch schedule");
  if (schedule == LIFT_BATCH_PER_ITEM && b->num_items > INT32_MAX)
    return set_error(LIFT_ERR_UNSUPPORTED, "more work items than CTAs in a grid");
  if (schedule == b->schedule) return LIFT_OK;
  // the next run captures the graph again; a launch of the old one may still
  // be in flight on some stream, so let the device drain first
  if (b->exec) cudaDeviceSynchronize();
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  b->exec = nullptr;
  b->graph = nullptr;
  b->schedule = schedule;
  return LIFT_OK;
}

int lift_batch_schedule(const lift_batch* b) { return b ? b->schedule : -1; }

lift_status lift_batch_info(const lift_batch* b, int64_t* items, int64_t* bytes, int64_t* grid) {
  if (!b) return set_error(LIFT_ERR_INVALID_ARG, "batch is NULL");
  if (items) *items = b->num_items;
  if (bytes) *bytes = b->bytes;
  if (grid) *grid = b->schedule == LIFT_BATCH_QUEUE ? b->grid : b->num_items;
  return LIFT_OK;
}

lift_status lift_batch_op_choice(const lift_batch* b, int64_t i, int* variant, int* mode,
                                 int64_t* item) {
  if (!b || i < 0 || i >= b->count) return set_error(LIFT_ERR_INVALID_ARG, "batch op index");
  if (variant) *variant = b->variant[i];
  if (mode) *mode = b->mode[i];
  if (item) *item = b->item[i];
  return LIFT_OK;
}

lift_status lift_batch_destroy(lift_batch* b) {
  if (!b) return LIFT_OK;
  cudaDeviceSynchronize();
  free_batch(b);
  return LIFT_OK;
}

}  // extern "C"
