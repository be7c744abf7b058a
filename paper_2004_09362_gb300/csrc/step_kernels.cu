// Step-faithful mode: one kernel launch per communication step of the schedule.
//
// A launch applies the step's block ops (plan.cpp) for every rank x at once.  An op
// names a placement; rank x works on block b = (x - dst_place) mod P, which is the same
// block index at the partner (a move by t^{l} changes a vector's placement, never its
// block index; eq. comm_op_0).  "Sending" is a coalesced 16-byte vector read of the
// partner rank's block; the read value is combined in registers with the own block
// (eq. distr_vectors_combination) and stored.  Every CTA owns one chunk of one block
// of one (op, rank) pair (short blocks: one thread per element and one to four ops).
// Combine ops batch 2 vectors per thread; same-type copies move raw 16-byte units, 6 per
// thread; a bf16 plan's first step keeps its 16-byte bf16 loads packed until the
// combine.  Every thread counts the bytes it reads from partners and the kernels add them to
// the step's counter slots, so the bytes a step actually moved are recorded.  The launches of one Allreduce
// are chained by programmatic dependent launch.  The same work functions serve the
// per-step launches, the persistent kernel and the no-allocation launches.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <string>
#include <type_traits>

#include "gar_internal.hpp"

namespace gar {

// SM count of the current device (cached per device ordinal).
int num_sms() {
  static int cache[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) {
    cudaGetLastError();
    dev = 0;
  }
  if (dev < 64 && cache[dev] > 0) return cache[dev];
  int v = 0;
  if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) {
    cudaGetLastError();
    v = 1;
  }
  if (dev < 64) cache[dev] = v;
  return v;
}

namespace {

// Launch shape, from sweeps on GB300: CTAs own 16384-element chunks of large vectors
// (smaller chunks ran up to 2.5x slower) and each thread issues the loads of 2 vectors
// before combining.  Launches of fewer than 4 CTAs per SM halve the chunk, down to one
// batch of loads per thread (P = 20 x 1 MiB fp32 S = 9 without allocation: 34 us at 2048
// elements, 36 at 4096 and 1024).
constexpr int kThreads = 256;
constexpr uint64_t kChunk = 16384;      // largest chunk (elements per CTA)
constexpr uint64_t kMinChunk = 2048;    // smallest chunk
constexpr uint64_t kMinCtas = 4;        // CTAs per SM below which the chunk is halved
constexpr int kUnroll = 2;              // 4-element vectors a thread loads at once
constexpr uint64_t kFlatBelow = 4 * kThreads * kUnroll;  // blocks shorter than this: element-major
// Element-major launches: threads per SM before a thread takes 2 or 4 ops instead of one.
// P = 127 x 9 KiB bf16 S = 10: 44.5 us with one op per thread throughout (and the next
// launch at the end); 33.3 us at 512
// threads, 36.8 at 256, 35.7 at 1024, 41.8 at 2048 (43.5 with up to 8 ops per thread).
// No-allocation launches are element-major only for blocks of fewer than 512 elements, or in
// all fewer than 2^18 elements (ops * n): a longer launch is bound by its 4-byte accesses.
// GB300, us a call in graph replay, fp32, element-major -> chunked: P = 64 blocks of 1200
// elements S = 6 165 -> 80, S = 12 57 -> 42, blocks of 800 S = 6 113 -> 76, P = 20 x 2000 S = 5
// 33 -> 17; but P = 64 x 500 S = 6 75 -> 72, x 160 33 -> 70, P = 5 x 2000 S = 3 5.6 -> 7.3.
constexpr uint64_t kNoAllocFlatBlock = 512;
constexpr uint64_t kNoAllocFlatItems = 1u << 18;
constexpr int kFlatGroup = 4;
constexpr uint64_t kFlatThreads = 512;
// Persistent steps: smallest piece of a block, and most pieces (see launch_desc).  The chunked
// steps run in CTAs of 256 threads, 2 per SM without spills, or 3, whose warps hide more of the
// loads' latency, where the largest step has 2^22 elements (ops * n) or more (2^24 in bf16
// plans of one or two result copies, whose code spills at 3), or, with more than two copies,
// more than 4 blocks (P * ops) per SM.  GB300, us call after call, 2 per SM -> 3
// (before: 3 per SM, every step cut into 16384 elements): P = 24 x 4 MiB int32 max S = 10 96 ->
// 93 (134), P = 18 x 1.8M fp32 S = 5 409 -> 333 (387), P = 64 x 851000 int32 S = 6 697 -> 586
// (604), P = 18 x 38000 S = 5 31 -> 27 (32), P = 13 x 1.6M bf16 S = 4 279 -> 243 (258); but
// P = 17 x 77000 fp32 S = 5 27 -> 29 (45), P = 12 x 160000 int32 S = 8 29 -> 33 (40), P = 33 x
// 69000 fp32 S = 11 41 -> 45 (57), P = 24 x 960000 bf16 S = 10 75 -> 79 (151).
constexpr int kPersistThreads = 256;
constexpr uint64_t kMinPiece = 2048;
constexpr uint64_t kMostPieces = 24;

// Counter upkeep of one launch, by its first CTA (after wait_prior_grid): zeroes the
// counters of the communication step that follows, and moves the first step's counts,
// which were added to a row of their own, to their place.  So every step's counters are
// zero when its launch starts, without a memset in the launch sequence.
struct CounterUpkeep {
  unsigned long long *zero;                // row to zero, or nullptr
  unsigned long long *move_from, *move_to; // row to move (and zero), or nullptr
};

template <int MAXP>
struct StepArgs {
  void *rank[MAXP];
  void *ws[NUM_WS_BUFS];             // QP0, QP1, QS slice bases (nullptr if unused)
  const StepOp *ops;                 // this launch's ops
  unsigned long long *bytes;         // the step's row of counters, or nullptr
  uint64_t q, rem, n_pad;
  uint64_t n;                        // elements per rank
  uint32_t chunk;                    // elements per CTA
  int P, partner, nops, nchunks;
  int group;                         // ops per thread (element-major mapping)
  int xor_group;                     // 1: placements and partners combine by XOR (Table 1b)
  int early;                         // 1: the next launch is this call's (element-major: it may start at once)
  // 1: work items in descending order.  Every second launch runs so, and then first reads
  // what its predecessor wrote last, which L2 still holds (P = 127 x 8 MiB bf16 S = 14:
  // 1114 us instead of 1132).
  int reverse;
  CounterUpkeep upkeep;
};

template <typename T> struct AccOf { using type = T; };
template <> struct AccOf<__nv_bfloat16> { using type = float; };

__device__ __forceinline__ float widen(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ float widen(float x) { return x; }
__device__ __forceinline__ int widen(int x) { return x; }
__device__ __forceinline__ void narrow(float x, __nv_bfloat16 *o) { *o = __float2bfloat16_rn(x); }
__device__ __forceinline__ void narrow(float x, float *o) { *o = x; }
__device__ __forceinline__ void narrow(int x, int *o) { *o = x; }

template <int OP> __device__ __forceinline__ float combine(float a, float b) {
  if (OP == GAR_SUM) return a + b;
  if (OP == GAR_MAX) return fmaxf(a, b);
  return fminf(a, b);
}
template <int OP> __device__ __forceinline__ int combine(int a, int b) {
  if (OP == GAR_SUM) return (int)((unsigned)a + (unsigned)b);
  if (OP == GAR_MAX) return a > b ? a : b;
  return a < b ? a : b;
}

// One element / four aligned elements of buffer `buf` (rank buffers hold T, workspace
// slices hold the accumulation type A).
template <typename T, typename A>
__device__ __forceinline__ A load1(uint8_t buf, const void *base, uint64_t e) {
  if (buf == BUF_RANK) return widen(static_cast<const T *>(base)[e]);
  return static_cast<const A *>(base)[e];
}

template <typename T, typename A>
__device__ __forceinline__ void load4(uint8_t buf, const void *base, uint64_t e, A (&v)[4]) {
  if (buf == BUF_RANK && sizeof(T) == 2) {
    const uint2 u = *reinterpret_cast<const uint2 *>(static_cast<const T *>(base) + e);
    v[0] = (A)__uint_as_float(u.x << 16);
    v[1] = (A)__uint_as_float(u.x & 0xffff0000u);
    v[2] = (A)__uint_as_float(u.y << 16);
    v[3] = (A)__uint_as_float(u.y & 0xffff0000u);
  } else {
    const A *p = (buf == BUF_RANK) ? reinterpret_cast<const A *>(static_cast<const T *>(base))
                                   : static_cast<const A *>(base);
    const int4 u = *reinterpret_cast<const int4 *>(p + e);
    v[0] = *reinterpret_cast<const A *>(&u.x);
    v[1] = *reinterpret_cast<const A *>(&u.y);
    v[2] = *reinterpret_cast<const A *>(&u.z);
    v[3] = *reinterpret_cast<const A *>(&u.w);
  }
}

template <typename T, typename A>
__device__ __forceinline__ void store1(uint8_t buf, void *base, uint64_t e, A v) {
  if (buf == BUF_RANK)
    narrow(v, static_cast<T *>(base) + e);
  else
    static_cast<A *>(base)[e] = v;
}

template <typename T, typename A>
__device__ __forceinline__ void store4(uint8_t buf, void *base, uint64_t e, const A (&v)[4]) {
  if (buf == BUF_RANK && sizeof(T) == 2) {
    __nv_bfloat16 h[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) narrow(v[k], &h[k]);
    uint2 u;
    u.x = (uint32_t)__bfloat16_as_ushort(h[0]) | ((uint32_t)__bfloat16_as_ushort(h[1]) << 16);
    u.y = (uint32_t)__bfloat16_as_ushort(h[2]) | ((uint32_t)__bfloat16_as_ushort(h[3]) << 16);
    *reinterpret_cast<uint2 *>(static_cast<T *>(base) + e) = u;
  } else {
    A *p = (buf == BUF_RANK) ? reinterpret_cast<A *>(static_cast<T *>(base)) : static_cast<A *>(base);
    int4 u;
    u.x = *reinterpret_cast<const int *>(&v[0]);
    u.y = *reinterpret_cast<const int *>(&v[1]);
    u.z = *reinterpret_cast<const int *>(&v[2]);
    u.w = *reinterpret_cast<const int *>(&v[3]);
    *reinterpret_cast<int4 *>(p + e) = u;
  }
}

template <typename A, int MAXP>
__device__ __forceinline__ void *buf_ptr(const StepArgs<MAXP> &a, uint8_t buf, int rank) {
  if (buf == BUF_RANK) return a.rank[rank];
  if (buf == BUF_NONE) return nullptr;
  return static_cast<char *>(a.ws[buf - BUF_QP0]) + (uint64_t)rank * a.n_pad * sizeof(A);
}

// v mod P for v in (-P, 2P).
__device__ __forceinline__ int wrap_rank(int v, int P) { return v < 0 ? v + P : (v >= P ? v - P : v); }

// Programmatic dependent launch: the step launches of one Allreduce are made with
// programmatic stream serialisation, so launch i+1's CTAs may become resident while
// launch i drains.  griddepcontrol.wait blocks until every prerequisite grid has
// completed and its memory is visible (a no-op without such a dependency); nothing but
// the kernel's parameters and the plan's op table, which never changes, is read before
// it.  launch_dependents lets the next launch start once every CTA of this one has issued
// it or exited.  Chunked launches issue it when their work is done: at the start, the
// waiting CTAs took slots from the running ones' (P = 127 x 8 MiB bf16 S = 14 1122 us
// instead of 1112, P = 20 x 1 MiB fp32 S = 9 without allocation 37.6 instead of 34.3).
// Element-major launches, whose CTAs are few and short, issue it at the start (P = 127 x
// 9 KiB bf16 S = 10 34.0 instead of 36.4), but for a call's last launch, whose successor
// is not ours.
__device__ __forceinline__ void wait_prior_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void allow_next_grid() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Per-launch parameters the work functions need besides the buffers.
struct LaunchView {
  const StepOp *ops;
  unsigned long long *bytes;  // the communication step's row of counters, or nullptr
  uint32_t chunk;             // elements per CTA item (chunked mapping)
  int nops, partner, nchunks;
  int group;                  // ops per thread (element-major mapping)
};

// Adds the bytes that a warp's threads have read from partners to a step's counters.
__device__ __forceinline__ void count_moved(unsigned long long *bytes, uint32_t moved) {
  if (bytes == nullptr) return;
  const uint32_t sum = __reduce_add_sync(0xffffffffu, moved);
  if ((threadIdx.x & 31) == 0 && sum)
    atomicAdd(bytes + (blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)) % STEP_BYTE_SLOTS * STEP_SLOT_STRIDE,
              (unsigned long long)sum);
}

// The same by one add of a CTA of NT threads (persistent kernel): every thread stages its
// count, and after a barrier one thread adds the sums of the warps.
template <int NT>
__device__ __forceinline__ void stage_moved(uint32_t *s_moved, uint32_t moved) {
  const uint32_t sum = __reduce_add_sync(0xffffffffu, moved);
  if ((threadIdx.x & 31) == 0) s_moved[threadIdx.x >> 5] = sum;
}
template <int NT>
__device__ __forceinline__ void add_moved(unsigned long long *bytes, const uint32_t *s_moved) {
  unsigned long long total = 0;
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) total += s_moved[w];
  if (total) atomicAdd(bytes + blockIdx.x % STEP_BYTE_SLOTS * STEP_SLOT_STRIDE, total);
}

// Elements [c0, c0 + len) of the block that op `op` touches at rank x, by the CTA's NT
// threads; returns the bytes that this thread has read from the partner.
template <typename T, int OP, int MAXP, int NT>
__device__ __forceinline__ uint32_t range_work(const StepArgs<MAXP> &a, const LaunchView &lv, const StepOp &op, int x,
                                           uint64_t c0, uint32_t len) {
  using A = typename AccOf<T>::type;
  constexpr bool kMixed = sizeof(T) != sizeof(A);  // rank buffers hold a narrower type than the slices
  // placements and ranks are in [0, P), partner offsets in (-P, P)
  const int b = a.xor_group ? (x ^ (int)op.dst_place) : wrap_rank(x - (int)op.dst_place, a.P);
  const uint64_t bstart = (uint64_t)b * a.q + ((uint64_t)b < a.rem ? (uint64_t)b : a.rem);
  const uint64_t blen = a.q + ((uint64_t)b < a.rem ? 1 : 0);
  if (c0 >= blen) return 0;
  const uint64_t lo = bstart + c0;
  const uint64_t hi = bstart + (blen < c0 + len ? blen : c0 + len);

  const bool has_recv = op.recv_place >= 0;
  const int partner = a.xor_group ? (x ^ lv.partner) : wrap_rank(x + lv.partner, a.P);
  const void *recv = has_recv ? buf_ptr<A>(a, op.recv_buf, partner) : nullptr;
  void *out0 = buf_ptr<A>(a, op.out0_buf, x);
  const void *own0 = buf_ptr<A>(a, op.out0_own, x);
  void *out1 = buf_ptr<A>(a, op.out1_buf, x);
  const void *own1 = buf_ptr<A>(a, op.out1_own, x);
  // An op with one source and one output is a copy (distribution steps, q* moves); between
  // buffers of one element type it moves raw 16-byte units (4 fp32 or 8 bf16 elements).
  const bool copy_only = !out1 && (has_recv != (own0 != nullptr));
  const uint8_t src_buf = has_recv ? op.recv_buf : op.out0_own;
  const bool raw = copy_only && (!kMixed || src_buf == op.out0_buf);
  // bf16 partner block + bf16 own block -> fp32 partial (the first reduction step of a
  // bf16 plan)
  const bool packed = kMixed && has_recv && !out1 && own0 != nullptr && op.recv_buf == BUF_RANK &&
                      op.out0_own == BUF_RANK && op.out0_buf != BUF_RANK;

  // Element offsets are the same in every buffer, and every buffer base is 16-byte
  // aligned, so one head/body/tail split serves all operands: `unit` elements per vector,
  // fewer than one unit at either end.
  const uint32_t unit = (kMixed && raw && src_buf == BUF_RANK) ? 8 : 4;
  uint64_t va = (lo + unit - 1) & ~(uint64_t)(unit - 1), vb = hi & ~(uint64_t)(unit - 1);
  if (va > hi) va = hi;
  if (vb < va) vb = va;
  const uint32_t head = (uint32_t)(va - lo), ends = head + (uint32_t)(hi - vb);
  uint32_t moved = 0;  // elements read, partner's or (without one) own
  for (uint32_t k = threadIdx.x; k < ends; k += NT) {
    const uint64_t e = k < head ? lo + k : vb + (k - head);
    A r = A(0);
    if (has_recv) r = load1<T, A>(op.recv_buf, recv, e);
    ++moved;
    A o0 = r, o1 = r;
    if (own0) o0 = load1<T, A>(op.out0_own, own0, e);
    if (own0 && has_recv) o0 = combine<OP>(o0, r);
    if (own1) o1 = load1<T, A>(op.out1_own, own1, e);
    if (own1 && has_recv) o1 = combine<OP>(o1, r);
    store1<T, A>(op.out0_buf, out0, e, o0);
    if (out1) store1<T, A>(op.out1_buf, out1, e, o1);
  }
  const uint32_t units = (uint32_t)((vb - va) / unit);
  if (raw) {
    // 6 units per thread in flight within the 40-register budget.  bf16 copies of 8-byte
    // units ran at about 4 TB/s (48 bytes in flight per thread) against 6.6 TB/s for fp32.
    constexpr int U = 6;
    const uint64_t off = va * (src_buf == BUF_RANK ? sizeof(T) : sizeof(A));
    const int4 *src = reinterpret_cast<const int4 *>(static_cast<const char *>(has_recv ? recv : own0) + off);
    int4 *dst = reinterpret_cast<int4 *>(static_cast<char *>(out0) + off);
    for (uint32_t k = threadIdx.x; k < units; k += U * NT) {
      int4 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k + u * NT < units) {
          v[u] = src[k + u * NT];
          moved += unit;
        }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k + u * NT < units) dst[k + u * NT] = v[u];
    }
  } else if (packed) {
    // Each lane reads 4 bf16 (8 bytes) of both operands and writes their 4 fp32 partials as
    // one 16-byte store, so every warp store covers 512 contiguous bytes.  Reading 8 bf16
    // per lane instead made each 16-byte store half of a 32-byte stretch, a warp store then
    // half-filled 32 sectors, and the step ran at 74 % of DRAM throughput (P = 127 x 8 MiB
    // bf16: whole Allreduce S = 14 1.190 -> 1.164 ms, S = 10 2.323 -> 2.288 ms).  4 units
    // per thread keep 64 bytes of loads in flight.
    constexpr int U = 4;
    const uint2 *rp = reinterpret_cast<const uint2 *>(static_cast<const T *>(recv) + va);
    const uint2 *wp = reinterpret_cast<const uint2 *>(static_cast<const T *>(own0) + va);
    float4 *dp = reinterpret_cast<float4 *>(static_cast<A *>(out0) + va);
    for (uint32_t k = threadIdx.x; k < units; k += U * NT) {
      uint2 rv[U], ov[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k + u * NT < units) {
          rv[u] = rp[k + u * NT];
          moved += 4;
          ov[u] = wp[k + u * NT];
        }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k + u * NT < units) {
          float4 f;
          f.x = combine<OP>(__uint_as_float(ov[u].x << 16), __uint_as_float(rv[u].x << 16));
          f.y = combine<OP>(__uint_as_float(ov[u].x & 0xffff0000u), __uint_as_float(rv[u].x & 0xffff0000u));
          f.z = combine<OP>(__uint_as_float(ov[u].y << 16), __uint_as_float(rv[u].y << 16));
          f.w = combine<OP>(__uint_as_float(ov[u].y & 0xffff0000u), __uint_as_float(rv[u].y & 0xffff0000u));
          dp[k + u * NT] = f;
        }
    }
  } else {
    // kUnroll aligned 4-element vectors per thread: every load of the batch is issued
    // before the first combine, so a thread keeps up to 3 * kUnroll 16-byte loads in flight.
    for (uint32_t k = threadIdx.x; k < units; k += kUnroll * NT) {
      A r[kUnroll][4], o0[kUnroll][4], o1[kUnroll][4];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u)
        if (k + u * NT < units) {
          const uint64_t e = va + 4 * (uint64_t)(k + u * NT);
          if (has_recv) load4<T, A>(op.recv_buf, recv, e, r[u]);
          moved += 4;
          if (own0) load4<T, A>(op.out0_own, own0, e, o0[u]);
          if (own1) load4<T, A>(op.out1_own, own1, e, o1[u]);
        }
#pragma unroll
      for (int u = 0; u < kUnroll; ++u)
        if (k + u * NT < units) {
          const uint64_t e = va + 4 * (uint64_t)(k + u * NT);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            o0[u][c] = own0 ? (has_recv ? combine<OP>(o0[u][c], r[u][c]) : o0[u][c]) : r[u][c];
            if (out1) o1[u][c] = own1 ? (has_recv ? combine<OP>(o1[u][c], r[u][c]) : o1[u][c]) : r[u][c];
          }
          store4<T, A>(op.out0_buf, out0, e, o0[u]);
          if (out1) store4<T, A>(op.out1_buf, out1, e, o1[u]);
        }
    }
  }
  return has_recv ? moved * (uint32_t)(op.recv_buf == BUF_RANK ? sizeof(T) : sizeof(A)) : 0;
}

// Chunked mapping: work item `item` = (chunk, rank x, op) is done by the whole CTA; returns
// the bytes that this thread has read from the partner.
template <typename T, int OP, int MAXP>
__device__ __forceinline__ uint32_t chunk_work(const StepArgs<MAXP> &a, const LaunchView &lv, uint32_t item) {
  const int chunk = (int)(item % (uint32_t)lv.nchunks);
  item /= (uint32_t)lv.nchunks;
  const StepOp op = lv.ops[item / (uint32_t)a.P];
  return range_work<T, OP, MAXP, kThreads>(a, lv, op, (int)(item % (uint32_t)a.P), (uint64_t)chunk * lv.chunk, lv.chunk);
}

// Element-major mapping, for small blocks: an op touches block b = (x - dst_place) mod P
// at every rank x, i.e. every element position exactly once across the P ranks, so
// work item g = (op group, element e) maps to rank x = (b(e) + dst_place) mod P.  One
// thread per item keeps every thread busy however short the blocks are; an item is
// `group` (1, 2 or 4) consecutive ops, which share the position's block index and keep
// their loads in flight together.  `ranks`: the rank pointers in shared memory, because
// the lanes of a warp work on several blocks, so on several ranks.  The ops are read
// before wait_prior_grid (they never change), the buffers after it.
template <typename T, int OP, int MAXP>
__device__ __forceinline__ void flat_work(const StepArgs<MAXP> &a, const LaunchView &lv, void *const *ranks,
                                          uint64_t g_first, uint64_t g_stride) {
  using A = typename AccOf<T>::type;
  const uint64_t groups = (uint64_t)((lv.nops + lv.group - 1) / lv.group);
  const uint64_t total = groups * a.n;
  const uint64_t big = a.rem * (a.q + 1);
  uint32_t moved = 0;
  // 32-bit index arithmetic when every index fits (the element-major launch serves
  // short blocks, so practically always): 64-bit division is a long software sequence.
  const bool narrow_idx = total + g_stride <= 0xffffffffull;
  auto slot = [&](uint8_t buf, int rank) -> char * {
    if (buf == BUF_RANK) return static_cast<char *>(ranks[rank]);
    return static_cast<char *>(a.ws[buf - BUF_QP0]) + (uint64_t)rank * a.n_pad * sizeof(A);
  };
  for (uint64_t g = g_first; g < total; g += g_stride) {
    int gi, b;
    uint64_t e;
    if (narrow_idx) {
      const uint32_t g32 = (uint32_t)g, n32 = (uint32_t)a.n;
      gi = (int)(g32 / n32);
      const uint32_t e32 = g32 - (uint32_t)gi * n32;
      e = e32;
      b = e32 < (uint32_t)big ? (int)(e32 / (uint32_t)(a.q + 1))
                              : (int)((uint32_t)a.rem + (e32 - (uint32_t)big) / (uint32_t)a.q);
    } else {
      gi = (int)(g / a.n);
      e = g - (uint64_t)gi * a.n;
      b = e < big ? (int)(e / (a.q + 1)) : (int)(a.rem + (e - big) / a.q);
    }
    const int first = gi * lv.group;
    const int count = min(lv.group, lv.nops - first);
    StepOp op[kFlatGroup];
#pragma unroll
    for (int k = 0; k < kFlatGroup; ++k)
      if (k < count) op[k] = lv.ops[first + k];
    wait_prior_grid();
    A r[kFlatGroup], o0[kFlatGroup], o1[kFlatGroup];
#pragma unroll
    for (int k = 0; k < kFlatGroup; ++k) {
      if (k >= count) break;
      const int x = a.xor_group ? (b ^ (int)op[k].dst_place) : wrap_rank(b + (int)op[k].dst_place, a.P);
      r[k] = o0[k] = o1[k] = A(0);
      if (op[k].recv_place >= 0) {
        const int partner = a.xor_group ? (x ^ lv.partner) : wrap_rank(x + lv.partner, a.P);
        r[k] = load1<T, A>(op[k].recv_buf, slot(op[k].recv_buf, partner), e);
        moved += (op[k].recv_buf == BUF_RANK) ? sizeof(T) : sizeof(A);
      }
      if (op[k].out0_own != BUF_NONE) o0[k] = load1<T, A>(op[k].out0_own, slot(op[k].out0_own, x), e);
      if (op[k].out1_own != BUF_NONE) o1[k] = load1<T, A>(op[k].out1_own, slot(op[k].out1_own, x), e);
    }
#pragma unroll
    for (int k = 0; k < kFlatGroup; ++k) {
      if (k >= count) break;
      const int x = a.xor_group ? (b ^ (int)op[k].dst_place) : wrap_rank(b + (int)op[k].dst_place, a.P);
      const bool has_recv = op[k].recv_place >= 0;
      if (op[k].out0_own == BUF_NONE) o0[k] = r[k];
      else if (has_recv) o0[k] = combine<OP>(o0[k], r[k]);
      store1<T, A>(op[k].out0_buf, slot(op[k].out0_buf, x), e, o0[k]);
      if (op[k].out1_buf != BUF_NONE) {
        if (op[k].out1_own == BUF_NONE) o1[k] = r[k];
        else if (has_recv) o1[k] = combine<OP>(o1[k], r[k]);
        store1<T, A>(op[k].out1_buf, slot(op[k].out1_buf, x), e, o1[k]);
      }
    }
  }
  wait_prior_grid();  // threads without an item: the grid must not complete before its predecessor
  count_moved(lv.bytes, moved);
}

template <int MAXP>
__device__ __forceinline__ LaunchView view_of(const StepArgs<MAXP> &a) {
  LaunchView lv;
  lv.ops = a.ops;
  lv.bytes = a.bytes;
  lv.chunk = a.chunk;
  lv.nops = a.nops;
  lv.partner = a.partner;
  lv.nchunks = a.nchunks;
  lv.group = a.group;
  return lv;
}

__device__ __forceinline__ void counter_upkeep(const CounterUpkeep &c) {
  static_assert(STEP_BYTE_SLOTS <= kThreads, "one thread per counter slot");
  if (threadIdx.x < STEP_BYTE_SLOTS) {
    const int at = threadIdx.x * STEP_SLOT_STRIDE;
    if (c.zero != nullptr) c.zero[at] = 0;
    if (c.move_from != nullptr) c.move_to[at] = atomicExch(c.move_from + at, 0ull);
  }
}

// At most 40 registers (6 CTAs per SM): the bf16 launches ran 5-8 % faster than at the
// 48 registers the compiler picks unbounded, fp32 the same.
template <typename T, int OP, int MAXP>
__global__ void __launch_bounds__(kThreads, 6) step_kernel(const __grid_constant__ StepArgs<MAXP> a) {
  wait_prior_grid();
  if (blockIdx.x == 0) counter_upkeep(a.upkeep);
  const uint32_t moved = chunk_work<T, OP, MAXP>(a, view_of(a), a.reverse ? gridDim.x - 1 - blockIdx.x : blockIdx.x);
  allow_next_grid();
  count_moved(a.bytes, moved);
}

template <typename T, int OP, int MAXP>
__global__ void __launch_bounds__(kThreads) step_kernel_flat(const __grid_constant__ StepArgs<MAXP> a) {
  __shared__ void *s_rank[MAXP];
  if (a.early) allow_next_grid();
  for (int x = threadIdx.x; x < a.P; x += kThreads) s_rank[x] = a.rank[x];
  __syncthreads();
  flat_work<T, OP, MAXP>(a, view_of(a), s_rank, (uint64_t)blockIdx.x * blockDim.x + threadIdx.x,
                         (uint64_t)gridDim.x * blockDim.x);
  if (blockIdx.x == 0) counter_upkeep(a.upkeep);
  if (!a.early) allow_next_grid();
}

// Launches a step kernel with programmatic stream serialisation (see above).
template <typename Args>
cudaError_t launch_pdl(void (*kernel)(Args), unsigned grid, gar_stream_t stream, const Args &a) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, a);
}

// ---------------------------------------------------------------------------
// Persistent step-faithful mode (GAR_STEP_PERSISTENT): one cooperative launch runs every
// step of the schedule; a grid-wide barrier between steps takes the place of the kernel
// boundary.  The barrier's waits are bounded: after spin_limit polls a CTA records a
// timeout in the barrier state and returns, and every other CTA stops at its next poll,
// so the kernel always ends and the context stays usable; the host reads the outcome
// with gar_plan_status.
// ---------------------------------------------------------------------------

// Device state of a plan's persistent launches, zero between launches but for the outcome:
// the last CTA to leave a launch writes the outcome and resets the rest, so no memset
// precedes a launch.
struct BarrierState {
  unsigned int count;   // CTA arrivals since the launch began
  unsigned int leaving; // CTAs that have finished
  int error;            // 1 once any CTA gave up waiting
  int error_launch;     // launch index after which the first timeout happened
  int outcome;          // `error` and `error_launch` of the launch that ended last
  int outcome_launch;
};

template <int MAXP>
struct PersistArgs {
  StepArgs<MAXP> s;                 // buffers and sizes (s.ops = whole op table)
  const LaunchDesc *launches;
  unsigned long long *step_bytes;   // S rows of STEP_ROW counters, then the first step's own
  BarrierState *bar;
  int nlaunch, nsteps;
  unsigned int spin_limit;          // polls before a wait gives up
  unsigned int phantom;             // arrivals expected beyond the grid (test hook, normally 0)
};

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned atom_add_acq_rel_gpu(unsigned *p, unsigned v) {
  unsigned old;
  asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
  return old;
}
__device__ __forceinline__ int ld_relaxed_int(const int *p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Grid-wide barrier number `launch` (0-based) with a bounded wait.  Every CTA adds one
// to the arrival count with acquire-release semantics (release: the CTA's writes of the
// step, ordered before it by __syncthreads, become visible with it; acquire: the CTA
// that arrives last reads the others' writes, having seen all their arrivals in the add
// itself) and polls the count with acquire loads until it reaches (launch + 1) *
// expected, the arrivals of this and every earlier barrier of the launch.  The count
// only grows within a launch, so no CTA resets it and the last arrival releases everyone
// at once.  Returns false (for the whole CTA) if this or any other CTA timed out.
// The CTA's staged byte counts of the step (bytes: its counters, or nullptr) are added on the
// way: by a warp beside the one that waits, so they may follow this arrival and precede the
// next, or, with `first`, before the arrival.
template <int NT>
__device__ bool grid_barrier(BarrierState *bar, unsigned expected, unsigned spin_limit, int launch,
                             unsigned long long *bytes, const uint32_t *s_moved, bool first) {
  __shared__ int s_ok;
  __syncthreads();
  if (bytes != nullptr && threadIdx.x == (first ? 0 : 32)) add_moved<NT>(bytes, s_moved);
  if (threadIdx.x == 0) {
    int ok = 1;
    const unsigned target = (unsigned)(launch + 1) * expected;
    unsigned now = atom_add_acq_rel_gpu(&bar->count, 1u) + 1u;
    unsigned polls = 0;
    while (now < target) {
      ++polls;
      if (polls >= spin_limit || ((polls & 63u) == 0 && ld_relaxed_int(&bar->error) != 0)) {
        ok = 0;
        break;
      }
      if (polls > 32) __nanosleep(32);
      now = ld_acquire_gpu(&bar->count);
    }
    if (!ok && atomicCAS(&bar->error, 0, 1) == 0) bar->error_launch = launch;
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// Counter row of a communication step: the step's own, but for the first step's, whose
// counts wait in row nsteps until a later launch moves them (see CounterUpkeep).
__host__ __device__ __forceinline__ unsigned long long *counter_row(unsigned long long *rows, int comm_step,
                                                                    int nsteps) {
  if (rows == nullptr || comm_step < 0) return nullptr;
  return rows + (size_t)(comm_step == 0 ? nsteps : comm_step) * STEP_ROW;
}
__host__ __device__ __forceinline__ CounterUpkeep upkeep_of(unsigned long long *rows, int launch, int next_comm_step,
                                                            int nsteps, int move_at = 1) {
  CounterUpkeep c{nullptr, nullptr, nullptr};
  if (rows == nullptr) return c;
  if (next_comm_step > 0) c.zero = rows + (size_t)next_comm_step * STEP_ROW;
  if (launch == move_at) {
    c.move_from = rows + (size_t)nsteps * STEP_ROW;
    c.move_to = rows;
  }
  return c;
}

// FLAT: element-major mapping (small blocks), else pieces of blocks.  PER_SM: CTAs per SM that
// its registers allow for.
template <typename T, int OP, int MAXP, bool FLAT, int PER_SM>
__global__ void __launch_bounds__(FLAT ? kThreads : kPersistThreads, PER_SM)
    step_kernel_persistent(const __grid_constant__ PersistArgs<MAXP> p) {
  __shared__ void *s_rank[FLAT ? MAXP : 1];
  __shared__ uint32_t s_moved[kPersistThreads / 32];
  if (FLAT) {
    for (int x = threadIdx.x; x < p.s.P; x += kThreads) s_rank[x] = p.s.rank[x];
    __syncthreads();
  }
  const unsigned expected = gridDim.x + p.phantom;
  bool ok = true;
  // The first step's counts are added beside barrier 0 and moved behind barrier 1; a launch of
  // two steps has no barrier 1: there the add comes before the arrival at barrier 0.
  const int move_at = p.nlaunch > 2 ? 2 : 1;
  LaunchDesc st = p.launches[0];  // fetched before the barrier that opens the step (never changes)
  for (int l = 0; l < p.nlaunch && ok; ++l) {
    LaunchView lv;
    lv.ops = p.s.ops + st.first_op;
    lv.nops = st.nops;
    lv.partner = st.partner;
    lv.bytes = counter_row(p.step_bytes, st.comm_step, p.nsteps);
    lv.chunk = (uint32_t)st.piece;
    lv.nchunks = st.pieces;
    lv.group = st.group;
    if (FLAT) {
      flat_work<T, OP, MAXP>(p.s, lv, s_rank, (uint64_t)blockIdx.x * kThreads + threadIdx.x,
                             (uint64_t)gridDim.x * kThreads);
    } else {
      uint32_t moved = 0;
      const uint32_t pieces = (uint32_t)st.pieces, items = pieces * (uint32_t)p.s.P * (uint32_t)st.nops;
      for (uint32_t item = blockIdx.x; item < items; item += gridDim.x) {
        const uint32_t blk = item / pieces, op = blk / (uint32_t)p.s.P;
        moved += range_work<T, OP, MAXP, kPersistThreads>(p.s, lv, lv.ops[op], (int)(blk - op * (uint32_t)p.s.P),
                                                          (uint64_t)(item - blk * pieces) * lv.chunk, lv.chunk);
      }
      stage_moved<kPersistThreads>(s_moved, moved);
    }
    unsigned long long *const bytes = FLAT ? nullptr : lv.bytes;  // (flat_work has added its own)
    if (l + 1 < p.nlaunch) {
      st = p.launches[l + 1];
      if (blockIdx.x == 0) counter_upkeep(upkeep_of(p.step_bytes, l, st.comm_step, p.nsteps, move_at));
      ok = grid_barrier<kPersistThreads>(p.bar, expected, p.spin_limit, l, bytes, s_moved, p.nlaunch == 2);
    } else {
      if (blockIdx.x == 0) counter_upkeep(upkeep_of(p.step_bytes, l, -1, p.nsteps, move_at));
      __syncthreads();
      if (bytes != nullptr && threadIdx.x == 32) add_moved<kPersistThreads>(bytes, s_moved);
    }
  }
  // The last CTA to leave records the outcome and resets the state for the next launch; a
  // launch that gave up also drops the first step's counts, which may not have been moved.
  __syncthreads();
  if (threadIdx.x == 0 && atom_add_acq_rel_gpu(&p.bar->leaving, 1u) == gridDim.x - 1) {
    const int error = ld_relaxed_int(&p.bar->error);
    p.bar->outcome = error;
    p.bar->outcome_launch = p.bar->error_launch;
    if (error != 0 && p.step_bytes != nullptr)
      for (int k = 0; k < STEP_BYTE_SLOTS; ++k) p.step_bytes[(size_t)p.nsteps * STEP_ROW + k * STEP_SLOT_STRIDE] = 0;
    p.bar->count = 0;
    p.bar->leaving = 0;
    p.bar->error = 0;
  }
}


// Elements per CTA of a chunked launch.  Distribution steps copy 2-byte elements with as
// many bytes per CTA as fp32 chunks hold; launches of few CTAs take smaller chunks; a last
// chunk shorter than 1/8 of a chunk is spread over the block's others (P = 127 x 8 MiB
// bf16: blocks of 33,026 elements became 16,384 + 16,384 + 258, a third of the CTAs nearly
// empty).
uint32_t pick_chunk(uint64_t maxblk, int P, int nops, int phase, size_t elem_bytes) {
  uint64_t chunk = (phase == 1 && elem_bytes == 2) ? 2 * kChunk : kChunk;
  const uint64_t min_ctas = kMinCtas * (uint64_t)num_sms();
  while (chunk > kMinChunk && ((maxblk + chunk - 1) / chunk) * P * nops < min_ctas) chunk /= 2;
  const uint64_t nch = (maxblk + chunk - 1) / chunk;
  if (nch > 1 && maxblk - (nch - 1) * chunk < chunk / 8) chunk = ((maxblk + nch - 2) / (nch - 1) + 7) / 8 * 8;
  return (uint32_t)chunk;
}

// Ops per thread of an element-major launch: one while the device has a thread for every
// (op, element), more beyond.
int pick_group(uint64_t n, int nops) {
  const uint64_t threads = kFlatThreads * (uint64_t)num_sms();
  int group = 1;
  while (group < kFlatGroup && (uint64_t)((nops + group - 1) / group) * n > threads) group *= 2;
  return group;
}

template <int MAXP>
StepArgs<MAXP> step_args(const gar_plan &pl, const Launch &ln, void *const *rank, void *workspace) {
  StepArgs<MAXP> a{};
  for (int x = 0; x < pl.P; ++x) a.rank[x] = rank[x];
  int slot = 0;
  for (int k = 0; k < NUM_WS_BUFS; ++k)
    if (pl.ws_used[k])
      a.ws[k] = static_cast<char *>(workspace) + (size_t)(slot++) * pl.P * pl.n_pad * acc_size(pl.dtype);
  a.q = pl.q;
  a.rem = pl.rem;
  a.n_pad = pl.n_pad;
  a.n = pl.n;
  a.P = pl.P;
  a.xor_group = pl.group == GAR_GROUP_XOR ? 1 : 0;
  a.partner = ln.partner;
  a.nops = ln.nops;
  return a;
}

// Mapping and grid of one launch; *flat: element-major.
template <int MAXP>
int step_grid(const gar_plan &pl, const Launch &ln, bool noalloc, StepArgs<MAXP> &a, bool *flat, unsigned *grid) {
  const uint64_t maxblk = pl.q + (pl.rem ? 1 : 0);
  *grid = 0;
  *flat = maxblk < kFlatBelow &&
          (!noalloc || maxblk < kNoAllocFlatBlock || (uint64_t)ln.nops * pl.n < kNoAllocFlatItems);
  if (maxblk == 0 || ln.nops == 0) return GAR_OK;
  if (*flat) {
    // blocks shorter than one CTA's worth of vectors: element-major launch
    a.group = pick_group(pl.n, ln.nops);
    const uint64_t total = (uint64_t)((ln.nops + a.group - 1) / a.group) * pl.n;
    *grid = (unsigned)std::min<uint64_t>((total + kThreads - 1) / kThreads, (uint64_t)num_sms() * 32);
    return GAR_OK;
  }
  a.chunk = pick_chunk(maxblk, pl.P, ln.nops, ln.phase, (size_t)elem_size(pl.dtype));
  a.nchunks = (int)((maxblk + a.chunk - 1) / a.chunk);
  const uint64_t g = (uint64_t)a.nchunks * (uint64_t)pl.P * (uint64_t)ln.nops;
  if (g > 0x7fffffffull) {
    set_error("step launch grid too large");
    return GAR_EINVAL;
  }
  *grid = (unsigned)g;
  return GAR_OK;
}

template <typename T, int OP, int MAXP>
int launch_typed(const gar_plan &pl, const Launch &ln, int launch_index, void *const *rank,
                 gar_stream_t stream) {
  StepArgs<MAXP> a = step_args<MAXP>(pl, ln, rank, pl.ws);
  a.ops = pl.d_ops + ln.first_op;
  a.bytes = counter_row(pl.d_step_bytes, ln.comm_step, pl.S);
  const bool last = launch_index + 1 == (int)pl.launches.size();
  a.upkeep = upkeep_of(pl.d_step_bytes, launch_index, last ? -1 : pl.launches[launch_index + 1].comm_step, pl.S);
  a.early = last ? 0 : 1;
  a.reverse = launch_index & 1;
  bool flat = false;
  unsigned grid = 0;
  if (int rc = step_grid(pl, ln, false, a, &flat, &grid)) return rc;
  if (grid == 0) return GAR_OK;
  const cudaError_t e = flat ? launch_pdl(step_kernel_flat<T, OP, MAXP>, grid, stream, a)
                             : launch_pdl(step_kernel<T, OP, MAXP>, grid, stream, a);
  if (e != cudaSuccess) return cuda_fail(e, "step kernel launch");
  return GAR_OK;
}

template <typename T, int MAXP>
int launch_op(const gar_plan &pl, const Launch &ln, int li, void *const *rank, gar_stream_t s) {
  switch (pl.op) {
    case GAR_SUM: return launch_typed<T, GAR_SUM, MAXP>(pl, ln, li, rank, s);
    case GAR_MAX: return launch_typed<T, GAR_MAX, MAXP>(pl, ln, li, rank, s);
    case GAR_MIN: return launch_typed<T, GAR_MIN, MAXP>(pl, ln, li, rank, s);
  }
  return GAR_EINVAL;
}

template <int MAXP>
int launch_dt(const gar_plan &pl, const Launch &ln, int li, void *const *rank, gar_stream_t s) {
  switch (pl.dtype) {
    case GAR_F32: return launch_op<float, MAXP>(pl, ln, li, rank, s);
    case GAR_BF16: return launch_op<__nv_bfloat16, MAXP>(pl, ln, li, rank, s);
    case GAR_I32: return launch_op<int, MAXP>(pl, ln, li, rank, s);
  }
  return GAR_EINVAL;
}

// CTAs per SM of a plan's persistent launches (see kPersistThreads).
int persist_per_sm(const gar_plan &pl) {
  int most_ops = 0;
  for (const Launch &ln : pl.launches) most_ops = std::max(most_ops, ln.nops);
  const uint64_t blocks = (uint64_t)most_ops * (uint64_t)pl.P, elements = (uint64_t)most_ops * pl.n;
  const bool few = pl.K <= 2;
  return elements >= (few && pl.dtype == GAR_BF16 ? 1u << 24 : 1u << 22) || (!few && blocks > 4 * (uint64_t)num_sms()) ? 3 : 2;
}

template <typename T, int OP, int MAXP>
int launch_persistent_typed(const gar_plan &pl, void *const *rank, gar_stream_t stream) {
  PersistArgs<MAXP> p{};
  p.s = step_args<MAXP>(pl, pl.launches[0], rank, pl.ws);
  p.s.ops = pl.d_ops;
  p.launches = static_cast<const LaunchDesc *>(pl.d_launches);
  p.step_bytes = pl.d_step_bytes;
  p.bar = static_cast<BarrierState *>(pl.d_barrier);
  p.nlaunch = (int)pl.launches.size();
  p.nsteps = pl.S;
  p.spin_limit = pl.barrier_spin_limit;
  p.phantom = pl.barrier_phantom;
  // As many CTAs as the largest step has work items, at most the co-resident maximum: a
  // small Allreduce then waits at its barriers for a few CTAs instead of several per SM.
  const uint64_t maxblk = pl.q + (pl.rem ? 1 : 0);
  const bool flat = maxblk < kFlatBelow;
  uint64_t need = 1;
  for (const Launch &ln : pl.launches) {
    const int group = pick_group(pl.n, ln.nops);
    need = std::max<uint64_t>(need, flat ? ((uint64_t)((ln.nops + group - 1) / group) * pl.n + kThreads - 1) / kThreads
                                         : (uint64_t)ln.nops * pl.P * ((maxblk + kMinPiece - 1) / kMinPiece));
  }
  const void *fn = flat   ? (const void *)step_kernel_persistent<T, OP, MAXP, true, 4>
                   : persist_per_sm(pl) == 3 ? (const void *)step_kernel_persistent<T, OP, MAXP, false, 3>
                                             : (const void *)step_kernel_persistent<T, OP, MAXP, false, 2>;
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, flat ? kThreads : kPersistThreads, 0);
  if (e != cudaSuccess || per_sm < 1) return cuda_fail(e == cudaSuccess ? cudaErrorInvalidConfiguration : e,
                                                       "persistent kernel occupancy");
  const unsigned grid = (unsigned)std::min<uint64_t>(need, (uint64_t)per_sm * (uint64_t)num_sms());
  void *args[] = {&p};
  e = cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(flat ? kThreads : kPersistThreads), args, 0, (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e, "persistent kernel launch");
  return GAR_OK;
}

template <typename T, int MAXP>
int launch_persistent_op(const gar_plan &pl, void *const *rank, gar_stream_t s) {
  switch (pl.op) {
    case GAR_SUM: return launch_persistent_typed<T, GAR_SUM, MAXP>(pl, rank, s);
    case GAR_MAX: return launch_persistent_typed<T, GAR_MAX, MAXP>(pl, rank, s);
    case GAR_MIN: return launch_persistent_typed<T, GAR_MIN, MAXP>(pl, rank, s);
  }
  return GAR_EINVAL;
}

template <int MAXP>
int launch_persistent_dt(const gar_plan &pl, void *const *rank, gar_stream_t s) {
  switch (pl.dtype) {
    case GAR_F32: return launch_persistent_op<float, MAXP>(pl, rank, s);
    case GAR_BF16: return launch_persistent_op<__nv_bfloat16, MAXP>(pl, rank, s);
    case GAR_I32: return launch_persistent_op<int, MAXP>(pl, rank, s);
  }
  return GAR_EINVAL;
}

}  // namespace

int launch_step(const gar_plan &pl, const Launch &ln, int launch_index, void *const *rank,
                gar_stream_t stream) {
  if (pl.P <= 128) return launch_dt<128>(pl, ln, launch_index, rank, stream);
  return launch_dt<GAR_MAX_P>(pl, ln, launch_index, rank, stream);
}

int launch_persistent(const gar_plan &pl, void *const *rank, gar_stream_t stream) {
  if (pl.P <= 128) return launch_persistent_dt<128>(pl, rank, stream);
  return launch_persistent_dt<GAR_MAX_P>(pl, rank, stream);
}

size_t barrier_state_bytes() { return sizeof(BarrierState); }

void barrier_outcome(const void *state, int *error, int *launch) {
  const BarrierState *st = static_cast<const BarrierState *>(state);
  *error = st->outcome;
  *launch = st->outcome_launch;
}

// A persistent step's blocks (P * nops of at most maxblk elements) are cut into equal pieces,
// as many as take the fewest batches of loads (and starts of pieces) in all rounds of the
// grid, so that every CTA reaches the barrier at about the same time.  (With at most 4 pieces,
// and one where there are more CTAs than blocks, P = 13 x 1.6M bf16 S = 4, 338 blocks, took 289
// us instead of 243.)
LaunchDesc launch_desc(const gar_plan &pl, const Launch &ln) {
  LaunchDesc d{ln.first_op, ln.nops, ln.partner, ln.comm_step, pick_group(pl.n, ln.nops), 1, 0};
  const uint64_t maxblk = pl.q + (pl.rem ? 1 : 0), blocks = (uint64_t)pl.P * (uint64_t)std::max(1, ln.nops);
  const uint64_t grid = (uint64_t)persist_per_sm(pl) * (uint64_t)num_sms();
  constexpr uint64_t batch = 4 * kUnroll * kPersistThreads;
  uint64_t best = ~0ull;
  for (uint64_t c = 1; c <= std::max<uint64_t>(kMostPieces, grid / blocks); ++c) {
    const uint64_t piece = std::max<uint64_t>(kMinPiece, ((maxblk + c - 1) / c + 7) / 8 * 8);
    const uint64_t pieces = (maxblk + piece - 1) / piece;
    const uint64_t cost = ((blocks * pieces + grid - 1) / grid) * ((piece + batch - 1) / batch + 1);
    if (cost < best) {
      best = cost;
      d.pieces = (int)pieces;
      d.piece = (int)piece;
    }
  }
  return d;
}

}  // namespace gar

// ---------------------------------------------------------------------------
// Step-faithful Allreduce without device allocation (gar_allreduce_noalloc).
//
// For callers that must not allocate device memory at call time -- code running
// under a caching allocator that owns all of the GPU's memory, or a host runtime with
// no allocator hook -- the workspace lives in one file-scope device array of fixed
// size instead of a caller-supplied buffer, and each launch receives its block ops by
// value in the kernel parameters instead of from a device table.  No cudaMalloc,
// cudaFree or memset is issued.  The array exists on a device once this file's device
// code is loaded there -- under CUDA's lazy module loading, at the first launch of any
// of its kernels, at gar_plan_prepare of a step-faithful mode, or at the first
// no-allocation call -- and stays until the process exits.  Nothing in it needs to
// start at zero: the schedule writes every workspace slot before it reads it.  All
// calls share the array, so two calls whose work overlaps on the GPU race.
// ---------------------------------------------------------------------------

static __device__ __align__(256) unsigned char g_noalloc_scratch[GAR_NOALLOC_SCRATCH_BYTES];

namespace gar {
namespace {

constexpr int kNoAllocMaxOps = 2 * GAR_NOALLOC_MAX_P;  // |transmit set| + K <= 2P per launch

struct NoAllocArgs {
  StepArgs<GAR_NOALLOC_MAX_P> s;
  StepOp ops[kNoAllocMaxOps];
};

// The step kernels' work with the ops read from the parameter block and no byte counting.
template <typename T, int OP>
__global__ void __launch_bounds__(kThreads, 6) step_kernel_noalloc(const __grid_constant__ NoAllocArgs a) {
  LaunchView lv = view_of(a.s);
  lv.ops = a.ops;
  wait_prior_grid();
  chunk_work<T, OP>(a.s, lv, a.s.reverse ? gridDim.x - 1 - blockIdx.x : blockIdx.x);
  allow_next_grid();
}

template <typename T, int OP>
__global__ void __launch_bounds__(kThreads) step_kernel_noalloc_flat(const __grid_constant__ NoAllocArgs a) {
  __shared__ void *s_rank[GAR_NOALLOC_MAX_P];
  if (a.s.early) allow_next_grid();
  for (int x = threadIdx.x; x < a.s.P; x += kThreads) s_rank[x] = a.s.rank[x];
  __syncthreads();
  LaunchView lv = view_of(a.s);
  lv.ops = a.ops;
  flat_work<T, OP>(a.s, lv, s_rank, (uint64_t)blockIdx.x * kThreads + threadIdx.x, (uint64_t)gridDim.x * kThreads);
  if (!a.s.early) allow_next_grid();
}

// Device address of the scratch array on the current device, looked up on every call
// with that device current: the lookup allocates nothing, and a cached address would be
// stale after cudaDeviceReset or in another context on the same device.
int noalloc_scratch(void **out);

}  // namespace

// Loads this file's device code on the current device (and with it the scratch array).
int load_step_module() {
  void *p = nullptr;
  return noalloc_scratch(&p);
}

namespace {

int noalloc_scratch(void **out) {
  void *p = nullptr;
  cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(no-allocation scratch)");
  *out = p;
  return GAR_OK;
}

template <typename T, int OP>
int noalloc_launch(const gar_plan &pl, int launch_index, void *const *rank, void *scratch, gar_stream_t stream) {
  const Launch &ln = pl.launches[launch_index];
  NoAllocArgs a{};
  a.s = step_args<GAR_NOALLOC_MAX_P>(pl, ln, rank, scratch);
  for (int k = 0; k < ln.nops; ++k) a.ops[k] = pl.ops[ln.first_op + k];
  a.s.early = launch_index + 1 < (int)pl.launches.size() ? 1 : 0;
  a.s.reverse = launch_index & 1;
  bool flat = false;
  unsigned grid = 0;
  if (int rc = step_grid(pl, ln, true, a.s, &flat, &grid)) return rc;
  if (grid == 0) return GAR_OK;
  const cudaError_t e = flat ? launch_pdl(step_kernel_noalloc_flat<T, OP>, grid, stream, a)
                             : launch_pdl(step_kernel_noalloc<T, OP>, grid, stream, a);
  if (e != cudaSuccess) return cuda_fail(e, "no-allocation step kernel launch");
  return GAR_OK;
}

template <typename T>
int noalloc_launch_op(const gar_plan &pl, int li, void *const *rank, void *scratch, gar_stream_t s) {
  switch (pl.op) {
    case GAR_SUM: return noalloc_launch<T, GAR_SUM>(pl, li, rank, scratch, s);
    case GAR_MAX: return noalloc_launch<T, GAR_MAX>(pl, li, rank, scratch, s);
    case GAR_MIN: return noalloc_launch<T, GAR_MIN>(pl, li, rank, scratch, s);
  }
  return GAR_EINVAL;
}

}  // namespace
}  // namespace gar

extern "C" int gar_allreduce_noalloc(gar_plan *pl, void *const *rank_buffers, gar_stream_t stream) {
  using namespace gar;
  if (pl == nullptr || rank_buffers == nullptr) {
    set_error("null plan or rank buffer array");
    return GAR_EINVAL;
  }
  if (pl->group != GAR_GROUP_CYCLIC) {
    set_error("gar_allreduce_noalloc supports the cyclic group only");
    return GAR_EINVAL;
  }
  if (pl->P > GAR_NOALLOC_MAX_P) {
    set_error("gar_allreduce_noalloc supports P <= " + std::to_string(GAR_NOALLOC_MAX_P) +
              ", plan has P=" + std::to_string(pl->P));
    return GAR_EINVAL;
  }
  if (pl->ws_bytes > (size_t)GAR_NOALLOC_SCRATCH_BYTES) {
    set_error("gar_allreduce_noalloc: plan needs " + std::to_string(pl->ws_bytes) +
              " bytes of workspace, the fixed scratch array holds " +
              std::to_string((size_t)GAR_NOALLOC_SCRATCH_BYTES));
    return GAR_EINVAL;
  }
  for (int x = 0; x < pl->P; ++x) {
    if (rank_buffers[x] == nullptr) {
      set_error("null rank buffer " + std::to_string(x));
      return GAR_EINVAL;
    }
    if (reinterpret_cast<uintptr_t>(rank_buffers[x]) % 16 != 0) {
      set_error("rank buffer " + std::to_string(x) + " is not 16-byte aligned");
      return GAR_EALIGN;
    }
    for (int y = 0; y < x; ++y)
      if (rank_buffers[y] == rank_buffers[x]) {
        set_error("two ranks share one buffer");
        return GAR_EINVAL;
      }
  }
  for (const Launch &ln : pl->launches)
    if (ln.nops > kNoAllocMaxOps) {
      set_error("gar_allreduce_noalloc: a launch has more block ops than the parameter block holds");
      return GAR_EINVAL;
    }
  if (pl->n == 0 || pl->P == 1) return GAR_OK;
  void *scratch = nullptr;
  int rc = noalloc_scratch(&scratch);
  if (rc) return rc;
  for (int li = 0; li < (int)pl->launches.size(); ++li) {
    switch (pl->dtype) {
      case GAR_F32: rc = noalloc_launch_op<float>(*pl, li, rank_buffers, scratch, stream); break;
      case GAR_BF16: rc = noalloc_launch_op<__nv_bfloat16>(*pl, li, rank_buffers, scratch, stream); break;
      case GAR_I32: rc = noalloc_launch_op<int>(*pl, li, rank_buffers, scratch, stream); break;
      default: rc = GAR_EINVAL;
    }
    if (rc) return rc;
  }
  return GAR_OK;
}
