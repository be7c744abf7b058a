// range_work of step_kernels.cu, compiled for the host and run thread by thread, for
// tests/test_step_count_host.py (which puts the file's device part in step_device.inc): every
// thread returns the bytes that it has read from its partner, and all threads together cover
// the range once.
#include <cuda_bf16.h>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#undef __launch_bounds__
#define __launch_bounds__(...)
struct Dim {
  unsigned x;
};
static Dim threadIdx, blockIdx, blockDim, gridDim;
static inline unsigned __reduce_add_sync(unsigned, unsigned v) { return v; }
template <typename T> static T atomicAdd(T *p, T v) { const T old = *p; *p += v; return old; }
template <typename T> static T atomicExch(T *p, T v) { const T old = *p; *p = v; return old; }
static inline void __syncthreads() {}
static inline float __uint_as_float(unsigned u) { float f; std::memcpy(&f, &u, 4); return f; }
static inline int min(int a, int b) { return a < b ? a : b; }

#include "step_device.inc"

namespace gar {
int cuda_fail(int, const char *) { return GAR_ECUDA; }
void set_error(const std::string &) {}
namespace {

int failures = 0;

// One op at rank x over elements [c0, c0 + len) of its block, by NT threads: the elements
// that a thread writes are those it has read.
template <typename T, int NT>
void check(const StepOp &op, int P, uint64_t n, int x, uint64_t c0, uint32_t len) {
  using A = typename AccOf<T>::type;
  StepArgs<128> a{};
  a.P = P;
  a.n = n;
  a.n_pad = (n + 63) / 64 * 64;
  a.q = n / P;
  a.rem = n % P;
  std::vector<std::vector<T>> rank(P);
  std::vector<std::vector<A>> ws(NUM_WS_BUFS);
  for (int r = 0; r < P; ++r) {
    rank[r].resize(a.n_pad + 8);
    a.rank[r] = (void *)(((uintptr_t)rank[r].data() + 15) & ~(uintptr_t)15);
  }
  for (int k = 0; k < NUM_WS_BUFS; ++k) {
    ws[k].resize(P * a.n_pad + 8);
    a.ws[k] = (void *)(((uintptr_t)ws[k].data() + 15) & ~(uintptr_t)15);
  }
  LaunchView lv{};
  lv.partner = 1;
  const int partner = (x + 1) % P;
  const bool recv = op.recv_place >= 0;
  const size_t out_size = op.out0_buf == BUF_RANK ? sizeof(T) : sizeof(A);
  const size_t in_size = op.recv_buf == BUF_RANK ? sizeof(T) : sizeof(A);
  char *out = (char *)(op.out0_buf == BUF_RANK ? a.rank[x] : (char *)a.ws[op.out0_buf - BUF_QP0] + x * a.n_pad * sizeof(A));
  // the sources hold ones, so that every element written changes
  for (int r = 0; r < P; ++r)
    for (uint64_t e = 0; e < a.n_pad; ++e) {
      if (r == partner || op.out0_own == BUF_RANK) ((T *)a.rank[r])[e] = T(1);
      for (int k = 0; k < NUM_WS_BUFS; ++k)
        if (r == partner || op.out0_own == BUF_QP0 + k) ((A *)a.ws[k])[r * a.n_pad + e] = A(1);
    }
  std::vector<char> zero(a.n_pad * out_size, 0);
  const int b = (x - op.dst_place + P) % P;
  const uint64_t lo = b * a.q + (b < (int)a.rem ? b : a.rem), blen = a.q + (b < (int)a.rem ? 1 : 0);
  uint64_t written = 0, want = blen > c0 ? std::min<uint64_t>(len, blen - c0) : 0;
  for (int t = 0; t < NT; ++t) {
    threadIdx.x = t;
    const bool in_place = op.out0_own == op.out0_buf;
    if (!in_place) std::memset(out, 0, zero.size());
    std::vector<char> before(out, out + zero.size());
    const uint32_t bytes = range_work<T, GAR_SUM, 128, NT>(a, lv, op, x, c0, len);
    uint64_t mine = 0;
    for (uint64_t e = 0; e < n; ++e)
      if (std::memcmp(out + e * out_size, before.data() + e * out_size, out_size) != 0) {
        ++mine;
        if (e < lo + c0 || e >= lo + c0 + want) ++failures;
      }
    if (bytes != (recv ? mine * in_size : 0)) {
      std::printf("thread %d: %u bytes counted, %llu elements read\n", t, bytes, (unsigned long long)mine);
      ++failures;
    }
    written += mine;
  }
  if (written != want) {
    std::printf("P=%d n=%llu c0=%llu len=%u: %llu of %llu elements\n", P, (unsigned long long)n, (unsigned long long)c0, len,
                (unsigned long long)written, (unsigned long long)want);
    ++failures;
  }
}

StepOp op_of(int recv_place, int recv_buf, int out0, int own0) {
  StepOp op{};
  op.recv_place = recv_place;
  op.dst_place = 1;
  op.recv_buf = recv_buf;
  op.out0_buf = out0;
  op.out0_own = own0;
  op.out1_buf = op.out1_own = BUF_NONE;
  return op;
}

template <typename T> void all_ranges(const StepOp &op) {
  for (uint64_t n : {7ull, 100ull, 3011ull})
    for (int x : {0, 2})
      for (uint64_t c0 : {0ull, 5ull, 512ull})
        for (uint32_t len : {1u, 64u, 515u, 4096u}) check<T, 32>(op, 3, n, x, c0, len);
}

}  // namespace
}  // namespace gar

int main() {
  using namespace gar;
  all_ranges<__nv_bfloat16>(op_of(0, BUF_RANK, BUF_QP0, BUF_RANK));  // packed first step
  all_ranges<__nv_bfloat16>(op_of(0, BUF_RANK, BUF_RANK, BUF_NONE));  // copy of 8-element units
  all_ranges<__nv_bfloat16>(op_of(0, BUF_QP0, BUF_QS, BUF_NONE));     // copy of 4-element units
  all_ranges<__nv_bfloat16>(op_of(0, BUF_QP0, BUF_RANK, BUF_NONE));   // rounding copy
  all_ranges<float>(op_of(0, BUF_QP0, BUF_QP1, BUF_QP0));             // combine
  all_ranges<int>(op_of(0, BUF_RANK, BUF_QP0, BUF_RANK));
  all_ranges<float>(op_of(-1, BUF_NONE, BUF_RANK, BUF_QP0));          // nothing received
  return failures != 0;
}
