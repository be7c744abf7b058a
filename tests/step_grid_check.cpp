// The mapping that step_kernels.cu chooses for a launch, for tests/test_step_grid_host.py
// (which puts the file's host rules in step_rules.inc and step_desc.inc): element-major or
// chunked, and the persistent kernel's shape.
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <string>

#include "gar_internal.hpp"

namespace gar {
void set_error(const std::string &) {}
int num_sms() { return 152; }
int elem_size(int dtype) { return dtype == GAR_BF16 ? 2 : 4; }
namespace {
struct Args {
  uint32_t chunk;
  int nchunks, group;
};
template <int> using StepArgs = Args;
#include "step_rules.inc"
}  // namespace
#include "step_desc.inc"
}  // namespace gar

// "flat": prints, for every line of block length, ranks, ops and mode, 1 where the launch is
// element-major.  "pieces": for every line of elements, ranks, ops, copies and type, the CTAs per
// SM, pieces per block and elements of a piece of the persistent kernel.
int main(int, char **argv) {
  if (argv[1][0] == 'p') {
    unsigned long long n;
    int P, nops, K, dtype;
    while (std::scanf("%llu %d %d %d %d", &n, &P, &nops, &K, &dtype) == 5) {
      gar_plan pl;
      pl.P = P;
      pl.n = n;
      pl.q = n / P;
      pl.rem = n % P;
      pl.K = K;
      pl.dtype = dtype;
      gar::Launch ln{};
      ln.nops = nops;
      pl.launches.push_back(ln);
      const gar::LaunchDesc d = gar::launch_desc(pl, ln);
      std::printf("%d %d %d\n", gar::persist_per_sm(pl), d.pieces, d.piece);
    }
    return 0;
  }
  int blk, P, nops, noalloc;
  while (std::scanf("%d %d %d %d", &blk, &P, &nops, &noalloc) == 4) {
    gar_plan pl;
    pl.P = P;
    pl.n = (uint64_t)blk * P;
    pl.q = blk;
    gar::Launch ln{};
    ln.nops = nops;
    gar::Args a{};
    bool flat = false;
    unsigned grid = 0;
    if (gar::step_grid<64>(pl, ln, noalloc != 0, a, &flat, &grid) != GAR_OK || grid == 0) return 1;
    std::printf("%d\n", (int)flat);
  }
}
