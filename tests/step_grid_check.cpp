// The mapping that step_kernels.cu chooses for a launch, for tests/test_step_grid_host.py
// (which puts the file's host rules in step_rules.inc): element-major or chunked.
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
}  // namespace gar

// prints, for every line of block length, ranks, ops and mode, 1 where the launch is element-major
int main() {
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
