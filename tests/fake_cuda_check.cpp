// Checks of the library's host code on a fake CUDA runtime, for tests/test_host_fake_cuda.py:
// the first argument names the check.  Prints what failed and exits 1.
#include "fake_cuda.hpp"

#include <cstdint>

namespace {

gar_plan *plan_of(int P, uint64_t n, int dtype, int steps) {
  gar_plan *pl = nullptr;
  CHECK(gar_plan_create(&pl, P, n, dtype, GAR_SUM, steps) == GAR_OK);
  return pl;
}

std::vector<void *> rows(int P) {
  std::vector<void *> r(P);
  for (int x = 0; x < P; ++x) r[x] = reinterpret_cast<void *>((uintptr_t)4096 * (x + 1));
  return r;
}

int form_of(gar_plan *pl) {
  gar_plan_info info;
  CHECK(gar_plan_get_info(pl, &info) == GAR_OK);
  return info.fused_form;
}

// Equal plans on two devices share one kernel, whose shared-memory limit and resident CTAs
// are each device's own.
void two_devices() {
  fake::blocks_per_sm = [](int dev) { return 1 + dev; };
  struct { int P; uint64_t n; int dtype, steps, form; } cases[] = {
      {127, 4608, GAR_BF16, 10, GAR_FORM_COOP}, {127, 1u << 20, GAR_BF16, 7, GAR_FORM_STREAM}};
  for (const auto &c : cases) {
    const std::vector<void *> r = rows(c.P);
    gar_plan *pl[2];
    for (int dev : {0, 1}) {
      fake::device = dev;
      pl[dev] = plan_of(c.P, c.n, c.dtype, c.steps);
      fake::launches.clear();
      CHECK(gar_allreduce(pl[dev], r.data(), GAR_FUSED, nullptr) == GAR_OK);
      CHECK(form_of(pl[dev]) == c.form);
      CHECK(fake::launches.size() == 1 && fake::launches[0].device == dev && fake::launches[0].smem > 48 * 1024);
      if (c.form == GAR_FORM_STREAM) CHECK(fake::launches[0].grid == 152u * (unsigned)(1 + dev));
    }
    fake::device = 0;
    CHECK(gar_allreduce(pl[0], r.data(), GAR_FUSED, nullptr) == GAR_OK);
    for (gar_plan *p : pl) gar_plan_destroy(p);
  }
}

}  // namespace

int main(int argc, char **argv) {
  const std::map<std::string, void (*)()> checks = {{"two_devices", two_devices}};
  CHECK(argc == 2 && checks.count(argv[1]));
  checks.at(argv[1])();
  return 0;
}
