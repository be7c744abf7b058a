// Checks of the library's host code on a fake CUDA runtime, for tests/test_host_fake_cuda.py:
// the first argument names the check.  Prints what failed and exits 1.
#include "fake_cuda.hpp"

#include <cstdint>
#include <thread>

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

// Plans that share a streaming kernel report their own failed waits, each failure once,
// also of a replay that the host made no call for; a capture is not waited for.
void wait_status() {
  const int P = 127, first = 16 * P + 16;            // gar_args of a program without rotation
  const std::vector<void *> r = rows(P);
  std::vector<gar_plan *> pl;
  uint64_t slot = 0;
  fake::Function *f = nullptr;
  fake::on_launch = [&](fake::Function &k, const fake::Launch &ln) {
    f = &k;
    std::memcpy(&slot, static_cast<char *>(ln.args[0]) + first, 8);
    return cudaSuccess;
  };
  // a kernel's wait that gives up, on the device
  auto give_up = [&](uint64_t s) {
    CHECK(f->globals.size() == 1);
    const std::string name = f->globals.begin()->first.second;
    ++reinterpret_cast<unsigned *>(f->globals.begin()->second.data())[name == "gar_gave_up" ? s : 0];
  };
  std::vector<uint64_t> slots;
  for (int k = 0; k < 2; ++k) {
    pl.push_back(plan_of(P, 1u << 20, GAR_BF16, 7));
    CHECK(gar_plan_status(pl[k]) == GAR_OK);
    CHECK(gar_allreduce(pl[k], r.data(), GAR_FUSED, nullptr) == GAR_OK && form_of(pl[k]) == GAR_FORM_STREAM);
    slots.push_back(slot);
  }
  give_up(slots[1]);
  CHECK(gar_plan_status(pl[0]) == GAR_OK);
  CHECK(gar_plan_status(pl[1]) == GAR_ETIMEOUT);
  CHECK(gar_plan_status(pl[1]) == GAR_OK);
  give_up(slots[0]);                                  // a replay
  CHECK(gar_plan_status(pl[1]) == GAR_OK);
  CHECK(gar_plan_status(pl[0]) == GAR_ETIMEOUT);
  fake::capture = cudaStreamCaptureStatusActive;
  fake::on_synchronize = [](cudaStream_t) { return cudaErrorStreamCaptureUnsupported; };
  CHECK(gar_plan_status(pl[0]) == GAR_OK);
  fake::capture = cudaStreamCaptureStatusNone;
  fake::on_synchronize = nullptr;
  // more plans than slots: nobody's failure is lost, and a destroyed plan's slot is free again
  while (pl.size() < 70) {
    pl.push_back(plan_of(P, 1u << 20, GAR_BF16, 7));
    CHECK(gar_allreduce(pl.back(), r.data(), GAR_FUSED, nullptr) == GAR_OK);
    CHECK(gar_plan_status(pl.back()) == GAR_OK);
    slots.push_back(slot);
  }
  CHECK(slots[69] == slots[5]);
  give_up(slots[69]);
  for (size_t k = 0; k < pl.size(); ++k) CHECK(gar_plan_status(pl[k]) == (k == 5 || k == 69 ? GAR_ETIMEOUT : GAR_OK));
  for (gar_plan *p : pl) gar_plan_destroy(p);
  gar_plan *again = plan_of(P, 1u << 20, GAR_BF16, 7);
  CHECK(gar_allreduce(again, r.data(), GAR_FUSED, nullptr) == GAR_OK && slot == 0);
  CHECK(gar_plan_status(again) == GAR_OK);
  gar_plan_destroy(again);
}

// A streaming kernel that spills is built with fewer groups, down to two; a forced number of
// groups is kept.
void stream_groups() {
  fake::local_bytes = 64;
  gar_plan *pl = plan_of(127, 1u << 20, GAR_BF16, 7);
  CHECK(gar_plan_prepare(pl, GAR_FUSED) == GAR_OK && form_of(pl) == GAR_FORM_STREAM);
  const std::vector<void *> r = rows(127);
  CHECK(gar_allreduce(pl, r.data(), GAR_FUSED, nullptr) == GAR_OK);
  const char *forced = std::getenv("GAR_TUNE_ST_GROUPS");
  CHECK(fake::launches[0].block == 128u * (forced ? std::atoi(forced) : 2));
  gar_plan_destroy(pl);
}

// Threads batch over shared plans, in more sets than a plan remembers.
void batched_threads() {
  std::vector<gar_plan *> pl;
  for (int P = 2; P < 14; ++P) pl.push_back(plan_of(P, 100, GAR_F32, GAR_STEPS_BO));
  alignas(8) static gar_batch_desc desc[1];
  std::vector<std::thread> threads;
  for (int t = 0; t < 4; ++t)
    threads.emplace_back([&, t] {
      for (int k = 0; k < 60; ++k) {
        gar_plan *set[2] = {pl[0], pl[1 + (5 * t + k) % 11]};
        CHECK(gar_allreduce_batched(set, 2, desc, 1, nullptr) == GAR_OK);
      }
    });
  for (std::thread &t : threads) t.join();
  CHECK(fake::compiles == 11 && fake::launches.size() == 240);
  for (gar_plan *p : pl) gar_plan_destroy(p);
}

// A knob that changes a batched kernel's source reaches plans that remember a kernel, and a
// knob of the single-thread or breadth-first form keeps a plan to that form.
void knobs() {
  gar_plan *pl = plan_of(5, 100, GAR_BF16, GAR_STEPS_BO);
  alignas(8) static gar_batch_desc desc[1];
  int compiles = 0;
  for (const char *hint : {".cs", ".cs", ".cg", ".cg", ".cs"}) {
    setenv("GAR_TUNE_LDH", hint, 1);
    CHECK(gar_allreduce_batched(&pl, 1, desc, 1, nullptr) == GAR_OK);
    compiles += compiles == 0 || (compiles == 1 && std::string(hint) == ".cg");
    CHECK(fake::compiles == compiles);
  }
  gar_plan_destroy(pl);
  struct { const char *knob; int P; uint64_t n; int steps, form; } cases[] = {
      {"", 127, 1u << 20, 7, GAR_FORM_STREAM},  {"GAR_TUNE_BF_WARPS", 127, 1u << 20, 7, GAR_FORM_BREADTH},
      {"GAR_TUNE_BF_ORDER", 127, 1u << 20, 7, GAR_FORM_BREADTH}, {"", 24, 100, 7, GAR_FORM_COOP},
      {"GAR_TUNE_DOUBLED", 24, 100, 7, GAR_FORM_SINGLE}, {"GAR_TUNE_FADD2", 24, 100, 10, GAR_FORM_SINGLE}};
  for (const auto &c : cases) {
    if (*c.knob) setenv(c.knob, "1", 1);
    pl = plan_of(c.P, c.n, GAR_BF16, c.steps);
    CHECK(gar_plan_prepare(pl, GAR_FUSED) == GAR_OK && form_of(pl) == c.form);
    if (*c.knob) unsetenv(c.knob);
    gar_plan_destroy(pl);
  }
}

// A plan that is compiled ahead names the form that it will run, and preparing it compiles
// nothing more.
void compiled_ahead() {
  struct { int P; uint64_t n; int dtype, steps, form; } cases[] = {
      {127, 212, GAR_BF16, 14, GAR_FORM_COOP},      {24, 9000, GAR_F32, 10, GAR_FORM_COOP},
      {127, 1u << 20, GAR_BF16, 7, GAR_FORM_STREAM}, {127, 1u << 18, GAR_BF16, 7, GAR_FORM_BREADTH},
      {24, 1u << 20, GAR_F32, 10, GAR_FORM_SINGLE}};
  for (const auto &c : cases) {
    const int before = fake::compiles;
    gar_plan *pl = plan_of(c.P, c.n, c.dtype, c.steps);
    CHECK(gar_plan_compile(pl, GAR_FUSED) == GAR_OK && form_of(pl) == c.form);
    size_t len = 0, prepared = 0;
    CHECK(gar_plan_fused_source(pl, nullptr, &len) == GAR_OK);
    CHECK(gar_plan_prepare(pl, GAR_FUSED) == GAR_OK && form_of(pl) == c.form);
    CHECK(gar_plan_fused_source(pl, nullptr, &prepared) == GAR_OK && prepared == len);
    CHECK(fake::compiles == before + 1);
    gar_plan_destroy(pl);
  }
}

// The line of the cooperative form and its tiles follow the device's SM count, also of a plan
// that was compiled ahead without one.
void sm_count() {
  struct { int sms; uint64_t n; int form; unsigned grid; } cases[] = {
      {152, 4864, GAR_FORM_COOP, 152}, {152, 4865, GAR_FORM_SINGLE, 0}, {76, 2432, GAR_FORM_COOP, 76},
      {76, 2433, GAR_FORM_SINGLE, 0},  {76, 300, GAR_FORM_COOP, 75},    {152, 300, GAR_FORM_COOP, 75},
      {76, 600, GAR_FORM_COOP, 75},    {152, 600, GAR_FORM_COOP, 150}};
  const std::vector<void *> r = rows(48);
  for (bool ahead : {false, true})
    for (const auto &c : cases) {
      fake::sms[0] = c.sms;
      fake::launches.clear();
      gar_plan *pl = plan_of(48, c.n, GAR_F32, 12);
      if (ahead) CHECK(gar_plan_compile(pl, GAR_FUSED) == GAR_OK);
      CHECK(gar_allreduce(pl, r.data(), GAR_FUSED, nullptr) == GAR_OK && form_of(pl) == c.form);
      if (c.form == GAR_FORM_COOP) CHECK(fake::launches[0].grid == c.grid);
      gar_plan_destroy(pl);
    }
}

// The ranks from which short vectors take the cooperative form.
void cooperative_ranks() {
  struct { int P, steps, group, form; } cases[] = {
      {15, 8, GAR_GROUP_CYCLIC, GAR_FORM_SINGLE}, {16, 8, GAR_GROUP_CYCLIC, GAR_FORM_COOP},
      {16, 7, GAR_GROUP_CYCLIC, GAR_FORM_SINGLE}, {19, 8, GAR_GROUP_CYCLIC, GAR_FORM_SINGLE},
      {19, 10, GAR_GROUP_CYCLIC, GAR_FORM_COOP},  {20, 8, GAR_GROUP_CYCLIC, GAR_FORM_COOP},
      {20, 5, GAR_GROUP_CYCLIC, GAR_FORM_SINGLE}, {16, 8, GAR_GROUP_XOR, GAR_FORM_SINGLE},
      {32, 7, GAR_GROUP_XOR, GAR_FORM_COOP},      {32, 10, GAR_GROUP_XOR, GAR_FORM_COOP}};
  for (const auto &c : cases) {
    gar_plan *pl = nullptr;
    CHECK(gar_plan_create_group(&pl, c.P, 100, GAR_F32, GAR_SUM, c.steps, c.group) == GAR_OK);
    CHECK(gar_plan_compile(pl, GAR_FUSED) == GAR_OK);
    if (form_of(pl) != c.form) std::printf("P = %d, S = %d, group %d\n", c.P, c.steps, c.group);
    CHECK(form_of(pl) == c.form);
    gar_plan_destroy(pl);
  }
}

// A plan whose vectors are cut by block boundaries runs wider vectors on host memory than on
// the device, from a kernel that gar_plan_prepare or the first host call builds; other plans
// share one kernel.
void host_width() {
  struct { int P; uint64_t n; int dtype, steps; bool apart; } cases[] = {
      {8, 200003, GAR_F32, 6, true}, {8, 200003, GAR_BF16, 6, false}, {8, 1u << 20, GAR_F32, 6, false},
      {8, 8 * 4096, GAR_F32, 6, false}, {24, 100, GAR_F32, 10, false}, {6, 79063, GAR_I32, 5, true},
      {8, 65535, GAR_F32, 6, false}, {8, 65537, GAR_F32, 6, true}};
  for (const auto &c : cases)
    for (bool device_first : {false, true}) {
      const std::vector<void *> r = rows(c.P);
      const std::vector<const void *> in(r.begin(), r.end());
      gar_plan *pl = plan_of(c.P, c.n, c.dtype, c.steps);
      auto run = [&](bool host) {
        fake::memory = host ? cudaMemoryTypeHost : cudaMemoryTypeDevice;
        fake::launches.clear();
        fake::on_launch = [](fake::Function &f, const fake::Launch &) {
          fake::last_source = f.source;
          return cudaSuccess;
        };
        CHECK((host ? gar_allreduce_host(pl, in.data(), r.data(), r.data(), GAR_FUSED, nullptr)
                    : gar_allreduce(pl, r.data(), GAR_FUSED, nullptr)) == GAR_OK);
        CHECK(fake::launches.size() == 1);
        return fake::last_source;
      };
      const int before = fake::compiles;
      std::string source[2];
      for (int k = 0; k < 2; ++k) {
        const bool host = device_first ? k == 1 : k == 0;
        if (host && c.apart && device_first) {        // captured before the kernel is there
          fake::capture = cudaStreamCaptureStatusActive;
          CHECK(run(true) == source[0] && fake::compiles == before + (device_first ? 0 : 1));
          fake::capture = cudaStreamCaptureStatusNone;
        }
        source[host] = run(host);
        CHECK(run(host) == source[host]);
      }
      CHECK((source[0] != source[1]) == c.apart);
      gar_plan *ready = plan_of(c.P, c.n, c.dtype, c.steps);
      CHECK(gar_plan_prepare(ready, GAR_FUSED) == GAR_OK);
      std::swap(pl, ready);
      fake::capture = cudaStreamCaptureStatusActive;
      CHECK(run(true) == source[1] && run(false) == source[0]);
      fake::capture = cudaStreamCaptureStatusNone;
      gar_plan_destroy(ready);
      if (!device_first) CHECK(fake::compiles == before + (c.apart ? 2 : 1));
      if (c.apart) {
        CHECK(source[0].find("#define GAR_W 1\n") != std::string::npos);
        CHECK(source[1].find("#define GAR_W 4\n") != std::string::npos);
      }
      gar_plan_destroy(pl);
    }
}

// A fused call on host memory shares its CTAs out over whole rounds of about 3 MB of loads.
void host_grid() {
  fake::memory = cudaMemoryTypeHost;
  struct { uint64_t n; unsigned grid; } cases[] = {
      {8 * 40000, 313}, {8 * 46000, 360}, {8 * 56000, 438}, {8 * 60000, 367}, {8 * 140000, 365}, {8 * 1000000, 373}};
  const int P = 8;                                   // 8192 bytes of loads a CTA: 367 for 3 MB
  const std::vector<void *> r = rows(P);
  const std::vector<const void *> in(r.begin(), r.end());
  fake::regs = 8;                                    // 32 bytes a thread
  for (const auto &c : cases) {
    gar_plan *pl = plan_of(P, c.n, GAR_F32, 6);
    fake::launches.clear();
    CHECK(gar_allreduce_host(pl, in.data(), r.data(), r.data(), GAR_FUSED, nullptr) == GAR_OK);
    if (fake::launches[0].grid != c.grid) std::printf("%llu positions: %u CTAs\n", (unsigned long long)c.n, fake::launches[0].grid);
    CHECK(fake::launches[0].grid == c.grid);
    gar_plan_destroy(pl);
  }
}

}  // namespace

int main(int argc, char **argv) {
  const std::map<std::string, void (*)()> checks = {{"two_devices", two_devices}, {"wait_status", wait_status}, {"stream_groups", stream_groups},
      {"batched_threads", batched_threads}, {"knobs", knobs},
      {"compiled_ahead", compiled_ahead}, {"sm_count", sm_count},
      {"cooperative_ranks", cooperative_ranks}, {"host_width", host_width},
      {"host_grid", host_grid}};
  CHECK(argc == 2 && checks.count(argv[1]));
  checks.at(argv[1])();
  return 0;
}
