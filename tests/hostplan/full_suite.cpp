// Expectation values on a device without room for the passes' tables (pass_suite.cpp's
// launchers): full_suite <dir> <n> <c128|c64> prints, for three calls without room and one with,
// the passes taken and the host allocations of the call, and whether all values agree.
#include <atomic>
#include <cstdlib>
#include <new>

static std::atomic<long> allocations{0};
void* operator new(std::size_t n) {
  ++allocations;
  if (void* p = std::malloc(n ? n : 1)) return p;
  throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }

#define cudaMalloc stub_malloc
#define main pass_main
#include "pass_suite.cpp"
#undef main
#undef cudaMalloc

static bool full = false;
extern "C" cudaError_t cudaMalloc(void** p, size_t n) { return full ? cudaErrorMemoryAllocation : stub_malloc(p, n); }

int main(int argc, char** argv) {
  const std::string dir = argv[1];
  const int n = std::atoi(argv[2]);
  const auto T = load<qf_term>(dir + "/terms.bin");
  const auto psi = load<char>(dir + "/state.bin");
  const qf_arot rot = {3, 4, 0.5, 0, 0};
  double re[4], im = 0.0, e = 0.0, g = 0.0;
  const double t = 0.3;
  qf_state* st = nullptr;
  if (qf_state_create(n, std::string(argv[3]) == "c64" ? QF_C64 : QF_C128, nullptr, nullptr, 0, &st)) return 2;
  if (qf_energy_grad(st, 1, &rot, 1, &t, 1, T.data(), T.size(), &e, &g)) return 3;  // plans the terms
  if (qf_state_copy_from_host(st, psi.data(), psi.size())) return 3;
  for (int k = 0; k < 4; ++k) {
    full = k < 3;
    g_passes = 0;
    const long before = allocations;
    if (qf_expectation(st, T.data(), T.size(), &re[k], &im)) return 4;
    const long made = allocations - before;
    std::printf("%d %ld ", g_passes, made);
  }
  const bool same = std::abs(re[0] - re[3]) < 1e-12 && re[0] == re[1] && re[0] == re[2];
  std::printf("%d\n", (int)same);
  qf_state_destroy(st);
  return stub::live_bytes() == 0 ? 0 : 5;
}
