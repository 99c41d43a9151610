// Grouped requests on a device without room for their item map: memory_suite <dir> prints the
// status and the grouped launches of a call whose allocations all fail, of one after it, and
// of one after the plans were dropped and made again.  memory_suite <dir> <n> <c128|c64> <det>
// <rows> prints the status and the device bytes a handle holds after a grouped call.
#define cudaMalloc stub_malloc
#define launch_small_eval stub_small_eval
#include "cuda_stub.cpp"
#undef cudaMalloc
#undef launch_small_eval

#include <vector>

static bool full = false;
static int grouped = 0;

extern "C" cudaError_t cudaMalloc(void** p, size_t n) { return full ? cudaErrorMemoryAllocation : stub_malloc(p, n); }
namespace qf {
cudaError_t launch_small_eval(const SmallEval& a, qf_dtype dt, int n_req, cudaStream_t s) {
  ++grouped;
  return stub_small_eval(a, dt, n_req, s);
}
}  // namespace qf

template <typename T>
static std::vector<T> load(const std::string& path) {
  FILE* f = std::fopen(path.c_str(), "rb");
  if (!f) std::exit(2);
  std::fseek(f, 0, SEEK_END);
  std::vector<T> v((size_t)std::ftell(f) / sizeof(T));
  std::fseek(f, 0, SEEK_SET);
  if (std::fread(v.data(), sizeof(T), v.size(), f) != v.size()) std::exit(2);
  std::fclose(f);
  return v;
}

static int held(const std::string& dir, int n, qf_dtype dt, uint64_t det, size_t rows) {
  const auto A = load<qf_arot>(dir + "/ansatz_fp.bin");
  const auto T = load<qf_term>(dir + "/terms_fp.bin");
  const auto t = load<double>(dir + "/t_fp.bin");
  std::vector<double> e(rows), g(t.size());
  qf_state* st = nullptr;
  if (qf_state_create(n, dt, nullptr, nullptr, 0, &st) != QF_OK) return 1;
  const qf_status s = qf_energy_grad_multi(st, det, A.data(), A.size(), t.data(), t.size() / rows, rows, T.data(),
                                           T.size(), e.data(), g.data());
  std::printf("%d %d %zu\n", (int)s, grouped, stub::live_bytes());
  return 0;
}

int main(int argc, char** argv) {
  const std::string dir = argv[1];
  if (argc > 5)
    return held(dir, std::atoi(argv[2]), std::string(argv[3]) == "c64" ? QF_C64 : QF_C128,
                std::strtoull(argv[4], nullptr, 0), std::strtoull(argv[5], nullptr, 0));
  const auto A = load<qf_arot>(dir + "/ansatz8.bin");
  const auto T = load<qf_term>(dir + "/terms8.bin");
  const auto t = load<double>(dir + "/t8.bin");
  const size_t rows = 4, npar = t.size() / rows;
  std::vector<double> e(rows), g(t.size());
  qf_state* st = nullptr;
  if (qf_state_create(8, QF_C128, nullptr, nullptr, 0, &st) != QF_OK) return 1;
  auto plan = [&] { return qf_energy_grad(st, 15, A.data(), A.size(), t.data(), npar, T.data(), T.size(), &e[0], g.data()); };
  auto call = [&] {
    grouped = 0;
    const qf_status s = qf_energy_grad_multi(st, 15, A.data(), A.size(), t.data(), npar, rows, T.data(), T.size(),
                                             e.data(), g.data());
    std::printf("%d %d ", (int)s, grouped);
  };
  if (plan() != QF_OK) return 1;
  full = true;
  call();
  full = false;
  call();
  qf_state_clear_plans(st);
  if (plan() != QF_OK) return 1;
  call();
  qf_state_destroy(st);
  std::printf("%zu\n", stub::live_bytes());
  return 0;
}
