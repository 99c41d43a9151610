// As support_suite.cpp (whose launchers it takes), with the device's own sums of a run's
// angles, and a deviation that counts an amplitude that is not a number.
//   circuit_suite <n> <det> <c128|c64> <rots.bin> [<det written by the owner in between>]
// prints the status, the largest deviation ("nan" if any is), the launches that visited a part
// of the state and the blocks that visited a part of their tiles.
#define launch_phase_run launch_phase_run_radians
#define main support_main
#include "support_suite.cpp"
#undef main
#undef launch_phase_run

namespace qf {
cudaError_t launch_phase_run(void* p, int n, const PhaseArgs& a, cudaStream_t) {
  const Amp psi{p, QF_C128};
  uint64_t total = 0;
  for (int k = 0; k < a.m; ++k) {
    if (!(std::fabs(a.th[k]) <= kPhaseMaxAngle)) std::abort();
    total += phase_turns(a.th[k]);
  }
  for (uint64_t b : visited(a.on, n, a.h < 0 ? 0 : 1ull << a.h)) {
    uint64_t odd = 0;
    for (int k = 0; k < a.m; ++k)
      if (par(a.z[k] & b)) odd += phase_turns(a.th[k]);
    const double phi = M_PI * phase_halves(total - 2 * odd);
    const cplx u = psi.get(b), v = psi.get(b ^ a.x), f = cplx(0, -1) * std::sin(phi);
    psi.set(b, std::cos(phi) * u + f * std::conj(kI[a.y]) * v);
    if (a.x) psi.set(b ^ a.x, std::cos(phi) * v + f * kI[a.y] * u);
  }
  return cudaSuccess;
}
}  // namespace qf

int main(int argc, char** argv) {
  const int n = std::atoi(argv[1]);
  const uint64_t det = std::strtoull(argv[2], nullptr, 0), N = 1ull << n;
  const qf_dtype dt = std::string(argv[3]) == "c64" ? QF_C64 : QF_C128;
  std::vector<qf_rot> R(1 << 16);
  FILE* f = std::fopen(argv[4], "rb");
  R.resize(std::fread(R.data(), sizeof(qf_rot), R.size(), f));
  std::fclose(f);
  qf_state* st = nullptr;
  if (qf_state_create(n, dt, nullptr, nullptr, 0, &st) != QF_OK) return 2;
  qf_set_basis(st, det);
  void* p = nullptr;
  qf_state_info(st, nullptr, nullptr, &p, nullptr);
  const uint64_t start = argc > 5 ? std::strtoull(argv[5], nullptr, 0) : det;
  if (argc > 5) qf::launch_zero_and_set(p, n, dt, start, nullptr);
  std::vector<cplx> ref(N, 0.0);
  ref[start] = 1.0;
  qf_status s = qf_apply_circuit(st, R.data(), R.size() / 2);
  if (s == QF_OK) s = qf_apply_circuit(st, R.data() + R.size() / 2, R.size() - R.size() / 2);
  const std::vector<uint64_t> at = all(n);
  for (const qf_rot& r : R) rotate(Amp{ref.data(), QF_C128}, at, r.x, r.z, std::cos(r.theta), std::sin(r.theta));
  double scale = 1, worst = 0;
  qf_state_info(st, nullptr, nullptr, nullptr, &scale);
  for (uint64_t b = 0; b < N; ++b) {
    const double d = std::abs(scale * Amp{p, dt}.get(b) - ref[b]);
    if (!(d <= worst)) worst = d;
    if (worst != worst) break;
  }
  std::printf("%d %.3g %d %d\n", (int)s, worst, parts, inner);
  qf_state_destroy(st);
  return 0;
}
