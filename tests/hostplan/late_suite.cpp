// Expectation passes of a Hamiltonian that another call has planned before (pass_suite.cpp's
// launchers): late_suite <dir> <n> <c128|c64> prints the value on a fresh handle and the value,
// passes and groups left over on a handle whose gradient call planned the terms.
#define main pass_main
#include "pass_suite.cpp"
#undef main

int main(int argc, char** argv) {
  const std::string dir = argv[1];
  const int n = std::atoi(argv[2]);
  const qf_dtype dt = std::string(argv[3]) == "c64" ? QF_C64 : QF_C128;
  const auto T = load<qf_term>(dir + "/terms.bin");
  const auto psi = load<char>(dir + "/state.bin");
  const qf_arot rot = {3, 4, 0.5, 0, 0};
  double re[2] = {0.0, 0.0}, im = 0.0, e = 0.0, g = 0.0;
  const double t = 0.3;
  for (int late = 0; late < 2; ++late) {
    qf_state* st = nullptr;
    if (qf_state_create(n, dt, nullptr, nullptr, 0, &st)) return 2;
    if (late && qf_energy_grad(st, 1, &rot, 1, &t, 1, T.data(), T.size(), &e, &g)) return 3;
    g_passes = 0;
    if (qf_state_copy_from_host(st, psi.data(), psi.size()) || qf_expectation(st, T.data(), T.size(), &re[late], &im))
      return 4;
    qf_state_destroy(st);
  }
  std::printf("%.17g %.17g %d %d\n", re[0], re[1], g_passes, g_rest);
  return stub::live_bytes() == 0 ? 0 : 5;
}
