// Circuits on a determinant, planned by the C ABI and carried out on the host exactly as
// launched: each pass touches only the tiles, outside patterns or pairs it is told to visit.
//   support_suite <n> <det> <c128|c64> <rots.bin> [<det written by the owner in between>]
// prints the status, the largest deviation from the rotations applied one by one, how many
// launches visited a part of the state and how many blocks a part of their tiles.  The launchers replaced here are those that
// cuda_stub.cpp, compiled with them renamed, would only record.
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <string>
#include <vector>

#include "qf.h"
#include "qf_internal.h"

typedef std::complex<double> cplx;
static int parts = 0, inner = 0;
static int par(uint64_t v) { return __builtin_parityll(v); }
static const cplx kI[4] = {{1, 0}, {0, 1}, {-1, 0}, {0, -1}};

struct Amp {  // amplitudes of either type
  void* p;
  qf_dtype dt;
  cplx get(uint64_t b) const {
    return dt == QF_C128 ? static_cast<cplx*>(p)[b] : cplx(static_cast<std::complex<float>*>(p)[b]);
  }
  void set(uint64_t b, cplx v) const {
    if (dt == QF_C128)
      static_cast<cplx*>(p)[b] = v;
    else
      static_cast<std::complex<float>*>(p)[b] = std::complex<float>(v);
  }
};
// The values of the bits outside `set` that a pass visits.
static std::vector<uint64_t> visited(const qf::Reached& on, int n, uint64_t set) {
  std::vector<uint64_t> v;
  if (on.nsup >= 0 && (!on.dense || *on.dense == 0)) {
    ++parts;
    for (uint64_t t = 0; t < (1ull << on.nsup); ++t) {
      uint64_t b = on.off;
      for (int i = 0; i < on.nsup; ++i)
        if ((t >> i) & 1) b ^= on.sup[i];
      if (b & set) std::abort();
      v.push_back(b);
    }
    return v;
  }
  for (uint64_t b = 0; b < (1ull << n); ++b)
    if (!(b & set)) v.push_back(b);
  return v;
}
static uint64_t expand(uint64_t o, const int* bits, int s) {
  uint64_t v = 0;
  for (int i = 0; i < s; ++i)
    if ((o >> i) & 1) v |= 1ull << bits[i];
  return v;
}
// A psi - i B P psi on the given indices (closed under ^ x).
static void rotate(const Amp& psi, const std::vector<uint64_t>& at, uint64_t x, uint64_t z, double A, double B) {
  std::vector<cplx> out(at.size());
  for (size_t k = 0; k < at.size(); ++k) {
    const uint64_t b = at[k], c = b ^ x;
    const cplx p = kI[__builtin_popcountll(x & z) & 3] * (par(z & c) ? -1.0 : 1.0) * psi.get(c);
    out[k] = A * psi.get(b) - cplx(0, 1) * B * p;
  }
  for (size_t k = 0; k < at.size(); ++k) psi.set(at[k], out[k]);
}
static std::vector<uint64_t> all(int n) {
  qf::Reached on{};
  on.nsup = -1;
  return visited(on, n, 0);
}

namespace qf {
cudaError_t launch_zero_and_set(void* p, int n, qf_dtype dt, uint64_t det, cudaStream_t) {
  for (uint64_t b = 0; b < (1ull << n); ++b) Amp{p, dt}.set(b, b == det ? 1.0 : 0.0);
  return cudaSuccess;
}
cudaError_t launch_rot(void* p, int n, qf_dtype dt, const RotArgs& a, cudaStream_t) {
  rotate(Amp{p, dt}, all(n), a.x, a.z, a.A, a.B);
  return cudaSuccess;
}
cudaError_t launch_tile(void* p, int n, qf_dtype dt, const TileArgs& a, cudaStream_t) {
  const uint64_t S = expand(~0ull, a.sbits, a.s);
  for (uint64_t base : visited(a.on, n, S)) {
    std::vector<uint64_t> at;
    for (uint64_t j = 0; j < (1ull << a.s); ++j) at.push_back(base | expand(j, a.sbits, a.s));
    for (int t = 0; t < a.m; ++t)
      rotate(Amp{p, dt}, at, expand(a.r[t].xl, a.sbits, a.s), expand(a.r[t].zl, a.sbits, a.s) | a.r[t].zout, a.r[t].A,
             a.r[t].B);
  }
  return cudaSuccess;
}
cudaError_t launch_sparse_on(void* p, int n, qf_dtype dt, const SparseArgs& a, const Reached& on, bool, cudaStream_t) {
  const Amp psi{p, dt};
  const uint64_t S = expand(~0ull, a.supp, a.u);
  for (uint64_t base : visited(on, n, S)) {
    const int c = (a.nzc > 0 ? par(a.zc[0] & base) : 0) | (a.nzc > 1 ? par(a.zc[1] & base) << 1 : 0);
    std::vector<cplx> v(a.nr);
    for (int r = 0; r < a.nr; ++r) v[r] = psi.get(base | a.pat[r]);
    for (int r = 0; r < a.nr; ++r) {
      cplx o = v[r];
      for (int q = 0; q < a.nr; ++q) o += cplx(a.M[c][r][q].x, a.M[c][r][q].y) * v[q];
      psi.set(base | a.pat[r], o);
    }
  }
  return cudaSuccess;
}
cudaError_t launch_sparse(void* p, int n, qf_dtype dt, const SparseArgs& a, bool r, cudaStream_t s) {
  Reached on{};
  on.nsup = -1;
  return launch_sparse_on(p, n, dt, a, on, r, s);
}
cudaError_t launch_block_pass(void* p, int n, qf_dtype dt, const BlockPass& a, cudaStream_t) {
  const Amp psi{p, dt};
  const bool part = a.on.nsup >= 0 && (!a.on.dense || *a.on.dense == 0);
  uint64_t t = 0;
  for (uint64_t base : visited(a.on, n, expand(~0ull, a.sbits, a.s))) {
    uint64_t in_tile = a.loff;
    for (int i = 0; part && i < a.on.nsup; ++i)
      if ((t >> i) & 1) in_tile ^= a.lsup[i];
    ++t;
    for (int b = 0; b < a.nb; ++b) {
      const BlockRec& R = a.b[b];
      uint64_t supp = 0;
      for (int i = 0; i < R.u; ++i) supp |= 1ull << R.supp[i];
      const bool some = part && R.nin < a.s - R.u;
      inner += some;
      auto patterns = [&](int q) {  // of pair q
        std::vector<uint64_t> js;
        if (!some) {
          for (uint64_t j = 0; j < (1ull << a.s); ++j)
            if (!(j & supp)) js.push_back(j);
          return js;
        }
        if (R.supp_mask != supp || R.omask != ((1ull << a.s) - 1 & ~supp)) std::abort();
        uint64_t w = in_tile;
        if (w >> R.supp[R.u - 1] & 1) w ^= supp;
        for (int l = 0; l < R.nlift; ++l)
          if ((w ^ R.pat[q][0]) >> (63 - __builtin_clzll(R.lift[l] & supp)) & 1) w ^= R.lift[l];
        if ((w ^ R.pat[q][0]) & supp) return js;
        for (uint64_t o = 0; o < (1ull << R.nin); ++o) {
          uint64_t j = w & R.omask;
          for (int i = 0; i < R.nin; ++i)
            if ((o >> i) & 1) j ^= R.in[i];
          js.push_back(j);
        }
        return js;
      };
      for (int q = 0; q < R.np; ++q)
        for (uint64_t j : patterns(q)) {
          const int c = par(R.zl & j) ^ par(R.zout & base);
          const double* m = R.M[c][q];
          const cplx l = R.turn ? cplx(0, 1) : cplx(1, 0);
          const uint64_t iu = base | expand(j | R.pat[q][0], a.sbits, a.s), iv = base | expand(j | R.pat[q][1], a.sbits, a.s);
          const cplx u = psi.get(iu), v = psi.get(iv);
          psi.set(iu, u + m[0] * u + l * m[1] * v);
          psi.set(iv, v + l * m[2] * u + m[3] * v);
        }
    }
  }
  return cudaSuccess;
}
cudaError_t launch_phase_run(void* p, int n, const PhaseArgs& a, cudaStream_t) {
  const Amp psi{p, QF_C128};
  for (uint64_t b : visited(a.on, n, a.h < 0 ? 0 : 1ull << a.h)) {
    double phi = 0;
    for (int k = 0; k < a.m; ++k) phi += par(a.z[k] & b) ? -a.th[k] : a.th[k];
    const cplx u = psi.get(b), v = psi.get(b ^ a.x), f = cplx(0, -1) * std::sin(phi);
    psi.set(b, std::cos(phi) * u + f * std::conj(kI[a.y]) * v);
    if (a.x) psi.set(b ^ a.x, std::cos(phi) * v + f * kI[a.y] * u);
  }
  return cudaSuccess;
}
cudaError_t launch_check_support(const void* p, int n, qf_dtype dt, const Support& s, unsigned* dense, cudaStream_t) {
  for (uint64_t b = 0; b < (1ull << n); ++b) {
    if (Amp{const_cast<void*>(p), dt}.get(b) == 0.0) continue;
    uint64_t w = b ^ s.off;
    for (int i = 0; i < s.d; ++i)
      if ((w >> (63 - __builtin_clzll(s.v[i]))) & 1) w ^= s.v[i];
    if (w) *dense = 1;
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
  std::vector<cplx> ref(N, 0.0);
  uint64_t start = det;
  if (argc > 5) {
    start = std::strtoull(argv[5], nullptr, 0);
    qf::launch_zero_and_set(p, n, dt, start, nullptr);
  }
  ref[start] = 1.0;
  // two calls: the second starts from what the first has reached
  qf_status s = qf_apply_circuit(st, R.data(), R.size() / 2);
  if (s == QF_OK) s = qf_apply_circuit(st, R.data() + R.size() / 2, R.size() - R.size() / 2);
  const std::vector<uint64_t> at = all(n);
  for (const qf_rot& r : R) rotate(Amp{ref.data(), QF_C128}, at, r.x, r.z, std::cos(r.theta), std::sin(r.theta));
  double scale = 1, worst = 0;
  qf_state_info(st, nullptr, nullptr, nullptr, &scale);
  for (uint64_t b = 0; b < N; ++b) worst = std::max(worst, std::abs(scale * Amp{p, dt}.get(b) - ref[b]));
  std::printf("%d %.3g %d %d\n", (int)s, worst, parts, inner);
  qf_state_destroy(st);
  return 0;
}
