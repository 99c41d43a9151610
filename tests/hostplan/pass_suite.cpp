// Expectation passes on the CUDA test double: the state, the plan's passes and the
// groups left to the per-group kernel are evaluated on the host with the kernels'
// own index arithmetic (thread by thread, pair by pair).
//   pass_suite <dir> <n> <c128|c64>   prints <psi|H|psi> of state.bin and terms.bin,
//                                     the pass count and the groups left over
#define launch_expect stub_launch_expect  // replaced below
#include "cuda_stub.cpp"
#undef launch_expect

#include <cmath>
#include <vector>

namespace {
int g_passes = 0, g_rest = 0;

struct Amp {
  const void* p;
  bool dbl;
  double re(uint64_t i) const { return dbl ? ((const double*)p)[2 * i] : ((const float*)p)[2 * i]; }
  double im(uint64_t i) const { return dbl ? ((const double*)p)[2 * i + 1] : ((const float*)p)[2 * i + 1]; }
};

template <typename T>
double run_passes(Amp psi, int n, const qf::ExpPass* passes, int npass, const qf::PassGroup* groups,
                  const qf::PassChunk* chunks, const qf::ExpChunk* tabs) {
  constexpr int S = qf::PassTile<T>::S, P = qf::PassTile<T>::P;
  double sum = 0.0;
  for (int p = 0; p < npass; ++p)
    for (uint64_t t = 0; t < (1ull << (n - S)); ++t) {
      uint64_t base = t;
      for (int i = 0; i < S; ++i)
        base = ((base >> passes[p].sbits[i]) << (passes[p].sbits[i] + 1)) | (base & ((1ull << passes[p].sbits[i]) - 1));
      auto at = [&](uint32_t j) {
        uint64_t b = base;
        for (int i = 0; i < S; ++i)
          if ((j >> i) & 1) b |= 1ull << passes[p].sbits[i];
        return b;
      };
      for (int g = passes[p].g0; g < passes[p].g1; ++g) {
        const qf::PassGroup& G = groups[g];
        const int flags = G.nchunk_flags & 7, nchunk = G.nchunk_flags >> 3;
        const uint32_t piv = G.hl < 0 ? 0u : 1u << G.hl;
        for (uint32_t tid = 0; tid < qf::kPassThreads; ++tid) {
          const uint32_t j0 = G.hl < 0 ? tid : ((tid >> G.hl) << (G.hl + 1)) | (tid & (piv - 1));
          for (int half = 0; half < (G.hl < 0 ? 2 : 1); ++half) {
            for (int k = 0; k < P; ++k) {
              uint32_t j = j0;  // k's bits on the bits above the thread's own, the pivot left out
              if (G.hl < 0) j += (uint32_t)(k + half * P) * qf::kPassThreads;
              for (int i = 0; G.hl >= 0 && i < S - 9; ++i)
                j |= (uint32_t)((k >> i) & 1) << (G.hl <= 8 || 8 + i >= G.hl ? 9 + i : 8 + i);
              const uint64_t b = at(j), b2 = at(j ^ G.xl);
              if (j >> S || (j ^ G.xl) >> S) std::exit(4);  // outside the tile
              const double re = psi.re(b) * psi.re(b2) + psi.im(b) * psi.im(b2);
              const double im = psi.im(b) * psi.re(b2) - psi.re(b) * psi.im(b2);
              for (int c = G.chunk; c < G.chunk + nchunk; ++c) {
                unsigned i = (unsigned)(chunks[c].kx[half] >> (4 * k)) & 15u;
                for (int q = 0; q < qf::kChunkTerms; ++q)
                  i ^= ((__builtin_popcount(chunks[c].zl[q] & j0) + __builtin_popcountll(chunks[c].zout[q] & base)) & 1)
                       << q;
                if (flags & 1) sum += tabs[c].tab[i].x * re;
                if (flags & 2) sum += tabs[c].tab[i].y * im;
              }
            }
          }
        }
      }
    }
  return sum;
}
}  // namespace

namespace qf {
cudaError_t launch_expect_passes(const void* psi, int n, qf_dtype dt, const ExpPass* passes, int npass,
                                 const PassGroup* groups, const PassChunk* chunks, const ExpChunk* tabs, double*, int,
                                 unsigned*, double* out, cudaStream_t) {
  g_passes = npass;
  out[0] = dt == QF_C128 ? run_passes<double>({psi, true}, n, passes, npass, groups, chunks, tabs)
                         : run_passes<float>({psi, false}, n, passes, npass, groups, chunks, tabs);
  return cudaSuccess;
}
cudaError_t launch_expect(const void* psi, int n, qf_dtype dt, const ExpGroup* groups, int ngroups,
                          const ExpChunk* chunks, double*, unsigned*, double* out, int, cudaStream_t) {
  const Amp a{psi, dt == QF_C128};
  g_rest = ngroups;
  out[0] = 0.0;
  for (int g = 0; g < ngroups; ++g)
    for (uint64_t b = 0; b < (1ull << n); ++b) {
      const ExpGroup& G = groups[g];
      if (G.h >= 0 && ((b >> G.h) & 1)) continue;
      const uint64_t b2 = b ^ G.x;
      for (int c = G.chunk0; c < G.chunk0 + G.nchunk; ++c) {
        unsigned i = 0;
        for (int q = 0; q < kChunkTerms; ++q) i |= (__builtin_popcountll(chunks[c].z[q] & b) & 1) << q;
        out[0] += chunks[c].tab[i].x * (a.re(b) * a.re(b2) + a.im(b) * a.im(b2));
        out[0] += chunks[c].tab[i].y * (a.im(b) * a.re(b2) - a.re(b) * a.im(b2));
      }
    }
  return cudaSuccess;
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

int main(int argc, char** argv) {
  if (argc < 4) return 1;
  const std::string dir = argv[1];
  const auto T = load<qf_term>(dir + "/terms.bin");
  const auto psi = load<char>(dir + "/state.bin");
  qf_state* st = nullptr;
  double re = 0.0, im = 0.0;
  if (qf_state_create(std::atoi(argv[2]), std::string(argv[3]) == "c64" ? QF_C64 : QF_C128, nullptr, nullptr, 0, &st) ||
      qf_state_copy_from_host(st, psi.data(), psi.size()) || qf_expectation(st, T.data(), T.size(), &re, &im)) {
    std::printf("#error %s\n", qf_last_error());
    return 3;
  }
  std::printf("%.17g %d %d\n", re, g_passes, g_rest);
  qf_state_destroy(st);
  return stub::live_bytes() == 0 ? 0 : 5;
}
