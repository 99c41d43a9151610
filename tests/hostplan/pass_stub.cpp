// The launchers of the passes that cuda_stub.cpp leaves out, recorded like its own, so that
// the planner built with both plans what the library launches.
#include "qf_internal.h"

namespace stub {
void mix(const void* p, size_t n);
}

namespace qf {
template <typename T> static void mixv(const T& v) { stub::mix(&v, sizeof(T)); }
static void mix_on(const Reached& on) {
  mixv(on.nsup);
  if (on.nsup < 0) return;
  mixv(on.off);
  stub::mix(on.sup, sizeof(uint64_t) * on.nsup);
}
cudaError_t launch_sparse_on(void* psi, int n, qf_dtype dt, const SparseArgs& a, const Reached& on, bool realst,
                             cudaStream_t s) {
  mix_on(on);
  return launch_sparse(psi, n, dt, a, realst, s);
}
cudaError_t launch_block_pass(void*, int n, qf_dtype, const BlockPass& a, cudaStream_t) {
  mixv(n), mixv(a.s), mixv(a.nb), mix_on(a.on);
  stub::mix(a.b, sizeof(BlockRec) * a.nb);
  return cudaSuccess;
}
cudaError_t launch_phase_run(void*, int n, const PhaseArgs& a, cudaStream_t) {
  mixv(n), mixv(a.m), mixv(a.x), mixv(a.y), mix_on(a.on);
  stub::mix(a.z, sizeof(uint64_t) * a.m);
  stub::mix(a.th, sizeof(double) * a.m);
  return cudaSuccess;
}
cudaError_t launch_check_support(const void*, int n, qf_dtype, const Support& s, unsigned*, cudaStream_t) {
  mixv(n), mixv(s.d), mixv(s.off);
  stub::mix(s.v, sizeof(uint64_t) * s.d);
  return cudaSuccess;
}
cudaError_t launch_expect_passes(const void*, int n, qf_dtype, const ExpPass*, int npass, const PassGroup*,
                                 const PassChunk*, const ExpChunk*, double*, int, unsigned*, double*, cudaStream_t) {
  mixv(n), mixv(npass);
  return cudaSuccess;
}
}  // namespace qf
