// CUDA kernels of libqf for GB300 (sm_103a).
//
// Every kernel streams the 2^n-amplitude state vector (interleaved complex,
// double2 for complex128, float2 for complex64).  The rotation kernels apply
// exp(-i theta P) (Eq. 9, with the factor -i theta of Eq. 11) as a pair swap
// b <-> b xor x with the phase i^{popc(x&z)} (-1)^{popc(z&b)} of the Pauli
// string (Eq. 10); the expectation kernels evaluate exact operator averaging
// (Eq. 18) with the terms grouped by X mask.  Reductions are FP64 for both
// state precisions and deterministic (fixed-order second stage).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstring>
#include <type_traits>
#include <vector>

#include "qf_internal.h"

namespace qf {

namespace {

template <typename T> struct Cx;
template <> struct Cx<double> { using V = double2; };
template <> struct Cx<float> { using V = float2; };

__device__ __forceinline__ double flip(double v, unsigned neg) {
  return __longlong_as_double(__double_as_longlong(v) ^ ((unsigned long long)(neg & 1u) << 63));
}
__device__ __forceinline__ float flip(float v, unsigned neg) {
  return __int_as_float(__float_as_int(v) ^ (int)((neg & 1u) << 31));
}

// i^k * v for k in 0..3, done with component swaps and sign-bit flips only.
template <typename V>
__device__ __forceinline__ V qturn(V v, unsigned k) {
  V o;
  o.x = flip((k & 1u) ? v.y : v.x, (k ^ (k >> 1)) & 1u);
  o.y = flip((k & 1u) ? v.x : v.y, (k >> 1) & 1u);
  return o;
}

// The form is a compile-time parameter: with a runtime form the compiler
// evaluates every branch, tripling the FP64 work of the one-FMA forms.
template <int F, typename T, typename V>
__device__ __forceinline__ V comb(V u, V w, T A, T B) {
  V o;
  if (F == FORM_A1) {
    o.x = fma(B, w.x, u.x);
    o.y = fma(B, w.y, u.y);
  } else if (F == FORM_B1) {
    o.x = fma(A, u.x, w.x);
    o.y = fma(A, u.y, w.y);
  } else {
    o.x = fma(B, w.x, A * u.x);
    o.y = fma(B, w.y, A * u.y);
  }
  return o;
}

__device__ __forceinline__ uint64_t ins0(uint64_t p, int h) {
  return ((p >> h) << (h + 1)) | (p & ((1ull << h) - 1ull));
}

__device__ __forceinline__ unsigned par64(uint64_t v) { return (unsigned)__popcll(v) & 1u; }

// ---------------------------------------------------------------------------
// deterministic block + grid reduction (the last block to finish sums the
// per-block partials in index order)

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

__device__ double block_sum(double v) {
  __shared__ double red[32];
  __syncthreads();
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) red[wid] = v;
  __syncthreads();
  const int nw = (blockDim.x + 31) >> 5;
  v = (threadIdx.x < nw) ? red[threadIdx.x] : 0.0;
  if (wid == 0) v = warp_sum(v);
  return v;  // valid in thread 0
}

__device__ void grid_finish(double v, double* partials, unsigned* counter, double* out) {
  __shared__ bool last;
  double bs = block_sum(v);
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = bs;
    __threadfence();
    unsigned t = atomicAdd(counter, 1u);
    last = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (last) {
    __threadfence();
    double s = 0.0;
    for (unsigned i = threadIdx.x; i < gridDim.x; i += blockDim.x) s += __ldcg(partials + i);
    s = block_sum(s);
    if (threadIdx.x == 0) {
      *out = s;
      *counter = 0u;
    }
  }
}

// Two sums at once (out[0], out[1]); partials holds 2 * gridDim.x doubles.
__device__ void grid_finish2(double v0, double v1, double* partials, unsigned* counter, double* out) {
  __shared__ bool last2;
  const double b0 = block_sum(v0);
  const double b1 = block_sum(v1);
  if (threadIdx.x == 0) {
    partials[2 * blockIdx.x] = b0;
    partials[2 * blockIdx.x + 1] = b1;
    __threadfence();
    unsigned t = atomicAdd(counter, 1u);
    last2 = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (last2) {
    __threadfence();
    double s0 = 0.0, s1 = 0.0;
    for (unsigned i = threadIdx.x; i < gridDim.x; i += blockDim.x) {
      s0 += __ldcg(partials + 2 * i);
      s1 += __ldcg(partials + 2 * i + 1);
    }
    s0 = block_sum(s0);
    s1 = block_sum(s1);
    if (threadIdx.x == 0) {
      out[0] = s0;
      out[1] = s1;
      *counter = 0u;
    }
  }
}

// ---------------------------------------------------------------------------
// state preparation

template <typename V>
__global__ void k_zero_and_set(V* psi, uint64_t N, uint64_t det) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < N; i += stride) {
    V v;
    v.x = (i == det) ? 1 : 0;
    v.y = 0;
    psi[i] = v;
  }
}

// out[2k], out[2k + 1] = the amplitude at idx[k] (0 where idx[k] < 0); packed:
// the real value stored in the imaginary slot, imaginary part 0.
// The same for a packed double-single state: (re hi, re lo, packed hi, packed lo).
__global__ void k_gather_ds(const float4* __restrict__ src, const int64_t* __restrict__ idx, int count,
                            double* __restrict__ out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= count) return;
  const int64_t i = idx[k];
  double re = 0.0;
  if (i >= 0) {
    const float4 v = src[i];
    re = (double)v.z + (double)v.w;
  }
  out[2 * k] = re;
  out[2 * k + 1] = 0.0;
}

template <typename V>
__global__ void k_gather(const V* __restrict__ src, const int64_t* __restrict__ idx, int count, int packed,
                         double* __restrict__ out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= count) return;
  const int64_t i = idx[k];
  double re = 0.0, im = 0.0;
  if (i >= 0) {
    const V v = src[i];
    if (packed) {
      re = (double)v.y;
    } else {
      re = (double)v.x;
      im = (double)v.y;
    }
  }
  out[2 * k] = re;
  out[2 * k + 1] = im;
}

template <typename T>
__global__ void k_scale(typename Cx<T>::V* psi, uint64_t N, T s) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < N; i += stride) {
    auto v = psi[i];
    v.x *= s;
    v.y *= s;
    psi[i] = v;
  }
}

// ---------------------------------------------------------------------------
// unfused rotation: one read + one write sweep of the state
//
// For the pair (b, b' = b xor x) with b's pivot bit h clear and par = popc(z&b) mod 2:
//   out[b]  = A u + B i^{3+3y+2par} v,     out[b'] = A v + B i^{3+y+2par} u,
// which is c u - i s (P psi)[b] etc. with A = c, B = s (up to the kept scale).
// Each thread takes the two pairs (b, b|1) so the partner amplitudes also form
// an aligned 2-vector (needs h >= 1).

template <typename T, int F>
__global__ void __launch_bounds__(256) k_rot_pair2(typename Cx<T>::V* __restrict__ psi, uint64_t nquads, uint64_t x,
                                                   uint64_t z, int h, int y, T A, T B) {
  using V = typename Cx<T>::V;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const unsigned z0 = (unsigned)(z & 1ull);
  for (uint64_t q = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; q < nquads; q += stride) {
    const uint64_t b0 = ins0(q << 1, h);  // even, pivot clear
    const uint64_t b1 = b0 | 1ull;
    const uint64_t c0 = b0 ^ x, c1 = b1 ^ x;
    const V u0 = psi[b0], u1 = psi[b1];
    const V v0 = psi[c0], v1 = psi[c1];
    const unsigned p0 = par64(z & b0), p1 = p0 ^ z0;
    psi[b0] = comb<F, T, V>(u0, qturn(v0, (3u + 3u * y + 2u * p0) & 3u), A, B);
    psi[b1] = comb<F, T, V>(u1, qturn(v1, (3u + 3u * y + 2u * p1) & 3u), A, B);
    psi[c0] = comb<F, T, V>(v0, qturn(u0, (3u + y + 2u * p0) & 3u), A, B);
    psi[c1] = comb<F, T, V>(v1, qturn(u1, (3u + y + 2u * p1) & 3u), A, B);
  }
}

// x == 1: the pair is the aligned 2-vector (2q, 2q+1).
template <typename T, int F>
__global__ void __launch_bounds__(256) k_rot_pair1(typename Cx<T>::V* __restrict__ psi, uint64_t npairs, uint64_t z,
                                                   int y, T A, T B) {
  using V = typename Cx<T>::V;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t q = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; q < npairs; q += stride) {
    const uint64_t b = q << 1;
    const V u = psi[b], v = psi[b | 1ull];
    const unsigned p = par64(z & b);
    psi[b] = comb<F, T, V>(u, qturn(v, (3u + 3u * y + 2u * p) & 3u), A, B);
    psi[b | 1ull] = comb<F, T, V>(v, qturn(u, (3u + y + 2u * p) & 3u), A, B);
  }
}

// x == 0: diagonal phase, out[b] = A u + B i^{3+2par} u.
template <typename T, int F>
__global__ void __launch_bounds__(256) k_rot_diag(typename Cx<T>::V* __restrict__ psi, uint64_t N, uint64_t z, T A,
                                                  T B) {
  using V = typename Cx<T>::V;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t b = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; b < N; b += stride) {
    const V u = psi[b];
    psi[b] = comb<F, T, V>(u, qturn(u, (3u + 2u * par64(z & b)) & 3u), A, B);
  }
}

// ---------------------------------------------------------------------------
// fused rotations in a shared-memory tile
//
// A tile is the 2^s amplitudes whose bits outside the tile bit set S are fixed
// (S holds the union of the pass's X supports plus low bits for coalescing).
// The tile is read once, all m rotations act on it in shared memory (the part
// of z outside S only flips the sign class of the whole tile), and it is
// written once.

// One rotation of a fused pass on the staged tile.
template <int F, typename T>
__device__ __forceinline__ void tile_rot(typename Cx<T>::V* tile, const TileRot& R, unsigned pout, unsigned tsize, T A,
                                         T B) {
  using V = typename Cx<T>::V;
  if (R.hl < 0) {
    for (unsigned j = threadIdx.x; j < tsize; j += blockDim.x) {
      const unsigned p = (__popc(R.zl & j) + pout) & 1u;
      const V u = tile[j];
      tile[j] = comb<F, T, V>(u, qturn(u, (3u + 2u * p) & 3u), A, B);
    }
  } else {
    const unsigned hmask = (1u << R.hl) - 1u;
    for (unsigned q = threadIdx.x; q < (tsize >> 1); q += blockDim.x) {
      const unsigned j = ((q >> R.hl) << (R.hl + 1)) | (q & hmask);
      const unsigned jp = j ^ R.xl;
      const unsigned p = (__popc(R.zl & j) + pout) & 1u;
      const V u = tile[j], v = tile[jp];
      tile[j] = comb<F, T, V>(u, qturn(v, (3u + 3u * R.y + 2u * p) & 3u), A, B);
      tile[jp] = comb<F, T, V>(v, qturn(u, (3u + R.y + 2u * p) & 3u), A, B);
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(256) k_tile(typename Cx<T>::V* __restrict__ psi, int n,
                                              const __grid_constant__ TileArgs a) {
  using V = typename Cx<T>::V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* tile = reinterpret_cast<V*>(smem_raw);
  uint64_t* hitab = reinterpret_cast<uint64_t*>(tile + (1 << a.s));
  const int s = a.s, l = a.l;
  const unsigned tsize = 1u << s, lmask = (1u << l) - 1u;
  for (int j = threadIdx.x; j < (1 << a.nhi); j += blockDim.x) {
    uint64_t off = 0;
    for (int i = 0; i < a.nhi; ++i)
      if ((j >> i) & 1) off |= 1ull << a.pos[i];
    hitab[j] = off;
  }
  const uint64_t ntiles = 1ull << (n - s);
  for (uint64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    uint64_t base = t;
    for (int i = 0; i < s; ++i) base = ins0(base, a.sbits[i]);
    __syncthreads();
#pragma unroll 8
    for (unsigned j = threadIdx.x; j < tsize; j += blockDim.x) tile[j] = psi[base | hitab[j >> l] | (j & lmask)];
    __syncthreads();
    for (int r = 0; r < a.m; ++r) {
      const TileRot R = a.r[r];
      const unsigned pout = par64(R.zout & base);
      const T A = (T)R.A, B = (T)R.B;
      if (R.form == FORM_A1)
        tile_rot<FORM_A1, T>(tile, R, pout, tsize, A, B);
      else if (R.form == FORM_B1)
        tile_rot<FORM_B1, T>(tile, R, pout, tsize, A, B);
      else
        tile_rot<FORM_AB, T>(tile, R, pout, tsize, A, B);
      __syncthreads();
    }
    for (unsigned j = threadIdx.x; j < tsize; j += blockDim.x) psi[base | hitab[j >> l] | (j & lmask)] = tile[j];
  }
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
}

// The outside patterns a pass visits (see Reached), after griddepcontrol.wait.
__device__ __forceinline__ bool on_part(const Reached& r) {
  return r.nsup >= 0 && (!r.dense || __ldcg(r.dense) == 0u);
}
__device__ __forceinline__ uint64_t reached(const Reached& r, uint64_t t) {
  uint64_t b = r.off;
  for (int i = 0; i < r.nsup; ++i) b ^= r.sup[i] & (0ull - ((t >> i) & 1ull));
  return b;
}

// ---------------------------------------------------------------------------
// fused rotation passes on tiles of 2^S amplitudes (S >= 10; k_tile below that)
//
// A CTA stages a tile by asynchronous copies, applies the pass's rotations in
// shared memory and writes it back; three CTAs per SM (large tiles) overlap one's
// copies with the others' rotations.  Thread tid takes the pairs j0 + o_k,
// (j0 ^ xl) ^ o_k, with o_k constants (TilePairs), so a pair costs one XOR and the
// rotation's multiply-adds; its sign is the thread's parity times a sign per k.
// complex128 is bound by the FP64 pipe (four multiply-adds per pair), complex64 by
// the state's read and write per pass.
// ADJ: psi and lam tiles side by side; each rotation first adds its overlap into the
// thread's own slot in shared memory, summed over the CTA once, after its last tile.

// The pairs of a thread for pivot case C (see PassPairs), in groups of U.
template <int S, int C> struct TilePairs {
  static constexpr int P = 1 << (S - 9), KB = S - 9, U = P < 4 ? P : 4;
  static __device__ __forceinline__ unsigned off(int k) {
    unsigned o = 0;
#pragma unroll
    for (int i = 0; i < KB; ++i)
      if ((k >> i) & 1) o |= 1u << (C == 0 ? 9 + i : 8 + i < 8 + C ? 8 + i : 9 + i);
    return o;
  }
};

// u' = A u + B i^{3+3y+2p} v, v' = A v + B i^{3+y+2p} u for y odd (YODD) and even; neg: p
// plus the sign y itself gives.  F: the coefficient form.
template <int F, bool YODD, typename T, typename V>
__device__ __forceinline__ void rot_pair(V& u, V& v, T A, T B, unsigned neg) {
  // the partner's image is (v, -u) for odd y, (i v, i u) for even y; signs go on the
  // coefficient or by the sign bit (a negated double that feeds a bit operation would
  // cost an FP64 addition)
  const V u0 = u, v0 = v;
  if (F == FORM_B1) {
    u.x = fma(A, u0.x, YODD ? flip(v0.x, neg) : flip(v0.y, neg ^ 1u));
    u.y = fma(A, u0.y, YODD ? flip(v0.y, neg) : flip(v0.x, neg));
    v.x = fma(A, v0.x, YODD ? flip(u0.x, neg ^ 1u) : flip(u0.y, neg ^ 1u));
    v.y = fma(A, v0.y, YODD ? flip(u0.y, neg ^ 1u) : flip(u0.x, neg));
  } else {
    const T b = flip(B, neg), c = flip(B, neg ^ 1u);
    const bool ab = F == FORM_AB;
    u.x = fma(YODD ? b : c, YODD ? v0.x : v0.y, ab ? A * u0.x : u0.x);
    u.y = fma(b, YODD ? v0.y : v0.x, ab ? A * u0.y : u0.y);
    v.x = fma(c, YODD ? u0.x : u0.y, ab ? A * v0.x : v0.x);
    v.y = fma(YODD ? c : b, YODD ? u0.y : u0.x, ab ? A * v0.y : v0.y);
  }
}

// Running sum of products a * b: FP64, or exact FP32 products in a float pair.
template <typename T> struct DotAcc;
template <> struct DotAcc<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double a, double b) { s = fma(a, b, s); }
  __device__ __forceinline__ double value() const { return s; }
};
template <> struct DotAcc<float> {
  float h = 0.f, l = 0.f;
  __device__ __forceinline__ void add(float a, float b) {
    const float p = __fmul_rn(a, b);
    const float e = fmaf(a, b, -p);
    const float t = __fadd_rn(h, p);
    const float bp = __fsub_rn(t, h);
    const float r = __fadd_rn(__fsub_rn(h, __fsub_rn(t, bp)), __fsub_rn(p, bp));
    l = __fadd_rn(l, __fadd_rn(r, e));
    h = t;
  }
  __device__ __forceinline__ double value() const { return (double)h + (double)l; }
};

// One rotation with X part xl != 0 on a tile; the thread's overlap when ADJ.
template <typename T, int S, int C, int F, bool YODD, bool ADJ>
__device__ __forceinline__ double tile_pairs(unsigned char* psi, unsigned char* lam, unsigned j0, unsigned xl,
                                             unsigned zl, unsigned neg0, T A, T B) {
  using V = typename Cx<T>::V;
  using TP = TilePairs<S, C>;
  constexpr unsigned sz = sizeof(V);
  DotAcc<T> even, odd;  // pairs of positive and negative sign
#pragma unroll 1
  for (int kb = 0; kb < TP::P; kb += TP::U) {
    const unsigned oh = TP::off(kb);
    const unsigned nh = neg0 ^ (unsigned)__popc(zl & oh);
    const unsigned a = (j0 + oh) * sz, b = ((j0 ^ xl) ^ oh) * sz;
#pragma unroll
    for (int k = 0; k < TP::U; ++k) {
      const unsigned o = TP::off(k);
      const unsigned neg = nh ^ (unsigned)__popc(zl & o);
      V* pu = reinterpret_cast<V*>(psi + a + o * sz);
      V* pv = reinterpret_cast<V*>(psi + (b ^ (o * sz)));
      V u = *pu, v = *pv;
      if (ADJ) {
        V* qu = reinterpret_cast<V*>(lam + a + o * sz);
        V* qv = reinterpret_cast<V*>(lam + (b ^ (o * sz)));
        V p = *qu, r = *qv;
        // even y: Im conj(p) v + Im conj(r) u; odd y: Re conj(r) u - Re conj(p) v
        V su = u, sv = v;  // psi with the pair's sign
        su.x = flip(su.x, neg);
        su.y = flip(su.y, neg);
        sv.x = flip(sv.x, neg);
        sv.y = flip(sv.y, neg);
        if (YODD) {
          even.add(r.x, su.x);
          even.add(r.y, su.y);
          odd.add(-p.x, sv.x);
          odd.add(-p.y, sv.y);
        } else {
          even.add(p.x, sv.y);
          even.add(-p.y, sv.x);
          odd.add(r.x, su.y);
          odd.add(-r.y, su.x);
        }
        rot_pair<F, YODD, T, V>(p, r, A, B, neg);
        *qu = p;
        *qv = r;
      }
      rot_pair<F, YODD, T, V>(u, v, A, B, neg);
      *pu = u;
      *pv = v;
    }
  }
  return ADJ ? even.value() + odd.value() : 0.0;
}

// A diagonal rotation: out = A u + B i^{3+2p} u.
template <typename T, int S, int F, bool ADJ>
__device__ __forceinline__ double tile_diag(unsigned char* psi, unsigned char* lam, unsigned zl, unsigned neg0, T A,
                                            T B) {
  using V = typename Cx<T>::V;
  DotAcc<T> acc;
#pragma unroll 4
  for (unsigned j = threadIdx.x; j < (1u << S); j += 256u) {
    const unsigned p = ((unsigned)__popc(zl & j) + neg0) & 1u;
    V* pu = reinterpret_cast<V*>(psi) + j;
    const V u = *pu;
    if (ADJ) {  // Im conj(lam) s psi
      V* qu = reinterpret_cast<V*>(lam) + j;
      const V q = *qu;
      acc.add(q.x, flip(u.y, p));
      acc.add(-q.y, flip(u.x, p));
      *qu = comb<F, T, V>(q, qturn(q, (3u + 2u * p) & 3u), A, B);
    }
    *pu = comb<F, T, V>(u, qturn(u, (3u + 2u * p) & 3u), A, B);
  }
  return ADJ ? acc.value() : 0.0;
}

// CTAs per SM.  complex128 forward takes small tiles and many CTAs: with the FP64 pipe
// saturated, two buffers of the same tile (3 CTAs) or one of twice the size gained
// nothing (28 qubits, 100 rotations: 122.9 ms against 124.4 and 129).
template <typename T, int S, bool ADJ> __host__ __device__ constexpr int tile_ctas() {
  return ADJ ? 2 : sizeof(T) == 8 || S == kTileSmall ? 6 : 3;
}
template <typename T, int S, bool ADJ>
__global__ void __launch_bounds__(256, tile_ctas<T, S, ADJ>())
    k_tile_pass(typename Cx<T>::V* __restrict__ psi, int n, const __grid_constant__ TileArgs a) {
  using V = typename Cx<T>::V;
  constexpr int L = sizeof(T) == 8 ? 3 : 4;
  constexpr unsigned E16 = 16 / sizeof(V), size = 1u << S;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* tp = smem_raw;                    // psi tile
  unsigned char* tl = smem_raw + sizeof(V) * size; // lam tile
  double* red = reinterpret_cast<double*>(tl + sizeof(V) * size);  // [rotation][thread]
  V* lam = reinterpret_cast<V*>(a.lam);
  __shared__ uint32_t hitab[1 << (S - L)];  // offsets of the tile's runs of 2^L amplitudes, in units of 2^L
  const unsigned tid = threadIdx.x;
  for (unsigned h = tid; h < (1u << (S - L)); h += 256u) {
    uint32_t off = 0;
#pragma unroll
    for (int i = L; i < S; ++i) off |= ((h >> (i - L)) & 1u) << (a.sbits[i] - L);
    hitab[h] = off;
  }
  if (ADJ)
    for (int r = 0; r < a.m; ++r) red[r * 256 + tid] = 0.0;
  // launched while the pass before it ends (programmatic dependent launch): all above
  // reads the arguments only; the states come from the passes before
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const bool part = on_part(a.on);
  const uint64_t ntiles = 1ull << (part ? a.on.nsup : n - S);
  auto base_of = [&](uint64_t t) {
    if (part) return reached(a.on, t);
#pragma unroll
    for (int i = 0; i < S; ++i) t = ins0(t, a.sbits[i]);
    return t;
  };
  auto copy_in = [&](uint64_t base, unsigned char* dst) {
#pragma unroll 8
    for (unsigned e = tid * E16; e < size; e += 256u * E16) {
      const uint64_t g = base | ((uint64_t)hitab[e >> L] << L) | (e & ((1u << L) - 1u));
      cp_async16(dst + e * sizeof(V), psi + g);
      if (ADJ) cp_async16(tl + e * sizeof(V), lam + g);
    }
  };
  for (uint64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const uint64_t base = base_of(t);
    __syncthreads();  // hitab; the last tile's writers are done
    copy_in(base, tp);
    cp_async_wait_all();
    __syncthreads();
    // the next pass may launch once every CTA is at its last tile's rotations
    if (t + gridDim.x >= ntiles) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int r = 0; r < a.m; ++r) {
      const TileRot& R = a.r[r];
      const unsigned xl = R.xl, zl = R.zl;
      const int hl = R.hl, form = R.form, y = R.y;
      const T A = (T)R.A, B = (T)R.B;
      const unsigned pout = par64(R.zout & base);
      double d = 0.0;
      if (hl < 0) {
        d = form == FORM_A1   ? tile_diag<T, S, FORM_A1, ADJ>(tp, tl, zl, pout, A, B)
            : form == FORM_B1 ? tile_diag<T, S, FORM_B1, ADJ>(tp, tl, zl, pout, A, B)
                              : tile_diag<T, S, FORM_AB, ADJ>(tp, tl, zl, pout, A, B);
      } else {
        const unsigned j0 = (unsigned)ins0(tid, hl);
        // the sign of pair k = 0: Z parity of j0, and the one y gives (odd y: - for 1 mod 4; even y: - for 0 mod 4)
        const unsigned zp = ((unsigned)__popc(zl & j0) + pout) & 1u;
        const unsigned ys = (y & 1) ? ((y & 2) ? 0u : 1u) : ((y & 2) ? 0u : 1u);
        auto go = [&](auto c) {
          constexpr int C = decltype(c)::value;
          auto run = [&](auto f, auto odd) {
            return tile_pairs<T, S, C, decltype(f)::value, decltype(odd)::value, ADJ>(tp, tl, j0, xl, zl, zp ^ ys, A,
                                                                                     B);
          };
          using A1 = std::integral_constant<int, FORM_A1>;
          using B1 = std::integral_constant<int, FORM_B1>;
          using AB = std::integral_constant<int, FORM_AB>;
          if (y & 1)
            d = form == FORM_A1 ? run(A1{}, std::true_type{}) : form == FORM_B1 ? run(B1{}, std::true_type{})
                                                                               : run(AB{}, std::true_type{});
          else
            d = form == FORM_A1 ? run(A1{}, std::false_type{}) : form == FORM_B1 ? run(B1{}, std::false_type{})
                                                                                : run(AB{}, std::false_type{});
        };
        switch (hl) {
          case 9: go(std::integral_constant<int, 1>{}); break;
          case 10: go(std::integral_constant<int, (S > 10 ? 2 : 1)>{}); break;
          case 11: go(std::integral_constant<int, (S > 11 ? 3 : 1)>{}); break;
          case 12: go(std::integral_constant<int, (S > 12 ? 4 : 1)>{}); break;
          default: go(std::integral_constant<int, 0>{});
        }
        // the overlap's sign: i^y's (y mod 4 >= 2) and the Z parity; tile_pairs took zp ^ ys
        if (ADJ) d = flip(d, ys ^ ((unsigned)y >> 1));
      }
      if (ADJ) red[r * 256 + tid] += d;
      __syncthreads();
    }
#pragma unroll 4
    for (unsigned e = tid * E16; e < size; e += 256u * E16) {
      const uint64_t g = base | ((uint64_t)hitab[e >> L] << L) | (e & ((1u << L) - 1u));
      *reinterpret_cast<float4*>(psi + g) = *reinterpret_cast<const float4*>(tp + e * sizeof(V));
      if (ADJ) *reinterpret_cast<float4*>(lam + g) = *reinterpret_cast<const float4*>(tl + e * sizeof(V));
    }
  }
  if (!ADJ) return;
  // the CTA's sums (a warp per rotation), then the last CTA's over the CTAs, in order
  __shared__ bool last;
  const int lane = tid & 31, warp = tid >> 5;
  for (int r = warp; r < a.m; r += 8) {
    double v = 0.0;
    for (int j = lane; j < 256; j += 32) v += red[r * 256 + j];
    v = warp_sum(v);
    if (lane == 0) a.partials[(size_t)r * gridDim.x + blockIdx.x] = v;
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicAdd(a.counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int r = warp; r < a.m; r += 8) {
    double v = 0.0;
    for (unsigned j = lane; j < gridDim.x; j += 32) v += __ldcg(a.partials + (size_t)r * gridDim.x + j);
    v = warp_sum(v);
    if (lane == 0) a.out[-r] = v;
  }
  if (tid == 0) *a.counter = 0u;
}

// Whether a state is zero outside a support (one read of the state, half a dense pass):
// a handle's amplitudes may sit in memory that its owner also writes.
struct SupportArg {
  int d;
  uint64_t off, v[QF_MAX_QUBITS];
  int top[QF_MAX_QUBITS];
};
template <typename V>
__global__ void __launch_bounds__(256) k_check_support(const V* __restrict__ psi, uint64_t N,
                                                       const __grid_constant__ SupportArg s, unsigned* dense) {
  bool out = false;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
#pragma unroll 8
  for (uint64_t b = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; b < N; b += stride) {
    const V a = psi[b];
    if (a.x == 0 && a.y == 0) continue;
    uint64_t w = b ^ s.off;
    for (int i = 0; i < s.d; ++i)
      if ((w >> s.top[i]) & 1) w ^= s.v[i];
    out = out || w != 0;
  }
  if (out) *dense = 1u;
}

// ---------------------------------------------------------------------------
// sparse composite block
//
// The composite of the block's rotations restricted to its support qubits is
// the identity except on a few "active" support patterns; only those
// amplitudes are read and written.  One thread per assignment of the
// non-support bits ("outside index").  The arguments hold M - I, so each output
// is v_r + sum_k (M - I)_rk v_k: the rounding then scales with the (small)
// change rather than with the amplitude, which keeps complex64 states close to
// unit norm.  REALST: the state is real (imaginary parts are
// exactly zero and stay zero), so only real parts are read and written.

template <int NR>
struct SpK {
  int u, nr, nzc, pad;
  int supp[kSparseMaxSupp];
  uint64_t pat[NR];
  uint64_t zc[2];
  double2 M[kSparseMaxCls][NR][NR];
  double2 Q[kSparseMaxCls][NR][NR];
};

__device__ __forceinline__ uint64_t sp_base(uint64_t o, const int* supp, int u) {
  for (int i = 0; i < u; ++i) o = ins0(o, supp[i]);
  return o;
}

template <int NR>
__device__ __forceinline__ unsigned sp_class(const SpK<NR>& a, uint64_t base) {
  unsigned cls = 0;
  if (a.nzc > 0) cls = par64(a.zc[0] & base);
  if (a.nzc > 1) cls |= par64(a.zc[1] & base) << 1;
  return cls;
}

// A forward block.  Each of its rotations pairs pattern r with r ^ x, so the composite is
// a 2x2 matrix per pair of rows: two entries a row, not the block's whole row (a double
// excitation of equal spins has 6 rows).  For commuting strings of an even number of Y
// (a Trotter step's) the diagonal is real and the rest imaginary, for an odd number (an
// excitation's) all is real: FP64 work, which bounds the kernel on large states, is 4
// multiply-adds a row.  Small ones are bound by the launches, so the next one's
// prologue overlaps (programmatic dependent launch), and on a state grown from a
// determinant only the outside patterns it has reached are visited (see Support).
// Trotter step at 20 qubits, complex128, 2445 blocks: whole rows and every pattern 38 ms,
// pairs and reached patterns 16 ms.
enum { PAIR_COMPLEX = 0, PAIR_TURN = 1, PAIR_REAL = 2 };
template <int NP>
struct PairK {
  int u, nzc;
  int supp[kSparseMaxSupp];
  uint64_t pat[NP][2], zc[2];
  Reached on;
  double2 M[kSparseMaxCls][NP][2][2];  // minus the identity
};

// out = own + the products of row `own`, in row order.
template <int F, bool REALST, typename T, typename V>
__device__ __forceinline__ V pair_row(V own, V first, V second, V m0, V m1, bool own_first) {
  V o = own;
  auto mul = [&](V m, V v, bool diag) {
    if (F == PAIR_COMPLEX || F == PAIR_REAL || diag) {
      o.x = fma(m.x, v.x, o.x);
      if (!REALST) o.y = fma(m.x, v.y, o.y);
    }
    if (F == PAIR_COMPLEX || (F == PAIR_TURN && !diag)) {
      o.x = fma(-m.y, v.y, o.x);
      o.y = fma(m.y, v.x, o.y);
    }
  };
  mul(m0, first, own_first);
  mul(m1, second, !own_first);
  return o;
}

template <typename T, int NP, int F, bool REALST>
__global__ void __launch_bounds__(256) k_pairs(typename Cx<T>::V* __restrict__ psi, int n,
                                               const __grid_constant__ PairK<NP> a) {
  using V = typename Cx<T>::V;
  __shared__ V M[kSparseMaxCls][NP][2][2];
  for (int i = threadIdx.x; i < kSparseMaxCls * NP * 4; i += blockDim.x) {
    const double2 d = (&a.M[0][0][0][0])[i];
    V m;
    m.x = (T)d.x;
    m.y = (T)d.y;
    (&M[0][0][0][0])[i] = m;
  }
  __syncthreads();
  // all above reads the arguments only
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const bool part = on_part(a.on);
  const uint64_t nout = 1ull << (part ? a.on.nsup : n - a.u);
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  T* pr = reinterpret_cast<T*>(psi);
  for (uint64_t o = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; o < nout; o += stride) {
    const uint64_t base = part ? reached(a.on, o) : sp_base(o, a.supp, a.u);
    unsigned cls = 0;
    if (a.nzc > 0) cls = par64(a.zc[0] & base);
    if (a.nzc > 1) cls |= par64(a.zc[1] & base) << 1;
    V v[NP][2];
#pragma unroll
    for (int p = 0; p < NP; ++p)
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const uint64_t at = base | a.pat[p][r];
        if (REALST) {
          v[p][r].x = pr[2 * at];
          v[p][r].y = 0;
        } else {
          v[p][r] = psi[at];
        }
      }
#pragma unroll
    for (int p = 0; p < NP; ++p)
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const V w = pair_row<F, REALST, T, V>(v[p][r], v[p][0], v[p][1], M[cls][p][r][0], M[cls][p][r][1], r == 0);
        const uint64_t at = base | a.pat[p][r];
        if (REALST)
          pr[2 * at] = w.x;
        else
          psi[at] = w;
      }
  }
}

// A run of commuting rotations of one X mask, too varied in Z for a composite (a Trotter
// step's one-electron flips, each with a Z on every other qubit; its diagonal): on the pair
// (b, b ^ x) their product is one rotation by phi(b), the sum of the angles with signs
// (-1)^{popc(z & b)}, added as whole numbers (phase_turns): the sum of all less twice those
// of odd parity: about ten integer operations a string and one FP64 sine and cosine a pair,
// where a rotation each takes four FP64 multiply-adds a string and pair.  At 20 qubits a
// launch takes 11 us, bound by its prologue and latency (barrier the top stall, FP64 pipe 18 %).
// Trotter step at 20 qubits, 3631 strings in 91 runs: 7.8 ms as tile passes, 1.5 ms here, each
// launch timed by itself; the whole step 5.91 ms with FP64 sums of the angles, 5.51 ms.
__global__ void __launch_bounds__(256) k_phase_run(double2* __restrict__ psi, int n,
                                                   const __grid_constant__ PhaseArgs a) {
  __shared__ uint64_t turn[kPhaseMax];
  __shared__ unsigned long long sum;
  static_assert(kPhaseMax <= 256, "a thread converts one angle");
  if (threadIdx.x == 0) sum = 0;
  __syncthreads();
  if ((int)threadIdx.x < a.m) {
    const uint64_t t = phase_turns(a.th[threadIdx.x]);
    turn[threadIdx.x] = t;
    atomicAdd(&sum, (unsigned long long)t);
  }
  __syncthreads();
  const uint64_t total = sum;
  // all above reads the arguments only
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const bool part = on_part(a.on);
  const uint64_t nout = 1ull << (part ? a.on.nsup : a.h < 0 ? n : n - 1);
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t o = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; o < nout; o += stride) {
    const uint64_t b = part ? reached(a.on, o) : a.h < 0 ? o : ins0(o, a.h);
    uint64_t odd = 0;
#pragma unroll 4
    for (int k = 0; k < a.m; ++k) odd += turn[k] & (0ull - (uint64_t)par64(a.z[k] & b));
    double sn, cs;
    sincospi(phase_halves(total - 2 * odd), &sn, &cs);
    const double2 u = psi[b];
    if (a.h < 0) {
      double2 w;
      w.x = fma(sn, u.y, cs * u.x);
      w.y = fma(-sn, u.x, cs * u.y);
      psi[b] = w;
      continue;
    }
    const double2 v = psi[b ^ a.x];
    // v' = cos v - i i^y sin u, u' = cos u - i conj(i^y) sin v
    const double s = (a.y & 2) ? -sn : sn;
    double2 p, q;
    if (a.y & 1) {
      p = make_double2(fma(-s, v.x, cs * u.x), fma(-s, v.y, cs * u.y));
      q = make_double2(fma(s, u.x, cs * v.x), fma(s, u.y, cs * v.y));
    } else {
      p = make_double2(fma(s, v.y, cs * u.x), fma(-s, v.x, cs * u.y));
      q = make_double2(fma(s, u.y, cs * v.x), fma(-s, u.x, cs * v.y));
    }
    psi[b] = p;
    psi[b ^ a.x] = q;
  }
}

// Consecutive forward blocks on tiles of 2^S amplitudes in shared memory (see k_tile_pass
// and k_pairs): one launch, and one read and write of the state, for up to kPassBlocks
// blocks, with a CTA barrier between them.  A thread takes one pair of rows at one
// outside pattern of the tile.  Trotter step at 20 qubits, complex128, 2445 blocks: 16 ms one
// launch each, 6.1 ms in 300 launches; 5.7 ms visiting only the outside patterns that go
// with a reached row of a pair (a quarter there: both spins' parities are fixed).
template <typename T, int S>
__global__ void __launch_bounds__(256, (sizeof(typename Cx<T>::V) << S) > 32768 ? 3 : 4)
    k_block_pass(typename Cx<T>::V* __restrict__ psi, int n, const __grid_constant__ BlockPass a) {
  using V = typename Cx<T>::V;
  constexpr int L = sizeof(T) == 8 ? 3 : 4;
  constexpr unsigned E16 = 16 / sizeof(V), size = 1u << S;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* tile = reinterpret_cast<V*>(smem_raw);
  __shared__ uint32_t hitab[1 << (S - L)];
  __shared__ T M[kPassBlocks][2][kPassPairs][4];
  const unsigned tid = threadIdx.x;
  for (unsigned h = tid; h < (1u << (S - L)); h += 256u) {
    uint32_t off = 0;
#pragma unroll
    for (int i = L; i < S; ++i) off |= ((h >> (i - L)) & 1u) << (a.sbits[i] - L);
    hitab[h] = off;
  }
  for (int i = tid; i < a.nb * 8 * kPassPairs; i += 256)
    (&M[0][0][0][0])[i] = (T)(&a.b[i / (8 * kPassPairs)].M[0][0][0])[i % (8 * kPassPairs)];
  // all above reads the arguments only
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const bool part = on_part(a.on);
  const uint64_t ntiles = 1ull << (part ? a.on.nsup : n - S);
  for (uint64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    uint64_t base = t;
    unsigned in_tile = a.loff;
    if (part) {
      base = reached(a.on, t);
      for (int i = 0; i < a.on.nsup; ++i) in_tile ^= a.lsup[i] & (0u - (unsigned)((t >> i) & 1ull));
    } else {
#pragma unroll
      for (int i = 0; i < S; ++i) base = ins0(base, a.sbits[i]);
    }
    __syncthreads();  // hitab and M; the last tile's writers are done
#pragma unroll 8
    for (unsigned e = tid * E16; e < size; e += 256u * E16)
      cp_async16(tile + e, psi + (base | ((uint64_t)hitab[e >> L] << L) | (e & ((1u << L) - 1u))));
    cp_async_wait_all();
    __syncthreads();
    if (t + gridDim.x >= ntiles) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int b = 0; b < a.nb; ++b) {
      const BlockRec& R = a.b[b];
      const bool some = part && R.nin < S - R.u;
      const int ob = some ? R.nin : S - R.u;
      const unsigned items = (unsigned)R.np << ob;
      const unsigned pout = par64(R.zout & base), zl = R.zl;
      for (unsigned i = tid; i < items; i += 256u) {
        const unsigned p = i >> ob;
        unsigned j = i & ((1u << ob) - 1u);
        if (some) {
          unsigned w = in_tile;
          if (w >> R.supp[R.u - 1] & 1u) w ^= R.supp_mask;  // x, the whole support: the lower row
          for (int q = 0; q < R.nlift; ++q) {
            const unsigned l = R.lift[q];
            w ^= l & (0u - (((w ^ R.pat[p][0]) >> (31 - __clz(l & R.supp_mask))) & 1u));
          }
          if ((w ^ R.pat[p][0]) & R.supp_mask) continue;
          w &= R.omask;
          for (int q = 0; q < ob; ++q) w ^= R.in[q] & (0u - ((j >> q) & 1u));
          j = w;
        } else {
          for (int q = 0; q < R.u; ++q) {
            const unsigned low = j & ((1u << R.supp[q]) - 1u);
            j = ((j - low) << 1) | low;
          }
        }
        const T* m = M[b][((unsigned)__popc(zl & j) + pout) & 1u][p];
        V* pu = tile + (j | R.pat[p][0]);
        V* pv = tile + (j | R.pat[p][1]);
        const V u = *pu, v = *pv;
        V x = u, y = v;
        if (R.turn) {
          x.x = fma(-m[1], v.y, fma(m[0], u.x, x.x));
          x.y = fma(m[1], v.x, fma(m[0], u.y, x.y));
          y.x = fma(m[3], v.x, fma(-m[2], u.y, y.x));
          y.y = fma(m[3], v.y, fma(m[2], u.x, y.y));
        } else {
          x.x = fma(m[1], v.x, fma(m[0], u.x, x.x));
          x.y = fma(m[1], v.y, fma(m[0], u.y, x.y));
          y.x = fma(m[3], v.x, fma(m[2], u.x, y.x));
          y.y = fma(m[3], v.y, fma(m[2], u.y, y.y));
        }
        *pu = x;
        *pv = y;
      }
      __syncthreads();
    }
#pragma unroll 4
    for (unsigned e = tid * E16; e < size; e += 256u * E16)
      *reinterpret_cast<float4*>(psi + (base | ((uint64_t)hitab[e >> L] << L) | (e & ((1u << L) - 1u)))) =
          *reinterpret_cast<const float4*>(tile + e);
  }
}

// ---------------------------------------------------------------------------
// expectation value, pair form
//
// For an X group g (x != 0) and the pair (b, b xor x) with b's pivot bit clear,
// w = conj(psi[b xor x]) psi[b]; the pair's contribution from term t is
//   2 c_t (-1)^{y/2} s_t(b) Re w          (y even)
//   2 c_t (-1)^{(y+1)/2} s_t(b) Im w      (y odd),
// s_t(b) = (-1)^{popc(z_t & b)}.  Terms are packed four per chunk with a 16-entry
// table over their sign pattern, so a chunk costs one lookup and one or two
// FMAs per pair.  The diagonal group (x = 0) uses |psi_b|^2 and c_t.

template <typename T>
__global__ void __launch_bounds__(256) k_expect(const typename Cx<T>::V* __restrict__ psi, int n,
                                                const ExpGroup* __restrict__ groups, int ngroups,
                                                const ExpChunk* __restrict__ chunks, double* partials,
                                                unsigned* counter, double* out) {
  using V = typename Cx<T>::V;
  const uint64_t hmask = (1ull << (n - 1)) - 1ull;
  const uint64_t total = (uint64_t)ngroups << (n - 1);
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  double acc = 0.0;
  // complex64: pair products and table weights in FP32, folded into the FP64
  // accumulator every 32 pairs (no per-pair FP64 conversions)
  float facc = 0.f;
  int nf = 0;
  for (uint64_t f = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; f < total; f += stride) {
    const int g = (int)(f >> (n - 1));
    const uint64_t p = f & hmask;
    const ExpGroup G = groups[g];
    if (G.h < 0) {
      const uint64_t b0 = p << 1;
      const V u0 = psi[b0], u1 = psi[b0 | 1ull];
      for (int c = 0; c < G.nchunk; ++c) {
        const ExpChunk* C = chunks + G.chunk0 + c;
        unsigned i0 = 0, i1 = 0;
#pragma unroll
        for (int t = 0; t < kChunkTerms; ++t) {
          const uint64_t zt = C->z[t];
          const unsigned pb = par64(zt & b0);
          i0 |= pb << t;
          i1 |= (pb ^ (unsigned)(zt & 1ull)) << t;
        }
        if constexpr (sizeof(T) == 4) {
          facc = fmaf(C->ftab[i0].x, fmaf(u0.x, u0.x, u0.y * u0.y), facc);
          facc = fmaf(C->ftab[i1].x, fmaf(u1.x, u1.x, u1.y * u1.y), facc);
        } else {
          acc = fma(C->tab[i0].x, fma((double)u0.x, u0.x, (double)u0.y * u0.y), acc);
          acc = fma(C->tab[i1].x, fma((double)u1.x, u1.x, (double)u1.y * u1.y), acc);
        }
      }
    } else {
      const uint64_t b = ins0(p, G.h);
      const V u = psi[b], v = psi[b ^ G.x];
      T rew = 0, imw = 0;
      if (G.flags & 1) rew = fma(u.x, v.x, u.y * v.y);
      if (G.flags & 2) imw = fma(u.y, v.x, -u.x * v.y);
      for (int c = 0; c < G.nchunk; ++c) {
        const ExpChunk* C = chunks + G.chunk0 + c;
        unsigned idx = 0;
#pragma unroll
        for (int t = 0; t < kChunkTerms; ++t) idx |= par64(C->z[t] & b) << t;
        if constexpr (sizeof(T) == 4) {
          const float2 D = C->ftab[idx];
          if (G.flags & 1) facc = fmaf(D.x, rew, facc);
          if (G.flags & 2) facc = fmaf(D.y, imw, facc);
        } else {
          const double2 D = C->tab[idx];
          if (G.flags & 1) acc = fma(D.x, rew, acc);
          if (G.flags & 2) acc = fma(D.y, imw, acc);
        }
      }
    }
    if constexpr (sizeof(T) == 4) {
      if (++nf == 32) {
        acc += (double)facc;
        facc = 0.f;
        nf = 0;
      }
    }
  }
  acc += (double)facc;
  grid_finish(acc, partials, counter, out);
}

// Tiled form for n > 10: a CTA takes tiles of 256 x P pairs of one X group
// (P = 4; 8 was slower for complex64 at 28 qubits), reads the group's descriptor
// once per tile, and every thread issues the loads of its P pairs before using
// them (P times the loads in flight of the flat loop).  A group of one term
// (flags bit 2: its table is +-tab[0]) puts the sign on the amplitude and the
// weight on the tile's sum, so a pair costs two multiply-adds.
template <typename T> struct ExpTile {
  static constexpr int P = 4;
  static constexpr int LOG = 10;  // log2(256 P)
};
constexpr int kExpTileLogMax = 10;

template <typename T>
__global__ void __launch_bounds__(256) k_expect_tiled(const typename Cx<T>::V* __restrict__ psi, int n,
                                                      const ExpGroup* __restrict__ groups, int ngroups,
                                                      const ExpChunk* __restrict__ chunks, double* partials,
                                                      unsigned* counter, double* out) {
  using V = typename Cx<T>::V;
  constexpr int kExpPairs = ExpTile<T>::P, kExpTileLog = ExpTile<T>::LOG;
  const int tb = n - 1 - kExpTileLog;  // log2(tiles per group)
  const uint64_t ntiles = (uint64_t)ngroups << tb;
  double acc = 0.0;
  float facc = 0.f;  // complex64: FP32 sums folded into acc once per tile
  for (uint64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int g = (int)(tile >> tb);
    const uint64_t p0 = ((tile & ((1ull << tb) - 1)) << kExpTileLog) + threadIdx.x;
    const ExpGroup G = groups[g];
    if (G.h < 0) {  // x = 0: |psi_b|^2 of both amplitudes of each pair
#pragma unroll
      for (int k = 0; k < kExpPairs; ++k) {
        const uint64_t b0 = (p0 + 256 * k) << 1;
        const V u0 = psi[b0], u1 = psi[b0 | 1ull];
        for (int c = 0; c < G.nchunk; ++c) {
          const ExpChunk* C = chunks + G.chunk0 + c;
          unsigned i0 = 0, i1 = 0;
#pragma unroll
          for (int t = 0; t < kChunkTerms; ++t) {
            const uint64_t zt = C->z[t];
            const unsigned pb = par64(zt & b0);
            i0 |= pb << t;
            i1 |= (pb ^ (unsigned)(zt & 1ull)) << t;
          }
          if constexpr (sizeof(T) == 4) {
            facc = fmaf(C->ftab[i0].x, fmaf(u0.x, u0.x, u0.y * u0.y), facc);
            facc = fmaf(C->ftab[i1].x, fmaf(u1.x, u1.x, u1.y * u1.y), facc);
          } else {
            acc = fma(C->tab[i0].x, fma((double)u0.x, u0.x, (double)u0.y * u0.y), acc);
            acc = fma(C->tab[i1].x, fma((double)u1.x, u1.x, (double)u1.y * u1.y), acc);
          }
        }
      }
    } else {
      uint64_t b[kExpPairs];
      V u[kExpPairs], v[kExpPairs];
#pragma unroll
      for (int k = 0; k < kExpPairs; ++k) {
        b[k] = ins0(p0 + 256 * k, G.h);
        u[k] = psi[b[k]];
        v[k] = psi[b[k] ^ G.x];
      }
      if (G.flags & 4) {  // one term: D = (-1)^{popc(z & b)} tab[0]
        const ExpChunk* C = chunks + G.chunk0;
        const uint64_t z = C->z[0];
        T gr = T(0), gi = T(0);
#pragma unroll
        for (int k = 0; k < kExpPairs; ++k) {
          const unsigned sg = par64(z & b[k]);
          const T ux = sg ? -u[k].x : u[k].x, uy = sg ? -u[k].y : u[k].y;
          if (G.flags & 1) gr = fma(ux, v[k].x, fma(uy, v[k].y, gr));
          if (G.flags & 2) gi = fma(uy, v[k].x, fma(-ux, v[k].y, gi));
        }
        if constexpr (sizeof(T) == 4) {
          const float2 D = C->ftab[0];
          facc = fmaf(D.x, gr, fmaf(D.y, gi, facc));
        } else {
          const double2 D = C->tab[0];
          acc = fma(D.x, gr, fma(D.y, gi, acc));
        }
      } else {
#pragma unroll
        for (int k = 0; k < kExpPairs; ++k) {
          T rew = 0, imw = 0;
          if (G.flags & 1) rew = fma(u[k].x, v[k].x, u[k].y * v[k].y);
          if (G.flags & 2) imw = fma(u[k].y, v[k].x, -u[k].x * v[k].y);
          for (int c = 0; c < G.nchunk; ++c) {
            const ExpChunk* C = chunks + G.chunk0 + c;
            unsigned idx = 0;
#pragma unroll
            for (int t = 0; t < kChunkTerms; ++t) idx |= par64(C->z[t] & b[k]) << t;
            if constexpr (sizeof(T) == 4) {
              const float2 D = C->ftab[idx];
              if (G.flags & 1) facc = fmaf(D.x, rew, facc);
              if (G.flags & 2) facc = fmaf(D.y, imw, facc);
            } else {
              const double2 D = C->tab[idx];
              if (G.flags & 1) acc = fma(D.x, rew, acc);
              if (G.flags & 2) acc = fma(D.y, imw, acc);
            }
          }
        }
      }
    }
    if constexpr (sizeof(T) == 4) {
      acc += (double)facc;
      facc = 0.f;
    }
  }
  grid_finish(acc, partials, counter, out);
}

// Passes (ExpPass): a CTA stages a tile of 2^S amplitudes (64 KB) in shared memory
// with asynchronous copies and evaluates every group of the pass on it, so the
// state is read once per pass instead of once per group (28 qubits, 500 strings: 55
// reads instead of 430); three CTAs per SM overlap one's copies with the others'
// sums.
// complex128 is bound by the FP64 pipe: two multiply-adds per pair and group, 75.6 ms
// of the 91.5 ms that 25 qubits, 1500 terms take (236 ms in the per-group kernel).
// complex64 is bound by shared-memory bandwidth (16 bytes per pair and group, 23 ms
// of the 46 ms that 28 qubits, 500 terms take; 178 ms in the per-group kernel) and,
// in passes of few groups, by the state's reads (55 reads: 18 ms); taking such passes
// in turn with large ones tile by tile was slower (56 ms: spills).
// complex64 sums stay in FP32 over four pairs, then join a float pair by TwoSum
// (converted to FP64 once per tile).
template <typename T> struct PassAcc {  // FP64 state: one running sum
  double s = 0.0;
  __device__ __forceinline__ void add(double w, double v) { s = fma(w, v, s); }
  __device__ __forceinline__ void add(double v) { s += v; }
  __device__ __forceinline__ double take() {
    const double v = s;
    s = 0.0;
    return v;
  }
};
template <> struct PassAcc<float> {
  float h = 0.f, l = 0.f;
  __device__ __forceinline__ void add(float w, float v) { add(w * v); }
  __device__ __forceinline__ void add(float v) {  // TwoSum, the error into l
    const float t = __fadd_rn(h, v);
    const float bp = __fsub_rn(t, h);
    l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(t, bp)), __fsub_rn(v, bp)));
    h = t;
  }
  __device__ __forceinline__ double take() {
    const double v = (double)h + (double)(isfinite(h) ? l : 0.f);  // TwoSum's error of an infinity is a NaN
    h = l = 0.f;
    return v;
  }
};

template <typename T> __device__ __forceinline__ T pass_weight(const ExpChunk* C, unsigned i, bool im);
template <> __device__ __forceinline__ double pass_weight<double>(const ExpChunk* C, unsigned i, bool im) {
  return im ? __ldg(&C->tab[i].y) : __ldg(&C->tab[i].x);
}
template <> __device__ __forceinline__ float pass_weight<float>(const ExpChunk* C, unsigned i, bool im) {
  return im ? __ldg(&C->ftab[i].y) : __ldg(&C->ftab[i].x);
}

// A thread's pairs of a group with pivot bit hl: j = j0 + o_k and j ^ xl, o_k running
// over the tile bits above the thread's own.  Those bits depend only on the case
// C = max(0, hl - 8) (the thread's 8 bits spread over bits 0..8 around a pivot up to
// bit 8, else the high bits leave out the pivot), so o_k is a constant: one load
// with an immediate offset and one XOR for the partner's address.
template <typename T, int C> struct PassPairs {
  static constexpr int P = PassTile<T>::P, KB = PassTile<T>::S - 9;
  static __device__ __forceinline__ unsigned off(int k) {
    unsigned o = 0;
#pragma unroll
    for (int i = 0; i < KB; ++i)
      if ((k >> i) & 1) o |= 1u << (C == 0 ? 9 + i : 8 + i < 8 + C ? 8 + i : 9 + i);
    return o;
  }
  template <typename F>
  static __device__ __forceinline__ void run(const unsigned char* tile, unsigned j0, unsigned xl, F&& f) {
    using V = typename Cx<T>::V;
    const unsigned a = j0 * sizeof(V), b = (j0 ^ xl) * sizeof(V);
#pragma unroll
    for (int k = 0; k < P; ++k) {
      const unsigned o = off(k) * (unsigned)sizeof(V);
      f(k, *reinterpret_cast<const V*>(tile + a + o), *reinterpret_cast<const V*>(tile + (b ^ o)));
    }
  }
};

// One-term group: the sum over the thread's pairs of +-Re w (+-Im w) times the term's
// weight w, which carries the thread's own sign.  Nibble 2^i of km is the sign of
// bit i of k; the sign of pair k is their product.
template <typename T, int C, bool IM>
__device__ __forceinline__ void pass_single(const unsigned char* tile, unsigned j0, unsigned xl, uint64_t km, T w,
                                            PassAcc<T>& acc) {
  using V = typename Cx<T>::V;
  if constexpr (sizeof(T) == 8) {  // two multiply-adds per pair, the sign on the amplitude
    T g = T(0);
    PassPairs<T, C>::run(tile, j0, xl, [&](int k, V u, const V& v) {
      const unsigned neg = (unsigned)(km >> (4 * k));
      u.x = flip(u.x, neg);
      u.y = flip(u.y, neg);
      g = IM ? fma(u.y, v.x, fma(-u.x, v.y, g)) : fma(u.x, v.x, fma(u.y, v.y, g));
    });
    acc.add(w, g);
  } else {  // four pairs as (t0 + e0 t1) + e1 (t2 + e0 t3) with e = +-1: no integer operation per pair
    const T e0 = flip(T(1), (unsigned)(km >> 4)), e1 = flip(T(1), (unsigned)(km >> 8));
    T g0 = T(0), g1 = T(0);
    PassPairs<T, C>::run(tile, j0, xl, [&](int k, const V& u, const V& v) {
      const T t = IM ? fma(u.y, v.x, -u.x * v.y) : fma(u.x, v.x, u.y * v.y);
      if ((k & 3) == 0) g0 = t;
      if ((k & 3) == 1) g0 = fma(e0, t, g0);
      if ((k & 3) == 2) g1 = t;
      if ((k & 3) == 3) acc.add(flip(w, (unsigned)(km >> (4 * (k & ~3)))), fma(e1, fma(e0, t, g1), g0));
    });
  }
}

// f(std::integral_constant<int, C>) for the group's case C.
template <typename T, typename F>
__device__ __forceinline__ void pass_case(int hl, F&& f) {
  switch (hl) {
    case 9: f(std::integral_constant<int, 1>{}); break;
    case 10: f(std::integral_constant<int, 2>{}); break;
    case 11: f(std::integral_constant<int, 3>{}); break;
    case 12: f(std::integral_constant<int, PassTile<T>::S - 9>{}); break;
    default: f(std::integral_constant<int, 0>{});
  }
}

template <typename T>
__global__ void __launch_bounds__(kPassThreads, 3)
    k_expect_pass(const typename Cx<T>::V* __restrict__ psi, int n, const ExpPass* __restrict__ passes, int npass,
                  const PassGroup* __restrict__ groups, const PassChunk* __restrict__ chunks,
                  const ExpChunk* __restrict__ tabs, double* partials, unsigned* counter, double* out) {
  using V = typename Cx<T>::V;
  constexpr int S = PassTile<T>::S, L = PassTile<T>::L, P = PassTile<T>::P, B = PassTile<T>::B;
  constexpr unsigned E16 = 16 / sizeof(V);  // amplitudes per 16-byte copy
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* tile = reinterpret_cast<V*>(smem_raw);
  __shared__ uint64_t hitab[1 << (S - L)];  // global offset of each run of 2^L amplitudes
  __shared__ uint8_t sbits[16];
  // the pass's groups: (xl, hl, nchunk << 19 | flags << 16 | first term's zl, chunk), the
  // first chunk's kx[0], the first term's weight and its sign on the current tile
  __shared__ int4 rec[kPassGroups];
  __shared__ uint64_t signs[kPassGroups];
  __shared__ T weight[kPassGroups];
  __shared__ uint8_t tsign[kPassGroups];
  const unsigned tid = threadIdx.x;
  const int tb = n - S;
  const uint64_t items = (uint64_t)npass << tb;
  int cur = -1, g0 = 0, ng = 0;
  double total = 0.0;
  PassAcc<T> acc;
  for (uint64_t item = blockIdx.x; item < items; item += gridDim.x) {
    const int p = (int)(item >> tb);
    __syncthreads();  // the last tile's readers are done
    if (p != cur) {
      cur = p;
      g0 = __ldg(&passes[p].g0);
      ng = __ldg(&passes[p].g1) - g0;
      if (tid < 16) sbits[tid] = passes[p].sbits[tid];
      // the groups' records: what a one-term group needs, in two 16-byte loads
      if (tid < (unsigned)ng) {
        const PassGroup G = groups[g0 + tid];
        const PassChunk& C = chunks[G.chunk];
        rec[tid] = make_int4((int)G.xl, G.hl, (G.nchunk_flags << 16) | (int)C.zl[0], G.chunk);
        const T w = pass_weight<T>(tabs + G.chunk, 0u, (G.nchunk_flags & 2) != 0);
        signs[tid] = C.kx[0];
        weight[tid] = w;
      }
      __syncthreads();
      for (unsigned h = tid; h < (1u << (S - L)); h += kPassThreads) {
        uint64_t off = 0;
#pragma unroll
        for (int i = L; i < S; ++i) off |= (uint64_t)((h >> (i - L)) & 1u) << sbits[i];
        hitab[h] = off;
      }
      __syncthreads();
    }
    uint64_t base = item & ((1ull << tb) - 1);
#pragma unroll
    for (int i = 0; i < S; ++i) base = ins0(base, sbits[i]);
#pragma unroll 8
    for (unsigned e = tid * E16; e < (1u << S); e += kPassThreads * E16)
      cp_async16(tile + e, psi + (base | hitab[e >> L] | (e & ((1u << L) - 1u))));
    if (tid < (unsigned)ng) tsign[tid] = (uint8_t)par64(__ldg(&chunks[rec[tid].w].zout[0]) & base);
    cp_async_wait_all();
    __syncthreads();
    for (int g = 0; g < ng; ++g) {
      const int4 raw = rec[g];
      const unsigned xl = (unsigned)raw.x;
      const int hl = raw.y, flags = (raw.z >> 16) & 7, nchunk = raw.z >> 19;
      const unsigned j0 = hl < 0 ? tid : (unsigned)ins0(tid, hl);
      // parity of chunk c's term t for the thread's first index in this tile
      auto sign0 = [&](const PassChunk* C, int t) {
        return ((unsigned)__popc(__ldg(&C->zl[t]) & j0) + par64(__ldg(&C->zout[t]) & base)) & 1u;
      };
      if ((flags & 4) && hl >= 0) {
        const uint64_t km = signs[g];
        const T w = flip(weight[g], (unsigned)__popc((unsigned)raw.z & 0xFFFFu & j0) + tsign[g]);
        pass_case<T>(hl, [&](auto c) {
          if (flags & 2)
            pass_single<T, decltype(c)::value, true>(smem_raw, j0, xl, km, w, acc);
          else
            pass_single<T, decltype(c)::value, false>(smem_raw, j0, xl, km, w, acc);
        });
        continue;
      }
      // Re w and Im w of the thread's pairs (diagonal: |psi|^2 of its amplitudes, in
      // two halves), then every chunk's table on them
      for (int half = 0; half < (hl < 0 ? 2 : 1); ++half) {
        T re[P], im[P];
        auto pairs = [&](int k, const V& u, const V& v) {
          re[k] = (flags & 1) ? fma(u.x, v.x, u.y * v.y) : T(0);
          im[k] = (flags & 2) ? fma(u.y, v.x, -u.x * v.y) : T(0);
        };
        if (hl < 0) {
#pragma unroll
          for (int k = 0; k < P; ++k) {
            const V u = tile[tid + kPassThreads * (k + half * P)];
            pairs(k, u, u);
          }
        } else {
          pass_case<T>(hl, [&](auto c) { PassPairs<T, decltype(c)::value>::run(smem_raw, j0, xl, pairs); });
        }
        for (int c = 0; c < nchunk; ++c) {
          const PassChunk* C = chunks + raw.w + c;
          const ExpChunk* W = tabs + raw.w + c;
          unsigned i0 = 0;
#pragma unroll
          for (int t = 0; t < kChunkTerms; ++t) i0 |= sign0(C, t) << t;
          const uint64_t kx = __ldg(&C->kx[half]);
#pragma unroll
          for (int k0 = 0; k0 < P; k0 += B) {
            T s = T(0);
#pragma unroll
            for (int k = k0; k < k0 + B; ++k) {
              const unsigned i = i0 ^ ((unsigned)(kx >> (4 * k)) & 15u);
              if (flags & 1) s = fma(pass_weight<T>(W, i, false), re[k], s);
              if (flags & 2) s = fma(pass_weight<T>(W, i, true), im[k], s);
            }
            acc.add(s);
          }
        }
      }
    }
    total += acc.take();
  }
  grid_finish(total, partials, counter, out);
}

// ---------------------------------------------------------------------------
// lam = H psi (gather form) fused with out[0] = Re <psi|lam>, out[1] = <psi|psi>
//
// lam[c] = sum_g D_g(c xor x_g) psi[c xor x_g], D_g(b) = sum_t c_t i^{y_t} s_t(b);
// D is read from the same 16-entry chunk tables (real part from even-y terms,
// imaginary part from odd-y terms).

template <typename T>
__global__ void __launch_bounds__(256) k_hpsi(const typename Cx<T>::V* __restrict__ psi,
                                              typename Cx<T>::V* __restrict__ lam, int n,
                                              const ExpGroup* __restrict__ groups, int ngroups,
                                              const ExpChunk* __restrict__ chunks, double* partials,
                                              unsigned* counter, double* out) {
  using V = typename Cx<T>::V;
  const uint64_t N = 1ull << n;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  double acc = 0.0, nrm = 0.0;
  for (uint64_t cidx = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; cidx < N; cidx += stride) {
    double lx = 0.0, ly = 0.0;
    for (int g = 0; g < ngroups; ++g) {
      const ExpGroup G = groups[g];
      const uint64_t b = cidx ^ G.x;
      const V v = psi[b];
      double dx = 0.0, dy = 0.0;
      for (int c = 0; c < G.nchunk; ++c) {
        const ExpChunk* C = chunks + G.chunk0 + c;
        unsigned idx = 0;
#pragma unroll
        for (int t = 0; t < kChunkTerms; ++t) idx |= par64(C->z[t] & b) << t;
        const double2 D = C->tab[idx];
        dx += D.x;
        dy += D.y;
      }
      const double vx = (double)v.x, vy = (double)v.y;
      lx = fma(dx, vx, lx);
      ly = fma(dx, vy, ly);
      if (G.flags & 2) {
        lx = fma(-dy, vy, lx);
        ly = fma(dy, vx, ly);
      }
    }
    const V u = psi[cidx];
    acc = fma((double)u.x, lx, fma((double)u.y, ly, acc));
    nrm = fma((double)u.x, (double)u.x, fma((double)u.y, (double)u.y, nrm));
    V w;
    w.x = (T)lx;
    w.y = (T)ly;
    lam[cidx] = w;
  }
  grid_finish2(acc, nrm, partials, counter, out);
}

// ---------------------------------------------------------------------------
// tiled H|psi>: lam[c] = sum_g D_g(c xor x_g) psi[c xor x_g], out[0] = Re <psi|lam>,
// out[1] = <psi|psi>.
//
// Output tiles are 2^TB contiguous amplitudes (TB = 8 + log2 E; each of the 256
// threads owns E of them: c = tid + 256 k).  For every class of groups sharing
// the high part xh of their X mask, the partner tile (tile xor xh) is staged in
// shared memory once and all groups of the class read it there.  For element k
// the partner index inside the tile is (tid ^ xl) | ((k ^ xl >> 8) << 8), and the
// sign pattern of the group's terms splits into a per-thread part and a part
// that depends on k only, so the inner loop is an XOR, a table load and an FMA.
// REALST: psi is real and every D is real, so only real parts are used.
// For float states each class's contribution is summed in FP32 and folded into
// FP64 accumulators once per class.

template <typename T> struct WTab;
template <> struct WTab<double> { using C = WChunk; using V2 = double2; };
template <> struct WTab<float> { using C = WChunkF; using V2 = float2; };

// A tile is a chain of one partner tile and one descriptor per class and group, so
// both come early: the next kHpsiStages - 1 classes' partner tiles are in flight as
// asynchronous copies, and 64 groups' descriptors at a time are staged in shared
// memory.  A group of one term needs no table: its weight and sign.
// 17 qubits, 400 terms (complex128): 748 us one class and one group at a time.
constexpr int kHpsiStages = 4;
constexpr int kHpsiBatch = 64;
struct HpsiRec {
  uint64_t x, z;   // z: the term's, in a group of one
  int chunk0, nchunk, flags, pad;  // flags: bit 0 a single term, bit 1 odd, bit 2 even
};
template <typename T, int E, bool REALST>
__global__ void __launch_bounds__(256, 2) k_hpsi_tiled(const typename Cx<T>::V* __restrict__ psi,
                                                    typename Cx<T>::V* __restrict__ lam, int n,
                                                    const HClass* __restrict__ classes, int nclasses,
                                                    const HGroup* __restrict__ groups,
                                                    const typename WTab<T>::C* __restrict__ chunks,
                                                    double* partials, unsigned* counter, double* out) {
  using V = typename Cx<T>::V;
  static_assert(E == 4 || E == 8, "tiles of 2^10 and 2^11 amplitudes");
  constexpr int TB = E == 4 ? 10 : 11;
  constexpr int KB = TB - 8;  // bits of k
  constexpr unsigned E16 = 16 / sizeof(V);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ HpsiRec rec[kHpsiBatch];
  __shared__ typename WTab<T>::V2 w1[kHpsiBatch];  // weight of a single term
  const unsigned tid = threadIdx.x;
  const uint64_t ntiles = 1ull << (n - TB);
  double acc_e = 0.0, acc_n = 0.0;
  for (uint64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    double lx[E], ly[E];
#pragma unroll
    for (int k = 0; k < E; ++k) lx[k] = ly[k] = 0.0;
    uint64_t xh_next = nclasses > 0 ? __ldg(&classes[0].xh) : 0;  // of the next class to copy
    auto copy_in = [&](int ci) {
      if (ci < nclasses) {
        V* dst = reinterpret_cast<V*>(smem_raw) + ((ci % kHpsiStages) << TB);
        const V* src = psi + ((t ^ xh_next) << TB);
#pragma unroll
        for (unsigned e = tid * E16; e < (1u << TB); e += 256u * E16) cp_async16(dst + e, src + e);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      if (ci + 1 < nclasses) xh_next = __ldg(&classes[ci + 1].xh);
    };
    __syncthreads();  // the last tile's readers are done
    for (int q = 0; q < kHpsiStages - 1; ++q) copy_in(q);
    int staged = 0;  // groups [staged - kHpsiBatch, staged) are in rec
    for (int ci = 0; ci < nclasses; ++ci) {
      const HClass C = classes[ci];
      const uint64_t pt = t ^ C.xh;
      const V* tile = reinterpret_cast<const V*>(smem_raw) + ((ci % kHpsiStages) << TB);
      asm volatile("cp.async.wait_group %0;" ::"n"(kHpsiStages - 2) : "memory");
      __syncthreads();  // this class's tile is there, and the last class's readers are done
      copy_in(ci + kHpsiStages - 1);
      T fx[E], fy[E];
#pragma unroll
      for (int k = 0; k < E; ++k) fx[k] = fy[k] = 0;
      for (int g = C.g0; g < C.g1; ++g) {
        if (g >= staged) {  // uniform over the CTA
          __syncthreads();
          if (tid < kHpsiBatch && g + (int)tid < classes[nclasses - 1].g1) {
            const HGroup H = groups[g + tid];
            const typename WTab<T>::C* W = chunks + H.chunk0;
            rec[tid] = HpsiRec{H.x, W->z[0], H.chunk0, H.nchunk, (H.terms == 1 ? 1 : 0) | (H.odd ? 2 : 4), 0};
            w1[tid] = W->tab[0];
          }
          staged = g + kHpsiBatch;
          __syncthreads();
        }
        const HpsiRec& G = rec[g - (staged - kHpsiBatch)];
        const unsigned xl = (unsigned)(G.x & ((1ull << TB) - 1ull));
        const unsigned xlo = xl & 255u, xhi = xl >> 8;
        if (G.flags & 1) {  // D = +-w, real (even y) or imaginary (odd y)
          const typename WTab<T>::V2 w = w1[g - (staged - kHpsiBatch)];
          const uint64_t z = G.z;
          const unsigned zk = (unsigned)(z >> 8) & ((1u << KB) - 1u);
          const unsigned s0 = par64((z >> TB) & pt) ^ ((unsigned)__popc((unsigned)z & 255u & (tid ^ xlo)) & 1u);
          const T d = flip((G.flags & 2) ? w.y : w.x, s0);
#pragma unroll
          for (int k = 0; k < E; ++k) {
            const unsigned kk = (unsigned)k ^ xhi;
            const V v = tile[(tid ^ xlo) | (kk << 8)];
            const T dk = flip(d, (unsigned)__popc(zk & kk));
            if (REALST || !(G.flags & 2)) {
              fx[k] = fma(dk, v.x, fx[k]);
              if (!REALST) fy[k] = fma(dk, v.y, fy[k]);
            } else {
              fx[k] = fma(-dk, v.y, fx[k]);
              fy[k] = fma(dk, v.x, fy[k]);
            }
          }
          continue;
        }
        T dx[E], dy[E];
        // the first table initialises D (no add of zero), later tables add to it
        for (int c = 0; c < G.nchunk; ++c) {
          const typename WTab<T>::C* W = chunks + G.chunk0 + c;
          unsigned ith = 0, col[KB];
#pragma unroll
          for (int j = 0; j < KB; ++j) col[j] = 0;
#pragma unroll
          for (int q = 0; q < kWideTerms; ++q) {
            const uint64_t z = W->z[q];
            const unsigned hp = par64((z >> TB) & pt);
            const unsigned tp = (unsigned)__popc((unsigned)z & 255u & (tid ^ xlo)) & 1u;
            ith |= (hp ^ tp) << q;
#pragma unroll
            for (int j = 0; j < KB; ++j) col[j] |= (unsigned)((z >> (8 + j)) & 1ull) << q;
          }
#pragma unroll
          for (int k = 0; k < E; ++k) {
            unsigned idx = ith;
            const unsigned kk = (unsigned)k ^ xhi;
#pragma unroll
            for (int j = 0; j < KB; ++j)
              if ((kk >> j) & 1u) idx ^= col[j];
            const typename WTab<T>::V2 d = W->tab[idx];
            if (c == 0) {
              dx[k] = d.x;
              if (!REALST) dy[k] = d.y;
            } else {
              dx[k] += d.x;
              if (!REALST) dy[k] += d.y;
            }
          }
        }
#pragma unroll
        for (int k = 0; k < E; ++k) {
          const V v = tile[(tid ^ xlo) | ((((unsigned)k ^ xhi)) << 8)];
          fx[k] = fma(dx[k], v.x, fx[k]);
          if (!REALST) {
            fy[k] = fma(dx[k], v.y, fy[k]);
            if (G.flags & 2) {
              fx[k] = fma(-dy[k], v.y, fx[k]);
              fy[k] = fma(dy[k], v.x, fy[k]);
            }
          }
        }
      }
#pragma unroll
      for (int k = 0; k < E; ++k) {
        lx[k] += (double)fx[k];
        if (!REALST) ly[k] += (double)fy[k];
      }
    }
#pragma unroll
    for (int k = 0; k < E; ++k) {
      const uint64_t cidx = (t << TB) + tid + 256u * k;
      const V u = psi[cidx];
      acc_e = fma((double)u.x, lx[k], fma((double)u.y, ly[k], acc_e));
      acc_n = fma((double)u.x, (double)u.x, fma((double)u.y, (double)u.y, acc_n));
      V w;
      w.x = (T)lx[k];
      w.y = (T)ly[k];
      lam[cidx] = w;
    }
  }
  grid_finish2(acc_e, acc_n, partials, counter, out);
}

// ---------------------------------------------------------------------------
// tiled H|psi> for a real complex128 state and real D_g, double-single arithmetic
//
// GB300 executes FP64 FMAs at 1/58 of the FP32 rate, and this gather needs one
// multiply-add per (X group, amplitude).  Here each staged partner amplitude
// and each table value is split into a pair of floats (hi + lo, ~48 bits), the
// product D * v is formed exactly in its leading part (p = dh*vh and its FMA
// residual) plus the cross terms dh*vl + dl*vh, and it is accumulated with an
// error-free TwoSum into a (hi, lo) float pair per output amplitude.  Per
// operation the relative error is about 2^-46; the pair is renormalised once per
// class and converted to FP64 when the tile is written.  Groups with more than
// eight terms contribute one product per eight-term table.

// The _rn intrinsics keep the compiler from contracting or reassociating the
// error-free transformations.
__device__ __forceinline__ void ds_mad(float& ah, float& al, float dh, float dl, float vh, float vl) {
  const float p = __fmul_rn(dh, vh);
  float e = fmaf(dh, vh, -p);
  e = fmaf(dh, vl, e);
  e = fmaf(dl, vh, e);
  const float s = __fadd_rn(ah, p);
  const float bp = __fsub_rn(s, ah);
  const float err = __fadd_rn(__fsub_rn(ah, __fsub_rn(s, bp)), __fsub_rn(p, bp));
  al = __fadd_rn(al, __fadd_rn(err, e));
  ah = s;
}

__global__ void __launch_bounds__(256) k_split_ds(const double2* __restrict__ psi, float2* __restrict__ out,
                                                  uint64_t N) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < N; i += stride) {
    const double v = psi[i].x;
    const float h = __double2float_rn(v);
    out[i] = make_float2(h, __double2float_rn(v - (double)h));
  }
}

// Tiles of 2^12 amplitudes; thread t owns c = t + 256 k (k < 16).  For group
// g with low X bits xl = xlo + 256 xhi the partner of element k is
// (t ^ xlo) + 256 (k ^ xhi), and the sign-pattern index of a table is
//   hp (tile part, uniform) ^ nl[(t^xlo) & 15] ^ nh[(t^xlo) >> 4] ^ kx[k].
__global__ void __launch_bounds__(256) k_hpsi_ds(const double2* __restrict__ psi, const float2* __restrict__ split,
                                                 double2* __restrict__ lam, int n,
                                                 const HClass* __restrict__ classes, int nclasses,
                                                 const HGroup* __restrict__ groups,
                                                 const WChunkS* __restrict__ chunks, double* partials,
                                                 unsigned* counter, double* out) {
  constexpr int TB = 12, E = 16;
  __shared__ float2 tile[1 << TB];
  const unsigned tid = threadIdx.x;
  const uint64_t ntiles = 1ull << (n - TB);
  double acc_e = 0.0, acc_n = 0.0;
  for (uint64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    float ah[E], al[E];
#pragma unroll
    for (int k = 0; k < E; ++k) ah[k] = al[k] = 0.f;
    for (int ci = 0; ci < nclasses; ++ci) {
      const HClass C = classes[ci];
      const uint64_t pt = t ^ C.xh;
      __syncthreads();
#pragma unroll
      for (int k = 0; k < E; ++k) tile[tid + 256u * k] = split[(pt << TB) + tid + 256u * k];
      __syncthreads();
      for (int g = C.g0; g < C.g1; ++g) {
        const HGroup G = groups[g];
        const unsigned xlo = (unsigned)G.x & 255u;
        const unsigned tx = tid ^ xlo;
        for (int c = 0; c < G.nchunk; ++c) {
          const WChunkS* W = chunks + G.chunk0 + c;
          unsigned ith = (unsigned)W->nl[tx & 15u] ^ (unsigned)W->nh[tx >> 4];
#pragma unroll
          for (int q = 0; q < kWideTerms; ++q) ith ^= par64(W->zh[q] & pt) << q;
          const uint4 kxw = *reinterpret_cast<const uint4*>(W->kx);
          const unsigned kw[4] = {kxw.x, kxw.y, kxw.z, kxw.w};
          const unsigned xhi = ((unsigned)G.x >> 8) & 15u;
#pragma unroll
          for (int k = 0; k < E; ++k) {
            const unsigned idx = ith ^ ((kw[k >> 2] >> (8 * (k & 3))) & 255u);
            const float2 d = W->tab[idx];
            const float2 v = tile[tx | (((unsigned)k ^ xhi) << 8)];
            ds_mad(ah[k], al[k], d.x, d.y, v.x, v.y);
          }
        }
      }
#pragma unroll
      for (int k = 0; k < E; ++k) {  // renormalise the pair once per class
        const float s = __fadd_rn(ah[k], al[k]);
        al[k] = __fsub_rn(al[k], __fsub_rn(s, ah[k]));
        ah[k] = s;
      }
    }
#pragma unroll
    for (int k = 0; k < E; ++k) {
      const uint64_t cidx = (t << TB) + tid + 256u * k;
      const double lx = (double)ah[k] + (double)al[k];
      const double2 u = psi[cidx];
      acc_e = fma(u.x, lx, acc_e);
      acc_n = fma(u.x, u.x, acc_n);
      lam[cidx] = make_double2(lx, 0.0);
    }
  }
  grid_finish2(acc_e, acc_n, partials, counter, out);
}

// ---------------------------------------------------------------------------
// adjoint step for one rotation: out = Im <lam|P|psi> (pre-rotation values),
// then psi and lam both get the rotation given in the arguments (the host passes
// -theta, i.e. exp(+i theta P)).
//
// Over the pair (b, b'): <lam|P|psi> gets i^y s(b) [(-1)^y conj(lam_b) psi_b' +
// conj(lam_b') psi_b].

template <typename T, int F>
__global__ void __launch_bounds__(256) k_adj_rot(typename Cx<T>::V* __restrict__ psi,
                                                 typename Cx<T>::V* __restrict__ lam, int n, uint64_t x, uint64_t z,
                                                 int h, int y, T A, T B, double* partials, unsigned* counter,
                                                 double* out) {
  using V = typename Cx<T>::V;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  double acc = 0.0;
  const unsigned ym = (unsigned)y & 3u;
  if (x == 0ull) {
    const uint64_t N = 1ull << n;
    for (uint64_t b = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; b < N; b += stride) {
      const V u = psi[b], p = lam[b];
      const unsigned pb = par64(z & b);
      // Im(conj(p) s u)
      const double im = fma((double)p.x, (double)u.y, -(double)p.y * (double)u.x);
      acc += flip(im, pb);
      psi[b] = comb<F, T, V>(u, qturn(u, (3u + 2u * pb) & 3u), A, B);
      lam[b] = comb<F, T, V>(p, qturn(p, (3u + 2u * pb) & 3u), A, B);
    }
  } else {
    const uint64_t npairs = 1ull << (n - 1);
    for (uint64_t q = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; q < npairs; q += stride) {
      const uint64_t b = ins0(q, h), bp = b ^ x;
      const V u = psi[b], v = psi[bp], p = lam[b], r = lam[bp];
      const unsigned pb = par64(z & b);
      double val;
      if ((ym & 1u) == 0u) {
        // Im z1 + Im z2, z1 = conj(p) v, z2 = conj(r) u
        const double i1 = fma((double)p.x, (double)v.y, -(double)p.y * (double)v.x);
        const double i2 = fma((double)r.x, (double)u.y, -(double)r.y * (double)u.x);
        val = flip(i1 + i2, (ym >> 1) ^ pb);
      } else {
        // Re z2 - Re z1
        const double r1 = fma((double)p.x, (double)v.x, (double)p.y * (double)v.y);
        const double r2 = fma((double)r.x, (double)u.x, (double)r.y * (double)u.y);
        val = flip(r2 - r1, ((ym >> 1) & 1u) ^ pb);
      }
      acc += val;
      psi[b] = comb<F, T, V>(u, qturn(v, (3u + 3u * y + 2u * pb) & 3u), A, B);
      psi[bp] = comb<F, T, V>(v, qturn(u, (3u + y + 2u * pb) & 3u), A, B);
      lam[b] = comb<F, T, V>(p, qturn(r, (3u + 3u * y + 2u * pb) & 3u), A, B);
      lam[bp] = comb<F, T, V>(r, qturn(p, (3u + y + 2u * pb) & 3u), A, B);
    }
  }
  grid_finish(acc, partials, counter, out);
}

// adjoint step for a sparse block: out = Im <lam|Q|psi>, then psi <- M psi,
// lam <- M lam on the active rows (the arguments hold M - I for the block's
// inverse composite M).  RQ: M is real and Q = i * (real matrix), the case of
// every fermionic excitation block, where Im <lam|Q|psi> = sum Qi_rk Re(conj(lam_r) psi_k).
template <typename T, int NR, bool RQ, bool REALST>
__global__ void __launch_bounds__(256) k_adj_sparse(typename Cx<T>::V* __restrict__ psi,
                                                    typename Cx<T>::V* __restrict__ lam, int n,
                                                    const __grid_constant__ SpK<NR> a, double* partials,
                                                    unsigned* counter, double* out) {
  using V = typename Cx<T>::V;
  __shared__ V M[kSparseMaxCls][NR][NR];
  __shared__ double2 Q[kSparseMaxCls][NR][NR];
  for (int i = threadIdx.x; i < kSparseMaxCls * NR * NR; i += blockDim.x) {
    const int c = i / (NR * NR), r = (i / NR) % NR, k = i % NR;
    V m;
    m.x = (T)a.M[c][r][k].x;
    m.y = (T)a.M[c][r][k].y;
    M[c][r][k] = m;
    Q[c][r][k] = a.Q[c][r][k];
  }
  __syncthreads();
  const uint64_t nout = 1ull << (n - a.u);
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  T* pr = reinterpret_cast<T*>(psi);
  T* lr = reinterpret_cast<T*>(lam);
  double acc = 0.0;
  for (uint64_t o = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; o < nout; o += stride) {
    const uint64_t base = sp_base(o, a.supp, a.u);
    const unsigned cls = sp_class(a, base);
    V v[NR], w[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      if (r < a.nr) {
        const uint64_t idx = base | a.pat[r];
        if (REALST) {
          v[r].x = pr[2 * idx];
          w[r].x = lr[2 * idx];
          v[r].y = w[r].y = 0;
        } else {
          v[r] = psi[idx];
          w[r] = lam[idx];
        }
      }
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      if (r < a.nr) {
        if (RQ) {
          // Re <lam_r|Qi v>, in the state's precision (FP64 accumulation across items)
          T sx = 0, sy = 0;
#pragma unroll
          for (int k = 0; k < NR; ++k)
            if (k < a.nr) {
              const T qi = (T)Q[cls][r][k].y;
              sx = fma(qi, v[k].x, sx);
              if (!REALST) sy = fma(qi, v[k].y, sy);
            }
          acc += (double)fma(w[r].x, sx, REALST ? (T)0 : w[r].y * sy);
        } else {
          double qx = 0.0, qy = 0.0;
#pragma unroll
          for (int k = 0; k < NR; ++k) {
            if (k < a.nr) {
              const double2 q = Q[cls][r][k];
              qx = fma(q.x, (double)v[k].x, fma(-q.y, (double)v[k].y, qx));
              qy = fma(q.x, (double)v[k].y, fma(q.y, (double)v[k].x, qy));
            }
          }
          acc = fma((double)w[r].x, qy, fma(-(double)w[r].y, qx, acc));
        }
      }
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      if (r < a.nr) {
        T ox = v[r].x, oy = v[r].y, px = w[r].x, py = w[r].y;
#pragma unroll
        for (int k = 0; k < NR; ++k) {
          if (k < a.nr) {
            const V m = M[cls][r][k];
            ox = fma(m.x, v[k].x, ox);
            px = fma(m.x, w[k].x, px);
            if (!REALST) {
              oy = fma(m.x, v[k].y, oy);
              py = fma(m.x, w[k].y, py);
            }
            if (!RQ) {
              ox = fma(-m.y, v[k].y, ox);
              oy = fma(m.y, v[k].x, oy);
              px = fma(-m.y, w[k].y, px);
              py = fma(m.y, w[k].x, py);
            }
          }
        }
        const uint64_t idx = base | a.pat[r];
        if (REALST) {
          pr[2 * idx] = ox;
          lr[2 * idx] = px;
        } else {
          V o1, o2;
          o1.x = ox;
          o1.y = oy;
          o2.x = px;
          o2.y = py;
          psi[idx] = o1;
          lam[idx] = o2;
        }
      }
    }
  }
  grid_finish(acc, partials, counter, out);
}

int g_sms = 0;

int sm_count() {
  if (g_sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
    if (g_sms <= 0) g_sms = 152;
  }
  return g_sms;
}

unsigned grid_for(uint64_t work, int per_sm) {
  const uint64_t cap = (uint64_t)sm_count() * per_sm;
  uint64_t g = (work + 255) / 256;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return (unsigned)g;
}

thread_local uint64_t t_launches = 0;

// opt-in per-launch event timing
struct ProfRec {
  unsigned kind;
  cudaEvent_t a, b;
};
thread_local unsigned t_prof_mask = 0;
thread_local std::vector<ProfRec> t_prof;
thread_local std::vector<cudaEvent_t> t_ev_pool;
thread_local size_t t_prof_used = 0;

cudaEvent_t pool_event(size_t i) {
  while (t_ev_pool.size() <= i) {
    cudaEvent_t e;
    cudaEventCreate(&e);
    t_ev_pool.push_back(e);
  }
  return t_ev_pool[i];
}

}  // namespace

void count_launch() { ++t_launches; }

// Records the start event of a launch of `kind` (if profiled); returns a slot.
int prof_pre(unsigned kind, cudaStream_t s) {
  if (!(t_prof_mask & kind)) return -1;
  ProfRec r{kind, pool_event(2 * t_prof_used), pool_event(2 * t_prof_used + 1)};
  ++t_prof_used;
  cudaEventRecord(r.a, s);
  t_prof.push_back(r);
  return (int)t_prof.size() - 1;
}

void prof_post(int slot, cudaStream_t s) {
  if (slot >= 0) cudaEventRecord(t_prof[slot].b, s);
}

int profile_begin(unsigned mask) {
  t_prof.clear();
  t_prof_used = 0;
  t_prof_mask = mask;
  return 0;
}

cudaError_t profile_read(unsigned mask, uint64_t* launches, double* total_ms) {
  uint64_t n = 0;
  double ms = 0.0;
  for (const ProfRec& r : t_prof) {
    if (!(r.kind & mask)) continue;
    cudaError_t e = cudaEventSynchronize(r.b);
    if (e != cudaSuccess) return e;
    float f = 0.f;
    e = cudaEventElapsedTime(&f, r.a, r.b);
    if (e != cudaSuccess) return e;
    ms += f;
    ++n;
  }
  if (launches) *launches = n;
  if (total_ms) *total_ms = ms;
  return cudaSuccess;
}

void profile_end() {
  t_prof_mask = 0;
  t_prof.clear();
  t_prof_used = 0;
}

int reduce_blocks(int n, qf_dtype) {
  const uint64_t cap = (uint64_t)sm_count() * 4;
  uint64_t g = ((1ull << n) / 2 + 255) / 256;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return (int)g;
}

cudaError_t launch_zero_and_set(void* psi, int n, qf_dtype dt, uint64_t det, cudaStream_t s) {
  return launch_zero_and_set_count(psi, 1ull << n, dt, det, s);
}

cudaError_t launch_zero_and_set_count(void* psi, uint64_t N, qf_dtype dt, uint64_t det, cudaStream_t s) {
  const int prof_slot_ = prof_pre(QF_K_SET, s);
  const unsigned g = grid_for(N, 8);
  if (dt == QF_C128)
    k_zero_and_set<double2><<<g, 256, 0, s>>>(static_cast<double2*>(psi), N, det);
  else
    k_zero_and_set<float2><<<g, 256, 0, s>>>(static_cast<float2*>(psi), N, det);
  prof_post(prof_slot_, s);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_gather(const void* src, qf_dtype dt, const int64_t* idx, int count, bool packed, bool ds,
                          double* out, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  if (ds && (dt != QF_C128 || !packed)) return cudaErrorInvalidValue;
  const unsigned g = (unsigned)((count + 255) / 256);
  if (ds)
    k_gather_ds<<<g, 256, 0, s>>>(static_cast<const float4*>(src), idx, count, out);
  else if (dt == QF_C128)
    k_gather<double2><<<g, 256, 0, s>>>(static_cast<const double2*>(src), idx, count, packed ? 1 : 0, out);
  else
    k_gather<float2><<<g, 256, 0, s>>>(static_cast<const float2*>(src), idx, count, packed ? 1 : 0, out);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_scale(void* psi, int n, qf_dtype dt, double scale, cudaStream_t s) {
  const int prof_slot_ = prof_pre(QF_K_SET, s);
  const uint64_t N = 1ull << n;
  const unsigned g = grid_for(N, 8);
  if (dt == QF_C128)
    k_scale<double><<<g, 256, 0, s>>>(static_cast<double2*>(psi), N, scale);
  else
    k_scale<float><<<g, 256, 0, s>>>(static_cast<float2*>(psi), N, (float)scale);
  prof_post(prof_slot_, s);
  count_launch();
  return cudaGetLastError();
}

template <typename T, int F>
static void rot_impl_f(void* psi, int n, const RotArgs& a, cudaStream_t s) {
  using V = typename Cx<T>::V;
  V* p = static_cast<V*>(psi);
  const uint64_t N = 1ull << n;
  if (a.x == 0ull) {
    k_rot_diag<T, F><<<grid_for(N, 8), 256, 0, s>>>(p, N, a.z, (T)a.A, (T)a.B);
  } else if (a.h == 0) {
    k_rot_pair1<T, F><<<grid_for(N / 2, 8), 256, 0, s>>>(p, N / 2, a.z, a.y, (T)a.A, (T)a.B);
  } else {
    k_rot_pair2<T, F><<<grid_for(N / 4, 8), 256, 0, s>>>(p, N / 4, a.x, a.z, a.h, a.y, (T)a.A, (T)a.B);
  }
}

template <typename T>
static void rot_impl(void* psi, int n, const RotArgs& a, cudaStream_t s) {
  if (a.form == FORM_A1)
    rot_impl_f<T, FORM_A1>(psi, n, a, s);
  else if (a.form == FORM_B1)
    rot_impl_f<T, FORM_B1>(psi, n, a, s);
  else
    rot_impl_f<T, FORM_AB>(psi, n, a, s);
}

cudaError_t launch_rot(void* psi, int n, qf_dtype dt, const RotArgs& a, cudaStream_t s) {
  const int prof_slot_ = prof_pre(QF_K_ROT, s);
  if (dt == QF_C128)
    rot_impl<double>(psi, n, a, s);
  else
    rot_impl<float>(psi, n, a, s);
  prof_post(prof_slot_, s);
  count_launch();
  return cudaGetLastError();
}

template <typename T>
static cudaError_t tile_impl(void* psi, int n, const TileArgs& a, cudaStream_t s) {
  using V = typename Cx<T>::V;
  const size_t smem = (sizeof(V) << a.s) + (sizeof(uint64_t) << a.nhi);
  const uint64_t ntiles = 1ull << (n - a.s);
  int per_sm = 4;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tile<T>, 256, smem);
  uint64_t g = (uint64_t)sm_count() * (uint64_t)std::max(1, per_sm);
  if (g > ntiles) g = ntiles;
  k_tile<T><<<(unsigned)g, 256, smem, s>>>(static_cast<V*>(psi), n, a);
  return cudaGetLastError();
}

template <typename T, int S, bool ADJ>
static cudaError_t tile_pass_t(void* psi, int n, const TileArgs& a, cudaStream_t s) {
  using V = typename Cx<T>::V;
  constexpr int tiles_held = ADJ ? 2 : 1;
  const size_t smem = (sizeof(V) << S) * tiles_held + (ADJ ? a.m * 256 * sizeof(double) : 0);
  constexpr size_t most = (sizeof(V) << S) * tiles_held + (ADJ ? kTileAdjRot * 256 * sizeof(double) : 0);
  const cudaError_t attr = smem_limit<k_tile_pass<T, S, ADJ>>(most);
  if (attr != cudaSuccess) return attr;
  if (ADJ && (a.m < 1 || a.m > kTileAdjRot)) return cudaErrorInvalidValue;
  const uint64_t tiles = 1ull << (n - S);
  uint64_t grid = std::min<uint64_t>(tiles, (uint64_t)sm_count() * tile_ctas<T, S, ADJ>());
  if (ADJ) grid = std::min<uint64_t>(grid, kTilePartials / a.m);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_tile_pass<T, S, ADJ>, static_cast<V*>(psi), n, a);
}

cudaError_t launch_tile(void* psi, int n, qf_dtype dt, const TileArgs& a, cudaStream_t s) {
  const bool adj = a.lam != nullptr;
  const int prof_slot_ = prof_pre(adj ? QF_K_ADJ_ROT : QF_K_TILE, s);
  cudaError_t e = cudaErrorInvalidValue;
  if (n < kTileSmall) {
    if (!adj) e = dt == QF_C128 ? tile_impl<double>(psi, n, a, s) : tile_impl<float>(psi, n, a, s);
  } else if (dt == QF_C128) {
    e = adj ? (a.s == 11   ? tile_pass_t<double, 11, true>(psi, n, a, s)
               : a.s == 10 ? tile_pass_t<double, 10, true>(psi, n, a, s)
                           : e)
            : (a.s == 11   ? tile_pass_t<double, 11, false>(psi, n, a, s)
               : a.s == 10 ? tile_pass_t<double, 10, false>(psi, n, a, s)
                           : e);
  } else {
    e = adj ? (a.s == 12   ? tile_pass_t<float, 12, true>(psi, n, a, s)
               : a.s == 10 ? tile_pass_t<float, 10, true>(psi, n, a, s)
                           : e)
            : (a.s == 13   ? tile_pass_t<float, 13, false>(psi, n, a, s)
               : a.s == 10 ? tile_pass_t<float, 10, false>(psi, n, a, s)
                           : e);
  }
  prof_post(prof_slot_, s);
  count_launch();
  return e;
}

cudaError_t launch_check_support(const void* psi, int n, qf_dtype dt, const Support& s, unsigned* dense,
                                 cudaStream_t stream) {
  SupportArg a;
  memset(&a, 0, sizeof(a));
  a.d = s.d;
  a.off = s.off;
  for (int i = 0; i < s.d; ++i) {
    a.v[i] = s.v[i];
    a.top[i] = 63 - __builtin_clzll(s.v[i]);
  }
  const uint64_t N = 1ull << n;
  const unsigned g = grid_for(N, 8);
  const int prof_slot_ = prof_pre(QF_K_TILE, stream);
  if (dt == QF_C128)
    k_check_support<<<g, 256, 0, stream>>>(static_cast<const double2*>(psi), N, a, dense);
  else
    k_check_support<<<g, 256, 0, stream>>>(static_cast<const float2*>(psi), N, a, dense);
  prof_post(prof_slot_, stream);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_phase_run(void* psi, int n, const PhaseArgs& a, cudaStream_t s) {
  const int prof_slot_ = prof_pre(QF_K_TILE, s);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid_for(1ull << (a.h < 0 ? n : n - 1), 8));
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_phase_run, static_cast<double2*>(psi), n, a);
  prof_post(prof_slot_, s);
  count_launch();
  return e;
}

template <typename T, int S>
static cudaError_t block_pass_t(void* psi, int n, const BlockPass& a, cudaStream_t s) {
  using V = typename Cx<T>::V;
  constexpr size_t smem = sizeof(V) << S;
  const cudaError_t attr = smem_limit<k_block_pass<T, S>>(smem);
  if (attr != cudaSuccess) return attr;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)std::min<uint64_t>(1ull << (n - S), (uint64_t)sm_count() * (smem > 32768 ? 3 : 4)));
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_block_pass<T, S>, static_cast<V*>(psi), n, a);
}

cudaError_t launch_block_pass(void* psi, int n, qf_dtype dt, const BlockPass& a, cudaStream_t s) {
  const int prof_slot_ = prof_pre(QF_K_SPARSE, s);
  const cudaError_t e = dt == QF_C128 ? (a.s == 11 ? block_pass_t<double, 11>(psi, n, a, s)
                                                   : block_pass_t<double, kTileSmall>(psi, n, a, s))
                                      : (a.s == 13 ? block_pass_t<float, 13>(psi, n, a, s)
                                                   : block_pass_t<float, kTileSmall>(psi, n, a, s));
  prof_post(prof_slot_, s);
  count_launch();
  return e;
}

template <int NR>
static SpK<NR> compact(const SparseArgs& a) {
  SpK<NR> k;
  memset(&k, 0, sizeof(k));
  k.u = a.u;
  k.nr = a.nr;
  k.nzc = a.nzc;
  for (int i = 0; i < kSparseMaxSupp; ++i) k.supp[i] = a.supp[i];
  for (int r = 0; r < NR && r < a.nr; ++r) k.pat[r] = a.pat[r];
  k.zc[0] = a.zc[0];
  k.zc[1] = a.zc[1];
  for (int c = 0; c < kSparseMaxCls; ++c)
    for (int r = 0; r < NR && r < a.nr; ++r)
      for (int q = 0; q < NR && q < a.nr; ++q) {
        k.M[c][r][q] = a.M[c][r][q];
        k.Q[c][r][q] = a.Q[c][r][q];
      }
  return k;
}

bool sparse_m_real(const SparseArgs& a) {
  for (int c = 0; c < a.ncls; ++c)
    for (int r = 0; r < a.nr; ++r)
      for (int k = 0; k < a.nr; ++k)
        if (a.M[c][r][k].y != 0.0) return false;
  return true;
}

bool sparse_q_imag(const SparseArgs& a) {
  for (int c = 0; c < a.ncls; ++c)
    for (int r = 0; r < a.nr; ++r)
      for (int k = 0; k < a.nr; ++k)
        if (a.Q[c][r][k].x != 0.0) return false;
  return true;
}

template <typename T, int NR>
static void sparse_adj(void* psi, void* lam, int n, const SparseArgs& a, bool realst, double* partials,
                       unsigned* counter, double* out, int nblocks, cudaStream_t s) {
  using V = typename Cx<T>::V;
  const SpK<NR> k = compact<NR>(a);
  V* p = static_cast<V*>(psi);
  V* l = static_cast<V*>(lam);
  const bool rq = sparse_m_real(a) && sparse_q_imag(a);
  if (rq && realst)
    k_adj_sparse<T, NR, true, true><<<nblocks, 256, 0, s>>>(p, l, n, k, partials, counter, out);
  else if (rq)
    k_adj_sparse<T, NR, true, false><<<nblocks, 256, 0, s>>>(p, l, n, k, partials, counter, out);
  else
    k_adj_sparse<T, NR, false, false><<<nblocks, 256, 0, s>>>(p, l, n, k, partials, counter, out);
}

template <typename T, int NP, int F>
static cudaError_t pairs_t(void* psi, int n, const SparseArgs& a, const uint64_t (*pat)[2], const int (*row)[2],
                           const Reached& on, bool realst, cudaStream_t s) {
  using V = typename Cx<T>::V;
  PairK<NP> k;
  memset(&k, 0, sizeof(k));
  k.u = a.u;
  k.nzc = a.nzc;
  for (int i = 0; i < a.u; ++i) k.supp[i] = a.supp[i];
  k.zc[0] = a.zc[0];
  k.zc[1] = a.zc[1];
  k.on = on;
  for (int p = 0; p < NP; ++p)
    for (int r = 0; r < 2; ++r) {
      k.pat[p][r] = pat[p][r];
      for (int c = 0; c < a.ncls; ++c)
        for (int q = 0; q < 2; ++q)
          if (row[p][r] >= 0 && row[p][q] >= 0) k.M[c][p][r][q] = a.M[c][row[p][r]][row[p][q]];
    }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid_for(1ull << (n - a.u), 8));
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  V* v = static_cast<V*>(psi);
  if (F == PAIR_REAL && realst) return cudaLaunchKernelEx(&cfg, k_pairs<T, NP, PAIR_REAL, true>, v, n, k);
  return cudaLaunchKernelEx(&cfg, k_pairs<T, NP, F, false>, v, n, k);
}
template <typename T, int NP>
static cudaError_t pairs_f(void* psi, int n, const SparseArgs& a, const uint64_t (*pat)[2], const int (*row)[2],
                           const Reached& on, int form, bool realst, cudaStream_t s) {
  return form == PAIR_REAL   ? pairs_t<T, NP, PAIR_REAL>(psi, n, a, pat, row, on, realst, s)
         : form == PAIR_TURN ? pairs_t<T, NP, PAIR_TURN>(psi, n, a, pat, row, on, false, s)
                             : pairs_t<T, NP, PAIR_COMPLEX>(psi, n, a, pat, row, on, false, s);
}
template <typename T>
static cudaError_t pairs(void* psi, int n, const SparseArgs& a, const Reached& on, bool realst, cudaStream_t s) {
  uint64_t x = 0, pat[2 * kSparseMaxRows][2];
  for (int i = 0; i < a.u; ++i) x |= 1ull << a.supp[i];
  int row[2 * kSparseMaxRows][2], np = 0;
  for (int r = 0; r < a.nr; ++r) {  // rows ascend, so a pair's lower row comes first
    int q = 0;
    while (q < a.nr && a.pat[q] != (a.pat[r] ^ x)) ++q;
    if (q < r) continue;
    const bool alone = q == a.nr, low = a.pat[r] < (a.pat[r] ^ x);
    pat[np][low ? 0 : 1] = a.pat[r];
    pat[np][low ? 1 : 0] = a.pat[r] ^ x;
    row[np][low ? 0 : 1] = r;
    row[np++][low ? 1 : 0] = alone ? -1 : q;
  }
  bool real = true, turn = true;
  for (int c = 0; c < a.ncls; ++c)
    for (int r = 0; r < a.nr; ++r)
      for (int q = 0; q < a.nr; ++q) {
        real = real && a.M[c][r][q].y == 0.0;
        turn = turn && (r == q ? a.M[c][r][q].y : a.M[c][r][q].x) == 0.0;
      }
  const int form = real ? PAIR_REAL : turn ? PAIR_TURN : PAIR_COMPLEX;
  cudaError_t e = cudaSuccess;
  for (int p = 0; p < np && e == cudaSuccess; p += 4) {  // the pairs are independent
    const int m = std::min(4, np - p);
    e = m == 1   ? pairs_f<T, 1>(psi, n, a, pat + p, row + p, on, form, realst, s)
        : m == 2 ? pairs_f<T, 2>(psi, n, a, pat + p, row + p, on, form, realst, s)
        : m == 3 ? pairs_f<T, 3>(psi, n, a, pat + p, row + p, on, form, realst, s)
                 : pairs_f<T, 4>(psi, n, a, pat + p, row + p, on, form, realst, s);
  }
  return e;
}

template <typename T>
static void sparse_adj_nr(void* psi, void* lam, int n, const SparseArgs& a, bool realst, double* partials,
                          unsigned* counter, double* out, int nblocks, cudaStream_t s) {
  if (a.nr <= 2)
    sparse_adj<T, 2>(psi, lam, n, a, realst, partials, counter, out, nblocks, s);
  else if (a.nr <= 4)
    sparse_adj<T, 4>(psi, lam, n, a, realst, partials, counter, out, nblocks, s);
  else
    sparse_adj<T, 8>(psi, lam, n, a, realst, partials, counter, out, nblocks, s);
}

cudaError_t launch_sparse_on(void* psi, int n, qf_dtype dt, const SparseArgs& a, const Reached& on, bool realst,
                             cudaStream_t s) {
  const int prof_slot_ = prof_pre(QF_K_SPARSE, s);
  const cudaError_t e = dt == QF_C128 ? pairs<double>(psi, n, a, on, realst, s)
                                      : pairs<float>(psi, n, a, on, realst, s);
  prof_post(prof_slot_, s);
  count_launch();
  return e;
}

cudaError_t launch_sparse(void* psi, int n, qf_dtype dt, const SparseArgs& a, bool realst, cudaStream_t s) {
  Reached all;
  memset(&all, 0, sizeof(all));
  all.nsup = -1;
  return launch_sparse_on(psi, n, dt, a, all, realst, s);
}

cudaError_t launch_expect(const void* psi, int n, qf_dtype dt, const ExpGroup* groups, int ngroups,
                          const ExpChunk* chunks, double* partials, unsigned* counter, double* out, int nblocks,
                          cudaStream_t s) {
  const int prof_slot_ = prof_pre(QF_K_EXPECT, s);
  const bool tiled = n > kExpTileLogMax;  // at least one whole tile per group
  if (dt == QF_C128) {
    if (tiled)
      k_expect_tiled<double><<<nblocks, 256, 0, s>>>(static_cast<const double2*>(psi), n, groups, ngroups, chunks,
                                                     partials, counter, out);
    else
      k_expect<double><<<nblocks, 256, 0, s>>>(static_cast<const double2*>(psi), n, groups, ngroups, chunks,
                                               partials, counter, out);
  } else {
    if (tiled)
      k_expect_tiled<float><<<nblocks, 256, 0, s>>>(static_cast<const float2*>(psi), n, groups, ngroups, chunks,
                                                    partials, counter, out);
    else
      k_expect<float><<<nblocks, 256, 0, s>>>(static_cast<const float2*>(psi), n, groups, ngroups, chunks,
                                              partials, counter, out);
  }
  prof_post(prof_slot_, s);
  count_launch();
  return cudaGetLastError();
}

template <typename T>
static cudaError_t expect_passes_t(const void* psi, int n, const ExpPass* passes, int npass, const PassGroup* groups,
                                   const PassChunk* chunks, const ExpChunk* tabs, double* partials, int max_blocks,
                                   unsigned* counter, double* out, cudaStream_t s) {
  using V = typename Cx<T>::V;
  constexpr size_t smem = sizeof(V) << PassTile<T>::S;
  const cudaError_t attr = smem_limit<k_expect_pass<T>>(smem);
  if (attr != cudaSuccess) return attr;
  const uint64_t items = (uint64_t)npass << (n - PassTile<T>::S);
  const uint64_t grid = std::min<uint64_t>({items, (uint64_t)sm_count() * 3, (uint64_t)max_blocks});
  k_expect_pass<T><<<(unsigned)grid, kPassThreads, smem, s>>>(static_cast<const V*>(psi), n, passes, npass, groups,
                                                              chunks, tabs, partials, counter, out);
  return cudaGetLastError();
}

cudaError_t launch_expect_passes(const void* psi, int n, qf_dtype dt, const ExpPass* passes, int npass,
                                 const PassGroup* groups, const PassChunk* chunks, const ExpChunk* tabs,
                                 double* partials, int max_blocks, unsigned* counter, double* out, cudaStream_t s) {
  if (npass <= 0 || n < (dt == QF_C128 ? PassTile<double>::S : PassTile<float>::S)) return cudaErrorInvalidValue;
  const int prof_slot_ = prof_pre(QF_K_EXPECT, s);
  const cudaError_t e = dt == QF_C128 ? expect_passes_t<double>(psi, n, passes, npass, groups, chunks, tabs, partials,
                                                                max_blocks, counter, out, s)
                                      : expect_passes_t<float>(psi, n, passes, npass, groups, chunks, tabs, partials,
                                                               max_blocks, counter, out, s);
  prof_post(prof_slot_, s);
  count_launch();
  return e;
}

cudaError_t launch_hpsi(const void* psi, void* lam, int n, qf_dtype dt, const ExpGroup* groups, int ngroups,
                        const ExpChunk* chunks, double* partials, unsigned* counter, double* out, int nblocks,
                        cudaStream_t s) {
  const int prof_slot_ = prof_pre(QF_K_HPSI, s);
  if (dt == QF_C128)
    k_hpsi<double><<<nblocks, 256, 0, s>>>(static_cast<const double2*>(psi), static_cast<double2*>(lam), n, groups,
                                           ngroups, chunks, partials, counter, out);
  else
    k_hpsi<float><<<nblocks, 256, 0, s>>>(static_cast<const float2*>(psi), static_cast<float2*>(lam), n, groups,
                                          ngroups, chunks, partials, counter, out);
  prof_post(prof_slot_, s);
  count_launch();
  return cudaGetLastError();
}

template <typename T, int E, bool REALST>
static cudaError_t hpsi_tiled_e(const void* psi, void* lam, int n, const HClass* classes, int nclasses,
                                const HGroup* groups, const void* chunks, double* partials, unsigned* counter,
                                double* out, int nblocks, cudaStream_t s) {
  using V = typename Cx<T>::V;
  using C = typename WTab<T>::C;
  const size_t smem = sizeof(V) * 256 * E * kHpsiStages;
  const uint64_t ntiles = (1ull << n) / (256 * E);
  const cudaError_t attr = smem_limit<k_hpsi_tiled<T, E, REALST>>(smem);
  if (attr != cudaSuccess) return attr;
  // persistent grid: exactly the blocks that are resident at once (a partial
  // second wave would leave most SMs idle at the end)
  int per_sm = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_hpsi_tiled<T, E, REALST>, 256, smem);
  if (per_sm < 1) per_sm = 1;
  uint64_t cap = (uint64_t)sm_count() * (uint64_t)per_sm;
  if (cap > (uint64_t)nblocks) cap = (uint64_t)nblocks;
  unsigned g = (unsigned)std::min<uint64_t>(ntiles, cap);
  k_hpsi_tiled<T, E, REALST><<<g, 256, smem, s>>>(static_cast<const V*>(psi), static_cast<V*>(lam), n, classes,
                                                  nclasses, groups, static_cast<const C*>(chunks), partials, counter,
                                                  out);
  return cudaGetLastError();
}

// Tiles of 2^10 amplitudes, and of 2^11 for a real state (fewer registers per amplitude).
template <typename T>
static cudaError_t hpsi_tiled_t(const void* psi, void* lam, int n, int tb, bool realst, const HClass* classes,
                                int nclasses, const HGroup* groups, const void* chunks, double* partials,
                                unsigned* counter, double* out, int nblocks, cudaStream_t s) {
  const auto f = tb == 11 && realst ? hpsi_tiled_e<T, 8, true>
                 : tb == 10         ? (realst ? hpsi_tiled_e<T, 4, true> : hpsi_tiled_e<T, 4, false>)
                                    : nullptr;
  if (!f) return cudaErrorInvalidValue;
  return f(psi, lam, n, classes, nclasses, groups, chunks, partials, counter, out, nblocks, s);
}
cudaError_t launch_hpsi_tiled(const void* psi, void* lam, int n, qf_dtype dt, int tb, bool realst,
                              const HClass* classes, int nclasses, const HGroup* groups, const void* chunks,
                              double* partials, unsigned* counter, double* out, int nblocks, cudaStream_t s) {
  const int prof_slot_ = prof_pre(QF_K_HPSI, s);
  cudaError_t e = (dt == QF_C128)
                      ? hpsi_tiled_t<double>(psi, lam, n, tb, realst, classes, nclasses, groups, chunks, partials,
                                             counter, out, nblocks, s)
                      : hpsi_tiled_t<float>(psi, lam, n, tb, realst, classes, nclasses, groups, chunks, partials,
                                            counter, out, nblocks, s);
  prof_post(prof_slot_, s);
  count_launch();
  return e;
}

cudaError_t launch_hpsi_ds(const void* psi, void* lam, void* split, int n, const HClass* classes, int nclasses,
                           const HGroup* groups, const WChunkS* chunks, double* partials, unsigned* counter,
                           double* out, int nblocks, cudaStream_t s) {
  const int prof_slot_ = prof_pre(QF_K_HPSI, s);
  const uint64_t N = 1ull << n;
  k_split_ds<<<grid_for(N, 8), 256, 0, s>>>(static_cast<const double2*>(psi), static_cast<float2*>(split), N);
  int per_sm = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_hpsi_ds, 256, 0);
  if (per_sm < 1) per_sm = 1;
  uint64_t cap = (uint64_t)sm_count() * (uint64_t)per_sm;
  if (cap > (uint64_t)nblocks) cap = (uint64_t)nblocks;
  const unsigned g = (unsigned)std::min<uint64_t>(1ull << (n - 12), cap);
  k_hpsi_ds<<<g, 256, 0, s>>>(static_cast<const double2*>(psi), static_cast<const float2*>(split),
                              static_cast<double2*>(lam), n, classes, nclasses, groups, chunks, partials, counter,
                              out);
  prof_post(prof_slot_, s);
  count_launch();
  count_launch();
  return cudaGetLastError();
}

template <typename T, int F>
static void adj_rot_f(void* psi, void* lam, int n, const RotArgs& a, double* partials, unsigned* counter, double* out,
                      int nblocks, cudaStream_t s) {
  using V = typename Cx<T>::V;
  k_adj_rot<T, F><<<nblocks, 256, 0, s>>>(static_cast<V*>(psi), static_cast<V*>(lam), n, a.x, a.z, a.h, a.y, (T)a.A,
                                          (T)a.B, partials, counter, out);
}

template <typename T>
static void adj_rot_t(void* psi, void* lam, int n, const RotArgs& a, double* partials, unsigned* counter, double* out,
                      int nblocks, cudaStream_t s) {
  if (a.form == FORM_A1)
    adj_rot_f<T, FORM_A1>(psi, lam, n, a, partials, counter, out, nblocks, s);
  else if (a.form == FORM_B1)
    adj_rot_f<T, FORM_B1>(psi, lam, n, a, partials, counter, out, nblocks, s);
  else
    adj_rot_f<T, FORM_AB>(psi, lam, n, a, partials, counter, out, nblocks, s);
}

cudaError_t launch_adj_rot(void* psi, void* lam, int n, qf_dtype dt, const RotArgs& a, double* partials,
                           unsigned* counter, double* out, int nblocks, cudaStream_t s) {
  const int prof_slot_ = prof_pre(QF_K_ADJ_ROT, s);
  if (dt == QF_C128)
    adj_rot_t<double>(psi, lam, n, a, partials, counter, out, nblocks, s);
  else
    adj_rot_t<float>(psi, lam, n, a, partials, counter, out, nblocks, s);
  prof_post(prof_slot_, s);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_adj_sparse(void* psi, void* lam, int n, qf_dtype dt, const SparseArgs& a, bool realst,
                              double* partials, unsigned* counter, double* out, int nblocks, cudaStream_t s) {
  const int prof_slot_ = prof_pre(QF_K_ADJ_SPARSE, s);
  if (dt == QF_C128)
    sparse_adj_nr<double>(psi, lam, n, a, realst, partials, counter, out, nblocks, s);
  else
    sparse_adj_nr<float>(psi, lam, n, a, realst, partials, counter, out, nblocks, s);
  prof_post(prof_slot_, s);
  count_launch();
  return cudaGetLastError();
}

}  // namespace qf

extern "C" uint64_t qf_kernel_launches(int reset) {
  const uint64_t v = qf::t_launches;
  if (reset) qf::t_launches = 0;
  return v;
}
