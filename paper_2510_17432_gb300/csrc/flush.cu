// Buffered accumulation (Sec. II.B time blocks, Sec. IV quasi-eigenstates, the Fermi-Dirac series):
//     acc_e += sum_{t < T} a_t(e) r_t phi_t        (e < n_acc)
// over T buffered Chebyshev vectors phi_t (consecutive state blocks) with real amplitudes a_t(e).
// Every coefficient family of the method is real up to a power of -i common to all accumulators:
// c_n(j tau~) = a_n (-i)^n with a_n = (2 - delta_n0) J_n (the factor e^{-i H0 t_j} stays out of the states),
// so the vector is turned by (-i)^n once per term (r_t: a swap and a sign of the amplitude) and one real
// multiply-add per component does the rest.  The coefficients C_n(E) of the quasi-eigenstates and a_n of the Fermi-Dirac series are real as they are.
//
// All states take the same coefficients, so a state block is a flat array of complex numbers here.  A
// thread holds the accumulators of one 16-byte unit (two complex64 or one complex128 number) in
// registers, streams the T terms past them, TB loads in flight, and reads and writes each accumulator
// once per window.  The amplitudes sit in shared memory, one broadcast load per two accumulators; of a
// time block's accumulators the early ones close first (n >= N(j tau~)), and groups of four closed ones
// are skipped.  Grid: (tiles of EB accumulators, unit blocks); the tiles of a unit block run side by side
// and share the buffered vectors through L2.
//
// Bound: HBM for complex64 -- 8 B per term and 8 B (write) or 16 B per accumulator and window, per
// number; FP64 issue for complex128 (2 FMAs per term, accumulator and number).  Whole blocks of 92 terms
// into 16 accumulators in one window, real amplitudes instead of complex ones (half the FMAs), and sums
// that start and end in the kernel took the flushes of 16 blocks on 8.3M sites from 64 to about 25 ms
// (complex64), and those of the 2.1M-site complex128 correlation from 145 to 69 ms with b going from 6 to 16.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "stencil.cuh"
#include "tbpm_internal.cuh"

namespace tbpm {
namespace {

constexpr int kFlushT = 96;  // terms per window: a whole time block of 16 Nyquist steps (N(16 pi) = 92)

struct FlushArgs {
  const void* phi;
  int T;
  int64_t stride;      // units between consecutive vectors and between accumulators
  void* acc;
  int nb;
  const double* amp;   // amplitude of term t and accumulator e at amp[(t * nb + e) * as]
  int as;
  int init;            // 1: the window starts the sums (nothing is read from acc)
  int64_t n_units;
};

template <typename R>
struct UnitOf;
template <>
struct UnitOf<float4> { using R = float; static constexpr int C = 2; };
template <>
struct UnitOf<float2> { using R = float; static constexpr int C = 1; };
template <>
struct UnitOf<double2> { using R = double; static constexpr int C = 1; };

__device__ __forceinline__ float2 part(float4 v, int k) { return k ? make_float2(v.z, v.w) : make_float2(v.x, v.y); }
__device__ __forceinline__ float2 part(float2 v, int) { return v; }
__device__ __forceinline__ double2 part(double2 v, int) { return v; }
__device__ __forceinline__ float4 join(const float2 (&p)[2]) { return make_float4(p[0].x, p[0].y, p[1].x, p[1].y); }
__device__ __forceinline__ float2 join(const float2 (&p)[1]) { return p[0]; }
__device__ __forceinline__ double2 join(const double2 (&p)[1]) { return p[0]; }
// amplitude as the multiply-add takes it: twice for the packed f32x2 FMA
__device__ __forceinline__ float2 twice(float a) { return make_float2(a, a); }
__device__ __forceinline__ double twice(double a) { return a; }
__device__ __forceinline__ float2 axpy(float2 a, float2 x, float2 y) { return __ffma2_rn(a, x, y); }
__device__ __forceinline__ double2 axpy(double a, double2 x, double2 y) {
  return make_double2(fma(a, x.x, y.x), fma(a, x.y, y.y));
}
template <typename V2>
__device__ __forceinline__ V2 turn(V2 x) {  // -i x
  V2 r;
  r.x = x.y;
  r.y = -x.x;
  return r;
}

// ROT: term t carries (-i)^t (the window starts at a multiple of four).
template <typename U, int EB, int TB, bool ROT>
__global__ void __launch_bounds__(kThreads, EB >= 16 ? 2 : 3) k_flush(FlushArgs f) {
  using R = typename UnitOf<U>::R;
  constexpr int C = UnitOf<U>::C;
  using V2 = std::conditional_t<sizeof(R) == 4, float2, double2>;
  using A = decltype(twice(R(0)));
  constexpr int G = EB < 4 ? EB : 4;  // accumulators skipped together
  __shared__ __align__(16) A cs[kFlushT][EB];
  __shared__ int open[kFlushT];       // first group with an open accumulator
  const int e0 = blockIdx.x * EB;
  const int ne = min(EB, f.nb - e0);
  for (int i = threadIdx.x; i < f.T; i += kThreads) open[i] = EB / G;
  __syncthreads();
  for (int i = threadIdx.x; i < f.T * EB; i += kThreads) {
    const int t = i / EB, e = i - t * EB;
    R a = e < ne ? (R)f.amp[((int64_t)t * f.nb + e0 + e) * f.as] : R(0);
    if (ROT && (t & 2)) a = -a;
    cs[t][e] = twice(a);
    if (a != R(0)) atomicMin(&open[t], e / G);
  }
  __syncthreads();
  const U* Phi = reinterpret_cast<const U*>(f.phi);
  U* Q = reinterpret_cast<U*>(f.acc);
  for (int64_t u = (int64_t)blockIdx.y * kThreads + threadIdx.x; u < f.n_units; u += (int64_t)gridDim.y * kThreads) {
    V2 ac[EB][C];
#pragma unroll
    for (int e = 0; e < EB; ++e) {
      U q{};
      if (!f.init && e < ne && TBPM_DBG_OK((int64_t)(e0 + e) * f.stride + u, f.nb * f.stride, TBPM_DBG_FLUSH)) q = __ldcs(Q + (int64_t)(e0 + e) * f.stride + u);
#pragma unroll
      for (int k = 0; k < C; ++k) ac[e][k] = part(q, k);
    }
    for (int t0 = 0; t0 < f.T; t0 += TB) {
      U x[TB];
#pragma unroll
      for (int j = 0; j < TB; ++j) {
        if (t0 + j < f.T && TBPM_DBG_OK((int64_t)(t0 + j) * f.stride + u, f.T * f.stride, TBPM_DBG_FLUSH)) x[j] = __ldg(Phi + (int64_t)(t0 + j) * f.stride + u);
        else x[j] = U{};
      }
#pragma unroll
      for (int j = 0; j < TB; ++j) {
        if (t0 + j >= f.T) break;  // uniform
        V2 v[C];
#pragma unroll
        for (int k = 0; k < C; ++k) v[k] = ROT && (j & 1) ? turn(part(x[j], k)) : part(x[j], k);
        const int lo = open[t0 + j];
#pragma unroll
        for (int g = 0; g < EB / G; ++g) {
          if (g >= lo && g * G < ne) {  // uniform
#pragma unroll
            for (int e = g * G; e < g * G + G; ++e) {
              const A a = cs[t0 + j][e];
#pragma unroll
              for (int k = 0; k < C; ++k) ac[e][k] = axpy(a, v[k], ac[e][k]);
            }
          }
        }
      }
    }
#pragma unroll
    for (int e = 0; e < EB; ++e) {
      if (e < ne && TBPM_DBG_OK((int64_t)(e0 + e) * f.stride + u, f.nb * f.stride, TBPM_DBG_FLUSH)) {
        __stcs(Q + (int64_t)(e0 + e) * f.stride + u, join(ac[e]));
      }
    }
  }
}

template <typename U, int EB, int TB>
void launch_flush(const FlushArgs& f, bool rot, dim3 grid, cudaStream_t st) {
  if (rot) k_flush<U, EB, TB, true><<<grid, kThreads, 0, st>>>(f);
  else k_flush<U, EB, TB, false><<<grid, kThreads, 0, st>>>(f);
}

}  // namespace

int flush_max_terms() { return kFlushT; }

int launch_flush(tbpm_ctx* ctx, int precision, int64_t n_numbers, const void* phi, int T, void* acc, int nb,
                 const double* amp, int amp_stride, bool rot, bool init, int tile) {
  if (T < 1 || T > kFlushT || nb < 1) {
    set_error("flush of %d terms into %d accumulators", T, nb);
    return TBPM_EINVAL;
  }
  FlushArgs f;
  f.phi = phi;
  f.T = T;
  f.acc = acc;
  f.nb = nb;
  f.amp = amp;
  f.as = amp_stride;
  f.init = init ? 1 : 0;
  // two complex64 numbers per unit where every block holds an even number of them (blocks are then
  // 16-byte aligned); an odd number only comes from one state on an odd number of sites
  const bool wide = precision == TBPM_C64 && n_numbers % 2 == 0;
  f.n_units = wide ? n_numbers / 2 : n_numbers;
  f.stride = f.n_units;
  const int eb = tile > 0 ? tile : (nb == 1 ? 1 : nb <= 4 ? 4 : 16);
  const int etiles = (nb + eb - 1) / eb;
  const int64_t want = std::max<int64_t>(1, (int64_t)ctx->num_sms * (eb == 16 ? 8 : 12) / etiles);
  const dim3 grid(etiles, (unsigned)std::min<int64_t>(std::min<int64_t>(want, (f.n_units + kThreads - 1) / kThreads),
                                                      65535));
  if (precision == TBPM_C128) {
    if (eb == 1) launch_flush<double2, 1, 8>(f, rot, grid, ctx->stream);
    else if (eb == 4) launch_flush<double2, 4, 4>(f, rot, grid, ctx->stream);
    else launch_flush<double2, 16, 4>(f, rot, grid, ctx->stream);
  } else if (wide) {
    if (eb == 1) launch_flush<float4, 1, 8>(f, rot, grid, ctx->stream);
    else if (eb == 4) launch_flush<float4, 4, 8>(f, rot, grid, ctx->stream);
    else launch_flush<float4, 16, 8>(f, rot, grid, ctx->stream);
  } else {
    if (eb == 1) launch_flush<float2, 1, 8>(f, rot, grid, ctx->stream);
    else if (eb == 4) launch_flush<float2, 4, 8>(f, rot, grid, ctx->stream);
    else launch_flush<float2, 16, 8>(f, rot, grid, ctx->stream);
  }
  TBPM_CK_LAUNCH(ctx);
  return TBPM_OK;
}

}  // namespace tbpm

TBPM_DEBUG_UNIT(flush)
