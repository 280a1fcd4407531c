// C ABI of the library: context, lattice construction on the device, initial states, and
// the drivers of the three propagation forms of Sec. II.A (sequential, moment-based,
// state-based with time blocks) and of the spectra of Sec. III.
#include <cuda_runtime.h>
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <functional>
#include <vector>

#include "tbpm_internal.cuh"

namespace tbpm {

static thread_local char g_err[1024];

void set_error(const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof g_err, fmt, ap);
  va_end(ap);
}
void clear_error() { g_err[0] = 0; }

int ensure(tbpm_ctx* ctx, DevBuf& b, size_t bytes) {
  if (bytes <= b.cap) return TBPM_OK;
  if (b.p) {
    TBPM_CK(cudaFreeAsync(b.p, ctx->stream));
    b.p = nullptr;
    b.cap = 0;
  }
  const size_t want = std::max<size_t>(256, bytes + (bytes >> 4));
  cudaError_t e = cudaMallocAsync(&b.p, want, ctx->stream);
  if (e != cudaSuccess) {
    cudaGetLastError();
    b.p = nullptr;
    set_error("device allocation of %zu bytes failed: %s", want, cudaGetErrorString(e));
    return TBPM_ENOMEM;
  }
  b.cap = want;
  return TBPM_OK;
}

static cudaEvent_t take_event(tbpm_ctx* ctx) {
  if (!ctx->event_pool.empty()) {
    cudaEvent_t e = ctx->event_pool.back();
    ctx->event_pool.pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  cudaEventCreate(&e);
  return e;
}

int phase_begin(tbpm_ctx* ctx, int kind) {
  static const char* const kNames[3] = {"recurrence", "reconstruction", "fused passes"};
  ctx->nvtx_open.push_back(nvtxRangeStartA(kNames[kind >= 0 && kind < 3 ? kind : 0]));
  if (!ctx->profiling) return -1;
  tbpm_ctx::Phase ph;
  ph.a = take_event(ctx);
  ph.b = take_event(ctx);
  ph.kind = kind;
  ph.launches = ctx->launches;
  cudaEventRecord(ph.a, ctx->stream);
  ctx->phases.push_back(ph);
  return (int)ctx->phases.size() - 1;
}

void phase_end(tbpm_ctx* ctx, int token) {
  if (!ctx->nvtx_open.empty()) {
    nvtxRangeEnd(ctx->nvtx_open.back());
    ctx->nvtx_open.pop_back();
  }
  if (token < 0 || token >= (int)ctx->phases.size()) return;
  tbpm_ctx::Phase& ph = ctx->phases[token];
  ph.launches = ctx->launches - ph.launches;
  cudaEventRecord(ph.b, ctx->stream);
}

static void release(tbpm_ctx* ctx, DevBuf& b) {
  if (b.p) cudaFreeAsync(b.p, ctx->stream);
  b.p = nullptr;
  b.cap = 0;
}

static std::vector<DevBuf*> workspaces(tbpm_ctx* ctx) {
  return {&ctx->ws_phi[0], &ctx->ws_phi[1], &ctx->ws_psi, &ctx->ws_acc, &ctx->ws_partials,
          &ctx->ws_counter, &ctx->ws_mu, &ctx->ws_table, &ctx->ws_aux, &ctx->ws_out,
          &ctx->ws_energies, &ctx->ws_recon, &ctx->ws_phi2[0], &ctx->ws_phi2[1],
          &ctx->ws_fused_partials, &ctx->ws_qe, &ctx->ws_qe_coef, &ctx->ws_xdot, &ctx->ws_blk, &ctx->ws_blk_coef,
          &ctx->ws_jpsi, &ctx->ws_ec, &ctx->ws_fermi, &ctx->ws_packets};
}

// Bytes that further allocations can have: free on the device, and idle in the pool that keeps freed memory.
static size_t memory_left(tbpm_ctx* ctx) {
  size_t free_b = 0, total_b = 0;
  cudaMemGetInfo(&free_b, &total_b);
  cudaMemPool_t pool;
  uint64_t reserved = 0, used = 0;
  if (cudaDeviceGetDefaultMemPool(&pool, ctx->device) != cudaSuccess ||
      cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &reserved) != cudaSuccess ||
      cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used) != cudaSuccess) {
    cudaGetLastError();
    return free_b;
  }
  return free_b + (size_t)(reserved > used ? reserved - used : 0);
}

static size_t kept_bytes(tbpm_ctx* ctx) {
  size_t sum = 0;
  for (DevBuf* b : workspaces(ctx)) sum += b->cap;
  return sum;
}

static int release_workspaces(tbpm_ctx* ctx) {
  for (DevBuf* b : workspaces(ctx)) release(ctx, *b);
  ctx->packet_cap = 0;  // the packet buffer's tags start anew with the next one
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  return TBPM_OK;
}

// Before a request that sizes its blocks by the memory there is: workspaces kept from earlier requests go where
// they are more than half of what is left, so that the request sees the device that a context's first one sees.
// (With less than that kept, a window that the first call could have in full fits again: at most a third of the
// memory is kept, and a window takes up to half of what is left.)
static int fresh_workspaces(tbpm_ctx* ctx) {
  return 2 * kept_bytes(ctx) > memory_left(ctx) ? release_workspaces(ctx) : TBPM_OK;
}

// Runs a request; where memory does not suffice, again without what earlier requests kept, and then in the form
// with the fewest state blocks (index lists instead of the full layout, one step per pass).
template <typename F>
static int with_memory(tbpm_ctx* ctx, F body) {
  int r = body();
  for (int lean = 0; lean < 2 && r == TBPM_ENOMEM; ++lean) {
    clear_error();
    TBPM_TRY(release_workspaces(ctx));
    ctx->lean = lean != 0;
    r = body();
  }
  ctx->lean = false;
  return r;
}

template <typename T>
static int dev_alloc(tbpm_ctx* ctx, T** p, size_t count) {
  cudaError_t e = cudaMallocAsync((void**)p, std::max<size_t>(1, count) * sizeof(T), ctx->stream);
  if (e != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    set_error("device allocation of %zu bytes failed: %s", count * sizeof(T), cudaGetErrorString(e));
    return TBPM_ENOMEM;
  }
  return TBPM_OK;
}

static int grid_for(tbpm_ctx* ctx, int64_t n, int threads, int per_sm = 16) {
  const int64_t b = (n + threads - 1) / threads;
  return (int)std::max<int64_t>(1, std::min<int64_t>(b, (int64_t)ctx->num_sms * per_sm));
}

// ------------------------------------------------------------------ lattice kernels
constexpr int kT = 256;

__device__ __forceinline__ double disorder_value(uint64_t seed, double W, int64_t i) {
  const uint32_t u = draw_u32(seed, (uint64_t)i, STREAM_DISORDER, 0);
  return W * ((double)(u >> 8) * 0x1p-24 - 0.5);
}

__device__ __forceinline__ bool vacant(uint64_t seed, uint64_t thr, int64_t i) {
  return (uint64_t)draw_u32(seed, (uint64_t)i, STREAM_VACANCY, 0) < thr;
}

struct Bounds3 {
  double emax, emin, deg;
};

__device__ __forceinline__ void block_bounds(Bounds3 v, Bounds3* part) {
  __shared__ Bounds3 sh[kT / 32];
  for (int off = 16; off >= 1; off >>= 1) {
    v.emax = fmax(v.emax, __shfl_xor_sync(0xffffffffu, v.emax, off));
    v.emin = fmin(v.emin, __shfl_xor_sync(0xffffffffu, v.emin, off));
    v.deg += __shfl_xor_sync(0xffffffffu, v.deg, off);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    Bounds3 r = sh[0];
    for (int w = 1; w < kT / 32; ++w) {
      r.emax = fmax(r.emax, sh[w].emax);
      r.emin = fmin(r.emin, sh[w].emin);
      r.deg += sh[w].deg;
    }
    part[blockIdx.x] = r;
  }
}

// Stencil path: V_i (FP64), degree and Gershgorin terms for every site.
__global__ void __launch_bounds__(kT) k_lattice_stencil(Geom g, uint64_t seed, double W, double abs_t,
                                                        double* v64, Bounds3* part) {
  Bounds3 acc{-INFINITY, INFINITY, 0.0};
  for (int64_t i = (int64_t)blockIdx.x * kT + threadIdx.x; i < g.n_full; i += (int64_t)gridDim.x * kT) {
    int deg = 0;
    for (int d = 0; d < g.z; ++d) deg += neighbour_full(g, i, d) >= 0;
    const double v = (W != 0.0) ? disorder_value(seed, W, i) : 0.0;
    if (v64) v64[i] = v;
    acc.emax = fmax(acc.emax, v + deg * abs_t);
    acc.emin = fmin(acc.emin, v - deg * abs_t);
    acc.deg += deg;
  }
  block_bounds(acc, part);
}

__global__ void k_bounds_final(const Bounds3* part, int n, double* out) {
  __shared__ Bounds3 sh[kT];
  Bounds3 acc{-INFINITY, INFINITY, 0.0};
  for (int i = threadIdx.x; i < n; i += kT) {
    acc.emax = fmax(acc.emax, part[i].emax);
    acc.emin = fmin(acc.emin, part[i].emin);
    acc.deg += part[i].deg;
  }
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int w = kT / 2; w >= 1; w >>= 1) {  // maxima, minima and a sum of integers: any order gives the same
    if (threadIdx.x < w) {
      Bounds3 &r = sh[threadIdx.x], o = sh[threadIdx.x + w];
      r.emax = fmax(r.emax, o.emax);
      r.emin = fmin(r.emin, o.emin);
      r.deg += o.deg;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[0] = sh[0].emax;
    out[1] = sh[0].emin;
    out[2] = sh[0].deg;
  }
}

// CSR path, pass 1: active-site counts per chunk of kChunk sites.
constexpr int kPer = 16;
constexpr int kChunk = kT * kPer;

__global__ void __launch_bounds__(kT) k_count_active(int64_t n_full, uint64_t seed, uint64_t thr,
                                                     int64_t* counts) {
  __shared__ int64_t sh[kT / 32];
  const int64_t base = (int64_t)blockIdx.x * kChunk + (int64_t)threadIdx.x * kPer;
  int64_t c = 0;
  for (int q = 0; q < kPer; ++q) {
    const int64_t i = base + q;
    if (i < n_full && !vacant(seed, thr, i)) ++c;
  }
  for (int off = 16; off >= 1; off >>= 1) c += __shfl_xor_sync(0xffffffffu, c, off);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int64_t t = 0;
    for (int w = 0; w < kT / 32; ++w) t += sh[w];
    counts[blockIdx.x] = t;
  }
}

// Exclusive scan of the chunk counts by one block: offs[0..n], offs[n] = total.
__global__ void k_scan_counts(const int64_t* counts, int64_t n, int64_t* offs) {
  __shared__ int64_t sh[1024];
  const int64_t per = (n + 1023) / 1024;
  const int64_t lo = threadIdx.x * per, hi = std::min<int64_t>(n, lo + per);
  int64_t s = 0;
  for (int64_t i = lo; i < hi; ++i) s += counts[i];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    const int64_t v = threadIdx.x >= off ? sh[threadIdx.x - off] : 0;
    __syncthreads();
    sh[threadIdx.x] += v;
    __syncthreads();
  }
  int64_t run = sh[threadIdx.x] - s;  // exclusive prefix of this thread's segment
  for (int64_t i = lo; i < hi; ++i) {
    offs[i] = run;
    run += counts[i];
  }
  if (threadIdx.x == 1023) offs[n] = sh[1023];
}

// CSR path, pass 2: compact index of every site (-1 if vacant) and full index of every active site.
__global__ void __launch_bounds__(kT) k_compact(int64_t n_full, uint64_t seed, uint64_t thr,
                                                const int64_t* offs, int64_t* compact, int64_t* full_of) {
  __shared__ int64_t sh[kT];
  const int64_t base = (int64_t)blockIdx.x * kChunk + (int64_t)threadIdx.x * kPer;
  unsigned flags = 0;
  int c = 0;
  for (int q = 0; q < kPer; ++q) {
    const int64_t i = base + q;
    if (i < n_full && !vacant(seed, thr, i)) {
      flags |= 1u << q;
      ++c;
    }
  }
  sh[threadIdx.x] = c;
  __syncthreads();
  for (int off = 1; off < kT; off <<= 1) {
    const int64_t v = threadIdx.x >= off ? sh[threadIdx.x - off] : 0;
    __syncthreads();
    sh[threadIdx.x] += v;
    __syncthreads();
  }
  int64_t k = offs[blockIdx.x] + sh[threadIdx.x] - c;
  for (int q = 0; q < kPer; ++q) {
    const int64_t i = base + q;
    if (i >= n_full) break;
    if (flags & (1u << q)) {
      compact[i] = k;
      full_of[k] = i;
      ++k;
    } else {
      compact[i] = -1;
    }
  }
}

// CSR path, pass 3: ELL neighbour lists, V_i and Gershgorin terms of every active site.
__global__ void __launch_bounds__(kT) k_build_ell(Geom g, int64_t n, const int64_t* full_of,
                                                  const int64_t* compact, uint64_t seed, double W,
                                                  double abs_t, int32_t* ell, double* v64, Bounds3* part) {
  Bounds3 acc{-INFINITY, INFINITY, 0.0};
  for (int64_t k = (int64_t)blockIdx.x * kT + threadIdx.x; k < n; k += (int64_t)gridDim.x * kT) {
    const int64_t i = full_of[k];
    int deg = 0;
    for (int d = 0; d < g.z; ++d) {
      const int64_t j = neighbour_full(g, i, d);
      const int64_t cj = j >= 0 ? compact[j] : -1;
      ell[k * g.z + d] = (int32_t)cj;
      deg += cj >= 0;
    }
    const double v = (W != 0.0) ? disorder_value(seed, W, i) : 0.0;
    if (v64) v64[k] = v;
    acc.emax = fmax(acc.emax, v + deg * abs_t);
    acc.emin = fmin(acc.emin, v - deg * abs_t);
    acc.deg += deg;
  }
  block_bounds(acc, part);
}

// Long-range lattices, pass 3: ELL lists from the taps (dx, dy, dz, ds) of sublattice 0; a
// honeycomb B site takes every tap mirrored, (x-dx, y-dy) of sublattice 1-ds, so slot d has the
// same length and weight on both sublattices.  Periodic directions wrap by modulo, open ones
// drop the tap.  Gershgorin radius = sum of |t_d| over the slots that reach active sites.
__global__ void __launch_bounds__(kT) k_build_ell_taps(Geom g, int64_t n, const int64_t* full_of,
                                                       const int64_t* compact, const int4* taps, const double* tabs,
                                                       uint64_t seed, double W, int32_t* ell, double* v64,
                                                       Bounds3* part) {
  Bounds3 acc{-INFINITY, INFINITY, 0.0};
  const bool hc = g.kind == TBPM_HONEYCOMB;
  auto wrap = [](int64_t v, int64_t L, int periodic, bool* ok) -> int64_t {
    if (v >= 0 && v < L) return v;
    if (!periodic) { *ok = false; return 0; }
    const int64_t r = v % L;
    return r < 0 ? r + L : r;
  };
  for (int64_t k = (int64_t)blockIdx.x * kT + threadIdx.x; k < n; k += (int64_t)gridDim.x * kT) {
    const int64_t i = full_of[k];
    int64_t x, y, zc = 0;
    int s = 0;
    if (hc) {
      s = (int)(i & 1);
      const int64_t c = i >> 1;
      x = c % g.Lx;
      y = c / g.Lx;
    } else {
      x = i % g.Lx;
      y = (i / g.Lx) % g.Ly;
      zc = i / (g.Lx * g.Ly);
    }
    const int64_t sg = s ? -1 : 1;
    double rad = 0.0;
    int deg = 0;
    for (int d = 0; d < g.z; ++d) {
      const int4 tp = taps[d];
      bool ok = true;
      const int64_t tx = wrap(x + sg * tp.x, g.Lx, g.pbc_x, &ok);
      const int64_t ty = wrap(y + sg * tp.y, g.Ly, g.pbc_y, &ok);
      const int64_t tz = wrap(zc + sg * tp.z, g.Lz, g.pbc_z, &ok);
      int64_t cj = -1;
      if (ok) {
        const int64_t j = hc ? 2 * (ty * g.Lx + tx) + (s ? 1 - tp.w : tp.w) : (tz * g.Ly + ty) * g.Lx + tx;
        cj = compact[j];
      }
      if (ell) ell[k * g.z + d] = (int32_t)cj;
      if (cj >= 0) {
        rad += tabs[d];
        ++deg;
      }
    }
    const double v = (W != 0.0) ? disorder_value(seed, W, i) : 0.0;
    if (v64) v64[k] = v;
    acc.emax = fmax(acc.emax, v + rad);
    acc.emin = fmin(acc.emin, v - rad);
    acc.deg += deg;
  }
  block_bounds(acc, part);
}

// D_i = (V_i - H0)/|H| in FP64 and rounded once to FP32.
__global__ void k_make_diag(int64_t n, const double* v64, double H0, double half, double* d64, float* d32) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double d = (v64[i] - H0) / half;
    if (d64) d64[i] = d;
    if (d32) d32[i] = (float)d;
  }
}

// ------------------------------------------------------------------ initial states
// exp(2 pi i u / 2^32) * (sh + sl) in FP32, and whether each part is surely the correctly rounded one.  The pair it
// is rounded from is within 2^-14 ulp of the exact value (6e-5 over all 2^32 draws and ten scales), so it is unless
// the pair lies within 2^-13 ulp of the middle between two floats.  The draw is reduced exactly to a quarter turn
// (an integer below 2^29, split exactly into two floats), sin and cos of the remainder |x| <= 1/4 (in units of pi)
// come from their Taylor series, whose first three (sine) and four (cosine) terms are summed in float pairs
// (h + l) and the rest in FP32, where their weight keeps the error below 2^-36, and the scale is applied to the
// pair before the one rounding.
struct F2 {
  float h, l;
};
// c + z s for float pairs with |c| >= |z s|
__host__ __device__ __forceinline__ F2 pair_step(F2 c, F2 z, F2 s) {
  const float p = z.h * s.h;
  const float e = fmaf(z.h, s.h, -p) + fmaf(z.l, s.h, z.h * s.l);
  const float h = c.h + p;
  return {h, (c.h - h) + p + (c.l + e)};
}
// c scaled by sh + sl and rounded; *sure is cleared next to a tie (and for zero and powers of two, whose
// neighbours are not symmetric)
__host__ __device__ __forceinline__ float scaled(F2 c, float sh, float sl, bool* sure) {
  const float lo = fmaf(c.h, sl, c.l * sh);
  const float v = fmaf(c.h, sh, lo);
  const float p = c.h * sh;
  const float r = (p - v) + (fmaf(c.h, sh, -p) + lo);  // what the rounding left, at most half an ulp
  uint32_t b;
  memcpy(&b, &v, 4);
  const uint32_t e = b & 0x7f800000u, half_bits = e - (24u << 23);
  float half;
  memcpy(&half, &half_bits, 4);
  if ((b & 0x007fffffu) == 0 || e < (64u << 23) || fabsf(r) > half * (1.f - 0x1p-12f)) *sure = false;
  return v;
}
__host__ __device__ __forceinline__ float2 unit_phase(uint32_t u, float sh, float sl, bool* sure) {
  const uint32_t q = (u + 0x20000000u) >> 30;
  const int r = (int)(u - (q << 30));  // [-2^29, 2^29)
  const float xi = (float)r;
  const F2 x = {xi * 0x1p-31f, (float)(r - (int)xi) * 0x1p-31f};
  F2 z;
  z.h = x.h * x.h;
  z.l = fmaf(x.h, x.h, -z.h) + 2.f * x.h * x.l;
  // pi^(2k+1)/(2k+1)! and pi^(2k)/(2k)!, alternating
  float t = fmaf(z.h, -2.19153535e-05f, 4.66302794e-04f);
  t = fmaf(z.h, t, -7.37043098e-03f);
  t = fmaf(z.h, t, 8.21458846e-02f);
  t = fmaf(z.h, t, -5.99264503e-01f);
  F2 s = pair_step({2.55016398f, 5.55786386e-08f}, z, {t, 0.f});
  s = pair_step({-5.16771269f, -9.16039227e-08f}, z, s);
  s = pair_step({3.14159274f, -8.74227766e-08f}, z, s);
  const float ph = x.h * s.h;  // sin = x s
  s = {ph, fmaf(x.h, s.h, -ph) + fmaf(x.l, s.h, x.h * s.l)};
  t = fmaf(z.h, -1.04638108e-04f, 1.9295743e-03f);
  t = fmaf(z.h, t, -2.58068908e-02f);
  t = fmaf(z.h, t, 2.35330626e-01f);
  F2 c = pair_step({-1.33526278f, 6.56655308e-09f}, z, {t, 0.f});
  c = pair_step({4.05871201f, 1.20801531e-07f}, z, c);
  c = pair_step({-4.93480206f, -1.45185794e-07f}, z, c);
  c = pair_step({1.f, 0.f}, z, c);
  const float cs = scaled(c, sh, sl, sure);
  const float sn = scaled(s, sh, sl, sure);
  const float a = (q & 1) ? sn : cs, b = (q & 1) ? cs : sn;  // quarter turns: (c, s), (-s, c), (-c, -s), (s, -c)
  return make_float2((q == 1 || q == 2) ? -a : a, q >= 2 && q < 4 ? -b : b);
}

// Random phases psi_i = exp(2 pi i u / 2^32) / sqrt(N), u = Philox(state_seed; i, 2, s).
// complex64 is bound by the draw (integer multiplies) and FP32 issue: 537M states take 3.5 ms against 31.1 ms
// with FP64 sincospi (GB300 issues two FP64 operations per clock and SM), which complex128 keeps and which settles
// the one draw in 2000 that lies next to a tie, so that every state is the FP64 one rounded once.
template <typename R>
__global__ void k_init_random(int64_t n, int Spad, int logS, int S, int s0, uint64_t seed, const int64_t* full_of,
                              const float* masked, double inv_sqrt_n, R* out, uint32_t* draws) {
  const int64_t total = n * Spad;
  const float sh = (float)inv_sqrt_n, sl = (float)(inv_sqrt_n - (double)sh);
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = e >> logS;
    const int s = (int)(e & (Spad - 1));
    R re = R(0), im = R(0);
    if (s < S && !(masked && isnan(masked[k]))) {  // vacant sites of the full layout stay zero
      const int64_t f = full_of ? full_of[k] : k;
      const uint32_t u = draw_u32(seed, (uint64_t)f, STREAM_PHASE, (uint32_t)(s0 + s));
      if constexpr (sizeof(R) == 4) {
        bool sure = true;
        const float2 v = unit_phase(u, sh, sl, &sure);
        re = v.x;
        im = v.y;
        if (!sure) {
          double sn, cs;
          sincospi((double)u * 0x1p-31, &sn, &cs);
          re = (R)(cs * inv_sqrt_n);
          im = (R)(sn * inv_sqrt_n);
        }
      } else {
        double sn, cs;
        sincospi((double)u * 0x1p-31, &sn, &cs);
        re = (R)(cs * inv_sqrt_n);
        im = (R)(sn * inv_sqrt_n);
      }
      if (draws) draws[(int64_t)s * n + k] = u;
    }
    if constexpr (sizeof(R) == 4) {
      reinterpret_cast<float2*>(out)[e] = make_float2(re, im);
    } else {
      reinterpret_cast<double2*>(out)[e] = make_double2(re, im);
    }
  }
}

template <typename R>
__global__ void k_init_sites(int64_t n, int Spad, int S, const int64_t* sites, const int64_t* full_of, R* out) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= S) return;
  const int64_t i = full_of ? full_of[sites[s]] : sites[s];
  out[2 * (i * Spad + s)] = R(1);
}

// D_i by full site index for the masked stencil, NaN at vacant sites.
__global__ void k_make_dfull(int64_t n_full, const int64_t* compact, const float* d32, float dconst, float* out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_full; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = compact[i];
    out[i] = c < 0 ? __int_as_float(0x7fc00000) : (d32 ? d32[c] : dconst);
  }
}

// State blocks of a full-layout pass back in the compact order of the active sites (16- or 8-byte units).
template <typename T>
__global__ void k_compact_states(int64_t n, int P, const int64_t* full_of, const T* in, T* out) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n * P; u += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = u / P;
    out[u] = in[full_of[k] * P + (u - k * P)];
  }
}

}  // namespace tbpm

using namespace tbpm;

// ====================================================================== C ABI
extern "C" {

const char* tbpm_last_error(void) { return g_err; }

int tbpm_create(tbpm_ctx** out, int device) {
  clear_error();
  if (!out) {
    set_error("tbpm_create: out is NULL");
    return TBPM_EINVAL;
  }
  *out = nullptr;
  int count = 0;
  TBPM_CK(cudaGetDeviceCount(&count));
  if (device < 0 || device >= count) {
    set_error("tbpm_create: device %d out of range (%d devices)", device, count);
    return TBPM_EINVAL;
  }
  TBPM_CK(cudaSetDevice(device));
  tbpm_ctx* ctx = new tbpm_ctx();
  ctx->device = device;
  cudaError_t e = cudaDeviceGetAttribute(&ctx->num_sms, cudaDevAttrMultiProcessorCount, device);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&ctx->stream, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaMallocHost((void**)&ctx->pinned, 4096);
  if (e == cudaSuccess) {
    // keep memory freed by stream-ordered frees in the pool instead of returning it to the
    // system at every synchronisation (re-mapping it made later allocations expensive)
    cudaMemPool_t pool;
    if (cudaDeviceGetDefaultMemPool(&pool, device) == cudaSuccess) {
      uint64_t keep = UINT64_MAX;
      cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    }
    cudaGetLastError();
  }
  if (e != cudaSuccess) {
    set_error("tbpm_create: %s", cudaGetErrorString(e));
    delete ctx;
    return TBPM_ECUDA;
  }
  ctx->pinned_cap = 4096;
  memset(ctx->pinned, 0, ctx->pinned_cap);
  *out = ctx;
  return TBPM_OK;
}

int tbpm_destroy(tbpm_ctx* ctx) {
  clear_error();
  if (!ctx) return TBPM_OK;
  cudaSetDevice(ctx->device);
  for (DevBuf* b : workspaces(ctx)) release(ctx, *b);
  cudaStreamSynchronize(ctx->stream);
  for (auto& g : ctx->graphs) cudaGraphExecDestroy(g.exec);
  ctx->graphs.clear();
  for (auto& ph : ctx->phases) {
    cudaEventDestroy(ph.a);
    cudaEventDestroy(ph.b);
  }
  for (cudaEvent_t e : ctx->event_pool) cudaEventDestroy(e);
  for (cudaEvent_t e : ctx->queue_ev)
    if (e) cudaEventDestroy(e);
  if (ctx->pinned) cudaFreeHost(ctx->pinned);
  cudaStreamDestroy(ctx->stream);
  delete ctx;
  return TBPM_OK;
}

void* tbpm_stream(tbpm_ctx* ctx) { return ctx ? (void*)ctx->stream : nullptr; }

int tbpm_sync(tbpm_ctx* ctx) {
  clear_error();
  if (!ctx) {
    set_error("tbpm_sync: ctx is NULL");
    return TBPM_EINVAL;
  }
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  return sweep_status(ctx);  // a fused sweep's bounded wait that expired since the last check
}

int64_t tbpm_launch_count(const tbpm_ctx* ctx) { return ctx ? ctx->launches : -1; }

int tbpm_set_fusion(tbpm_ctx* ctx, int enable) {
  clear_error();
  if (!ctx) {
    set_error("tbpm_set_fusion: ctx is NULL");
    return TBPM_EINVAL;
  }
  if (enable < -1 || enable > 10) {
    set_error("tbpm_set_fusion: mode %d unknown (-1..10)", enable);
    return TBPM_EINVAL;
  }
  ctx->fusion = enable;
  ctx->resident = false;  // a chosen mode names the passes
  return TBPM_OK;
}

int tbpm_set_resident(tbpm_ctx* ctx, int enable) {
  clear_error();
  if (!ctx) {
    set_error("tbpm_set_resident: ctx is NULL");
    return TBPM_EINVAL;
  }
  ctx->resident = enable != 0;
  return TBPM_OK;
}

int tbpm_set_block_buffering(tbpm_ctx* ctx, int enable) {
  clear_error();
  if (!ctx) {
    set_error("tbpm_set_block_buffering: ctx is NULL");
    return TBPM_EINVAL;
  }
  ctx->buffer_blocks = enable != 0;
  return TBPM_OK;
}

int tbpm_set_graphs(tbpm_ctx* ctx, int enable) {
  clear_error();
  if (!ctx) {
    set_error("tbpm_set_graphs: ctx is NULL");
    return TBPM_EINVAL;
  }
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  ctx->use_graphs = enable != 0;
  if (!ctx->use_graphs) {
    for (auto& g : ctx->graphs) cudaGraphExecDestroy(g.exec);
    ctx->graphs.clear();
    ctx->graph_seen.clear();
  }
  return TBPM_OK;
}

int tbpm_fusion_report(tbpm_ctx* ctx, double ms_per_step[16]) {
  clear_error();
  if (!ctx || !ms_per_step) {
    set_error("tbpm_fusion_report: invalid argument");
    return TBPM_EINVAL;
  }
  for (int m = 0; m < 16; ++m) ms_per_step[m] = -1.0;
  for (auto& t : ctx->fusion_timings)
    if (t.first >= 0 && t.first < 16) ms_per_step[t.first] = t.second;
  return TBPM_OK;
}

int tbpm_set_pass_states(tbpm_ctx* ctx, int max_states) {
  clear_error();
  if (!ctx || max_states < 0) {
    set_error("tbpm_set_pass_states: invalid argument");
    return TBPM_EINVAL;
  }
  ctx->max_pass_states = max_states;
  return TBPM_OK;
}

int tbpm_profile(tbpm_ctx* ctx, int enable) {
  clear_error();
  if (!ctx) {
    set_error("tbpm_profile: ctx is NULL");
    return TBPM_EINVAL;
  }
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  for (auto& ph : ctx->phases) {
    ctx->event_pool.push_back(ph.a);
    ctx->event_pool.push_back(ph.b);
  }
  ctx->phases.clear();
  ctx->profiling = enable != 0;
  return TBPM_OK;
}

int tbpm_profile_read(tbpm_ctx* ctx, double out[6]) {
  clear_error();
  if (!ctx || !out) {
    set_error("tbpm_profile_read: NULL argument");
    return TBPM_EINVAL;
  }
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  for (int k = 0; k < 6; ++k) out[k] = 0.0;
  for (auto& ph : ctx->phases) {
    float ms = 0.f;
    TBPM_CK(cudaEventElapsedTime(&ms, ph.a, ph.b));
    out[2 * ph.kind] += ms;
    out[2 * ph.kind + 1] += (double)ph.launches;
  }
  return TBPM_OK;
}

int64_t tbpm_truncation_order(double tau) { return truncation_order_host(tau); }

}  // extern "C"

// ------------------------------------------------------------------ lattice construction
// Taps of a long-range lattice: every (dx, dy, dz, ds) from a site of sublattice 0 with
// 0 < r <= cutoff, in (dz, dy, dx, ds) order, and its weight t(r)/t = exp(-(r - 1)/decay).
// r^2 is exact in FP64 for these integer and half-integer coordinates.
static int make_taps(const tbpm_lattice_desc& d, std::vector<int>& off, std::vector<double>& wrel) {
  const bool hc = d.kind == TBPM_HONEYCOMB, cu = d.kind == TBPM_CUBIC;
  const int R = (int)ceil(d.cutoff) + 2;
  const double c2 = d.cutoff * d.cutoff;
  off.clear();
  wrel.clear();
  for (int dz = cu ? -R : 0; dz <= (cu ? R : 0); ++dz)
    for (int dy = -R; dy <= R; ++dy)
      for (int dx = -R; dx <= R; ++dx)
        for (int ds = 0; ds <= (hc ? 1 : 0); ++ds) {
          double r2;
          if (hc) {
            const double u = 1.5 * (dx + dy) + ds, v = (double)(dx - dy);
            r2 = u * u + 0.75 * v * v;
          } else {
            r2 = (double)dx * dx + (double)dy * dy + (double)dz * dz;
          }
          if (r2 == 0.0 || r2 > c2) continue;
          off.insert(off.end(), {dx, dy, dz, ds});
          wrel.push_back(exp(-(sqrt(r2) - 1.0) / d.decay));
        }
  if (wrel.empty()) {
    set_error("cutoff %g keeps no neighbour (nearest-neighbour distance is 1)", d.cutoff);
    return TBPM_EINVAL;
  }
  if (wrel.size() > 1024) {
    set_error("cutoff %g gives %zu neighbours per site (at most 1024)", d.cutoff, wrel.size());
    return TBPM_EUNSUPPORTED;
  }
  return TBPM_OK;
}

static int build_lattice(tbpm_ctx* ctx, tbpm_lattice* lat) {
  const tbpm_lattice_desc& d = lat->desc;
  Geom& g = lat->geom;
  g.kind = d.kind;
  g.Lx = d.L[0];
  g.Ly = d.kind == TBPM_CUBIC || d.kind == TBPM_SQUARE || d.kind == TBPM_HONEYCOMB ? d.L[1] : 1;
  g.Lz = d.kind == TBPM_CUBIC ? d.L[2] : 1;
  g.pbc_x = d.pbc[0] != 0;
  g.pbc_y = d.pbc[1] != 0;
  g.pbc_z = d.pbc[2] != 0;
  g.z = d.kind == TBPM_SQUARE ? 4 : d.kind == TBPM_HONEYCOMB ? 3 : 6;
  g.row_sites = d.kind == TBPM_HONEYCOMB ? 2 * g.Lx : g.Lx;
  g.n_rows = g.Ly * g.Lz;
  g.n_full = g.row_sites * g.n_rows;
  const double abs_t = fabs(d.t);
  const bool vac = d.vacancy_frac > 0.0;
  const bool lr = d.cutoff > 0.0;
  lat->path = (d.path == TBPM_PATH_AUTO) ? (vac || lr ? TBPM_PATH_CSR : TBPM_PATH_STENCIL) : d.path;
  if (vac && lat->path == TBPM_PATH_STENCIL) {
    set_error("vacancies need the CSR path");
    return TBPM_EINVAL;
  }
  if (lr && lat->path == TBPM_PATH_STENCIL) {
    set_error("long-range hopping runs on the CSR path");
    return TBPM_EINVAL;
  }
  std::vector<double> wrel;
  int4* d_taps = nullptr;
  double* d_tabs = nullptr;
  struct Release {  // frees the tap tables on every return path
    cudaStream_t st;
    int4** a;
    double** b;
    ~Release() {
      if (*a) cudaFreeAsync(*a, st);
      if (*b) cudaFreeAsync(*b, st);
    }
  } release{ctx->stream, &d_taps, &d_tabs};
  if (lr) {
    TBPM_TRY(make_taps(d, lat->tap_off, wrel));
    g.z = (int)wrel.size();
    lat->tap_t.resize(wrel.size());
    std::vector<double> tabs(wrel.size());
    std::vector<float> w32(wrel.size());
    for (size_t k = 0; k < wrel.size(); ++k) {
      lat->tap_t[k] = d.t * wrel[k];
      tabs[k] = abs_t * wrel[k];
      w32[k] = (float)wrel[k];
    }
    const size_t z = wrel.size();
    // current-operator weights t_k (r_j - r_i)_a per direction and sublattice; a honeycomb B site
    // takes every tap mirrored, so its bond vectors are the negatives
    std::vector<double> jw(6 * z);
    const double h = sqrt(3.0) / 2.0;
    for (size_t k = 0; k < z; ++k) {
      const int* o = &lat->tap_off[4 * k];
      double dv[3];
      if (d.kind == TBPM_HONEYCOMB) {
        dv[0] = 1.5 * (o[0] + o[1]) + o[3];
        dv[1] = h * (o[0] - o[1]);
        dv[2] = 0.0;
      } else {
        dv[0] = o[0];
        dv[1] = o[1];
        dv[2] = o[2];
      }
      for (int a = 0; a < 3; ++a) {
        jw[(a * 2 + 0) * z + k] = lat->tap_t[k] * dv[a];
        jw[(a * 2 + 1) * z + k] = (d.kind == TBPM_HONEYCOMB ? -1.0 : 1.0) * lat->tap_t[k] * dv[a];
      }
    }
    TBPM_TRY(dev_alloc(ctx, &lat->jw, 6 * z));
    TBPM_CK(cudaMemcpyAsync(lat->jw, jw.data(), 6 * z * sizeof(double), cudaMemcpyHostToDevice, ctx->stream));
    TBPM_TRY(dev_alloc(ctx, &lat->wrel64, z));
    TBPM_TRY(dev_alloc(ctx, &lat->wrel32, z));
    TBPM_TRY(dev_alloc(ctx, &d_taps, z));
    TBPM_TRY(dev_alloc(ctx, &d_tabs, z));
    TBPM_CK(cudaMemcpyAsync(lat->wrel64, wrel.data(), z * sizeof(double), cudaMemcpyHostToDevice, ctx->stream));
    TBPM_CK(cudaMemcpyAsync(lat->wrel32, w32.data(), z * sizeof(float), cudaMemcpyHostToDevice, ctx->stream));
    TBPM_CK(cudaMemcpyAsync(d_taps, lat->tap_off.data(), z * sizeof(int4), cudaMemcpyHostToDevice, ctx->stream));
    TBPM_CK(cudaMemcpyAsync(d_tabs, tabs.data(), z * sizeof(double), cudaMemcpyHostToDevice, ctx->stream));
    // the pageable sources above must outlive the copies
    TBPM_CK(cudaStreamSynchronize(ctx->stream));
  }
  lat->has_v = d.W != 0.0;
  const uint64_t thr = vac ? (uint64_t)floor(d.vacancy_frac * 4294967296.0) : 0;

  TBPM_TRY(ensure(ctx, ctx->ws_aux, sizeof(Bounds3) * (size_t)ctx->num_sms * 16 + 64));
  Bounds3* part = (Bounds3*)ctx->ws_aux.p;
  int nb = 0;
  if (lat->path == TBPM_PATH_STENCIL) {
    lat->n_sites = g.n_full;
    if (lat->has_v) TBPM_TRY(dev_alloc(ctx, &lat->v64, lat->n_sites));
    nb = grid_for(ctx, g.n_full, kT);
    k_lattice_stencil<<<nb, kT, 0, ctx->stream>>>(g, d.seed, d.W, abs_t, lat->v64, part);
    TBPM_CK_LAUNCH(ctx);
  } else {
    const int64_t nchunks = (g.n_full + kChunk - 1) / kChunk;
    int64_t *counts = nullptr, *offs = nullptr;
    TBPM_TRY(dev_alloc(ctx, &counts, nchunks));
    TBPM_TRY(dev_alloc(ctx, &offs, nchunks + 1));
    k_count_active<<<(unsigned)nchunks, kT, 0, ctx->stream>>>(g.n_full, d.seed, thr, counts);
    TBPM_CK_LAUNCH(ctx);
    k_scan_counts<<<1, 1024, 0, ctx->stream>>>(counts, nchunks, offs);
    TBPM_CK_LAUNCH(ctx);
    int64_t n_active = 0;
    TBPM_CK(cudaMemcpyAsync(&n_active, offs + nchunks, sizeof(int64_t), cudaMemcpyDeviceToHost, ctx->stream));
    TBPM_CK(cudaStreamSynchronize(ctx->stream));
    if (n_active <= 0) {
      cudaFreeAsync(counts, ctx->stream);
      cudaFreeAsync(offs, ctx->stream);
      set_error("lattice has no active sites");
      return TBPM_EINVAL;
    }
    if (n_active >= (int64_t)INT32_MAX) {
      set_error("CSR path supports fewer than 2^31 active sites");
      return TBPM_EUNSUPPORTED;
    }
    lat->n_sites = n_active;
    TBPM_TRY(dev_alloc(ctx, &lat->compact, g.n_full));
    TBPM_TRY(dev_alloc(ctx, &lat->full_of, n_active));
    // clean long-range lattices that the tap kernel serves build their ELL lists only when a
    // pass needs them (complex128, one state, exports): at D_H ~ 230 they outweigh the states
    const bool lazy_ell = lr && d.path == TBPM_PATH_AUTO && !vac && d.kind != TBPM_CUBIC;
    if (!lazy_ell) TBPM_TRY(dev_alloc(ctx, &lat->ell, (size_t)n_active * g.z));
    if (lat->has_v) TBPM_TRY(dev_alloc(ctx, &lat->v64, n_active));
    k_compact<<<(unsigned)nchunks, kT, 0, ctx->stream>>>(g.n_full, d.seed, thr, offs, lat->compact, lat->full_of);
    TBPM_CK_LAUNCH(ctx);
    cudaFreeAsync(counts, ctx->stream);
    cudaFreeAsync(offs, ctx->stream);
    nb = grid_for(ctx, n_active, kT);
    if (lr) {
      k_build_ell_taps<<<nb, kT, 0, ctx->stream>>>(g, n_active, lat->full_of, lat->compact, d_taps, d_tabs, d.seed,
                                                    d.W, lat->ell, lat->v64, part);
      TBPM_CK_LAUNCH(ctx);
    } else {
      k_build_ell<<<nb, kT, 0, ctx->stream>>>(g, n_active, lat->full_of, lat->compact, d.seed, d.W, abs_t,
                                               lat->ell, lat->v64, part);
      TBPM_CK_LAUNCH(ctx);
    }
  }
  if (lr && d.path == TBPM_PATH_AUTO) TBPM_TRY(build_tap_table(lat));
  double* res = (double*)((char*)ctx->ws_aux.p + sizeof(Bounds3) * (size_t)ctx->num_sms * 16);
  k_bounds_final<<<1, kT, 0, ctx->stream>>>(part, nb, res);
  TBPM_CK_LAUNCH(ctx);
  TBPM_CK(cudaMemcpyAsync(ctx->pinned, res, 3 * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  lat->E_max = ctx->pinned[0];
  lat->E_min = ctx->pinned[1];
  lat->n_bonds = (int64_t)ctx->pinned[2];
  if (!(lat->E_max > lat->E_min)) {
    set_error("degenerate spectrum (no hopping between active sites)");
    return TBPM_EINVAL;
  }
  lat->H0 = (lat->E_max + lat->E_min) / 2.0;
  lat->half = (1.0 + 0.01) * (lat->E_max - lat->E_min) / 2.0;
  if (lat->has_v) {
    TBPM_TRY(dev_alloc(ctx, &lat->d32, lat->n_sites));
    k_make_diag<<<grid_for(ctx, lat->n_sites, kT), kT, 0, ctx->stream>>>(lat->n_sites, lat->v64, lat->H0,
                                                                        lat->half, nullptr, lat->d32);
    TBPM_CK_LAUNCH(ctx);
  }
  return TBPM_OK;
}

// ELL lists of a long-range lattice built on first need (see build_lattice).
int tbpm::ensure_ell(tbpm_ctx* ctx, tbpm_lattice* lat) {
  if (lat->ell || lat->tap_t.empty()) return TBPM_OK;
  const Geom& g = lat->geom;
  const size_t z = lat->tap_t.size();
  std::vector<double> tabs(z);
  for (size_t k = 0; k < z; ++k) tabs[k] = fabs(lat->tap_t[k]);
  const int nb = grid_for(ctx, lat->n_sites, kT);
  int4* d_taps = nullptr;
  double* d_tabs = nullptr;
  Bounds3* part = nullptr;
  int r = dev_alloc(ctx, &lat->ell, (size_t)lat->n_sites * g.z);
  if (r == TBPM_OK) r = dev_alloc(ctx, &d_taps, z);
  if (r == TBPM_OK) r = dev_alloc(ctx, &d_tabs, z);
  if (r == TBPM_OK) r = dev_alloc(ctx, &part, (size_t)nb);
  if (r == TBPM_OK) {
    cudaMemcpyAsync(d_taps, lat->tap_off.data(), z * sizeof(int4), cudaMemcpyHostToDevice, ctx->stream);
    cudaMemcpyAsync(d_tabs, tabs.data(), z * sizeof(double), cudaMemcpyHostToDevice, ctx->stream);
    k_build_ell_taps<<<nb, kT, 0, ctx->stream>>>(g, lat->n_sites, lat->full_of, lat->compact, d_taps, d_tabs,
                                                  lat->desc.seed, lat->desc.W, lat->ell, nullptr, part);
    ctx->launches++;
    const cudaError_t e = cudaGetLastError();
    const cudaError_t es = cudaStreamSynchronize(ctx->stream);  // the host tables must outlive the copies
    if (e != cudaSuccess || es != cudaSuccess) {
      set_error("ELL build: %s", cudaGetErrorString(e != cudaSuccess ? e : es));
      r = TBPM_ECUDA;
    }
  }
  for (void* q : {(void*)d_taps, (void*)d_tabs, (void*)part})
    if (q) cudaFreeAsync(q, ctx->stream);
  if (r != TBPM_OK && lat->ell) {
    cudaFreeAsync(lat->ell, ctx->stream);
    lat->ell = nullptr;
  }
  return r;
}

static int ensure_d64(tbpm_lattice* lat) {
  if (!lat->has_v || lat->d64) return TBPM_OK;
  tbpm_ctx* ctx = lat->ctx;
  TBPM_TRY(dev_alloc(ctx, &lat->d64, lat->n_sites));
  k_make_diag<<<grid_for(ctx, lat->n_sites, kT), kT, 0, ctx->stream>>>(lat->n_sites, lat->v64, lat->H0, lat->half,
                                                                      lat->d64, nullptr);
  TBPM_CK_LAUNCH(ctx);
  return TBPM_OK;
}

static int ensure_dfull(tbpm_lattice* lat) {
  if (lat->dfull) return TBPM_OK;
  tbpm_ctx* ctx = lat->ctx;
  TBPM_TRY(dev_alloc(ctx, &lat->dfull, lat->geom.n_full));
  k_make_dfull<<<grid_for(ctx, lat->geom.n_full, kT), kT, 0, ctx->stream>>>(
      lat->geom.n_full, lat->compact, lat->d32, (float)((0.0 - lat->H0) / lat->half), lat->dfull);
  TBPM_CK_LAUNCH(ctx);
  return TBPM_OK;
}

static void free_lattice_mem(tbpm_lattice* lat) {
  tbpm_ctx* ctx = lat->ctx;
  void* ps[] = {lat->d32, lat->d64, lat->v64, lat->ell, lat->compact, lat->full_of, lat->wrel32, lat->wrel64,
                lat->jw, lat->dfull};
  for (void* p : ps)
    if (p) cudaFreeAsync(p, ctx->stream);
}

extern "C" {

int tbpm_lattice_create(tbpm_ctx* ctx, const tbpm_lattice_desc* desc, tbpm_lattice** out) {
  clear_error();
  TBPM_NVTX_CALL(ctx);
  if (!ctx || !desc || !out) {
    set_error("tbpm_lattice_create: NULL argument");
    return TBPM_EINVAL;
  }
  *out = nullptr;
  const tbpm_lattice_desc& d = *desc;
  if (d.kind < TBPM_SQUARE || d.kind > TBPM_CUBIC) {
    set_error("unknown lattice kind %d", d.kind);
    return TBPM_EINVAL;
  }
  const int dims = d.kind == TBPM_CUBIC ? 3 : 2;
  for (int k = 0; k < dims; ++k)
    if (d.L[k] < 1 || d.L[k] > (1LL << 31)) {
      set_error("lattice size L[%d] = %lld out of range", k, (long long)d.L[k]);
      return TBPM_EINVAL;
    }
  if (!(d.t == d.t) || d.t == 0.0 || !isfinite(d.t) || !isfinite(d.W) || d.W < 0.0) {
    set_error("hopping t must be finite and non-zero, W finite and >= 0");
    return TBPM_EINVAL;
  }
  if (!(d.vacancy_frac >= 0.0 && d.vacancy_frac < 1.0)) {
    set_error("vacancy_frac must lie in [0, 1)");
    return TBPM_EINVAL;
  }
  if (!(d.cutoff >= 0.0 && d.cutoff <= 12.0) || (d.cutoff > 0.0 && !(d.decay > 0.0 && isfinite(d.decay)))) {
    set_error("cutoff must lie in [0, 12], and decay be finite and > 0 when cutoff > 0");
    return TBPM_EINVAL;
  }
  if (d.path < TBPM_PATH_AUTO || d.path > TBPM_PATH_CSR) {
    set_error("unknown path %d", d.path);
    return TBPM_EINVAL;
  }
  if (d.kind == TBPM_CUBIC && (double)d.L[1] * (double)d.L[2] >= 2147483648.0) {
    set_error("cubic lattice: Ly*Lz must be below 2^31");
    return TBPM_EINVAL;
  }
  double nf = (double)d.L[0] * (double)d.L[1] * (d.kind == TBPM_CUBIC ? (double)d.L[2] : 1.0) *
              (d.kind == TBPM_HONEYCOMB ? 2.0 : 1.0);
  if (nf > 4.0e9) {
    set_error("lattice too large (%.3g sites)", nf);
    return TBPM_EINVAL;
  }
  TBPM_CK(cudaSetDevice(ctx->device));
  tbpm_lattice* lat = new tbpm_lattice();
  lat->ctx = ctx;
  lat->desc = d;
  if (d.kind != TBPM_CUBIC) lat->desc.L[2] = 1;
  int r = build_lattice(ctx, lat);
  if (r != TBPM_OK) {
    free_lattice_mem(lat);
    delete lat;
    return r;
  }
  *out = lat;
  return TBPM_OK;
}

int tbpm_lattice_destroy(tbpm_lattice* lat) {
  clear_error();
  if (!lat) return TBPM_OK;
  tbpm_ctx* ctx = lat->ctx;
  cudaSetDevice(ctx->device);
  free_lattice_mem(lat);
  cudaStreamSynchronize(lat->ctx->stream);
  delete lat;
  return TBPM_OK;
}

int tbpm_lattice_info(const tbpm_lattice* lat, tbpm_lattice_props* out) {
  clear_error();
  if (!lat || !out) {
    set_error("tbpm_lattice_info: NULL argument");
    return TBPM_EINVAL;
  }
  out->n_full = lat->geom.n_full;
  out->n_sites = lat->n_sites;
  out->n_bonds = lat->n_bonds;
  out->path = lat->path;
  out->coordination = lat->geom.z;
  out->E_min = lat->E_min;
  out->E_max = lat->E_max;
  out->H0 = lat->H0;
  out->half_width = lat->half;
  return TBPM_OK;
}

int tbpm_lattice_export(const tbpm_lattice* lat, int64_t* compact, double* V, int32_t* nbr) {
  clear_error();
  if (!lat) {
    set_error("tbpm_lattice_export: NULL lattice");
    return TBPM_EINVAL;
  }
  tbpm_ctx* ctx = lat->ctx;
  TBPM_CK(cudaSetDevice(ctx->device));
  const int64_t n = lat->n_sites, nf = lat->geom.n_full;
  const int z = lat->geom.z;
  if (compact) {
    if (lat->compact) {
      TBPM_CK(cudaMemcpyAsync(compact, lat->compact, nf * sizeof(int64_t), cudaMemcpyDeviceToHost, ctx->stream));
    } else {
      for (int64_t i = 0; i < nf; ++i) compact[i] = i;
    }
  }
  if (V) {
    if (lat->v64) {
      TBPM_CK(cudaMemcpyAsync(V, lat->v64, n * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    } else {
      for (int64_t i = 0; i < n; ++i) V[i] = 0.0;
    }
  }
  if (nbr) {
    TBPM_TRY(ensure_ell(ctx, const_cast<tbpm_lattice*>(lat)));
    if (lat->ell) {
      TBPM_CK(cudaMemcpyAsync(nbr, lat->ell, n * z * sizeof(int32_t), cudaMemcpyDeviceToHost, ctx->stream));
    } else {
      for (int64_t i = 0; i < n; ++i)
        for (int d = 0; d < z; ++d) nbr[i * z + d] = (int32_t)neighbour_full(lat->geom, i, d);
    }
  }
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  return TBPM_OK;
}

int tbpm_debug_status(tbpm_ctx* ctx, uint64_t words[3]) {
  clear_error();
  if (!ctx || !words) {
    set_error("tbpm_debug_status: NULL argument");
    return TBPM_EINVAL;
  }
#ifdef TBPM_DEBUG
  TBPM_CK(cudaSetDevice(ctx->device));
  TBPM_CK(cudaDeviceSynchronize());
  words[0] = 0;
  for (const unsigned long long w : {debug_take_cheb(), debug_take_resident(), debug_take_march(), debug_take_flush(),
                                     debug_take_taps()})  // every unit's word is cleared, the first one reported
    if (words[0] == 0) words[0] = w;
  words[1] = debug_take_sweep();
  words[2] = debug_take_serve();
  return TBPM_OK;
#else
  words[0] = words[1] = words[2] = 0;
  set_error("tbpm_debug_status: this library was built without TBPM_DEBUG (use libtbpm_debug.so)");
  return TBPM_EUNSUPPORTED;
#endif
}

int tbpm_lattice_taps(const tbpm_lattice* lat, int32_t* offsets, double* t) {
  clear_error();
  if (!lat) {
    set_error("tbpm_lattice_taps: NULL lattice");
    return TBPM_EINVAL;
  }
  const int z = lat->geom.z;
  if (!lat->tap_t.empty()) {
    if (offsets)
      for (int k = 0; k < 4 * z; ++k) offsets[k] = lat->tap_off[k];
    if (t)
      for (int k = 0; k < z; ++k) t[k] = lat->tap_t[k];
    return TBPM_OK;
  }
  // nearest-neighbour lattices: the fixed neighbour order of a sublattice-0 site
  static const int sq[4][4] = {{1, 0, 0, 0}, {-1, 0, 0, 0}, {0, 1, 0, 0}, {0, -1, 0, 0}};
  static const int hc[3][4] = {{0, 0, 0, 1}, {-1, 0, 0, 1}, {0, -1, 0, 1}};
  static const int cu[6][4] = {{1, 0, 0, 0}, {-1, 0, 0, 0}, {0, 1, 0, 0}, {0, -1, 0, 0}, {0, 0, 1, 0}, {0, 0, -1, 0}};
  const int(*tab)[4] = lat->geom.kind == TBPM_SQUARE ? sq : lat->geom.kind == TBPM_HONEYCOMB ? hc : cu;
  for (int d = 0; d < z; ++d) {
    if (offsets)
      for (int c = 0; c < 4; ++c) offsets[4 * d + c] = tab[d][c];
    if (t) t[d] = lat->desc.t;
  }
  return TBPM_OK;
}

}  // extern "C"

// ------------------------------------------------------------------ request plumbing
namespace {

struct Plan {
  int precision;
  int S, Spad, logS, spt, P, logP;
  size_t elem;        // bytes per complex element
  size_t state_bytes; // one block of Spad states
  double tau;
  int s0;             // index of the block's first state among the request's states (Philox sub-stream)
  int64_t n;          // sites of a state block: the active sites, or all of them in the full layout
  bool full;          // vacancy lattice on the masked stencil: blocks by full site index, vacant sites zero
};

void set_layout(const tbpm_lattice* lat, Plan* pl, bool full) {
  pl->full = full;
  pl->n = full ? lat->geom.n_full : lat->n_sites;
  pl->state_bytes = (size_t)pl->n * pl->Spad * pl->elem;
}

// Whether a nearest-neighbour vacancy lattice takes the masked register sweep: automatic path, a shape
// the sweep takes, and at most half the sites vacant.  In the full layout a step costs 8 B per
// (site + vacancy) and 4 / S B of D_i where the index lists cost 24 + (4 z + 4) / S B per site, so the
// sweep would win beyond half as well; the rule keeps the extra state memory below the lists' own scale.
bool masked_sweep_ok(const tbpm_lattice* lat, const Plan& pl) {
  return lat->path == TBPM_PATH_CSR && lat->desc.path == TBPM_PATH_AUTO && lat->desc.vacancy_frac > 0.0 &&
         2 * lat->n_sites >= lat->geom.n_full && sweep_shape_ok(lat, pl.precision, pl.Spad);
}

// The register sweep carries this plan's recurrence.
bool sweep_ok(const tbpm_lattice* lat, const Plan& pl) {
  return (lat->path == TBPM_PATH_STENCIL || pl.full) && sweep_shape_ok(lat, pl.precision, pl.Spad);
}

int ilog2(int v) {
  int r = 0;
  while ((1 << r) < v) ++r;
  return r;
}

int make_plan(const tbpm_lattice* lat, const tbpm_request* req, Plan* pl) {
  if (!lat || !req) {
    set_error("NULL lattice or request");
    return TBPM_EINVAL;
  }
  if (req->precision != TBPM_C64 && req->precision != TBPM_C128) {
    set_error("unknown precision %d", req->precision);
    return TBPM_EINVAL;
  }
  if (req->n_states < 1 || req->n_states > 32) {
    set_error("n_states must lie in [1, 32] (got %d)", req->n_states);
    return TBPM_EINVAL;
  }
  if (req->states == TBPM_STATES_SITES) {
    if (!req->sites) {
      set_error("site states need a site list");
      return TBPM_EINVAL;
    }
    for (int s = 0; s < req->n_states; ++s)
      if (req->sites[s] < 0 || req->sites[s] >= lat->n_sites) {
        set_error("site %lld out of range", (long long)req->sites[s]);
        return TBPM_EINVAL;
      }
  } else if (req->states != TBPM_STATES_RANDOM) {
    set_error("unknown state kind %d", req->states);
    return TBPM_EINVAL;
  }
  pl->precision = req->precision;
  pl->S = req->n_states;
  pl->logS = ilog2(pl->S);
  pl->Spad = 1 << pl->logS;
  pl->spt = (req->precision == TBPM_C64 && pl->Spad >= 2) ? 2 : 1;
  pl->P = pl->Spad / pl->spt;
  pl->logP = ilog2(pl->P);
  pl->elem = req->precision == TBPM_C64 ? 8 : 16;
  set_layout(lat, pl, false);
  pl->tau = req->tau == 0.0 ? M_PI : req->tau;
  pl->s0 = 0;
  if (!(pl->tau > 0.0) || !isfinite(pl->tau)) {
    set_error("tau must be positive");
    return TBPM_EINVAL;
  }
  return TBPM_OK;
}

int init_states(tbpm_ctx* ctx, const tbpm_lattice* lat, const tbpm_request* req, const Plan& pl, void* dst,
                uint32_t* draws) {
  const int64_t n = pl.n;
  const int64_t* full_of = pl.full ? nullptr : lat->full_of;
  const float* masked = pl.full ? lat->dfull : nullptr;
  if (req->states == TBPM_STATES_RANDOM) {
    const double inv = 1.0 / sqrt((double)lat->n_sites);
    const int nb = grid_for(ctx, n * pl.Spad, kT, 32);
    if (pl.precision == TBPM_C64)
      k_init_random<float><<<nb, kT, 0, ctx->stream>>>(n, pl.Spad, pl.logS, pl.S, pl.s0, req->state_seed, full_of,
                                                       masked, inv, (float*)dst, draws);
    else
      k_init_random<double><<<nb, kT, 0, ctx->stream>>>(n, pl.Spad, pl.logS, pl.S, pl.s0, req->state_seed, full_of,
                                                        masked, inv, (double*)dst, draws);
    TBPM_CK_LAUNCH(ctx);
  } else {
    TBPM_CK(cudaMemsetAsync(dst, 0, pl.state_bytes, ctx->stream));
    TBPM_TRY(ensure(ctx, ctx->ws_aux, sizeof(int64_t) * 32));
    TBPM_CK(cudaMemcpyAsync(ctx->ws_aux.p, req->sites, sizeof(int64_t) * pl.S, cudaMemcpyHostToDevice, ctx->stream));
    if (pl.precision == TBPM_C64)
      k_init_sites<float><<<1, 32, 0, ctx->stream>>>(n, pl.Spad, pl.S, (const int64_t*)ctx->ws_aux.p,
                                                     pl.full ? lat->full_of : nullptr, (float*)dst);
    else
      k_init_sites<double><<<1, 32, 0, ctx->stream>>>(n, pl.Spad, pl.S, (const int64_t*)ctx->ws_aux.p, nullptr,
                                                      (double*)dst);
    TBPM_CK_LAUNCH(ctx);
  }
  return TBPM_OK;
}

int64_t tiles_of(const tbpm_lattice* lat, const Plan& pl) {
  if (lat->path == TBPM_PATH_CSR && !pl.full) return (lat->n_sites * pl.P + 255) / 256;
  return lat->geom.n_rows * ((lat->geom.row_sites * pl.P + 255) / 256);
}

int base_args(tbpm_ctx* ctx, tbpm_lattice* lat, const Plan& pl, RecurrenceArgs* a, int comps) {
  memset(a, 0, sizeof(*a));
  a->geom = lat->geom;
  a->path = pl.full ? TBPM_PATH_STENCIL : lat->path;
  a->wrel = lat->wrel64 ? (pl.precision == TBPM_C128 ? (const void*)lat->wrel64 : (const void*)lat->wrel32) : nullptr;
  if (lat->taps && pl.precision == TBPM_C64 && pl.Spad >= 2) {
    a->taps = lat->taps.get();
  }
  if (!a->taps) TBPM_TRY(ensure_ell(ctx, lat));
  a->ell = lat->ell;
  if (pl.full) {
    TBPM_TRY(ensure_dfull(lat));
    a->diag = lat->dfull;
    a->masked = 1;
  } else if (lat->has_v) {
    if (pl.precision == TBPM_C128) TBPM_TRY(ensure_d64(lat));
    a->diag = pl.precision == TBPM_C128 ? (const void*)lat->d64 : (const void*)lat->d32;
  } else {
    a->diag = nullptr;
  }
  a->diag_const = (0.0 - lat->H0) / lat->half;
  a->thop = lat->desc.t / lat->half;
  set_float_coefficients(a);
  a->n_sites = pl.n;
  a->S = pl.Spad;
  a->P = pl.P;
  a->logP = pl.logP;
  a->n_tiles = tiles_of(lat, pl);
  a->nblocks = recurrence_blocks(ctx, pl.precision, pl.Spad);
  TBPM_TRY(ensure(ctx, ctx->ws_partials, sizeof(double) * (size_t)a->nblocks * pl.Spad * comps));
  a->partials = (double*)ctx->ws_partials.p;
  if (!ctx->ws_counter.p) {
    TBPM_TRY(ensure(ctx, ctx->ws_counter, 256));
    TBPM_CK(cudaMemsetAsync(ctx->ws_counter.p, 0, ctx->ws_counter.cap, ctx->stream));
  }
  a->counter = (unsigned*)ctx->ws_counter.p;
  if (a->taps) {
    TBPM_TRY(ensure(ctx, ctx->ws_fused_partials, taps_partials_bytes(*a)));
    a->tap_partials = (double*)ctx->ws_fused_partials.p;
  }
  return TBPM_OK;
}

// Fusion mode for a moment request: ctx->fusion, or under -1 the fastest mode measured on this
// lattice shape (a few passes of each applicable mode on scratch buffers; cached per shape).
int choose_fusion(tbpm_ctx* ctx, tbpm_lattice* lat, const tbpm_request* req, const Plan& pl, int64_t M, int* mode) {
  if (ctx->fusion >= 0) {
    *mode = ctx->fusion;
    return TBPM_OK;
  }
  *mode = 0;
  if (!fused_applicable(lat, pl.precision, pl.Spad)) {  // square, vacancy and one-state sweeps: no other fused pass
    *mode = 8;
    return TBPM_OK;
  }
  if (M / 2 < 64) return TBPM_OK;
  const Geom& g = lat->geom;
  const std::vector<int64_t> key = {g.kind, g.Lx, g.Ly, g.Lz, g.pbc_x | (g.pbc_y << 1) | (g.pbc_z << 2), lat->path,
                                    pl.Spad, pl.precision, lat->has_v ? 1 : 0};
  for (auto& kv : ctx->fusion_choice)
    if (kv.first == key) {
      *mode = kv.second;
      return TBPM_OK;
    }
  TBPM_TRY(ensure(ctx, ctx->ws_phi[0], pl.state_bytes));
  TBPM_TRY(ensure(ctx, ctx->ws_phi[1], pl.state_bytes));
  TBPM_TRY(ensure(ctx, ctx->ws_phi2[0], pl.state_bytes));
  TBPM_TRY(ensure(ctx, ctx->ws_phi2[1], pl.state_bytes));
  const int Ms = 64;  // scratch moments: steps 1 .. 31
  TBPM_TRY(ensure(ctx, ctx->ws_aux, sizeof(double) * 2 * (size_t)Ms * pl.Spad));
  TBPM_CK(cudaMemsetAsync(ctx->ws_aux.p, 0, sizeof(double) * 2 * (size_t)Ms * pl.Spad, ctx->stream));
  TBPM_TRY(init_states(ctx, lat, req, pl, ctx->ws_phi[0].p, nullptr));
  TBPM_TRY(init_states(ctx, lat, req, pl, ctx->ws_phi[1].p, nullptr));
  RecurrenceArgs a;
  TBPM_TRY(base_args(ctx, lat, pl, &a, 3));
  a.mu = (double*)ctx->ws_aux.p;
  a.M = Ms;
  cudaEvent_t e0, e1;
  TBPM_CK(cudaEventCreate(&e0));
  TBPM_CK(cudaEventCreate(&e1));
  const int modes[] = {0, 4, 5, 8};
  double best_ms = 1e300;
  ctx->fusion_timings.clear();
  // 24 steps per mode after 8 warm-up steps (multiples of every mode's steps per pass)
  int r = TBPM_OK;
  for (int m : modes) {
    const int K = m == 0 ? 1 : fused_steps(m);
    const int passes = 24 / K;  // 24 steps per measurement, after 8 warm-up steps
    float ms = 0.f;
    for (int rep = 0; rep < 2 && r == TBPM_OK; ++rep) {
      const int np = rep == 0 ? 8 / K : passes;
      if (rep == 1) cudaEventRecord(e0, ctx->stream);
      for (int i = 0; i < np && r == TBPM_OK; ++i) {
        if (m == 0) {
          a.cur = ctx->ws_phi[0].p;
          a.prev_out = ctx->ws_phi[1].p;
          a.step = 1 + (i % 16);
          r = launch_moment_step(ctx, a, pl.precision, false);
        } else {
          r = launch_fused_pass(ctx, lat, a, ctx->ws_phi[0].p, ctx->ws_phi[1].p, ctx->ws_phi2[0].p, ctx->ws_phi2[1].p,
                                1 + (i % 8) * K, m);
        }
      }
      if (rep == 1) cudaEventRecord(e1, ctx->stream);
    }
    if (r != TBPM_OK) break;
    if (cudaEventSynchronize(e1) == cudaSuccess) cudaEventElapsedTime(&ms, e0, e1);
    const double per_step = ms / 24.0;
    ctx->fusion_timings.push_back({m, per_step});
    if (per_step < best_ms) {
      best_ms = per_step;
      *mode = m;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  TBPM_TRY(r);
  ctx->fusion_choice.push_back({key, *mode});
  return TBPM_OK;
}

// Bounded launch queue (ctx->max_queue > 0, never while a graph is being captured): every 64
// launches record an event and wait for the one recorded 64 launches before.
void throttle_queue(tbpm_ctx* ctx, bool capturing) {
  if (ctx->max_queue <= 0 || capturing) return;
  if (++ctx->queue_count % 64 != 0) return;
  const int k = (int)((ctx->queue_count / 64) & 1);
  if (!ctx->queue_ev[k]) cudaEventCreateWithFlags(&ctx->queue_ev[k], cudaEventDisableTiming);
  if (ctx->queue_live[k]) cudaEventSynchronize(ctx->queue_ev[k]);
  cudaEventRecord(ctx->queue_ev[k], ctx->stream);
  ctx->queue_live[k] = true;
}

// Whether the resident kernel runs this moment request: a small lattice, unless a fusion mode has been chosen since
// (tbpm_set_resident).  Where the register sweep takes the lattice as well, the resident kernel is faster alone,
// but its grid must be resident as a whole: requests of several contexts overlap only as far as several grids fit,
// while sweeps and one-step passes fill each other's gaps. Requests of 512 moments a second from one and from eight
// contexts, one-step or sweep before -> resident: honeycomb pairs 64 x 64 x 8 states 506 / 3591 -> 1292 / 3962, 100
// x 100 x 4 693 / 4737 -> 1379 / 3225, 250 x 250 x 8 247 / 849 -> 493 / 503 (sweep now 302 / 998).  So honeycomb
// pairs, which had the sweep, go resident up to 70,000 site-states, where no number of contexts is slower; other
// kinds gained at both ends (300 x 300 square, 8 states 156 / 361 -> 566 / 812) but for complex128 honeycombs,
// whose FP64 time does not overlap: 160 x 160 x 4 states 160 / 340 -> 216 / 260, so four states and more stop at
// 90,000 (below it, two states on 110 x 110 cells 438 / 1294 -> 951 / 1043; four contexts 960 -> 1036).  Cubic
// lattices near the kernel's limit gain little alone and lose from eight contexts (60^3, 8 states: one step per
// launch before 259 / 476, resident 377 / 399, march 322 / 767), so they stop at 1.5M. Blocks of one or two states
// leave the shared-memory reads half empty and stop where the sweep is as fast alone (us per step, resident /
// sweep: two states 819k site-states 5.5 / 6.1, 1.44M 7.5 / 7.0; one state 262k 4.5 / 4.3, 33k 2.1 / 2.9).
bool use_resident(tbpm_ctx* ctx, const tbpm_lattice* lat, const Plan& pl, int64_t steps) {
  if (ctx->lean || !ctx->resident) return false;
  if (fused_applicable(lat, pl.precision, pl.Spad) && pl.n * pl.Spad > 70000) return false;
  if (lat->geom.kind == TBPM_CUBIC && pl.n * pl.Spad > 1500000) return false;
  if (pl.precision == TBPM_C128 && lat->geom.kind == TBPM_HONEYCOMB && pl.Spad >= 4 && pl.n * pl.Spad > 90000) return false;
  if (pl.Spad <= 2 && pl.n * pl.Spad > (pl.Spad == 1 ? 200000 : 1000000) && sweep_ok(lat, pl)) return false;
  return resident_applicable(ctx, lat, pl.precision, pl.Spad, steps);
}

// Moments of all Spad states into d_mu [Spad][M][2].
int run_moments(tbpm_ctx* ctx, tbpm_lattice* lat, const tbpm_request* req, const Plan& pl_in, int64_t M,
                double* d_mu) {
  if (M < 2 || (M & 1)) {
    set_error("n_moments must be even and >= 2 (got %lld)", (long long)M);
    return TBPM_EINVAL;
  }
  Plan pl = pl_in;
  if (use_resident(ctx, lat, pl, M / 2)) {
    TBPM_TRY(ensure(ctx, ctx->ws_phi[0], pl.state_bytes));
    TBPM_TRY(init_states(ctx, lat, req, pl, ctx->ws_phi[0].p, nullptr));
    RecurrenceArgs a;
    TBPM_TRY(base_args(ctx, lat, pl, &a, 3));
    a.mu = d_mu;
    a.M = (int)M;
    const int tok = phase_begin(ctx, 0);
    const int r = launch_resident(ctx, lat, a, pl.precision, ctx->ws_phi[0].p, M / 2);
    phase_end(ctx, tok);
    if (r != TBPM_EUNSUPPORTED) return r;
    clear_error();
  }
  int fmode = 0;
  if (!ctx->lean) TBPM_TRY(choose_fusion(ctx, lat, req, pl, M, &fmode));
  const int64_t steps = M / 2;
  const int K = fused_steps(fmode);
  if (fmode >= 8 && steps - 1 >= K && masked_sweep_ok(lat, pl)) {
    set_layout(lat, &pl, true);
    TBPM_TRY(ensure_dfull(lat));
  }
  const int band = (fmode == 9 ? 192 : fmode == 10 ? 256 : 128) / std::max(1, pl.Spad / 2);
  // the masked, square and one-state sweeps have 128 threads in every mode
  const bool wide_ok = pl.full || fmode == 8 || lat->geom.kind != TBPM_HONEYCOMB || pl.Spad < 2 || lat->geom.Lx >= band;
  const bool sweep = fmode >= 8 && steps - 1 >= K && wide_ok && sweep_ok(lat, pl);
  const bool fuse = !sweep && fmode > 0 && fused_applicable(lat, pl.precision, pl.Spad) && steps - 1 >= K;
  TBPM_TRY(ensure(ctx, ctx->ws_phi[0], pl.state_bytes));
  TBPM_TRY(ensure(ctx, ctx->ws_phi[1], pl.state_bytes));
  if (fuse || sweep) {
    TBPM_TRY(ensure(ctx, ctx->ws_phi2[0], pl.state_bytes));
    TBPM_TRY(ensure(ctx, ctx->ws_phi2[1], pl.state_bytes));
  }
  TBPM_TRY(init_states(ctx, lat, req, pl, ctx->ws_phi[0].p, nullptr));
  RecurrenceArgs a;
  TBPM_TRY(base_args(ctx, lat, pl, &a, 3));
  a.mu = d_mu;
  a.M = (int)M;
  // the pass sequence: step n reads cur = phi_n and overwrites prev (phi_{n-1}) with phi_{n+1}
  bool capturing = false;
  auto body = [&]() -> int {
    void* cur = ctx->ws_phi[0].p;
    void* prev = ctx->ws_phi[1].p;
    void* pair_out[2] = {ctx->ws_phi2[0].p, ctx->ws_phi2[1].p};
    int64_t n = 0;
    auto advance = [&](int steps_done) {
      std::swap(prev, pair_out[0]);
      std::swap(cur, pair_out[1]);
      n += steps_done;
    };
    if (sweep) {
      // every step through the register sweep: the first pass starts from phi_0 alone, the last
      // one may need fewer steps and stores no state
      const int ftok = phase_begin(ctx, 2);
      while (n < steps) {
        const int nk = (int)std::min<int64_t>(K, steps - n);
        const bool last = n + K >= steps;
        TBPM_TRY(launch_sweep_pass(ctx, lat, a, prev, cur, last ? nullptr : pair_out[0], last ? nullptr : pair_out[1],
                                   (int)n, nk, fmode));
        throttle_queue(ctx, capturing);
        advance(K);
      }
      phase_end(ctx, ftok);
      return TBPM_OK;
    }
    auto unfused = [&]() -> int {
      a.cur = cur;
      a.prev_out = prev;
      a.step = (int)n;
      TBPM_TRY(launch_moment_step(ctx, a, pl.precision, n == 0));
      throttle_queue(ctx, capturing);
      std::swap(cur, prev);
      ++n;
      return TBPM_OK;
    };
    TBPM_TRY(unfused());  // phi_1 = H~ phi_0, m_0, m_1
    if (fuse) {
      const int ftok = phase_begin(ctx, 2);
      while (n + K <= steps) {
        TBPM_TRY(launch_fused_pass(ctx, lat, a, prev, cur, pair_out[0], pair_out[1], (int)n, fmode));
        throttle_queue(ctx, capturing);
        advance(K);
      }
      phase_end(ctx, ftok);
    }
    while (n < steps) TBPM_TRY(unfused());
    return TBPM_OK;
  };
  const int tok = phase_begin(ctx, 0);
  if (!ctx->use_graphs || ctx->profiling) {
    TBPM_TRY(body());
  } else {
    auto bits = [](double v) {
      uint64_t u;
      memcpy(&u, &v, 8);
      return u;
    };
    const Geom& g = lat->geom;
    // every device pointer the captured passes read must be part of the key: a graph replays
    // only where those same addresses are allocated again (a lattice created anew at the same
    // addresses holds the same data there); a missing one would replay freed memory.  The tap table
    // is copied into the captured launches: cutoff and decay fix it
    const std::vector<uint64_t> key = {
        (uint64_t)ctx->ws_phi[0].p, (uint64_t)ctx->ws_phi[1].p, (uint64_t)ctx->ws_phi2[0].p,
        (uint64_t)ctx->ws_phi2[1].p, (uint64_t)d_mu, (uint64_t)lat, (uint64_t)lat->d32, (uint64_t)lat->d64,
        (uint64_t)lat->ell, (uint64_t)lat->dfull, (uint64_t)pl.full, (uint64_t)a.partials, (uint64_t)a.counter, (uint64_t)ctx->ws_fused_partials.p,
        (uint64_t)M, (uint64_t)fmode, (uint64_t)pl.precision, (uint64_t)pl.Spad, bits(a.thop), bits(a.diag_const),
        (uint64_t)g.Lx, (uint64_t)g.Ly, (uint64_t)g.Lz, (uint64_t)g.kind,
        (uint64_t)(g.pbc_x | (g.pbc_y << 1) | (g.pbc_z << 2)), (uint64_t)lat->path, (uint64_t)pl.n,
        (uint64_t)(a.taps != nullptr), bits(lat->desc.cutoff), bits(lat->desc.decay),
        (uint64_t)lat->wrel32, (uint64_t)lat->wrel64};
    tbpm_ctx::Graph* hit = nullptr;
    for (auto& e : ctx->graphs)
      if (e.key == key) hit = &e;
    if (!hit) {
      bool seen = false;
      for (auto& k : ctx->graph_seen) seen = seen || k == key;
      if (!seen) {
        // first time: run eagerly (this also sizes every workspace the sequence touches)
        if (ctx->graph_seen.size() >= 16) ctx->graph_seen.erase(ctx->graph_seen.begin());
        ctx->graph_seen.push_back(key);
        TBPM_TRY(body());
      } else {
        cudaGraph_t graph = nullptr;
        const int64_t l0 = ctx->launches;
        TBPM_CK(cudaStreamBeginCapture(ctx->stream, cudaStreamCaptureModeThreadLocal));
        capturing = true;
        const int r = body();
        capturing = false;
        const cudaError_t ec = cudaStreamEndCapture(ctx->stream, &graph);
        const int64_t kernels = ctx->launches - l0;
        ctx->launches = l0;
        if (r != TBPM_OK) {
          if (graph) cudaGraphDestroy(graph);
          return r;
        }
        TBPM_CK(ec);
        cudaGraphExec_t exec = nullptr;
        const cudaError_t ei = cudaGraphInstantiate(&exec, graph, 0);
        cudaGraphDestroy(graph);
        TBPM_CK(ei);
        if (ctx->graphs.size() >= 8) {
          cudaGraphExecDestroy(ctx->graphs.front().exec);
          ctx->graphs.erase(ctx->graphs.begin());
        }
        ctx->graphs.push_back({key, exec, kernels});
        hit = &ctx->graphs.back();
      }
    }
    if (hit) {
      TBPM_CK(cudaGraphLaunch(hit->exec, ctx->stream));
      ctx->launches += hit->kernels;
    }
  }
  phase_end(ctx, tok);
  return TBPM_OK;
}

// Coefficient table of one time block of bb steps: coef[n][j] = c_n((j+1) tau), zero once n >= N((j+1) tau);
// n_per[j] = N((j+1) tau).  amp: the real amplitudes a_n as the flush takes them, c_n = a_n (-i)^n.  The
// factor exp(-i H0 t) of the whole propagation is left out of the states -- it multiplies what is formed from
// them, in FP64 (k_turn_rows): rounded to FP32 in every block, its error was the same each time and added up.
void block_coefficients(double tau, int bb, std::vector<double>* coef, std::vector<int>* n_per,
                        std::vector<double>* amp) {
  n_per->resize(bb);
  for (int j = 0; j < bb; ++j) (*n_per)[j] = (int)truncation_order_host((j + 1) * tau);
  const int nt = *std::max_element(n_per->begin(), n_per->end());
  coef->assign((size_t)nt * bb * 2, 0.0);
  amp->assign((size_t)nt * bb, 0.0);
  std::vector<double> J(nt + 1);
  for (int j = 0; j < bb; ++j) {
    bessel_j_host((j + 1) * tau, nt, J.data());
    for (int n = 0; n < (*n_per)[j]; ++n) {
      const double a = n == 0 ? J[0] : 2.0 * J[n];
      (*amp)[(size_t)n * bb + j] = a;
      (*coef)[((size_t)n * bb + j) * 2 + (n & 1)] = (n & 3) == 1 || (n & 3) == 2 ? -a : a;  // (-i)^n a
    }
  }
}

// Largest b (<= 256, <= n_steps) whose accumulators fit in 80% of the memory there is, beside 34 blocks for a
// window of 32 terms and 4 for the recurrence; what is over goes to a longer window.
int64_t block_cap(tbpm_ctx* ctx, const Plan& pl, int64_t n_steps) {
  const double have = (double)(memory_left(ctx) + ctx->ws_acc.cap + ctx->ws_blk.cap);
  const int64_t by_mem = (int64_t)std::max<double>(1.0, 0.8 * have / (double)pl.state_bytes - 4.0 - 34.0);
  return std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(by_mem, 256), n_steps));
}

// Slots of a window in the buffer b: at most n_terms and what a flush takes, and b at most half the memory it and
// all further buffers can have.
int window_slots(tbpm_ctx* ctx, const DevBuf& b, const Plan& pl, int64_t n_terms) {
  const int64_t fit = (int64_t)(0.5 * (double)(memory_left(ctx) + b.cap) / (double)pl.state_bytes) - 2;
  const int64_t T = std::min<int64_t>(std::min<int64_t>(flush_max_terms(), fit), n_terms);
  return (int)(T >= 4 && T < n_terms ? T / 4 * 4 : T);  // a further window starts at a multiple of four terms
}

// Measured per-pass costs of the state-based form (Sec. II.B: "obtained via benchmarking prior
// to the main calculation"), in milliseconds.  Buffered blocks: t_amxsy = the recurrence into a buffer
// slot plus its share of the flush's slot reads, t_axpy = the flush's extra cost per accumulator and
// term.  Unbuffered ones: t_amxsy = one recurrence pass with no accumulator open, t_axpy = the extra time
// per open accumulator.  Each pass runs once to warm up and once timed where a state block is large
// enough for one launch to be timed well (16 MiB: tens of microseconds), three times otherwise; the
// contents of the scratch blocks do not matter.  (Both sets of passes, three times each on zeroed blocks,
// had made the choice of b 12 % of a 256-step correlation on 8.3M sites.)
int measure_pass_costs(tbpm_ctx* ctx, tbpm_lattice* lat, const tbpm_request* req, const Plan& pl, int k_acc,
                       double* t_amxsy, double* t_axpy) {
  TBPM_TRY(ensure(ctx, ctx->ws_phi[0], pl.state_bytes));
  TBPM_TRY(ensure(ctx, ctx->ws_phi[1], pl.state_bytes));
  TBPM_TRY(ensure(ctx, ctx->ws_psi, pl.state_bytes));
  TBPM_TRY(ensure(ctx, ctx->ws_acc, pl.state_bytes * (size_t)k_acc));
  AccumArgs g;
  memset(&g, 0, sizeof(g));
  TBPM_TRY(base_args(ctx, lat, pl, &g.r, 3));
  g.acc = ctx->ws_acc.p;
  g.acc_stride = pl.n * (int64_t)pl.Spad;
  g.psi = ctx->ws_psi.p;
  g.j_done = -1;
  g.r.cur = ctx->ws_phi[0].p;
  g.r.prev_out = ctx->ws_phi[1].p;
  const bool sweep = sweep_ok(lat, pl);
  // terms per timed flush: enough that the accumulators' own traffic weighs little
  const int Tm = ctx->buffer_blocks && k_acc >= 2 ? window_slots(ctx, ctx->ws_blk, pl, 24) : 0;
  const bool buffered = Tm >= 4 && ensure(ctx, ctx->ws_blk, pl.state_bytes * (size_t)Tm) == TBPM_OK &&
                        ensure(ctx, ctx->ws_blk_coef, sizeof(double) * (size_t)Tm * k_acc) == TBPM_OK;
  std::vector<std::function<int()>> pass;
  if (buffered) {
    // tiny amplitudes, not zeros: the flush skips closed accumulators
    TBPM_CK(cudaMemsetAsync(ctx->ws_blk_coef.p, 0x3c, sizeof(double) * (size_t)Tm * k_acc, ctx->stream));
    char* const w0 = (char*)ctx->ws_blk.p;
    g.r.next = w0;
    pass.push_back([&, w0]() -> int {
      if (!sweep) return launch_accum_step(ctx, g, pl.precision, ACC_REGULAR);
      void* const w[4] = {w0, w0 + pl.state_bytes, w0 + 2 * pl.state_bytes, w0 + 3 * pl.state_bytes};
      return launch_sweep_window(ctx, lat, g.r, ctx->ws_phi[1].p, ctx->ws_phi[0].p, w, false);
    });
    // both flushes in the 16-accumulator tile of the block sizes being chosen between, so that
    // the difference is the cost of the extra accumulators, not of another kernel
    for (const int k : {1, k_acc})
      pass.push_back([&, k]() -> int {
        return launch_flush(ctx, pl.precision, pl.n * pl.Spad, ctx->ws_blk.p, Tm, ctx->ws_acc.p, k,
                            (const double*)ctx->ws_blk_coef.p, 1, true, true, 16);
      });
  } else {
    TBPM_TRY(ensure(ctx, ctx->ws_table, sizeof(double) * 2 * (size_t)k_acc));
    TBPM_CK(cudaMemsetAsync(ctx->ws_table.p, 0, sizeof(double) * 2 * (size_t)k_acc, ctx->stream));
    TBPM_TRY(init_states(ctx, lat, req, pl, ctx->ws_phi[0].p, nullptr));
    TBPM_TRY(init_states(ctx, lat, req, pl, ctx->ws_phi[1].p, nullptr));
    TBPM_CK(cudaMemsetAsync(ctx->ws_acc.p, 0, pl.state_bytes * (size_t)k_acc, ctx->stream));
    g.coef = (const double*)ctx->ws_table.p;
    for (const int k : {0, k_acc})
      pass.push_back([&, k]() -> int {
        g.b = k;
        return launch_accum_step(ctx, g, pl.precision, ACC_REGULAR);
      });
  }
  const int reps = pl.state_bytes >= (16u << 20) ? 1 : 3;
  const int np = (int)pass.size();
  cudaEvent_t e[4];
  for (int k = 0; k <= np; ++k) TBPM_CK(cudaEventCreate(&e[k]));
  int r = TBPM_OK;
  for (int timed = 0; timed < 2 && r == TBPM_OK; ++timed) {
    cudaEventRecord(e[0], ctx->stream);
    for (int k = 0; k < np; ++k) {
      for (int i = 0; i < reps && r == TBPM_OK; ++i) r = pass[k]();
      cudaEventRecord(e[k + 1], ctx->stream);
    }
  }
  double ms[3] = {0.0, 0.0, 0.0};
  if (r == TBPM_OK && cudaEventSynchronize(e[np]) == cudaSuccess)
    for (int k = 0; k < np; ++k) {
      float t = 0.f;
      cudaEventElapsedTime(&t, e[k], e[k + 1]);
      ms[k] = (double)t / reps;
    }
  for (int k = 0; k <= np; ++k) cudaEventDestroy(e[k]);
  TBPM_TRY(r);
  if (buffered) {
    *t_amxsy = ms[0] / (sweep ? 4 : 1) + ms[1] / Tm;
    *t_axpy = std::max(1e-6, (ms[2] - ms[1]) / ((double)(k_acc - 1) * Tm));
  } else {
    *t_amxsy = ms[0];
    *t_axpy = std::max(1e-6, (ms[1] - ms[0]) / k_acc);
  }
  return TBPM_OK;
}

// b_opt = argmin_b C(b) with measured costs (Sec. II.B), capped by memory.
int choose_block(tbpm_ctx* ctx, tbpm_lattice* lat, const tbpm_request* req, const Plan& pl, int64_t n_steps,
                 int64_t* b, double* t_amxsy, double* t_axpy) {
  int64_t cap = block_cap(ctx, pl, n_steps);
  // buffered blocks: one flush serves 16 accumulators per pass over the buffer; past that every
  // further 16 re-read the buffer, which the linear cost model does not see
  if (ctx->buffer_blocks) cap = std::min<int64_t>(cap, 16);
  double ta = 0, tx = 0;
  TBPM_TRY(measure_pass_costs(ctx, lat, req, pl, (int)std::min<int64_t>(cap, 8), &ta, &tx));
  if (t_amxsy) *t_amxsy = ta;
  if (t_axpy) *t_axpy = tx;
  *b = tbpm_block_opt(n_steps, pl.tau, ta, tx, cap);
  return TBPM_OK;
}

// State-based propagation in blocks of b steps; b = 1 is the sequential form.
// d_C [Spad][n_steps+1][2].  The hook sees each finished time block: psi~(t_{start+1}) ..
// psi~(t_{start+bb}) as bb consecutive state blocks, without the common factor:
// psi(t) = e^{-i H0 t} psi~(t).  init (device, optional) replaces the request's initial states.
using BlockHook = std::function<int(int64_t /*start*/, int /*bb*/, const void* /*first state block*/)>;

// The Chebyshev vectors phi_0 .. phi_{n_terms-1} in windows of T buffer slots: slot 2 holds phi_0 on
// entry, slot 2 + k holds term n0 + k, slots 0 and 1 carry the two latest vectors of the previous
// window; flush(n0, nt) takes the nt terms from n0 on out of slot 2 ....  Where the register sweep
// applies, four terms at a time come from one window pass (phi_n and phi_{n-1} read once for four
// slots), else one term per pass.
using WindowFlush = std::function<int(int64_t /*n0*/, int /*nt*/)>;

int walk_windows(tbpm_ctx* ctx, tbpm_lattice* lat, const RecurrenceArgs& r, const Plan& pl, char* slots, int T,
                 int64_t n_terms, const WindowFlush& flush) {
  const bool sweep = sweep_ok(lat, pl);
  AccumArgs g;
  memset(&g, 0, sizeof(g));
  g.r = r;
  g.j_done = -1;
  auto slot = [&](int64_t k) { return (void*)(slots + (size_t)k * pl.state_bytes); };
  int64_t n0 = 0;
  auto slot_of = [&](int64_t m) { return m >= n0 ? slot(2 + (m - n0)) : (m == n0 - 1 ? slot(1) : slot(0)); };
  for (int64_t n = 1; n < n_terms;) {
    if (n - n0 == T) {
      TBPM_TRY(flush(n0, T));
      TBPM_CK(cudaMemcpyAsync(slot(0), slot(T), pl.state_bytes, cudaMemcpyDeviceToDevice, ctx->stream));
      TBPM_CK(cudaMemcpyAsync(slot(1), slot(T + 1), pl.state_bytes, cudaMemcpyDeviceToDevice, ctx->stream));
      n0 = n;
    }
    void* const cur = slot_of(n - 1);
    void* const prev = n >= 2 ? slot_of(n - 2) : cur;  // not read by the first step
    if (sweep) {
      const int cnt = (int)std::min<int64_t>(4, std::min<int64_t>(n_terms - n, T - (n - n0)));
      void* w[4] = {nullptr, nullptr, nullptr, nullptr};
      for (int l = 0; l < cnt; ++l) w[l] = slot_of(n + l);
      TBPM_TRY(launch_sweep_window(ctx, lat, r, prev, cur, w, n == 1));
      n += cnt;
      continue;
    }
    g.r.cur = cur;
    g.r.prev_out = prev;
    g.r.next = slot_of(n);
    TBPM_TRY(launch_accum_step(ctx, g, pl.precision, n == 1 ? ACC_FIRST : ACC_REGULAR));
    ++n;
  }
  return flush(n0, (int)(n_terms - n0));
}

int run_blocks(tbpm_ctx* ctx, tbpm_lattice* lat, const tbpm_request* req, const Plan& pl, int64_t n_steps,
               int64_t b, double* d_C, double tau_signed = 0.0, const BlockHook& hook = nullptr,
               const void* init = nullptr, bool corr = true) {
  const double tau = tau_signed != 0.0 ? tau_signed : pl.tau;
  if (n_steps < 1) {
    set_error("n_steps must be >= 1");
    return TBPM_EINVAL;
  }
  b = std::max<int64_t>(1, std::min<int64_t>(b, n_steps));
  if (corr) TBPM_TRY(ensure(ctx, ctx->ws_psi, pl.state_bytes));
  TBPM_TRY(ensure(ctx, ctx->ws_phi[0], pl.state_bytes));
  TBPM_TRY(ensure(ctx, ctx->ws_phi[1], pl.state_bytes));
  TBPM_TRY(ensure(ctx, ctx->ws_acc, pl.state_bytes * (size_t)b));
  if (corr) {
    if (init)
      TBPM_CK(cudaMemcpyAsync(ctx->ws_psi.p, init, pl.state_bytes, cudaMemcpyDeviceToDevice, ctx->stream));
    else
      TBPM_TRY(init_states(ctx, lat, req, pl, ctx->ws_psi.p, nullptr));
    TBPM_CK(cudaMemcpyAsync(ctx->ws_phi[0].p, ctx->ws_psi.p, pl.state_bytes, cudaMemcpyDeviceToDevice, ctx->stream));
  } else if (!init) {
    TBPM_TRY(init_states(ctx, lat, req, pl, ctx->ws_phi[0].p, nullptr));
  } else if (init != ctx->ws_phi[0].p) {
    TBPM_CK(cudaMemcpyAsync(ctx->ws_phi[0].p, init, pl.state_bytes, cudaMemcpyDeviceToDevice, ctx->stream));
  }

  AccumArgs g;
  memset(&g, 0, sizeof(g));
  TBPM_TRY(base_args(ctx, lat, pl, &g.r, 3));
  const int C_len = (int)(n_steps + 1);
  auto turn = [&]() -> int {  // C(t_j) = e^{-i H0 t_j} <psi|psi~(t_j)>
    return corr ? launch_turn_rows(ctx, d_C, pl.Spad, C_len, -lat->H0 / lat->half * tau) : TBPM_OK;
  };
  // C(0) = <psi|psi>
  if (corr) TBPM_TRY(launch_dot(ctx, g.r, pl.precision, ctx->ws_psi.p, ctx->ws_psi.p, d_C, C_len));

  std::vector<double> coef_full, coef_last, amp_full, amp_last;
  std::vector<int> nper_full, nper_last;
  block_coefficients(tau, (int)b, &coef_full, &nper_full, &amp_full);
  const int64_t last_len = n_steps % b;
  if (last_len) block_coefficients(tau, (int)last_len, &coef_last, &nper_last, &amp_last);
  const size_t tab_bytes = (coef_full.size() + coef_last.size()) * sizeof(double);
  TBPM_TRY(ensure(ctx, ctx->ws_table, tab_bytes));
  double* tab_full = (double*)ctx->ws_table.p;
  double* tab_last = tab_full + coef_full.size();
  TBPM_CK(cudaMemcpyAsync(tab_full, coef_full.data(), coef_full.size() * sizeof(double), cudaMemcpyHostToDevice,
                          ctx->stream));
  if (last_len)
    TBPM_CK(cudaMemcpyAsync(tab_last, coef_last.data(), coef_last.size() * sizeof(double), cudaMemcpyHostToDevice,
                            ctx->stream));
  TBPM_CK(cudaStreamSynchronize(ctx->stream));  // host vectors go out of scope below

  g.acc = ctx->ws_acc.p;
  g.acc_stride = pl.n * (int64_t)pl.Spad;
  g.psi = corr ? ctx->ws_psi.p : nullptr;
  g.C = corr ? d_C : nullptr;
  g.C_len = C_len;

  // Buffered accumulation: the recurrence writes phi_n into a window of T buffer slots, and
  // every T terms one flush adds sum_t c_t(j) phi_t to every accumulator of the block (each
  // accumulator crosses HBM once per T terms instead of once per term); C(t_j) = <psi|acc_j>
  // for the whole block comes from one block inner product at its end.  Where the register sweep
  // applies, this pays even for b = 1: the sequential form then buffers too; otherwise the
  // sequential form keeps its fused one-accumulator pass.
  int T = 0;
  if (ctx->buffer_blocks && (b >= 2 || sweep_ok(lat, pl)))
    T = window_slots(ctx, ctx->ws_blk, pl, *std::max_element(nper_full.begin(), nper_full.end()));
  if (T >= 4) {
    TBPM_TRY(ensure(ctx, ctx->ws_blk, pl.state_bytes * (size_t)(T + 2)));
    // amplitudes, full block then last block
    std::vector<double> cz = amp_full;
    cz.insert(cz.end(), amp_last.begin(), amp_last.end());
    TBPM_TRY(ensure(ctx, ctx->ws_blk_coef, cz.size() * sizeof(double)));
    TBPM_CK(cudaMemcpyAsync(ctx->ws_blk_coef.p, cz.data(), cz.size() * sizeof(double), cudaMemcpyHostToDevice,
                            ctx->stream));
    TBPM_CK(cudaStreamSynchronize(ctx->stream));
    char* slots = (char*)ctx->ws_blk.p;
    char* const terms = slots + 2 * pl.state_bytes;
    int64_t start = 0;
    while (start < n_steps) {
      const int bb = (int)std::min<int64_t>(b, n_steps - start);
      const std::vector<int>& nper = (bb == b) ? nper_full : nper_last;
      const double* amp = (const double*)ctx->ws_blk_coef.p + ((bb == b) ? 0 : amp_full.size());
      const int Nb = *std::max_element(nper.begin(), nper.end());
      // the block starts from the last state of the one before
      const char* first = start == 0 ? (const char*)ctx->ws_phi[0].p
                                     : (const char*)ctx->ws_acc.p + (size_t)(b - 1) * pl.state_bytes;
      TBPM_CK(cudaMemcpyAsync(terms, first, pl.state_bytes, cudaMemcpyDeviceToDevice, ctx->stream));
      TBPM_TRY(walk_windows(ctx, lat, g.r, pl, slots, T, Nb, [&](int64_t n0, int nt) -> int {
        return launch_flush(ctx, pl.precision, pl.n * pl.Spad, terms, nt, ctx->ws_acc.p, bb, amp + (size_t)n0 * bb, 1,
                            true, n0 == 0);
      }));
      if (corr)
        TBPM_TRY(launch_xdot(ctx, pl.precision, pl.Spad, pl.n, ctx->ws_psi.p, 1, ctx->ws_acc.p, bb, d_C,
                             C_len, 0, 1, start + 1));
      if (hook) TBPM_TRY(hook(start, bb, ctx->ws_acc.p));
      start += bb;
    }
    return turn();
  }

  int64_t start = 0;
  while (start < n_steps) {
    const int bb = (int)std::min<int64_t>(b, n_steps - start);
    const std::vector<int>& nper = (bb == b) ? nper_full : nper_last;
    const double* tab = (bb == b) ? tab_full : tab_last;
    const int Nb = *std::max_element(nper.begin(), nper.end());
    g.b = bb;
    for (int n = 0; n < Nb; ++n) {
      int j_lo = 0;
      while (j_lo < bb && nper[j_lo] <= n) ++j_lo;
      std::vector<int> done;
      for (int j = j_lo; j < bb; ++j)
        if (nper[j] - 1 == n) done.push_back(j);
      const int mode = (n == Nb - 1) ? ACC_NOSPMV : (n == 0 ? ACC_FIRST : ACC_REGULAR);
      g.r.cur = ctx->ws_phi[n & 1].p;
      g.r.prev_out = ctx->ws_phi[(n + 1) & 1].p;
      g.coef = tab + (size_t)n * bb * 2;
      g.j_lo = j_lo;
      g.first_term = n == 0;
      if (!corr) done.clear();
      g.j_done = done.empty() ? -1 : done[0];
      g.j_global = done.empty() ? 0 : (int)(start + done[0] + 1);
      TBPM_TRY(launch_accum_step(ctx, g, pl.precision, mode));
      for (size_t q = 1; q < done.size(); ++q) {
        const int j = done[q];
        const char* accj = (const char*)ctx->ws_acc.p + (size_t)j * pl.state_bytes;
        TBPM_TRY(launch_dot(ctx, g.r, pl.precision, ctx->ws_psi.p, accj, d_C + (start + j + 1) * 2, C_len));
      }
    }
    if (hook) TBPM_TRY(hook(start, bb, ctx->ws_acc.p));
    // the block's last state starts the next block
    const char* last = (const char*)ctx->ws_acc.p + (size_t)(bb - 1) * pl.state_bytes;
    TBPM_CK(cudaMemcpyAsync(ctx->ws_phi[0].p, last, pl.state_bytes, cudaMemcpyDeviceToDevice, ctx->stream));
    start += bb;
  }
  return turn();
}

// Time blocks, quasi-eigenstates and the conductivity of a vacancy lattice take the full layout where the masked
// sweep applies and memory is ample: `blocks` state blocks of the request, six of the propagation (16-fold
// roundings of the allocations included), and twice a window of eight terms, all of them for every site.
int take_full_layout(tbpm_ctx* ctx, tbpm_lattice* lat, Plan* pl, int64_t blocks) {
  if (!ctx->buffer_blocks || ctx->lean || !masked_sweep_ok(lat, *pl)) return TBPM_OK;
  set_layout(lat, pl, true);
  const double have = (double)(memory_left(ctx) + kept_bytes(ctx));
  if (((double)blocks + 6.0) * 1.07 + 20.0 > have / (double)pl->state_bytes) set_layout(lat, pl, false);
  return pl->full ? ensure_dfull(lat) : TBPM_OK;
}

// Correlation of all Spad states into d_C [Spad][n_steps+1][2].
int run_correlation(tbpm_ctx* ctx, tbpm_lattice* lat, const tbpm_request* req, const Plan& pl_in, double* d_C) {
  Plan pl = pl_in;
  const int64_t n_steps = req->n_steps;
  if (n_steps < 1 || n_steps > (1 << 24)) {
    set_error("n_steps out of range");
    return TBPM_EINVAL;
  }
  if (req->form == TBPM_CONCURRENT_M) {
    const int64_t need = truncation_order_host(n_steps * pl.tau);
    int64_t M = std::max<int64_t>(req->n_moments, need);
    M += (M & 1);
    TBPM_TRY(ensure(ctx, ctx->ws_mu, sizeof(double) * 2 * (size_t)M * pl.Spad));
    double* mu = (double*)ctx->ws_mu.p;
    TBPM_TRY(run_moments(ctx, lat, req, pl, M, mu));
    const int n_terms = (int)need + 8;
    const size_t tab = sizeof(double) * (size_t)n_terms * (n_steps + 1);
    TBPM_TRY(ensure(ctx, ctx->ws_table, tab + sizeof(int) * (n_steps + 1)));
    double* table = (double*)ctx->ws_table.p;
    int* nper = (int*)((char*)ctx->ws_table.p + tab);
    TBPM_TRY(launch_bessel_table(ctx, pl.tau, (int)n_steps, n_terms, table, nper));
    TBPM_TRY(launch_corr_from_moments(ctx, table, nper, (int)n_steps, n_terms, mu, pl.Spad, (int)M,
                                      lat->H0 / lat->half, pl.tau, d_C));
    return TBPM_OK;
  }
  TBPM_TRY(take_full_layout(ctx, lat, &pl, std::max<int64_t>(16, req->time_block)));
  if (req->form == TBPM_SEQUENTIAL) return run_blocks(ctx, lat, req, pl, n_steps, 1, d_C);
  if (req->form == TBPM_CONCURRENT_S) {
    int64_t b = req->time_block;
    if (b <= 0) TBPM_TRY(choose_block(ctx, lat, req, pl, n_steps, &b, nullptr, nullptr));
    return run_blocks(ctx, lat, req, pl, n_steps, b, d_C);
  }
  set_error("unknown form %d", req->form);
  return TBPM_EINVAL;
}

// Quasi-eigenstates (Sec. IV) of all Spad states into ws_qe: [nE][n_sites][Spad].
int run_qe(tbpm_ctx* ctx, tbpm_lattice* lat, const tbpm_request* req, const Plan& pl, const double* d_E, int nE) {
  const int64_t n_steps = req->n_steps;
  if (n_steps < 1 || n_steps > (1 << 22) || nE < 1 || nE > 4096) {
    set_error("quasi-eigenstates need 1 <= n_steps and 1 <= n_energies <= 4096");
    return TBPM_EINVAL;
  }
  const double tphys = pl.tau / lat->half;
  TBPM_TRY(ensure(ctx, ctx->ws_qe, pl.state_bytes * (size_t)nE));
  const size_t phase_bytes = sizeof(double) * 2 * (size_t)nE * (n_steps + 1);
  if (req->form == TBPM_CONCURRENT_E) {
    const int64_t need = truncation_order_host(n_steps * pl.tau);
    const int n_table = (int)need + 8;
    const size_t tab = sizeof(double) * (size_t)n_table * (n_steps + 1);
    TBPM_TRY(ensure(ctx, ctx->ws_table, tab + sizeof(int) * (n_steps + 1)));
    TBPM_TRY(ensure(ctx, ctx->ws_qe_coef, phase_bytes + sizeof(double) * 2 * (size_t)need * nE));
    double* table = (double*)ctx->ws_table.p;
    int* nper = (int*)((char*)ctx->ws_table.p + tab);
    double* phase = (double*)ctx->ws_qe_coef.p;
    double* coef = phase + 2 * (size_t)nE * (n_steps + 1);
    TBPM_TRY(launch_bessel_table(ctx, pl.tau, (int)n_steps, n_table, table, nper));
    TBPM_TRY(launch_qe_coefficients(ctx, table, (int)n_steps, (int)need, d_E, nE, lat->H0, tphys, phase, coef));
    // buffered accumulation: the recurrence fills a window of T slots, and every T terms one flush
    // adds sum_t C_t(E) phi_t to all N_E accumulators
    const int T = window_slots(ctx, ctx->ws_acc, pl, need);
    if (T >= 4) {
      TBPM_TRY(ensure(ctx, ctx->ws_acc, pl.state_bytes * (size_t)(T + 2)));
      char* const terms = (char*)ctx->ws_acc.p + 2 * pl.state_bytes;
      TBPM_TRY(init_states(ctx, lat, req, pl, terms, nullptr));
      RecurrenceArgs ra;
      TBPM_TRY(base_args(ctx, lat, pl, &ra, 3));
      const int tok = phase_begin(ctx, 0);
      TBPM_TRY(walk_windows(ctx, lat, ra, pl, (char*)ctx->ws_acc.p, T, need, [&](int64_t n0, int nt) -> int {
        return launch_flush(ctx, pl.precision, pl.n * pl.Spad, terms, nt, ctx->ws_qe.p, nE, coef + 2 * (size_t)n0 * nE, 2,
                            false, n0 == 0);
      }));
      phase_end(ctx, tok);
      return TBPM_OK;
    }
    // memory for a slot only: each pass copies phi_n into it and the flush follows at once
    TBPM_TRY(ensure(ctx, ctx->ws_phi[0], pl.state_bytes));
    TBPM_TRY(ensure(ctx, ctx->ws_phi[1], pl.state_bytes));
    TBPM_TRY(init_states(ctx, lat, req, pl, ctx->ws_phi[0].p, nullptr));
    TBPM_TRY(ensure(ctx, ctx->ws_acc, pl.state_bytes));
    TBPM_TRY(ensure(ctx, ctx->ws_aux, 2 * sizeof(double)));
    const double one[2] = {1.0, 0.0};
    TBPM_CK(cudaMemcpyAsync(ctx->ws_aux.p, one, sizeof(one), cudaMemcpyHostToDevice, ctx->stream));
    AccumArgs g;
    memset(&g, 0, sizeof(g));
    TBPM_TRY(base_args(ctx, lat, pl, &g.r, 3));
    g.acc = ctx->ws_acc.p;
    g.acc_stride = pl.n * (int64_t)pl.Spad;
    g.b = 1;
    g.j_lo = 0;
    g.j_done = -1;
    g.first_term = 1;  // the slot is written, not accumulated
    g.coef = (const double*)ctx->ws_aux.p;
    const int tok = phase_begin(ctx, 0);
    for (int64_t n = 0; n < need; ++n) {
      const int mode = (n == need - 1) ? ACC_NOSPMV : (n == 0 ? ACC_FIRST : ACC_REGULAR);
      g.r.cur = ctx->ws_phi[n & 1].p;
      g.r.prev_out = ctx->ws_phi[(n + 1) & 1].p;
      TBPM_TRY(launch_accum_step(ctx, g, pl.precision, mode));
      TBPM_TRY(launch_flush(ctx, pl.precision, pl.n * pl.Spad, ctx->ws_acc.p, 1, ctx->ws_qe.p, nE,
                            coef + 2 * (size_t)n * nE, 2, false, n == 0));
    }
    phase_end(ctx, tok);
    return TBPM_OK;
  }
  if (req->form != TBPM_SEQUENTIAL && req->form != TBPM_CONCURRENT_S) {
    set_error("quasi-eigenstates: form must be SEQUENTIAL, CONCURRENT_S or CONCURRENT_E");
    return TBPM_EINVAL;
  }
  // explicit states psi~(+-t_j), each folded into the N_E accumulators with (tau/2pi) e^{+-i (E - H0) t_j}
  TBPM_TRY(ensure(ctx, ctx->ws_qe_coef, phase_bytes));
  double* phase = (double*)ctx->ws_qe_coef.p;
  {
    const int64_t tot = (int64_t)nE * (n_steps + 1);
    (void)tot;
    TBPM_TRY(launch_qe_phases(ctx, d_E, nE, lat->H0, tphys, (int)n_steps, phase));
  }
  TBPM_CK(cudaMemsetAsync(ctx->ws_qe.p, 0, pl.state_bytes * (size_t)nE, ctx->stream));
  RecurrenceArgs ra;
  TBPM_TRY(base_args(ctx, lat, pl, &ra, 3));
  const int width = (int)(n_steps + 1);
  const double scale = tphys / (2.0 * M_PI);
  int64_t b = req->form == TBPM_SEQUENTIAL ? 1 : req->time_block;
  if (b <= 0) TBPM_TRY(choose_block(ctx, lat, req, pl, n_steps, &b, nullptr, nullptr));
  TBPM_TRY(ensure(ctx, ctx->ws_psi, pl.state_bytes));
  TBPM_TRY(init_states(ctx, lat, req, pl, ctx->ws_psi.p, nullptr));
  for (int dir = 0; dir < 2; ++dir) {
    const double sgn = dir == 0 ? 1.0 : -1.0;
    BlockHook hook = [&](int64_t start, int bb, const void* first) -> int {
      for (int j = 0; j < bb; ++j)
        TBPM_TRY(launch_qe_axpy(ctx, ra, pl.precision, (const char*)first + (size_t)j * pl.state_bytes,
                                ctx->ws_qe.p, phase, width, (int)(start + j + 1), sgn, scale, nE));
      return TBPM_OK;
    };
    TBPM_TRY(run_blocks(ctx, lat, req, pl, n_steps, b, nullptr, sgn * pl.tau, hook, ctx->ws_psi.p, false));
    if (dir == 0)  // j = 0 term, tau a(E,0) psi, once
      TBPM_TRY(launch_qe_axpy(ctx, ra, pl.precision, ctx->ws_psi.p, ctx->ws_qe.p, phase, width, 0, 1.0, scale, nE));
  }
  return TBPM_OK;
}

// The overlaps O(E) = <psi|Psi(E)> that the conductivity divides by, in 64 bits where FP32 does not do.  Psi(E) in
// complex64 gives O with an absolute error that does not shrink with O: the rounding of H~ and of C_n(E), 1e-8 to
// 1e-7 of O's mean 1 / (2 |H|) over the window, and the recurrence's own, about 8e-9 of it on 1e5 sites and falling
// as 1 / sqrt(N).  Next to the Dirac point of a sample with few vacancies O passes through zero between energies: at
// |O| = 2e-4 of the mean (380 x 200 cells, W = 1.7, 127 steps) C(t, E) was 1.3e-4 off, now 6e-7.  The line lies
// where the recurrence's share passes 1e-7 of O: a tenth of the mean at 2e5 sites, falling with 1 / sqrt(N) to 0.03
// (the first two shares stay) and 0.5 for small samples and site states.  Below it, all overlaps of the request are
// formed again from the complex128 moments of the same states, need / 2 steps in FP64: on 2.1M sites and 128 time
// steps 26 ms beside the 16 ms of 9 energies.  Long-range lattices keep the complex64 overlaps (an FP64 step of 235
// neighbours costs more than the request).
int refine_overlaps(tbpm_ctx* ctx, tbpm_lattice* lat, const tbpm_request* req, const Plan& pl, const double* d_E,
                    int nE, double* nrm) {
  if (pl.precision != TBPM_C64 || !lat->tap_t.empty()) return TBPM_OK;
  std::vector<double> h(2 * (size_t)pl.S * nE);
  TBPM_CK(cudaMemcpyAsync(h.data(), nrm, sizeof(double) * h.size(), cudaMemcpyDeviceToHost, ctx->stream));
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  double least = INFINITY;
  for (size_t k = 0; k < h.size(); k += 2) least = std::min(least, hypot(h[k], h[k + 1]));
  const double n_eff = req->states == TBPM_STATES_SITES ? 1.0 : (double)lat->n_sites;
  const double line = std::min(0.5, std::max(0.03, 0.1 * sqrt(2e5 / n_eff)));
  if (!(least < line / (2.0 * lat->half))) return TBPM_OK;
  tbpm_request r128 = *req;
  r128.precision = TBPM_C128;
  r128.form = TBPM_CONCURRENT_M;
  r128.n_moments = 0;
  Plan p128;
  TBPM_TRY(make_plan(lat, &r128, &p128));
  int r = ensure(ctx, ctx->ws_out, sizeof(double) * 2 * (size_t)p128.Spad * (req->n_steps + 1));
  if (r == TBPM_OK) r = run_correlation(ctx, lat, &r128, p128, (double*)ctx->ws_out.p);
  if (r == TBPM_ENOMEM) {  // no room for two complex128 blocks: the complex64 overlaps stay
    clear_error();
    return TBPM_OK;
  }
  TBPM_TRY(r);
  return launch_ec_overlap(ctx, (const double*)ctx->ws_out.p, d_E, nE, pl.Spad * nE, (int)req->n_steps,
                           pl.tau / lat->half, nrm);
}

// Electronic conductivity (Sec. V) along `direction` for all Spad states and nE energies.
// Leaves C(t_j, E_k) in ws_out as [Spad][nE][n_steps+1][2] and sigma in ws_ec (after the
// 2*Spad*nE norms) as [Spad][nE].  Returns the sigma pointer through *d_sigma.
int run_ec(tbpm_ctx* ctx, tbpm_lattice* lat, const tbpm_request* req, const Plan& pl_in, const double* d_E, int nE,
           int direction, double** d_C_out, double** d_sigma) {
  Plan pl = pl_in;
  const int64_t n_steps = req->n_steps;
  const int dims = lat->desc.kind == TBPM_CUBIC ? 3 : 2;
  if (direction < 0 || direction >= dims) {
    set_error("direction %d out of range for a %d-dimensional lattice", direction, dims);
    return TBPM_EINVAL;
  }
  if (req->form != TBPM_SEQUENTIAL && req->form != TBPM_CONCURRENT_S && req->form != TBPM_CONCURRENT_M) {
    set_error("conductivity: form must be SEQUENTIAL, CONCURRENT_S or CONCURRENT_M");
    return TBPM_EINVAL;
  }
  if (n_steps < 1 || n_steps > (1 << 20) || nE < 1 || nE > 4096 || (int64_t)nE * pl.Spad > 65536) {
    set_error("conductivity needs 1 <= n_steps <= 2^20, 1 <= n_energies <= 4096 and n_energies * states <= 65536");
    return TBPM_EINVAL;
  }
  // quasi-eigenstates: energy-based form for few energies, state-based otherwise (Sec. IV)
  tbpm_request qreq = *req;
  qreq.form = nE <= 200 ? TBPM_CONCURRENT_E : TBPM_CONCURRENT_S;
  qreq.time_block = 0;
  TBPM_TRY(take_full_layout(ctx, lat, &pl, nE + std::max<int64_t>(16, req->time_block)));
  TBPM_TRY(run_qe(ctx, lat, &qreq, pl, d_E, nE));
  const int rows = pl.Spad * nE;
  const int64_t W = n_steps + 1;
  TBPM_TRY(ensure(ctx, ctx->ws_ec, sizeof(double) * 3 * (size_t)rows));
  double* nrm = (double*)ctx->ws_ec.p;
  double* sigma = nrm + 2 * (size_t)rows;
  TBPM_TRY(ensure(ctx, ctx->ws_psi, pl.state_bytes));
  TBPM_TRY(ensure(ctx, ctx->ws_jpsi, pl.state_bytes));
  TBPM_TRY(init_states(ctx, lat, req, pl, ctx->ws_psi.p, nullptr));
  const int64_t n = pl.n;
  // <psi|Psi(E)> before the kets are overwritten
  TBPM_TRY(launch_xdot(ctx, pl.precision, pl.Spad, n, ctx->ws_psi.p, 1, ctx->ws_qe.p, nE, nrm, nE, 0, 1, 0));
  TBPM_TRY(refine_overlaps(ctx, lat, req, pl, d_E, nE, nrm));
  TBPM_TRY(ensure(ctx, ctx->ws_phi[0], pl.state_bytes));
  TBPM_TRY(ensure(ctx, ctx->ws_phi[1], pl.state_bytes));
  // |psi_2(E)> = J |Psi(E)> in place (through one scratch block), |psi_1> = J |psi>
  for (int k = 0; k < nE; ++k) {
    char* qk = (char*)ctx->ws_qe.p + (size_t)k * pl.state_bytes;
    TBPM_TRY(launch_current(ctx, lat, pl.precision, pl.Spad, direction, qk, ctx->ws_phi[0].p, pl.full));
    TBPM_CK(cudaMemcpyAsync(qk, ctx->ws_phi[0].p, pl.state_bytes, cudaMemcpyDeviceToDevice, ctx->stream));
  }
  TBPM_TRY(launch_current(ctx, lat, pl.precision, pl.Spad, direction, ctx->ws_psi.p, ctx->ws_jpsi.p, pl.full));
  const void* kets = ctx->ws_qe.p;
  TBPM_TRY(ensure(ctx, ctx->ws_out, sizeof(double) * 2 * (size_t)rows * W));
  double* C = (double*)ctx->ws_out.p;
  const int tok = phase_begin(ctx, 0);
  if (req->form == TBPM_CONCURRENT_M) {
    // m_n(E) = <J psi|T_n(H~)|J Psi(E)> (Eq. dc_mom), n < N(t~_tot)
    const int64_t Nn = truncation_order_host(n_steps * pl.tau);
    TBPM_TRY(ensure(ctx, ctx->ws_mu, sizeof(double) * 2 * (size_t)rows * Nn));
    double* m = (double*)ctx->ws_mu.p;
    TBPM_CK(cudaMemcpyAsync(ctx->ws_phi[0].p, ctx->ws_jpsi.p, pl.state_bytes, cudaMemcpyDeviceToDevice, ctx->stream));
    AccumArgs g;
    memset(&g, 0, sizeof(g));
    TBPM_TRY(base_args(ctx, lat, pl, &g.r, 3));
    g.b = 0;
    g.j_done = -1;
    // buffered: the recurrence fills a window of slots and one block inner product
    // gives the window's moments against all kets (each ket read once per window, not per term)
    const int T = ctx->buffer_blocks ? window_slots(ctx, ctx->ws_blk, pl, Nn) : 0;
    if (T >= 4) {
      TBPM_TRY(ensure(ctx, ctx->ws_blk, pl.state_bytes * (size_t)(T + 2)));
      char* const terms = (char*)ctx->ws_blk.p + 2 * pl.state_bytes;
      TBPM_CK(cudaMemcpyAsync(terms, ctx->ws_jpsi.p, pl.state_bytes, cudaMemcpyDeviceToDevice, ctx->stream));
      TBPM_TRY(walk_windows(ctx, lat, g.r, pl, (char*)ctx->ws_blk.p, T, Nn, [&](int64_t n0, int nt) -> int {
        return launch_xdot(ctx, pl.precision, pl.Spad, n, terms, nt, kets, nE, m, (int64_t)nE * Nn, 1, Nn, n0);
      }));
    } else {
    TBPM_TRY(launch_xdot(ctx, pl.precision, pl.Spad, n, ctx->ws_phi[0].p, 1, kets, nE, m, (int64_t)nE * Nn, 0, Nn, 0));
    for (int64_t k = 0; k + 1 < Nn; ++k) {
      g.r.cur = ctx->ws_phi[k & 1].p;
      g.r.prev_out = ctx->ws_phi[(k + 1) & 1].p;
      TBPM_TRY(launch_accum_step(ctx, g, pl.precision, k == 0 ? ACC_FIRST : ACC_REGULAR));
      TBPM_TRY(launch_xdot(ctx, pl.precision, pl.Spad, n, ctx->ws_phi[(k + 1) & 1].p, 1, kets, nE, m,
                           (int64_t)nE * Nn, 0, Nn, k + 1));
    }
    }
    phase_end(ctx, tok);
    const int n_table = (int)Nn + 8;
    const size_t tab = sizeof(double) * (size_t)n_table * W;
    TBPM_TRY(ensure(ctx, ctx->ws_table, tab + sizeof(int) * (size_t)W));
    double* table = (double*)ctx->ws_table.p;
    int* nper = (int*)((char*)ctx->ws_table.p + tab);
    TBPM_TRY(launch_bessel_table(ctx, pl.tau, (int)n_steps, n_table, table, nper));
    TBPM_TRY(launch_ec_corr_from_moments(ctx, table, nper, (int)n_steps, m, rows, (int)Nn, lat->H0 / lat->half,
                                         pl.tau, C));
  } else {
    // psi_1(t_j) = e^{-iHt_j} J psi in time blocks; each block's b states meet all N_E kets at once
    int64_t b = req->form == TBPM_SEQUENTIAL ? 1 : req->time_block;
    if (b <= 0) TBPM_TRY(choose_block(ctx, lat, req, pl, n_steps, &b, nullptr, nullptr));
    BlockHook hook = [&](int64_t start, int bb, const void* first) -> int {
      return launch_xdot(ctx, pl.precision, pl.Spad, n, first, bb, kets, nE, C, (int64_t)nE * W, 1, W, start + 1);
    };
    TBPM_TRY(run_blocks(ctx, lat, req, pl, n_steps, b, nullptr, 0.0, hook, ctx->ws_jpsi.p, false));
    TBPM_TRY(launch_xdot(ctx, pl.precision, pl.Spad, n, ctx->ws_jpsi.p, 1, kets, nE, C, (int64_t)nE * W, 0, W, 0));
    TBPM_TRY(launch_turn_rows(ctx, C, rows, W, lat->H0 / lat->half * pl.tau));
    phase_end(ctx, tok);
  }
  const double area = lat->desc.kind == TBPM_HONEYCOMB ? 3.0 * sqrt(3.0) / 4.0 : 1.0;
  TBPM_TRY(launch_ec_finish(ctx, C, nrm, d_E, nE, rows, (int)n_steps, pl.tau / lat->half, area, sigma));
  *d_C_out = C;
  *d_sigma = sigma;
  return TBPM_OK;
}

// Chebyshev coefficients of the Fermi-Dirac function (or its square root) on the lattice's
// spectral window into ws_fermi; *coef = device complex table [n_terms][2], truncated at
// 1 + max{n : |a_n| > 1e-14} within n_cap = min(2^14, 12|H|/kT + 64) orders.
int fermi_series(tbpm_ctx* ctx, const tbpm_lattice* lat, double mu, double kT, int sqrt_f, const double** coef,
                 int* n_terms) {
  if (!(kT > 0.0) || !isfinite(kT) || !isfinite(mu)) {
    set_error("Fermi-Dirac operator needs kT > 0 and a finite mu");
    return TBPM_EINVAL;
  }
  const double want = 12.0 * lat->half / kT + 64.0;
  const int n_cap = (int)std::min<double>(16384.0, std::max<double>(64.0, ceil(want)));
  const int K = std::max(2 * n_cap, 1024);
  TBPM_TRY(ensure(ctx, ctx->ws_fermi, sizeof(double) * ((size_t)K + 2 * (size_t)n_cap)));
  double* scratch = (double*)ctx->ws_fermi.p;
  double* table = scratch + K;
  TBPM_TRY(launch_fermi_coefficients(ctx, mu, kT, lat->H0, lat->half, sqrt_f, n_cap, K, scratch, table));
  std::vector<double> h(2 * (size_t)n_cap);
  TBPM_CK(cudaMemcpyAsync(h.data(), table, sizeof(double) * h.size(), cudaMemcpyDeviceToHost, ctx->stream));
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  int last = 0;
  for (int n = n_cap - 1; n >= 0; --n)
    if (fabs(h[2 * (size_t)n]) > 1e-14) {
      last = n;
      break;
    }
  *coef = table;
  *n_terms = last + 1;
  return TBPM_OK;
}

// Workspaces of the response drivers are given back between their phases only where memory is short
// (a block above an eighth of what is left): freeing and allocating them again on every call cost
// 7 of 85 ms of the optical conductivity of 2.1M sites.
void release_if_tight(tbpm_ctx* ctx, DevBuf& b) {
  if (b.cap <= memory_left(ctx) / 8) return;
  release(ctx, b);
  cudaStreamSynchronize(ctx->stream);  // the pool counts the block as idle from here on
}

// out = sum_{n < n_terms} coef_n T_n(H~) X for one state block of plan pc.  The recurrence runs
// in b0 (which holds X on entry and is overwritten) and b1; out is distinct from both.
int apply_series_bufs(tbpm_ctx* ctx, tbpm_lattice* lat, const Plan& pc, void* b0, void* b1, void* out,
                      const double* coef, int n_terms) {
  AccumArgs g;
  memset(&g, 0, sizeof(g));
  TBPM_TRY(base_args(ctx, lat, pc, &g.r, 3));
  g.acc = out;
  g.acc_stride = lat->n_sites * (int64_t)pc.Spad;
  g.b = 1;
  g.j_lo = 0;
  g.j_done = -1;
  // buffered: terms go into a window of slots and one flush adds sum_n a_n T_n phi to
  // the output per window (as the buffered time blocks)
  const int T = ctx->buffer_blocks ? window_slots(ctx, ctx->ws_blk, pc, n_terms) : 0;
  if (T >= 4) {
    TBPM_TRY(ensure(ctx, ctx->ws_blk, pc.state_bytes * (size_t)(T + 2)));
    char* const terms = (char*)ctx->ws_blk.p + 2 * pc.state_bytes;
    TBPM_CK(cudaMemcpyAsync(terms, b0, pc.state_bytes, cudaMemcpyDeviceToDevice, ctx->stream));
    TBPM_TRY(walk_windows(ctx, lat, g.r, pc, (char*)ctx->ws_blk.p, T, n_terms, [&](int64_t n0, int nt) -> int {
      return launch_flush(ctx, pc.precision, pc.n * pc.Spad, terms, nt, out, 1, coef + 2 * (size_t)n0, 2, false, n0 == 0);
    }));
    release_if_tight(ctx, ctx->ws_blk);  // the callers' next step sizes its blocks by the free memory
    return TBPM_OK;
  }
  void* buf[2] = {b0, b1};
  for (int n = 0; n < n_terms; ++n) {
    const int mode = (n == n_terms - 1) ? ACC_NOSPMV : (n == 0 ? ACC_FIRST : ACC_REGULAR);
    g.r.cur = buf[n & 1];
    g.r.prev_out = buf[(n + 1) & 1];
    g.coef = coef + 2 * (size_t)n;
    g.first_term = n == 0;
    TBPM_TRY(launch_accum_step(ctx, g, pc.precision, mode));
  }
  return TBPM_OK;
}

// Largest power-of-two number of states per pass (<= cap) for which `blocks` state blocks of
// that width fit in 85% of the memory there is, kept workspaces included; 0 when not even one state fits.
int states_per_pass(tbpm_ctx* ctx, const tbpm_lattice* lat, size_t elem, int cap, double blocks) {
  const double have = (double)(memory_left(ctx) + kept_bytes(ctx));
  int k = cap;
  while (k >= 1 && blocks * (double)lat->n_sites * k * elem > 0.85 * have) k >>= 1;
  return k;
}

// Optical conductivity (op 0: X = J_alpha, O = J_beta) or dynamical polarization (op 1:
// X = rho(q), O = rho(-q)) correlation C(t_j) = <psi_1(t_j)|X|psi_2(t_j)> of the plan's Sh states
// (the request's states pl.s0 .. pl.s0 + S - 1) into ws_out [Sh][n_steps+1][2]; the pair plan's
// time step is returned in *tphys.  Live memory: three pair blocks during the Fermi-Dirac series,
// 2 + b during the propagation.
int run_response(tbpm_ctx* ctx, tbpm_lattice* lat, const tbpm_request* req, const Plan& pl, int op, int alpha,
                 int beta, const double q[3], double mu, double kT, double** d_C, double* tphys) {
  const int64_t n_steps = req->n_steps;
  const int Sh = pl.Spad;
  tbpm_request rc = *req;
  rc.n_states = 2 * Sh;
  rc.states = TBPM_STATES_RANDOM;
  Plan pc;
  TBPM_TRY(make_plan(lat, &rc, &pc));
  pc.tau = req->tau == 0.0 ? M_PI / 2 : req->tau;
  *tphys = pc.tau / lat->half;
  const int64_t n = lat->n_sites;
  const double* coef = nullptr;
  int nf = 0;
  TBPM_TRY(fermi_series(ctx, lat, mu, kT, 0, &coef, &nf));
  const double2* phase = nullptr;
  if (op == 1) {
    TBPM_TRY(ensure(ctx, ctx->ws_ec, sizeof(double2) * (size_t)n));
    phase = (const double2*)ctx->ws_ec.p;
    TBPM_TRY(launch_density_phases(ctx, lat, q, (double2*)ctx->ws_ec.p));
  }
  // O psi, formed from psi (twice: before the series and for the split after it)
  auto make_states = [&]() -> int {
    TBPM_TRY(ensure(ctx, ctx->ws_psi, pl.state_bytes));
    TBPM_TRY(init_states(ctx, lat, req, pl, ctx->ws_psi.p, nullptr));
    if (op == 0) {
      TBPM_TRY(ensure(ctx, ctx->ws_jpsi, pl.state_bytes));
      TBPM_TRY(launch_current(ctx, lat, pl.precision, Sh, beta, ctx->ws_psi.p, ctx->ws_jpsi.p, false));
    }
    return TBPM_OK;
  };
  TBPM_TRY(make_states());
  TBPM_TRY(ensure(ctx, ctx->ws_phi[0], pc.state_bytes));
  TBPM_TRY(launch_pair_init(ctx, pl.precision, n, Sh, ctx->ws_psi.p, op == 0 ? ctx->ws_jpsi.p : nullptr, phase,
                            ctx->ws_phi[0].p));
  release_if_tight(ctx, ctx->ws_psi);
  release_if_tight(ctx, ctx->ws_jpsi);
  TBPM_TRY(ensure(ctx, ctx->ws_phi[1], pc.state_bytes));
  TBPM_TRY(ensure(ctx, ctx->ws_phi2[1], pc.state_bytes));
  // F = f(H) X, consuming X in ws_phi[0]
  TBPM_TRY(apply_series_bufs(ctx, lat, pc, ctx->ws_phi[0].p, ctx->ws_phi[1].p, ctx->ws_phi2[1].p, coef, nf));
  release_if_tight(ctx, ctx->ws_phi[0]);
  TBPM_TRY(make_states());
  TBPM_TRY(launch_pair_split(ctx, pl.precision, n, Sh, ctx->ws_psi.p, op == 0 ? ctx->ws_jpsi.p : nullptr, phase,
                             ctx->ws_phi2[1].p));
  release_if_tight(ctx, ctx->ws_psi);
  release_if_tight(ctx, ctx->ws_jpsi);
  release_if_tight(ctx, ctx->ws_phi2[0]);
  std::swap(ctx->ws_phi[0], ctx->ws_phi2[1]);  // Y(0) = [f psi | (1 - f) O psi] starts the propagation
  const int64_t W = n_steps + 1;
  TBPM_TRY(ensure(ctx, ctx->ws_out, sizeof(double) * 2 * (size_t)W * Sh));
  double* C = (double*)ctx->ws_out.p;
  const int tok = phase_begin(ctx, 0);
  TBPM_TRY(launch_xmy(ctx, lat, pl.precision, Sh, alpha, phase, ctx->ws_phi[0].p, 1, pc.state_bytes, C, W, 0));
  int64_t b = req->form == TBPM_SEQUENTIAL ? 1 : req->time_block;
  if (b <= 0) {
    // time the passes on copies, leaving Y(0) in ws_phi[0] untouched
    std::swap(ctx->ws_phi[0], ctx->ws_phi2[0]);
    const int r = choose_block(ctx, lat, &rc, pc, n_steps, &b, nullptr, nullptr);
    std::swap(ctx->ws_phi[0], ctx->ws_phi2[0]);
    release_if_tight(ctx, ctx->ws_phi2[0]);
    release_if_tight(ctx, ctx->ws_psi);
    TBPM_TRY(r);
  }
  BlockHook hook = [&](int64_t start, int bb, const void* first) -> int {
    return launch_xmy(ctx, lat, pl.precision, Sh, alpha, phase, first, bb, pc.state_bytes, C, W, start + 1);
  };
  TBPM_TRY(run_blocks(ctx, lat, &rc, pc, n_steps, b, nullptr, 0.0, hook, ctx->ws_phi[0].p, false));
  phase_end(ctx, tok);
  *d_C = C;
  return TBPM_OK;
}

int copy_rows(tbpm_ctx* ctx, double* dst, const double* src, int S, size_t row_doubles, cudaMemcpyKind kind) {
  TBPM_CK(cudaMemcpyAsync(dst, src, sizeof(double) * row_doubles * S, kind, ctx->stream));
  return TBPM_OK;
}

int run_dos(tbpm_ctx* ctx, tbpm_lattice* lat, const tbpm_request* req, const Plan& pl, const double* d_E,
            int64_t nE, double* d_D) {
  if (nE < 1) {
    set_error("n_energies must be >= 1");
    return TBPM_EINVAL;
  }
  if (req->dos_method == TBPM_DOS_JACKSON) {
    const int64_t M = req->n_moments;
    TBPM_TRY(ensure(ctx, ctx->ws_mu, sizeof(double) * 2 * (size_t)std::max<int64_t>(M, 2) * pl.Spad));
    double* mu = (double*)ctx->ws_mu.p;
    TBPM_TRY(run_moments(ctx, lat, req, pl, M, mu));
    const int tok = phase_begin(ctx, 1);
    const int r = (req->recon == TBPM_RECON_TENSOR)
                      ? launch_dos_jackson_tensor(ctx, mu, pl.S, (int)M, d_E, nE, lat->H0, lat->half, d_D)
                      : launch_dos_jackson_fp64(ctx, mu, pl.S, (int)M, d_E, nE, lat->H0, lat->half, d_D);
    phase_end(ctx, tok);
    return r;
  }
  if (req->dos_method == TBPM_DOS_FOURIER) {
    TBPM_TRY(ensure(ctx, ctx->ws_out, sizeof(double) * 2 * (size_t)(req->n_steps + 1) * pl.Spad));
    double* C = (double*)ctx->ws_out.p;
    TBPM_TRY(run_correlation(ctx, lat, req, pl, C));
    return launch_dos_fourier(ctx, C, pl.S, (int)req->n_steps, d_E, nE, pl.tau / lat->half, req->window, d_D);
  }
  set_error("unknown dos_method %d", req->dos_method);
  return TBPM_EINVAL;
}

}  // namespace

namespace tbpm {
int lattice_ensure_d64(tbpm_lattice* lat) {
  TBPM_TRY(ensure_d64(lat));
  TBPM_CK(cudaStreamSynchronize(lat->ctx->stream));
  return TBPM_OK;
}

int init_request_states(tbpm_ctx* ctx, const tbpm_lattice* lat, const tbpm_request* req, void* dst) {
  Plan pl;
  TBPM_TRY(make_plan(lat, req, &pl));
  return init_states(ctx, lat, req, pl, dst, nullptr);
}
}  // namespace tbpm

// ====================================================================== C ABI: hot path
extern "C" {

int tbpm_states_export(tbpm_ctx* ctx, const tbpm_lattice* lat_c, const tbpm_request* req, void* out,
                       uint32_t* draws) {
  clear_error();
  if (!ctx) {
    set_error("NULL context");
    return TBPM_EINVAL;
  }
  tbpm_lattice* lat = const_cast<tbpm_lattice*>(lat_c);
  Plan pl;
  TBPM_TRY(make_plan(lat, req, &pl));
  TBPM_CK(cudaSetDevice(ctx->device));
  const int64_t n = lat->n_sites;
  TBPM_TRY(ensure(ctx, ctx->ws_phi[0], pl.state_bytes));
  uint32_t* d_draws = nullptr;
  if (draws && req->states == TBPM_STATES_RANDOM) {
    TBPM_TRY(ensure(ctx, ctx->ws_out, sizeof(uint32_t) * (size_t)n * pl.Spad));
    d_draws = (uint32_t*)ctx->ws_out.p;
  }
  TBPM_TRY(init_states(ctx, lat, req, pl, ctx->ws_phi[0].p, d_draws));
  if (out) {
    for (int s = 0; s < pl.S; ++s)
      TBPM_CK(cudaMemcpy2DAsync((char*)out + (size_t)s * n * pl.elem, pl.elem, (const char*)ctx->ws_phi[0].p + s * pl.elem,
                                pl.Spad * pl.elem, pl.elem, n, cudaMemcpyDeviceToHost, ctx->stream));
  }
  if (d_draws)
    TBPM_CK(cudaMemcpyAsync(draws, d_draws, sizeof(uint32_t) * n * pl.S, cudaMemcpyDeviceToHost, ctx->stream));
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  return TBPM_OK;
}

int tbpm_moment_pass_kind(tbpm_ctx* ctx, const tbpm_lattice* lat_c, const tbpm_request* req, int* kind) {
  clear_error();
  if (!ctx || !lat_c || !req || !kind) {
    set_error("tbpm_moment_pass_kind: NULL argument");
    return TBPM_EINVAL;
  }
  tbpm_lattice* lat = const_cast<tbpm_lattice*>(lat_c);
  Plan pl;
  TBPM_TRY(make_plan(lat, req, &pl));
  if (lat->taps && pl.precision == TBPM_C64 && pl.Spad >= 2) {
    *kind = TBPM_PASS_TAPS;
    return TBPM_OK;
  }
  const int m = ctx->fusion;  // -1: autotuned on first use, reported as the mode it would time first
  const int64_t M = req->n_moments > 0 ? req->n_moments : truncation_order_host(req->n_steps * pl.tau);
  if (use_resident(ctx, lat, pl, M / 2)) {
    *kind = TBPM_PASS_RESIDENT;
    return TBPM_OK;
  }
  if (m > 0 && fused_applicable(lat, pl.precision, pl.Spad) && M / 2 - 1 >= fused_steps(m)) {
    const int band = (m == 8 ? 128 : m == 9 ? 192 : 256) / (pl.Spad / 2);
    *kind = (m >= 8 && m <= 10 && lat->geom.Lx >= band) ? TBPM_PASS_SWEEP
            : (m >= 3) ? TBPM_PASS_ROWS : TBPM_PASS_TILES;
    return TBPM_OK;
  }
  if ((m >= 8 || m == -1) && !fused_applicable(lat, pl.precision, pl.Spad) && M / 2 - 1 >= 4 &&
      (sweep_ok(lat, pl) || masked_sweep_ok(lat, pl))) {
    *kind = TBPM_PASS_SWEEP;
    return TBPM_OK;
  }
  *kind = lat->path == TBPM_PATH_CSR ? TBPM_PASS_ELL : TBPM_PASS_STENCIL;
  return TBPM_OK;
}

int tbpm_moments_device(tbpm_ctx* ctx, const tbpm_lattice* lat_c, const tbpm_request* req, double* d_mu) {
  clear_error();
  TBPM_NVTX_CALL(ctx);
  if (!ctx || !d_mu) {
    set_error("NULL argument");
    return TBPM_EINVAL;
  }
  tbpm_lattice* lat = const_cast<tbpm_lattice*>(lat_c);
  Plan pl;
  TBPM_TRY(make_plan(lat, req, &pl));
  TBPM_CK(cudaSetDevice(ctx->device));
  const int64_t M = req->n_moments;
  return with_memory(ctx, [&]() -> int {
    if (pl.Spad == pl.S) return run_moments(ctx, lat, req, pl, M, d_mu);
    TBPM_TRY(ensure(ctx, ctx->ws_mu, sizeof(double) * 2 * (size_t)std::max<int64_t>(M, 2) * pl.Spad));
    TBPM_TRY(run_moments(ctx, lat, req, pl, M, (double*)ctx->ws_mu.p));
    return copy_rows(ctx, d_mu, (double*)ctx->ws_mu.p, pl.S, 2 * (size_t)M, cudaMemcpyDeviceToDevice);
  });
}

int tbpm_moments(tbpm_ctx* ctx, const tbpm_lattice* lat_c, const tbpm_request* req, double* mu) {
  clear_error();
  TBPM_NVTX_CALL(ctx);
  if (!ctx || !mu) {
    set_error("NULL argument");
    return TBPM_EINVAL;
  }
  tbpm_lattice* lat = const_cast<tbpm_lattice*>(lat_c);
  Plan pl;
  TBPM_TRY(make_plan(lat, req, &pl));
  TBPM_CK(cudaSetDevice(ctx->device));
  const int64_t M = req->n_moments;
  TBPM_TRY(with_memory(ctx, [&]() -> int {
    TBPM_TRY(ensure(ctx, ctx->ws_mu, sizeof(double) * 2 * (size_t)std::max<int64_t>(M, 2) * pl.Spad));
    return run_moments(ctx, lat, req, pl, M, (double*)ctx->ws_mu.p);
  }));
  TBPM_TRY(copy_rows(ctx, mu, (double*)ctx->ws_mu.p, pl.S, 2 * (size_t)M, cudaMemcpyDeviceToHost));
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  return sweep_status(ctx);
}

int tbpm_correlation_device(tbpm_ctx* ctx, const tbpm_lattice* lat_c, const tbpm_request* req, double* d_C) {
  clear_error();
  TBPM_NVTX_CALL(ctx);
  if (!ctx || !d_C) {
    set_error("NULL argument");
    return TBPM_EINVAL;
  }
  tbpm_lattice* lat = const_cast<tbpm_lattice*>(lat_c);
  Plan pl;
  TBPM_TRY(make_plan(lat, req, &pl));
  TBPM_CK(cudaSetDevice(ctx->device));
  const size_t row = 2 * (size_t)(req->n_steps + 1);
  TBPM_TRY(fresh_workspaces(ctx));
  return with_memory(ctx, [&]() -> int {
    if (pl.Spad == pl.S) return run_correlation(ctx, lat, req, pl, d_C);
    TBPM_TRY(ensure(ctx, ctx->ws_out, sizeof(double) * row * pl.Spad));
    TBPM_TRY(run_correlation(ctx, lat, req, pl, (double*)ctx->ws_out.p));
    return copy_rows(ctx, d_C, (double*)ctx->ws_out.p, pl.S, row, cudaMemcpyDeviceToDevice);
  });
}

int tbpm_correlation(tbpm_ctx* ctx, const tbpm_lattice* lat_c, const tbpm_request* req, double* C) {
  clear_error();
  TBPM_NVTX_CALL(ctx);
  if (!ctx || !C) {
    set_error("NULL argument");
    return TBPM_EINVAL;
  }
  tbpm_lattice* lat = const_cast<tbpm_lattice*>(lat_c);
  Plan pl;
  TBPM_TRY(make_plan(lat, req, &pl));
  TBPM_CK(cudaSetDevice(ctx->device));
  if (req->n_steps < 1) {
    set_error("n_steps must be >= 1");
    return TBPM_EINVAL;
  }
  const size_t row = 2 * (size_t)(req->n_steps + 1);
  TBPM_TRY(fresh_workspaces(ctx));
  TBPM_TRY(with_memory(ctx, [&]() -> int {
    TBPM_TRY(ensure(ctx, ctx->ws_out, sizeof(double) * row * pl.Spad));
    return run_correlation(ctx, lat, req, pl, (double*)ctx->ws_out.p);
  }));
  TBPM_TRY(copy_rows(ctx, C, (double*)ctx->ws_out.p, pl.S, row, cudaMemcpyDeviceToHost));
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  return sweep_status(ctx);
}

int tbpm_dos_device(tbpm_ctx* ctx, const tbpm_lattice* lat_c, const tbpm_request* req, const double* d_E,
                    int64_t nE, double* d_D) {
  clear_error();
  TBPM_NVTX_CALL(ctx);
  if (!ctx || !d_E || !d_D) {
    set_error("NULL argument");
    return TBPM_EINVAL;
  }
  tbpm_lattice* lat = const_cast<tbpm_lattice*>(lat_c);
  Plan pl;
  TBPM_TRY(make_plan(lat, req, &pl));
  TBPM_CK(cudaSetDevice(ctx->device));
  if (req->dos_method != TBPM_DOS_JACKSON) TBPM_TRY(fresh_workspaces(ctx));
  return with_memory(ctx, [&]() -> int { return run_dos(ctx, lat, req, pl, d_E, nE, d_D); });
}

int tbpm_dos(tbpm_ctx* ctx, const tbpm_lattice* lat_c, const tbpm_request* req, const double* energies,
             int64_t nE, double* D) {
  clear_error();
  TBPM_NVTX_CALL(ctx);
  if (!ctx || !energies || !D) {
    set_error("NULL argument");
    return TBPM_EINVAL;
  }
  tbpm_lattice* lat = const_cast<tbpm_lattice*>(lat_c);
  Plan pl;
  TBPM_TRY(make_plan(lat, req, &pl));
  TBPM_CK(cudaSetDevice(ctx->device));
  if (nE < 1) {
    set_error("n_energies must be >= 1");
    return TBPM_EINVAL;
  }
  if (req->dos_method != TBPM_DOS_JACKSON) TBPM_TRY(fresh_workspaces(ctx));
  double* dD = nullptr;
  TBPM_TRY(with_memory(ctx, [&]() -> int {
    TBPM_TRY(ensure(ctx, ctx->ws_energies, sizeof(double) * (size_t)nE * (1 + pl.S)));
    double* dE = (double*)ctx->ws_energies.p;
    dD = dE + nE;
    TBPM_CK(cudaMemcpyAsync(dE, energies, sizeof(double) * nE, cudaMemcpyHostToDevice, ctx->stream));
    return run_dos(ctx, lat, req, pl, dE, nE, dD);
  }));
  TBPM_CK(cudaMemcpyAsync(D, dD, sizeof(double) * nE * pl.S, cudaMemcpyDeviceToHost, ctx->stream));
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  return sweep_status(ctx);
}

// Adjacency operator y_i = sum_{j in nbr(i)} x_j through the hot-path recurrence kernel
// (first-term mode with zero diagonal and unit hopping); debug export for exact index tests.
int tbpm_apply_hopping(tbpm_ctx* ctx, const tbpm_lattice* lat_c, int precision, int n_states, const void* x,
                       void* y) {
  clear_error();
  if (!ctx || !lat_c || !x || !y) {
    set_error("NULL argument");
    return TBPM_EINVAL;
  }
  tbpm_lattice* lat = const_cast<tbpm_lattice*>(lat_c);
  tbpm_request req;
  memset(&req, 0, sizeof(req));
  req.precision = precision;
  req.n_states = n_states;
  req.states = TBPM_STATES_RANDOM;
  Plan pl;
  TBPM_TRY(make_plan(lat, &req, &pl));
  if (pl.Spad != pl.S) {
    set_error("tbpm_apply_hopping needs a power-of-two number of states");
    return TBPM_EINVAL;
  }
  TBPM_CK(cudaSetDevice(ctx->device));
  TBPM_TRY(ensure(ctx, ctx->ws_phi[0], pl.state_bytes));
  TBPM_TRY(ensure(ctx, ctx->ws_phi[1], pl.state_bytes));
  TBPM_TRY(ensure(ctx, ctx->ws_mu, sizeof(double) * 4 * pl.Spad));
  TBPM_CK(cudaMemcpyAsync(ctx->ws_phi[0].p, x, pl.state_bytes, cudaMemcpyHostToDevice, ctx->stream));
  RecurrenceArgs a;
  TBPM_TRY(base_args(ctx, lat, pl, &a, 3));
  a.diag = nullptr;
  a.diag_const = 0.0;
  a.thop = 1.0;
  set_float_coefficients(&a);
  a.mu = (double*)ctx->ws_mu.p;
  a.M = 2;
  a.cur = ctx->ws_phi[0].p;
  a.prev_out = ctx->ws_phi[1].p;
  TBPM_TRY(launch_moment_step(ctx, a, pl.precision, true));
  TBPM_CK(cudaMemcpyAsync(y, ctx->ws_phi[1].p, pl.state_bytes, cudaMemcpyDeviceToHost, ctx->stream));
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  return TBPM_OK;
}

// Block-size autotuner: measures t_amxsy and t_axpy on this lattice and request, then minimises
// the Tab. I cost model (Sec. II.B) under the memory cap.
int tbpm_block_autotune(tbpm_ctx* ctx, const tbpm_lattice* lat_c, const tbpm_request* req, int64_t n_steps,
                        int64_t* b_opt, double times_ms[2]) {
  clear_error();
  TBPM_NVTX_CALL(ctx);
  if (!ctx || !lat_c || !req || !b_opt || n_steps < 1) {
    set_error("tbpm_block_autotune: invalid argument");
    return TBPM_EINVAL;
  }
  tbpm_lattice* lat = const_cast<tbpm_lattice*>(lat_c);
  Plan pl;
  TBPM_TRY(make_plan(lat, req, &pl));
  TBPM_CK(cudaSetDevice(ctx->device));
  double ta = 0, tx = 0;
  TBPM_TRY(fresh_workspaces(ctx));
  TBPM_TRY(with_memory(ctx, [&]() -> int {
    set_layout(lat, &pl, false);
    TBPM_TRY(take_full_layout(ctx, lat, &pl, 16));
    return choose_block(ctx, lat, req, pl, n_steps, b_opt, &ta, &tx);
  }));
  if (times_ms) {
    times_ms[0] = ta;
    times_ms[1] = tx;
  }
  return sweep_status(ctx);  // the timed passes have ended
}

int tbpm_quasi_eigenstates(tbpm_ctx* ctx, const tbpm_lattice* lat_c, const tbpm_request* req, const double* energies,
                           int64_t nE, void* out) {
  clear_error();
  TBPM_NVTX_CALL(ctx);
  if (!ctx || !energies || !out || nE < 1) {
    set_error("tbpm_quasi_eigenstates: invalid argument");
    return TBPM_EINVAL;
  }
  tbpm_lattice* lat = const_cast<tbpm_lattice*>(lat_c);
  Plan pl;
  TBPM_TRY(make_plan(lat, req, &pl));
  TBPM_CK(cudaSetDevice(ctx->device));
  TBPM_TRY(fresh_workspaces(ctx));
  TBPM_TRY(with_memory(ctx, [&]() -> int {
    TBPM_TRY(ensure(ctx, ctx->ws_energies, sizeof(double) * (size_t)nE));
    TBPM_CK(cudaMemcpyAsync(ctx->ws_energies.p, energies, sizeof(double) * nE, cudaMemcpyHostToDevice, ctx->stream));
    set_layout(lat, &pl, false);
    TBPM_TRY(take_full_layout(ctx, lat, &pl, nE + std::max<int64_t>(16, req->time_block)));
    TBPM_TRY(run_qe(ctx, lat, req, pl, (const double*)ctx->ws_energies.p, (int)nE));
    return pl.full ? ensure(ctx, ctx->ws_phi[0], pl.state_bytes) : TBPM_OK;
  }));
  const int64_t n = lat->n_sites;
  for (int64_t k = 0; k < nE; ++k) {
    const char* block = (const char*)ctx->ws_qe.p + (size_t)k * pl.state_bytes;
    if (pl.full) {  // back to the compact order of the active sites
      const int nb = grid_for(ctx, n * pl.P, kT);
      if (pl.spt == 2)
        k_compact_states<<<nb, kT, 0, ctx->stream>>>(n, pl.P, lat->full_of, (const float4*)block,
                                                     (float4*)ctx->ws_phi[0].p);
      else
        k_compact_states<<<nb, kT, 0, ctx->stream>>>(n, pl.P, lat->full_of, (const float2*)block,
                                                     (float2*)ctx->ws_phi[0].p);
      TBPM_CK_LAUNCH(ctx);
      block = (const char*)ctx->ws_phi[0].p;
    }
    for (int s = 0; s < pl.S; ++s)
      TBPM_CK(cudaMemcpy2DAsync((char*)out + ((size_t)k * pl.S + s) * n * pl.elem, pl.elem, block + s * pl.elem,
                                pl.Spad * pl.elem, pl.elem, n, cudaMemcpyDeviceToHost, ctx->stream));
  }
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  return sweep_status(ctx);
}

int tbpm_conductivity(tbpm_ctx* ctx, const tbpm_lattice* lat_c, const tbpm_request* req, int direction,
                      const double* energies, int64_t nE, double* C, double* sigma) {
  return tbpm_conductivity_overlap(ctx, lat_c, req, direction, energies, nE, C, sigma, nullptr);
}

int tbpm_conductivity_overlap(tbpm_ctx* ctx, const tbpm_lattice* lat_c, const tbpm_request* req, int direction,
                              const double* energies, int64_t nE, double* C, double* sigma, double* overlap) {
  clear_error();
  TBPM_NVTX_CALL(ctx);
  if (!ctx || !energies || !sigma || nE < 1 || nE > 4096) {
    set_error("tbpm_conductivity: invalid argument");
    return TBPM_EINVAL;
  }
  tbpm_lattice* lat = const_cast<tbpm_lattice*>(lat_c);
  if (lat) TBPM_TRY(ensure_ell(ctx, lat));  // the current operator reads the ELL lists
  Plan pl;
  TBPM_TRY(make_plan(lat, req, &pl));
  TBPM_CK(cudaSetDevice(ctx->device));
  double *d_C = nullptr, *d_sigma = nullptr;
  TBPM_TRY(fresh_workspaces(ctx));
  TBPM_TRY(with_memory(ctx, [&]() -> int {
    TBPM_TRY(ensure(ctx, ctx->ws_energies, sizeof(double) * (size_t)nE));
    TBPM_CK(cudaMemcpyAsync(ctx->ws_energies.p, energies, sizeof(double) * nE, cudaMemcpyHostToDevice, ctx->stream));
    return run_ec(ctx, lat, req, pl, (const double*)ctx->ws_energies.p, (int)nE, direction, &d_C, &d_sigma);
  }));
  // rows s*nE + k of the first S states are contiguous
  const size_t rows = (size_t)pl.S * nE;
  if (C)
    TBPM_CK(cudaMemcpyAsync(C, d_C, sizeof(double) * 2 * rows * (req->n_steps + 1), cudaMemcpyDeviceToHost,
                            ctx->stream));
  TBPM_CK(cudaMemcpyAsync(sigma, d_sigma, sizeof(double) * rows, cudaMemcpyDeviceToHost, ctx->stream));
  // <psi|Psi(E)> of every state and energy, [Spad][nE][2] at the head of the EC workspace
  if (overlap)
    TBPM_CK(cudaMemcpyAsync(overlap, ctx->ws_ec.p, sizeof(double) * 2 * rows, cudaMemcpyDeviceToHost, ctx->stream));
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  return sweep_status(ctx);
}

int tbpm_fermi_apply(tbpm_ctx* ctx, const tbpm_lattice* lat_c, const tbpm_request* req, double mu, double kT,
                     int sqrt_f, void* out) {
  clear_error();
  TBPM_NVTX_CALL(ctx);
  if (!ctx || !out) {
    set_error("tbpm_fermi_apply: invalid argument");
    return TBPM_EINVAL;
  }
  tbpm_lattice* lat = const_cast<tbpm_lattice*>(lat_c);
  Plan pl;
  TBPM_TRY(make_plan(lat, req, &pl));
  TBPM_CK(cudaSetDevice(ctx->device));
  TBPM_TRY(fresh_workspaces(ctx));
  TBPM_TRY(with_memory(ctx, [&]() -> int {
    const double* coef = nullptr;
    int nf = 0;
    TBPM_TRY(fermi_series(ctx, lat, mu, kT, sqrt_f ? 1 : 0, &coef, &nf));
    TBPM_TRY(ensure(ctx, ctx->ws_phi[0], pl.state_bytes));
    TBPM_TRY(ensure(ctx, ctx->ws_phi[1], pl.state_bytes));
    TBPM_TRY(ensure(ctx, ctx->ws_phi2[0], pl.state_bytes));
    TBPM_TRY(init_states(ctx, lat, req, pl, ctx->ws_phi[0].p, nullptr));
    return apply_series_bufs(ctx, lat, pl, ctx->ws_phi[0].p, ctx->ws_phi[1].p, ctx->ws_phi2[0].p, coef, nf);
  }));
  const int64_t n = lat->n_sites;
  for (int s = 0; s < pl.S; ++s)
    TBPM_CK(cudaMemcpy2DAsync((char*)out + (size_t)s * n * pl.elem, pl.elem,
                              (const char*)ctx->ws_phi2[0].p + s * pl.elem, pl.Spad * pl.elem, pl.elem, n,
                              cudaMemcpyDeviceToHost, ctx->stream));
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  return sweep_status(ctx);
}

namespace {
// Shared checks and the state-chunk loop of the OC, DP and CD entry points: `pass` runs the
// request's states s0 .. s0 + k - 1 with the chunk's plan.
int response_chunks(tbpm_ctx* ctx, tbpm_lattice* lat, const tbpm_request* req, int64_t min_steps,
                    double pair_blocks, const std::function<int(const tbpm_request*, const Plan&)>& pass) {
  Plan pl;
  TBPM_TRY(make_plan(lat, req, &pl));
  if (req->n_steps < min_steps || req->n_steps > (1 << 22)) {
    set_error("n_steps must lie in [%lld, 2^22]", (long long)min_steps);
    return TBPM_EINVAL;
  }
  if (req->form != TBPM_SEQUENTIAL && req->form != TBPM_CONCURRENT_S) {
    set_error("this quantity takes the SEQUENTIAL or CONCURRENT_S form");
    return TBPM_EINVAL;
  }
  int cap = std::min(pl.Spad, 16);
  if (ctx->max_pass_states > 0)
    while (cap > ctx->max_pass_states) cap >>= 1;
  TBPM_TRY(fresh_workspaces(ctx));
  const int k = states_per_pass(ctx, lat, pl.elem, cap, pair_blocks);
  if (k < 1) {
    set_error("not enough device memory for one state of %lld sites", (long long)lat->n_sites);
    return TBPM_ENOMEM;
  }
  for (int s0 = 0; s0 < pl.S; s0 += k) {
    tbpm_request rq = *req;
    rq.n_states = std::min(k, pl.S - s0);
    if (req->states == TBPM_STATES_SITES) rq.sites = req->sites + s0;
    Plan pk;
    TBPM_TRY(make_plan(lat, &rq, &pk));
    pk.s0 = s0;
    TBPM_TRY(with_memory(ctx, [&]() -> int { return pass(&rq, pk); }));
  }
  return TBPM_OK;
}
}  // namespace

int tbpm_optical_conductivity(tbpm_ctx* ctx, const tbpm_lattice* lat_c, const tbpm_request* req, int alpha,
                              int beta, double mu, double kT, double omega_max, int64_t n_omega, double* C,
                              double* sigma) {
  clear_error();
  TBPM_NVTX_CALL(ctx);
  if (!ctx || !req || !sigma || n_omega < 2 || n_omega > (1 << 20) || !(omega_max > 0.0)) {
    set_error("tbpm_optical_conductivity: invalid argument (n_omega in [2, 2^20], omega_max > 0)");
    return TBPM_EINVAL;
  }
  tbpm_lattice* lat = const_cast<tbpm_lattice*>(lat_c);
  if (!lat) {
    set_error("tbpm_optical_conductivity: lattice is NULL");
    return TBPM_EINVAL;
  }
  TBPM_TRY(ensure_ell(ctx, lat));  // the current operator reads the ELL lists
  const int dims = lat->desc.kind == TBPM_CUBIC ? 3 : 2;
  if (alpha < 0 || alpha >= dims || beta < 0 || beta >= dims) {
    set_error("directions must lie in [0, %d)", dims);
    return TBPM_EINVAL;
  }
  TBPM_CK(cudaSetDevice(ctx->device));
  const double area = lat->desc.kind == TBPM_HONEYCOMB ? 3.0 * sqrt(3.0) / 4.0 : 1.0;
  const int64_t W = req->n_steps + 1;
  const double q0[3] = {0, 0, 0};
  // 3 pair blocks = 6 single blocks live at a time, plus room for b >= 2 accumulators
  return response_chunks(ctx, lat, req, 1, 8.0, [&](const tbpm_request* rq, const Plan& pk) -> int {
    double* d_C = nullptr;
    double tphys = 0.0;
    TBPM_TRY(run_response(ctx, lat, rq, pk, 0, alpha, beta, q0, mu, kT, &d_C, &tphys));
    TBPM_TRY(ensure(ctx, ctx->ws_recon, sizeof(double) * 2 * (size_t)n_omega * pk.S));
    double* d_sig = (double*)ctx->ws_recon.p;
    TBPM_TRY(launch_oc_spectrum(ctx, d_C, pk.S, (int)rq->n_steps, omega_max / (double)(n_omega - 1), (int)n_omega,
                                kT, tphys, area, rq->window, d_sig));
    if (C)
      TBPM_CK(cudaMemcpyAsync(C + 2 * (size_t)pk.s0 * W, d_C, sizeof(double) * 2 * (size_t)pk.S * W,
                              cudaMemcpyDeviceToHost, ctx->stream));
    TBPM_CK(cudaMemcpyAsync(sigma + 2 * (size_t)pk.s0 * n_omega, d_sig, sizeof(double) * 2 * (size_t)pk.S * n_omega,
                            cudaMemcpyDeviceToHost, ctx->stream));
    TBPM_CK(cudaStreamSynchronize(ctx->stream));
    return sweep_status(ctx);
  });
}

int tbpm_polarization(tbpm_ctx* ctx, const tbpm_lattice* lat_c, const tbpm_request* req, const double q[3], double mu,
                      double kT, const double* omegas, int64_t n_omega, double* C, double* Pi) {
  clear_error();
  TBPM_NVTX_CALL(ctx);
  if (!ctx || !req || !q || !omegas || !Pi || n_omega < 1 || n_omega > (1 << 20)) {
    set_error("tbpm_polarization: invalid argument");
    return TBPM_EINVAL;
  }
  tbpm_lattice* lat = const_cast<tbpm_lattice*>(lat_c);
  TBPM_CK(cudaSetDevice(ctx->device));
  const double area = lat->desc.kind == TBPM_HONEYCOMB ? 3.0 * sqrt(3.0) / 4.0 : 1.0;
  const int64_t W = req->n_steps + 1;
  return response_chunks(ctx, lat, req, 1, 8.0, [&](const tbpm_request* rq, const Plan& pk) -> int {
    double* d_C = nullptr;
    double tphys = 0.0;
    TBPM_TRY(run_response(ctx, lat, rq, pk, 1, 0, 0, q, mu, kT, &d_C, &tphys));
    TBPM_TRY(ensure(ctx, ctx->ws_energies, sizeof(double) * (size_t)n_omega));
    TBPM_CK(cudaMemcpyAsync(ctx->ws_energies.p, omegas, sizeof(double) * n_omega, cudaMemcpyHostToDevice,
                            ctx->stream));
    TBPM_TRY(ensure(ctx, ctx->ws_recon, sizeof(double) * 2 * (size_t)n_omega * pk.S));
    double* d_pi = (double*)ctx->ws_recon.p;
    TBPM_TRY(launch_dp_spectrum(ctx, d_C, pk.S, (int)rq->n_steps, (const double*)ctx->ws_energies.p, (int)n_omega,
                                tphys, area, rq->window, d_pi));
    if (C)
      TBPM_CK(cudaMemcpyAsync(C + 2 * (size_t)pk.s0 * W, d_C, sizeof(double) * 2 * (size_t)pk.S * W,
                              cudaMemcpyDeviceToHost, ctx->stream));
    TBPM_CK(cudaMemcpyAsync(Pi + 2 * (size_t)pk.s0 * n_omega, d_pi, sizeof(double) * 2 * (size_t)pk.S * n_omega,
                            cudaMemcpyDeviceToHost, ctx->stream));
    TBPM_CK(cudaStreamSynchronize(ctx->stream));
    return sweep_status(ctx);
  });
}

int tbpm_charge_density(tbpm_ctx* ctx, const tbpm_lattice* lat_c, const tbpm_request* req, double mu, double kT,
                        double* rho) {
  clear_error();
  TBPM_NVTX_CALL(ctx);
  if (!ctx || !req || !rho) {
    set_error("tbpm_charge_density: invalid argument");
    return TBPM_EINVAL;
  }
  tbpm_lattice* lat = const_cast<tbpm_lattice*>(lat_c);
  TBPM_CK(cudaSetDevice(ctx->device));
  double tau = req->tau;
  if (tau == 0.0) {
    const double occ = std::min(lat->E_max, mu + 20.0 * kT) - lat->E_min;
    if (!(occ > 0.0)) {
      set_error("charge density: no occupied states below mu");
      return TBPM_EINVAL;
    }
    tau = M_PI * lat->half / occ;
  }
  const int64_t n = lat->n_sites;
  // live: three state blocks in the series, then 2 + b blocks and the FP64 accumulator (2 blocks)
  return response_chunks(ctx, lat, req, 0, 6.0, [&](const tbpm_request* rq, const Plan& pl) -> int {
    Plan pc = pl;
    pc.tau = tau;
    const double* coef = nullptr;
    int nf = 0;
    TBPM_TRY(fermi_series(ctx, lat, mu, kT, 1, &coef, &nf));
    TBPM_TRY(ensure(ctx, ctx->ws_phi[0], pl.state_bytes));
    TBPM_TRY(ensure(ctx, ctx->ws_phi[1], pl.state_bytes));
    TBPM_TRY(ensure(ctx, ctx->ws_phi2[0], pl.state_bytes));
    TBPM_TRY(init_states(ctx, lat, rq, pl, ctx->ws_phi[0].p, nullptr));
    // phi = f^{1/2}(H) psi into ws_phi2[0], consuming psi in ws_phi[0]
    TBPM_TRY(apply_series_bufs(ctx, lat, pl, ctx->ws_phi[0].p, ctx->ws_phi[1].p, ctx->ws_phi2[0].p, coef, nf));
    std::swap(ctx->ws_phi[0], ctx->ws_phi2[0]);
    release_if_tight(ctx, ctx->ws_phi2[0]);
    const int64_t elems = n * pl.Spad;
    TBPM_TRY(ensure(ctx, ctx->ws_ec, sizeof(double) * (size_t)elems));
    double* z = (double*)ctx->ws_ec.p;
    TBPM_CK(cudaMemsetAsync(z, 0, sizeof(double) * (size_t)elems, ctx->stream));
    const int tok = phase_begin(ctx, 0);
    TBPM_TRY(launch_abs2py(ctx, pl.precision, ctx->ws_phi[0].p, 1, pl.state_bytes, elems, 0.5, z));
    if (rq->n_steps >= 1) {
      int64_t b = rq->form == TBPM_SEQUENTIAL ? 1 : rq->time_block;
      if (b <= 0) {
        std::swap(ctx->ws_phi[0], ctx->ws_phi2[0]);
        const int r = choose_block(ctx, lat, rq, pc, rq->n_steps, &b, nullptr, nullptr);
        std::swap(ctx->ws_phi[0], ctx->ws_phi2[0]);
        release_if_tight(ctx, ctx->ws_phi2[0]);
        release_if_tight(ctx, ctx->ws_psi);
        TBPM_TRY(r);
      }
      BlockHook hook = [&](int64_t, int bb, const void* first) -> int {
        return launch_abs2py(ctx, pl.precision, first, bb, pl.state_bytes, elems, 1.0, z);
      };
      TBPM_TRY(run_blocks(ctx, lat, rq, pc, rq->n_steps, b, nullptr, 0.0, hook, ctx->ws_phi[0].p, false));
    }
    phase_end(ctx, tok);
    TBPM_TRY(ensure(ctx, ctx->ws_out, sizeof(double) * (size_t)n * pl.S));
    const double wsum = 0.5 + (double)rq->n_steps;
    TBPM_TRY(launch_cd_finish(ctx, z, n, pl.S, pl.Spad, (double)n / wsum, (double*)ctx->ws_out.p));
    TBPM_CK(cudaMemcpyAsync(rho + (size_t)pl.s0 * n, ctx->ws_out.p, sizeof(double) * (size_t)n * pl.S,
                            cudaMemcpyDeviceToHost, ctx->stream));
    TBPM_CK(cudaStreamSynchronize(ctx->stream));
    return sweep_status(ctx);
  });
}

// ---------------------------------------------------------------- cost model (Sec. II.B, Tab. I)
int tbpm_block_counts(int64_t n_steps, int64_t b, double tau, int64_t out[3]) {
  clear_error();
  if (n_steps < 1 || b < 1 || !out || !(tau > 0)) {
    set_error("tbpm_block_counts: invalid argument");
    return TBPM_EINVAL;
  }
  int64_t amxsy = 0, axpy = 0;
  std::vector<int64_t> N(std::min(b, n_steps) + 1);
  for (int64_t j = 1; j <= std::min(b, n_steps); ++j) N[j] = truncation_order_host(j * tau);
  for (int64_t start = 0; start < n_steps; start += b) {
    const int64_t bb = std::min(b, n_steps - start);
    int64_t mx = 0;
    for (int64_t j = 1; j <= bb; ++j) {
      axpy += N[j];
      mx = std::max(mx, N[j]);
    }
    amxsy += mx;
  }
  out[0] = amxsy;
  out[1] = axpy;
  out[2] = n_steps;
  return TBPM_OK;
}

int64_t tbpm_block_opt(int64_t n_steps, double tau, double t_amxsy, double t_axpy, int64_t b_max) {
  clear_error();
  if (n_steps < 1 || !(tau > 0)) return 1;
  b_max = std::max<int64_t>(1, std::min(b_max, n_steps));
  std::vector<int64_t> N(b_max + 1), pre(b_max + 1, 0);
  for (int64_t j = 1; j <= b_max; ++j) {
    N[j] = truncation_order_host(j * tau);
    pre[j] = pre[j - 1] + N[j];
  }
  int64_t best = 1;
  double best_c = -1;
  for (int64_t b = 1; b <= b_max; ++b) {
    const int64_t full = n_steps / b, rest = n_steps % b;
    const double am = (double)full * N[b] + (rest ? (double)N[rest] : 0.0);
    const double ax = (double)full * pre[b] + (rest ? (double)pre[rest] : 0.0);
    const double c = am * t_amxsy + ax * t_axpy;
    if (best_c < 0 || c < best_c) {
      best_c = c;
      best = b;
    }
  }
  return best;
}

}  // extern "C"
