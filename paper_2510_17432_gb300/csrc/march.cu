// One Chebyshev step on the simple-cubic stencil as a march along z, with or without the moment inner
// products: phi_{n+1} = 2 H~ phi_n - phi_{n-1} (phi_1 = H~ phi_0).
//
// A CTA owns a tile of TX x TY columns and up to four state pairs of each, and walks a segment of planes.
// Planes of phi_n (with a rim of one column), phi_{n-1} and D stream through shared-memory rings by
// cp.async, kAhead planes ahead; a thread takes its four neighbours in the plane and its own unit of the
// next plane from the ring and keeps the one of the plane before in a register.  One barrier per plane.
// A unit so costs two copies and a store plus its share of the rim, where the line-by-line pass gathered
// six neighbours through L1 with 64-bit offsets each (270 instructions per unit and warp), and the bytes in
// flight do not depend on registers: with the loads of one plane ahead in registers the same march took as
// long as the line pass.
//
// Bound: shared-memory instructions (the copies and six reads of a unit) at about 0.6 of HBM's copy rate.
// Measured, us per step, line pass -> march: 101 x 103 x 99, 32 states 243 -> 195; 150^3, one state 81 -> 42;
// 20 x 300 x 300, 4 states (short lines) 251 -> 41; 128^3, 8 states 110 -> 97; 100 x 90 x 80, 4 complex128
// states 188 -> 122.
// The row sweep's temporal blocking is not carried over: with four steps per pass a tile would need a rim
// of four columns on each side (a 16 x 8 tile would form 3 times its own columns).
#include <cuda_runtime.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "stencil.cuh"
#include "tbpm_internal.cuh"

namespace tbpm {
namespace {

constexpr int kAhead = 2;            // planes copied ahead of the one that is needed next
constexpr int kSlots = kAhead + 2;   // the plane in use, the next one, and those ahead (a power of two)

struct MarchArgs {
  const void* cur;
  const void* prev;
  void* out;
  const void* diag;
  double th, dc;       // coefficients of this step (x2 past the first)
  float thf, dcf;
  int64_t Lx, Ly, Lz;
  int pbc_x, pbc_y, pbc_z;
  int P, logPC, logTX, logTY;
  int ntx, ntiles, nch, nz, zlen;
  // moments
  double* partials;    // [gridDim.x][PC SPT 2]
  unsigned* counter;
  double* mu;
  int M, step;
};

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double2 add2(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 fma2(float a, float2 x, float2 y) { return __ffma2_rn(make_float2(a, a), x, y); }
__device__ __forceinline__ double2 fma2(double a, double2 x, double2 y) {
  return make_double2(fma(a, x.x, y.x), fma(a, x.y, y.y));
}
__device__ __forceinline__ float2 fma2(float2 a, float2 x, float2 y) { return __ffma2_rn(a, x, y); }
__device__ __forceinline__ double2 fma2(double2 a, double2 x, double2 y) {
  return make_double2(fma(a.x, x.x, y.x), fma(a.y, x.y, y.y));
}

// B bytes (4, 8 or 16) from global to shared memory (a shared-space address), n of them data and the rest zeros
template <int B>
__device__ __forceinline__ void copy_async(uint32_t d, const void* src, uint32_t n) {
  if constexpr (B == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], %3, %2;" ::"r"(d), "l"(src), "r"(n), "n"(B) : "memory");
}

template <typename R, int SPT, bool FIRST, bool MOM>
__global__ void __launch_bounds__(kThreads, 4) k_cubic_march(MarchArgs a) {
  using V2 = std::conditional_t<sizeof(R) == 4, float2, double2>;
  struct __align__(sizeof(V2) * SPT) PK {  // SPT complex numbers
    V2 c[SPT];
  };
  constexpr int NV = 2 * SPT;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ double red[kWarps][8][NV];
  __shared__ unsigned ticket;
  const PK* cur = reinterpret_cast<const PK*>(a.cur);
  const PK* prev = reinterpret_cast<const PK*>(a.prev);
  PK* out = reinterpret_cast<PK*>(a.out);
  const R* diag = reinterpret_cast<const R*>(a.diag);
  const int logPC = a.logPC, PC = 1 << logPC, TX = 1 << a.logTX, TY = 1 << a.logTY, tid = threadIdx.x;
  const int pitch = (TX + 2) << logPC, slice = (TY + 2) * pitch;
  PK* plane = reinterpret_cast<PK*>(smraw);                              // [kSlots][slice]
  PK* pring = plane + kSlots * slice;                                        // phi_{n-1}: [kSlots][kThreads]
  R* dring = reinterpret_cast<R*>(pring + (FIRST ? 0 : kSlots * kThreads));  // D: [kSlots][kThreads]
  // the chunks of a tile run side by side: a chunk's 64-byte run is half of a 128-byte line, which L2 fetches whole
  const int chunk = blockIdx.x % a.nch, rest = blockIdx.x / a.nch;
  const int tile = rest % a.ntiles, zs = rest / a.ntiles;
  const int64_t x0 = (int64_t)(tile % a.ntx) << a.logTX, y0 = (int64_t)(tile / a.ntx) << a.logTY;
  const int w = (int)min((int64_t)TX, a.Lx - x0), h = (int)min((int64_t)TY, a.Ly - y0);  // columns of this tile
  const int p = tid & (PC - 1), x = (tid >> logPC) & (TX - 1), y = tid >> (logPC + a.logTX);
  const bool own = x < w && y < h;
  const int64_t pstride = a.Lx * a.Ly * a.P;  // units per plane
  const int64_t n_units = a.Lz * pstride;     // debug build: every unit's index is checked against it
  const int64_t site = (y0 + y) * a.Lx + x0 + x;  // within a plane
  const int64_t oo = site * a.P + (chunk << logPC) + p;
  const int so = ((y + 1) * (TX + 2) + x + 1) * PC + p;
  // the rim: columns above, below, left and right of the tile; its right edge is at column w, its upper at row h
  const int k = tid >> logPC;
  int rx = 0, ry = 0;
  bool rim = true;
  if (k < w) { rx = k; ry = -1; }
  else if (k < 2 * w) { rx = k - w; ry = h; }
  else if (k < 2 * w + h) { rx = -1; ry = k - 2 * w; }
  else if (k < 2 * (w + h)) { rx = w; ry = k - 2 * w - h; }
  else rim = false;
  const int sr = ((ry + 1) * (TX + 2) + rx + 1) * PC + p;
  bool rim_data = rim;
  int64_t ro = 0;
  {
    int64_t gx = x0 + rx, gy = y0 + ry;
    if (gx < 0 || gx >= a.Lx) {
      rim_data = rim_data && a.pbc_x;
      gx = gx < 0 ? gx + a.Lx : gx - a.Lx;
    }
    if (gy < 0 || gy >= a.Ly) {
      rim_data = rim_data && a.pbc_y;
      gy = gy < 0 ? gy + a.Ly : gy - a.Ly;
    }
    ro = (gy * a.Lx + gx) * a.P + (chunk << logPC) + p;
  }
  const int Lz = (int)a.Lz, z0 = zs * a.zlen, z1 = min(z0 + a.zlen, Lz);
  const R th = sizeof(R) == 4 ? (R)a.thf : (R)a.th, dc = sizeof(R) == 4 ? (R)a.dcf : (R)a.dc;
  // running sources of the copies of phi_n, one plane at a time: plane zc, own unit and rim; nothing (zeros)
  // beyond an open boundary, back to plane 0 beyond a periodic one
  const PK* src_own = cur + (own ? oo : 0) + z0 * pstride;
  const PK* src_rim = cur + (rim_data ? ro : 0) + z0 * pstride;
  const uint32_t sm = (uint32_t)__cvta_generic_to_shared(smraw);
  const uint32_t d_own = sm + (uint32_t)(so * sizeof(PK)), d_rim = sm + (uint32_t)(sr * sizeof(PK));
  const uint32_t slice_bytes = (uint32_t)(slice * sizeof(PK));
  int zc = z0;
  uint32_t n_own = sizeof(PK), n_rim = rim_data ? sizeof(PK) : 0;  // bytes with data
  auto copy_plane = [&](int slot) {
    if (zc > z1) return;  // the segment's last plane needs the one above it, no further
    if (zc == Lz) {
      src_own -= a.Lz * pstride;
      src_rim -= a.Lz * pstride;
      if (!a.pbc_z) n_own = n_rim = 0;
    }
    if (own && (n_own == 0 || TBPM_DBG_OK(src_own - cur, n_units, TBPM_DBG_MARCH)))
      copy_async<sizeof(PK)>(d_own + slot * slice_bytes, src_own, n_own);
    if (rim && (n_rim == 0 || TBPM_DBG_OK(src_rim - cur, n_units, TBPM_DBG_MARCH)))
      copy_async<sizeof(PK)>(d_rim + slot * slice_bytes, src_rim, n_rim);
    src_own += pstride;
    src_rim += pstride;
    ++zc;
  };
  PK m1{}, c0{};
  if (own && (z0 > 0 || a.pbc_z) && TBPM_DBG_OK(oo + (z0 > 0 ? z0 - 1 : Lz - 1) * pstride, n_units, TBPM_DBG_MARCH)) m1 = cur[oo + (z0 > 0 ? z0 - 1 : Lz - 1) * pstride];
  // phi_{n-1} and D of plane zo: each thread its own
  const PK* pp = prev + (own ? oo : 0) + z0 * pstride;
  const R* dp = diag ? diag + (own ? site : 0) + z0 * (a.Lx * a.Ly) : nullptr;
  const uint32_t d_prev = (uint32_t)__cvta_generic_to_shared(pring + tid), d_d = (uint32_t)__cvta_generic_to_shared(dring + tid);
  int zo = z0;
  auto copy_own = [&](int slot) {
    if (own && zo < z1) {
      if (!FIRST && TBPM_DBG_OK(pp - prev, n_units, TBPM_DBG_MARCH)) copy_async<sizeof(PK)>(d_prev + slot * (uint32_t)(kThreads * sizeof(PK)), pp, sizeof(PK));
      if (diag && TBPM_DBG_OK(dp - diag, a.Lz * a.Lx * a.Ly, TBPM_DBG_MARCH)) copy_async<sizeof(R)>(d_d + slot * (uint32_t)(kThreads * sizeof(R)), dp, sizeof(R));
    }
    pp += pstride;
    dp += a.Lx * a.Ly;
    ++zo;
  };
  // groups in flight: plane z0, then (plane z0 + 1 + k, own data of z0 + k) for k = 0 .. kAhead
  copy_plane(0);
#pragma unroll
  for (int k2 = 0; k2 < kAhead; ++k2) {
    copy_plane(1 + k2);
    copy_own(k2);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory");
  __syncthreads();  // plane z0 (in the first group) is there for everybody
  if (own) c0 = plane[so];
  PK* dst = out + oo + z0 * pstride;
  V2 acc[NV];       // packed halves of this thread's sums over at most 32 planes
  double tot[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    acc[q] = V2{};
    tot[q] = 0.0;
  }
  auto fold = [&]() {
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      tot[q] += (double)(acc[q].x + acc[q].y);
      acc[q] = V2{};
    }
  };
  int folded = 0;
  for (int zb = z0; zb < z1; zb += kSlots) {
#pragma unroll
    for (int s0 = 0; s0 < kSlots; ++s0) {  // plane z = zb + s0 in slot s0
      if (zb + s0 >= z1) break;
      constexpr int kWrap = kSlots - 1;
      // the slot of plane z - 1 is free since the last barrier
      copy_plane((s0 + 1 + kAhead) & kWrap);
      copy_own((s0 + kAhead) & kWrap);
      asm volatile("cp.async.commit_group;" ::: "memory");
      // own copies of plane z + 1 and of phi_{n-1}, D of z
      asm volatile("cp.async.wait_group %0;" ::"n"(kAhead) : "memory");
      if (own) {
        const PK* s = plane + s0 * slice + so;
        const PK p1 = plane[((s0 + 1) & kWrap) * slice + so];
        const PK xp = s[PC], xm = s[-PC], yp = s[pitch], ym = s[-pitch];
        R d = dc;
        if (diag) {
          d = dring[s0 * kThreads + tid];
          if (!FIRST) d = d + d;
        }
        PK pv{};
        if (!FIRST) pv = pring[s0 * kThreads + tid];
        PK o;
#pragma unroll
        for (int q = 0; q < SPT; ++q) {
          const V2 hs = add2(add2(add2(add2(add2(xp.c[q], xm.c[q]), yp.c[q]), ym.c[q]), p1.c[q]), m1.c[q]);
          V2 neg = pv.c[q];
          neg.x = -neg.x;
          neg.y = -neg.y;
          o.c[q] = fma2(d, c0.c[q], fma2(th, hs, neg));
          if constexpr (MOM) {
            acc[2 * q] = fma2(c0.c[q], c0.c[q], acc[2 * q]);
            acc[2 * q + 1] = fma2(o.c[q], c0.c[q], acc[2 * q + 1]);
          }
        }
        if (TBPM_DBG_OK(dst - out, n_units, TBPM_DBG_MARCH)) {
          if constexpr (sizeof(PK) == 16 && sizeof(R) == 4) __stcs(reinterpret_cast<float4*>(dst), *reinterpret_cast<const float4*>(&o));
          else __stcs(reinterpret_cast<V2*>(dst), o.c[0]);
        }
        m1 = c0;
        c0 = p1;
      }
      if (MOM && ++folded == 32) {
        folded = 0;
        fold();
      }
      dst += pstride;
      __syncthreads();  // plane z + 1 is there for everybody; plane z's slot may be filled again
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  fold();
  if constexpr (MOM) {
    // CTA sums per pair of the chunk, FP64, in a fixed order; the last CTA adds them over the CTAs of each chunk
    const int lane = tid & 31, warp = tid >> 5;
    double v[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = tot[q];
#pragma unroll
    for (int q = 0; q < NV; ++q)
      for (int off = 16; off >= PC; off >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], off);
    if (lane < PC)
#pragma unroll
      for (int q = 0; q < NV; ++q) red[warp][lane][q] = v[q];
    __syncthreads();
    const int per = PC * NV;
    if (tid < per) {
      double t = 0.0;
      for (int k2 = 0; k2 < kWarps; ++k2) t += red[k2][tid / NV][tid % NV];
      a.partials[(size_t)blockIdx.x * per + tid] = t;
      __threadfence();
    }
    __syncthreads();
    if (tid == 0) ticket = atomicAdd(a.counter, 1u);
    __syncthreads();
    if (ticket != gridDim.x - 1) return;
    __threadfence();
    const int blocks = a.ntiles * a.nz;  // CTAs of a chunk: every nch-th
    for (int q = warp; q < a.P * NV; q += kWarps) {
      const int pair = q / NV, c = pair >> logPC, i = (pair & (PC - 1)) * NV + q % NV;
      double t = 0.0;
      for (int b = lane; b < blocks; b += 32) t += __ldcg(a.partials + ((size_t)b * a.nch + c) * per + i);
      for (int off = 16; off >= 1; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
      if (lane == 0) {  // q = 2 s + comp: the odd inner product is real
        const int s = q >> 1, comp = q & 1, n = a.step;
        double* ms = a.mu + (size_t)s * a.M * 2 + 2 * comp;
        ms[4 * n] = FIRST ? t : 2.0 * t - ms[0];
        ms[4 * n + 1] = FIRST ? 0.0 : -ms[1];
      }
    }
    if (tid == 0) *a.counter = 0u;
  }
}

template <typename R, int SPT, bool MOM>
void* march_fn(bool first) {
  return first ? (void*)k_cubic_march<R, SPT, true, MOM> : (void*)k_cubic_march<R, SPT, false, MOM>;
}

}  // namespace

// One cubic step (moments: with the inner products of step ra.step): ra.cur, ra.prev_out -> ra.next or ra.prev_out.
int launch_cubic_march(tbpm_ctx* ctx, const RecurrenceArgs& ra, int precision, bool first, bool moments) {
  MarchArgs a;
  memset(&a, 0, sizeof(a));
  a.cur = ra.cur;
  a.prev = ra.prev_out;
  a.out = ra.next ? ra.next : ra.prev_out;
  a.diag = ra.diag;
  a.th = first ? ra.thop : 2.0 * ra.thop;
  a.dc = first ? ra.diag_const : 2.0 * ra.diag_const;
  a.thf = first ? ra.th1f : ra.th2f;
  a.dcf = first ? ra.dc1f : ra.dc2f;
  a.Lx = ra.geom.Lx;
  a.Ly = ra.geom.Ly;
  a.Lz = ra.geom.Lz;
  a.pbc_x = ra.geom.pbc_x;
  a.pbc_y = ra.geom.pbc_y;
  a.pbc_z = ra.geom.pbc_z;
  a.P = ra.P;
  const int spt = precision == TBPM_C64 && ra.S >= 2 ? 2 : 1;
  // up to four units of a site per CTA (a 64-byte run); the tile that wastes the fewest threads at the
  // lattice's edges, the wider one of two equals
  while ((1 << a.logPC) < std::min(4, ra.P)) ++a.logPC;
  double best = -1.0;
  for (int lx = 6; lx >= 2; --lx) {
    const int ly = 8 - a.logPC - lx;
    if (ly < 2 || ly > 6) continue;  // at least 4 x 4 columns: the rim has at most as many as the tile
    const int64_t tx = (a.Lx + (1 << lx) - 1) >> lx, ty = (a.Ly + (1 << ly) - 1) >> ly;
    const double rim = 1.0 / (1 << lx) + 1.0 / (1 << ly);
    const double eff = (double)(a.Lx * a.Ly) / (double)((tx << lx) * (ty << ly)) / (1.0 + 0.5 * rim);
    if (eff > best + 1e-9) {
      best = eff;
      a.logTX = lx;
      a.logTY = ly;
    }
  }
  const int64_t ntx = (a.Lx + (1 << a.logTX) - 1) >> a.logTX, nty = (a.Ly + (1 << a.logTY) - 1) >> a.logTY;
  const int64_t chunks = ra.P >> a.logPC, cols = ntx * nty * chunks;
  if (cols > 1 << 24) return TBPM_EUNSUPPORTED;  // the caller takes the line pass
  // segments of planes: as many as fill whole waves of the resident CTAs best, against two more planes read each
  const size_t unit = precision == TBPM_C64 ? 8 * (size_t)spt : 16;
  const size_t smem = kSlots * (unit * ((size_t)((1 << a.logTX) + 2) * ((1 << a.logTY) + 2) << a.logPC) +
                                (first ? 0 : unit * kThreads) + (ra.diag ? unit / (2 * spt) * kThreads : 0));
  void* fn;
  if (precision == TBPM_C128) fn = moments ? march_fn<double, 1, true>(first) : march_fn<double, 1, false>(first);
  else if (spt == 2) fn = moments ? march_fn<float, 2, true>(first) : march_fn<float, 2, false>(first);
  else fn = moments ? march_fn<float, 1, true>(first) : march_fn<float, 1, false>(first);
  TBPM_CK(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024));
  const int64_t slots = (int64_t)ctx->num_sms * std::max<int64_t>(1, std::min<int64_t>(4, (220 << 10) / (int64_t)smem));
  int64_t nz = 1;
  best = -1.0;
  for (int64_t k = 1; k <= std::min<int64_t>(a.Lz, 4 * slots / cols + 2); ++k) {
    const int64_t len = (a.Lz + k - 1) / k, segs = (a.Lz + len - 1) / len, ctas = cols * segs;
    const int64_t waves = (ctas + slots - 1) / slots;
    const double eff = (double)ctas / (double)(waves * slots) * (double)len / (double)(len + 2);
    if (eff > best + 1e-9) {
      best = eff;
      nz = k;
    }
  }
  a.ntx = (int)ntx;
  a.ntiles = (int)(ntx * nty);
  a.nch = (int)chunks;
  a.zlen = (int)((a.Lz + nz - 1) / nz);
  a.nz = (int)((a.Lz + a.zlen - 1) / a.zlen);
  const int64_t grid = cols * a.nz;
  const int PC = 1 << a.logPC;
  if (moments) {
    TBPM_TRY(ensure(ctx, ctx->ws_fused_partials, sizeof(double) * (size_t)grid * PC * spt * 2));
    a.partials = (double*)ctx->ws_fused_partials.p;
    a.counter = ra.counter;
    a.mu = ra.mu;
    a.M = ra.M;
    a.step = ra.step;
  }
  void* args[] = {&a};
  const cudaError_t e = cudaLaunchKernel(fn, dim3((unsigned)grid), dim3(kThreads), args, smem, ctx->stream);
  ctx->launches++;
  if (e != cudaSuccess) {
    set_error("kernel launch: %s", cudaGetErrorString(e));
    return TBPM_ECUDA;
  }
  return TBPM_OK;
}

}  // namespace tbpm

TBPM_DEBUG_UNIT(march)
