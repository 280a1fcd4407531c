// Matrix-free moment pass for clean long-range lattices (square and honeycomb): H applied
// from the lattice's taps, every neighbour within the cutoff with t(r) = t exp(-(r-1)/decay),
// fused with the moments of the cost-halving identity (Sec. II.A, Eq. cheby_prod):
//     phi_{n+1} = 2 H~ phi_n - phi_{n-1},  A_n = <phi_n|phi_n>,  B_n = <phi_{n+1}|phi_n>.
//
// The paper's test Hamiltonians are dense (D_H up to 230 non-zeros per row, Sec. IV); with a
// few states the CSR/ELL form of such a matrix reads ~4 D_H bytes of indices per site and
// step, more than the states themselves.  Here the taps are the same for every site, so no
// index is stored: a CTA stages a halo'd tile of phi_n (one 16-byte pack = two complex64
// states per site; 64 cells of two sites by 32 rows) in shared memory and each thread computes
// both sites of a cell in 8 consecutive rows.  A cell is the honeycomb's unit cell, or two
// neighbouring sites of a square lattice: both are two neighbouring packs of a row, so one
// kernel serves both.
//
// The pass has 2 (D_H - 1) FMAs per site-update against 24 bytes and is bound by FP32 FMAs only
// if the shared loads, 4 cycles a warp each, stay below them.  A column of source packs
// (cell offset, source site) therefore runs through a circular window of 8 rows in registers:
// step k loads one pack and applies one tap of each of the cell's two sites to 8 rows, 32 packed
// FMAs a load.  D_H = 235, 4.8M sites, 2 states: 235 -> 190 us per launch, 0.58 of the FP32 FMA
// peak; the column loop itself runs at 0.93 of it (139 us, by repeating it), the remaining 50 us are
// the staging and the epilogue of 1189 tiles, during which an SM has at most one other tile to work on.
// What was measured on the way (us): one pack, 8 rows, weights from shared memory 222; no test for
// zero weights, whose branches made the compiler move the sums about, and the previous state
// requested two rows ahead of its use 209; weights from the constant bank 201; no spills 195; sums in
// FP32 pairs instead of FP64 (two FP64 operations a clock and SM) and a carried row wrap 190.
// Tiles of 32 cells, three CTAs to an SM, took 215; a start staggered by half a tile and prefetching
// the previous state into L2 changed nothing.
//
// Reductions: compensated FP32 (value + error) per thread and through the lanes, FP64 from the warps'
// sums on, per-CTA partials and a fixed-order sum by the last CTA to finish.
#include <cuda_runtime.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <vector>

#include "tbpm_internal.cuh"
#include "stencil.cuh"

namespace tbpm {
namespace {

// Rows per thread and depth of the register window.  Per column of n taps a thread loads n + 7
// packs for 32 n packed FMAs; one site of 16 rows in pieces of 8, 4, 2 and 1 taps (the previous
// split) loaded n + 15 a piece, more shared-memory cycles than FMA cycles at D_H = 235 (4372 against
// 3568 a warp; now about 1900).  The union of the two sites' runs costs 7 % more FMAs there.  With
// both sites of 16 rows the sums alone take 128 registers, one CTA of 8 warps per SM.
constexpr int kTapWin = 8;
constexpr int kTapRB = 4;                        // row blocks per tile
constexpr int kTapTY = kTapWin * kTapRB;         // rows per tile
constexpr int kTapTX = 64;                       // cells per tile along x (two warps)
constexpr int kTapThreads = kTapTX * kTapRB;
constexpr int kTapMaxSmem = 226 * 1024;         // beside the sums' static shared memory
constexpr int kTapStage = 5;                     // groups of rows the staging is split into

__device__ __forceinline__ int64_t tap_wrap(int64_t v, int64_t L, int periodic, bool* ok) {
  if (v >= 0 && v < L) return v;
  if (!periodic) {
    *ok = false;
    return 0;
  }
  const int64_t r = v % L;
  return r < 0 ? r + L : r;
}

// MOM: fuse the moment sums (moment pass); without it the kernel is the plain recurrence step
// that the accumulation passes pair with an accumulate-only pass.
template <bool FIRST, bool MOM>
__global__ void __launch_bounds__(kTapThreads, 2) k_taps_moment(RecurrenceArgs a, const __grid_constant__ TapTable tp) {
  extern __shared__ float4 smem[];
  const int RX = tp.rx, RY = tp.ry;
  const int TW = kTapTX + 2 * RX, TH = kTapTY + 2 * RY, RS = 2 * TW;
  float4* tile = smem;

  const int P = a.P;
  const int p = (int)(blockIdx.x % (unsigned)P);
  const unsigned tile_id = blockIdx.x / (unsigned)P;
  const int64_t LS = a.geom.kind == TBPM_HONEYCOMB ? 2 * a.geom.Lx : a.geom.Lx, Ly = a.geom.Ly;  // sites of a row
  const unsigned ntx = (unsigned)((LS + 2 * kTapTX - 1) / (2 * kTapTX));
  const int64_t x0 = (int64_t)(tile_id % ntx) * kTapTX, y0 = (int64_t)(tile_id / ntx) * kTapTY;
  const float4* cur = reinterpret_cast<const float4*>(a.cur);
  float4* po = reinterpret_cast<float4*>(a.prev_out);

  // stage phi_n of the tile and its halo (wrapped on periodic sides, zero on open ones) with
  // asynchronous 16-byte copies, all in flight at once; a thread walks down a group of rows of
  // one site column, whose wrap is computed once
  for (int e = threadIdx.x; e < RS * kTapStage; e += kTapThreads) {
    const int g = e / RS, c = e - g * RS;
    const int ty0 = TH * g / kTapStage, ty1 = TH * (g + 1) / kTapStage;
    bool okx = true;
    const int64_t gx = tap_wrap(2 * (x0 - RX) + c, LS, a.geom.pbc_x, &okx);
    const float4* colsrc = cur + gx * P + p;
    const int64_t rstride = LS * P;
    // the row's wrap is carried along: one compare a row
    int64_t gy = y0 - RY + ty0;
    // open sides: rows [first, last) of the walk exist
    const int first = a.geom.pbc_y ? 0 : (int)-gy, last = a.geom.pbc_y || Ly - gy > TH ? TH : (int)(Ly - gy);
    if (a.geom.pbc_y) gy = tap_wrap(gy, Ly, 1, &okx);
    const float4* src = colsrc + gy * rstride;
    unsigned dst = (unsigned)__cvta_generic_to_shared(tile + ty0 * RS + (c & 1) * TW + (c >> 1));
    for (int i = 0; i < ty1 - ty0; ++i, dst += (unsigned)(RS * sizeof(float4))) {
      const bool ok = okx && i >= first && i < last && TBPM_DBG_OK(src - cur, Ly * rstride, TBPM_DBG_TAPS);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(ok ? src : cur), "r"(ok ? 16 : 0)
                   : "memory");
      src += rstride;
      if (++gy == Ly) {
        gy = 0;
        src = colsrc;
      }
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int xl = threadIdx.x % kTapTX, rb = threadIdx.x / kTapTX;  // cell and row block of this thread
  const float4* base = tile + (RY + rb * kTapWin) * RS + RX + xl;
  // the two states of a pack are two FP32 pairs; each takes one packed FMA with the tap's weight
  // in both halves
  float2 lo[2][kTapWin], hi[2][kTapWin];
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int o = 0; o < kTapWin; ++o) lo[s][o] = hi[s][o] = make_float2(0.f, 0.f);
  for (int c = 0; c < tp.n_cols; ++c) {
    const int4 hd = tp.col[c];  // pack offset of the first row, taps, first weight
    const float4* col = base + hd.x;
    const float4* w = tp.w + hd.z;
    int left = hd.y;
    float4 win[kTapWin];
#pragma unroll
    for (int j = 0; j < kTapWin - 1; ++j, col += RS) win[j] = *col;
    for (;;) {
#pragma unroll
      for (int j = 0; j < kTapWin; ++j, col += RS) {
        win[(j + kTapWin - 1) % kTapWin] = *col;
        const float4 wk = w[j];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const float2 w2 = s ? make_float2(wk.z, wk.w) : make_float2(wk.x, wk.y);
#pragma unroll
          for (int o = 0; o < kTapWin; ++o) {
            const float4 v = win[(j + o) % kTapWin];
            lo[s][o] = __ffma2_rn(w2, make_float2(v.x, v.y), lo[s][o]);
            hi[s][o] = __ffma2_rn(w2, make_float2(v.z, v.w), hi[s][o]);
          }
        }
        if (--left == 0) break;
      }
      if (left == 0) break;
      w += kTapWin;
    }
  }

  // phi_{n+1} = d phi_n + th h (- phi_{n-1}) and the moment sums of the two states
  const float th = FIRST ? a.th1f : a.th2f;
  Pair32 v[4];  // per state |phi|^2 and Re <out|phi>
#pragma unroll
  for (int k = 0; k < 4; ++k) v[k] = sum_of(0.f);
  const int64_t x = 2 * (x0 + xl), yb = y0 + rb * kTapWin;
  const int64_t rstep = LS * P;
  float4* prev = po + (yb * LS + x) * P + p;
  float4* next = (a.next ? reinterpret_cast<float4*>(a.next) : po) + (prev - po);
  const float* diag = a.diag ? reinterpret_cast<const float*>(a.diag) + yb * LS + x : nullptr;
  const float dc = FIRST ? a.dc1f : a.dc1f + a.dc1f;
  const int nx = x + 1 < LS ? 2 : x < LS ? 1 : 0, ny = (int)(Ly - yb < kTapWin ? Ly - yb : kTapWin);
  // two rows at a time: their phi_{n-1} and on-site terms are all requested before the first is used
  // (four rows spill)
#pragma unroll
  for (int o2 = 0; o2 < kTapWin; o2 += 2) {
    float4 pv[2][2];
    float dd[2][2];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const bool in = o2 + i < ny && s < nx &&
                        TBPM_DBG_OK(prev + (o2 + i) * rstep + s * P - po, Ly * rstep, TBPM_DBG_TAPS);
        pv[i][s] = !FIRST && in ? __ldcs(prev + (o2 + i) * rstep + s * P) : make_float4(0.f, 0.f, 0.f, 0.f);
        dd[i][s] = diag && in ? __ldg(diag + (o2 + i) * LS + s) : 0.f;
      }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int o = o2 + i;
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        if (o < ny && s < nx) {
          const float4 ph = base[o * RS + s * TW];
          const float d = diag ? (FIRST ? dd[i][s] : dd[i][s] + dd[i][s]) : dc;
          const float2 l = lo[s][o], h = hi[s][o];
          float4 out;
          out.x = d * ph.x + th * l.x;
          out.y = d * ph.y + th * l.y;
          out.z = d * ph.z + th * h.x;
          out.w = d * ph.w + th * h.y;
          if (!FIRST) {
            out.x -= pv[i][s].x;
            out.y -= pv[i][s].y;
            out.z -= pv[i][s].z;
            out.w -= pv[i][s].w;
          }
          if (TBPM_DBG_OK(prev + o * rstep + s * P - po, Ly * rstep, TBPM_DBG_TAPS)) next[o * rstep + s * P] = out;
          if constexpr (MOM) {
            v[0] = add(v[0], sum_of(ph.x * ph.x + ph.y * ph.y));
            v[1] = add(v[1], sum_of(out.x * ph.x + out.y * ph.y));
            v[2] = add(v[2], sum_of(ph.z * ph.z + ph.w * ph.w));
            v[3] = add(v[3], sum_of(out.z * ph.z + out.w * ph.w));
          }
        }
      }
    }
  }
  if constexpr (!MOM) return;

  // CTA sums (fixed trees), per-CTA partials, the last CTA sums them in CTA order
  __shared__ double red[kTapThreads / 32][4];
  __shared__ unsigned ticket;
  reduce_lanes<4>(v, 1, 0, lane, [&](int k, double t) { red[warp][k] = t; });
  __syncthreads();
  if (threadIdx.x < 4) {
    double s = 0.0;
    for (int w = 0; w < kTapThreads / 32; ++w) s += red[w][threadIdx.x];
    a.tap_partials[(size_t)blockIdx.x * 4 + threadIdx.x] = s;
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) ticket = atomicAdd(a.counter, 1u);
  __syncthreads();
  if (ticket != gridDim.x - 1) return;
  __threadfence();
  // <phi_0|phi_0> and <phi_1|phi_0> are the pass' first sums; H~ is Hermitian, so the imaginary parts
  // are zero
  const int64_t ntiles = gridDim.x / (unsigned)P;
  const int M = a.M, n = a.step;
  for (int q = warp; q < 4 * P; q += kTapThreads / 32) {
    const int pp = q / 4, k = q % 4, c = k & 1;
    double s = 0.0;
    for (int64_t t = lane; t < ntiles; t += 32) s += __ldcg(a.tap_partials + (size_t)(t * P + pp) * 4 + k);
    for (int off = 16; off >= 1; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) {
      double* ms = a.mu + (size_t)(2 * pp + k / 2) * M * 2;
      double* m = ms + (FIRST ? 0 : 4 * n) + 2 * c;
      m[0] = FIRST ? s : 2.0 * s - ms[2 * c];
      m[1] = 0.0;
    }
  }
  if (threadIdx.x == 0) *a.counter = 0u;
}

int64_t tap_grid(const RecurrenceArgs& a) {
  const int64_t LS = a.geom.kind == TBPM_HONEYCOMB ? 2 * a.geom.Lx : a.geom.Lx;
  return ((LS + 2 * kTapTX - 1) / (2 * kTapTX)) * ((a.geom.Ly + kTapTY - 1) / kTapTY) * a.P;
}

size_t tap_tile_bytes(int rx, int ry) { return (size_t)(kTapTY + 2 * ry) * 2 * (kTapTX + 2 * rx) * 16; }

}  // namespace

size_t taps_partials_bytes(const RecurrenceArgs& a) { return sizeof(double) * 4 * (size_t)tap_grid(a); }

static int launch_taps(tbpm_ctx* ctx, const RecurrenceArgs& a, bool first, bool mom) {
  const size_t smem = tap_tile_bytes(a.taps->rx, a.taps->ry);
  const int64_t grid = tap_grid(a);
  if (grid <= 0 || grid >= (1LL << 31) || smem > (size_t)kTapMaxSmem) {
    set_error("tap kernel: grid %lld or shared memory %zu out of range", (long long)grid, smem);
    return TBPM_EUNSUPPORTED;
  }
  void* fn = first ? (mom ? (void*)k_taps_moment<true, true> : (void*)k_taps_moment<true, false>)
                   : (mom ? (void*)k_taps_moment<false, true> : (void*)k_taps_moment<false, false>);
  // the limit is the kernel's, not the launch's: another thread's smaller lattice must not lower it in between
  TBPM_CK(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kTapMaxSmem));
  RecurrenceArgs aa = a;
  void* args[] = {&aa, const_cast<TapTable*>(a.taps)};
  const cudaError_t e = cudaLaunchKernel(fn, dim3((unsigned)grid), dim3(kTapThreads), args, smem, ctx->stream);
  ctx->launches++;
  if (e != cudaSuccess) {
    set_error("tap kernel launch: %s", cudaGetErrorString(e));
    return TBPM_ECUDA;
  }
  return TBPM_OK;
}

int launch_taps_moment(tbpm_ctx* ctx, const RecurrenceArgs& a, bool first) { return launch_taps(ctx, a, first, true); }

int launch_taps_step(tbpm_ctx* ctx, const RecurrenceArgs& a, bool first) { return launch_taps(ctx, a, first, false); }

// Columns of the taps of a cell's two sites: (cell offset, source site) -> a run along y with one
// weight per site and step (0 where a site has no such tap).  Sublattice 1 of the honeycomb takes
// each tap mirrored, (-dx, -dy, 1-ds), as the ELL builder does; site 1 of a pair of square sites
// sees the source one site further left.  The tile halo is the largest offset of any tap.
// Lattices whose tile would not fit shared memory, cubic lattices and lattices with vacancies keep
// the ELL path only.
int build_tap_table(tbpm_lattice* lat) {
  const tbpm_lattice_desc& d = lat->desc;
  if (lat->tap_t.empty() || d.kind == TBPM_CUBIC || d.vacancy_frac > 0.0) return TBPM_OK;
  const size_t z = lat->tap_t.size();
  std::map<std::pair<int, int>, std::map<int, float2>> runs;  // (dx, ds) -> dy -> weights
  int rx = 0, ry = 0;
  for (int sub = 0; sub < 2; ++sub) {
    for (size_t k = 0; k < z; ++k) {
      int dx = lat->tap_off[4 * k], dy = lat->tap_off[4 * k + 1], ds = lat->tap_off[4 * k + 3];
      if (d.kind != TBPM_HONEYCOMB) {
        ds = (sub + dx) & 1;
        dx = (sub + dx - ds) / 2;
      } else if (sub == 1) {
        dx = -dx;
        dy = -dy;
        ds = 1 - ds;
      }
      float2& w = runs[{dx, ds}][dy];  // a new entry is zero
      (sub ? w.y : w.x) += (float)(lat->tap_t[k] / d.t);
      rx = std::max(rx, std::abs(dx));
      ry = std::max(ry, std::abs(dy));
    }
  }
  if (tap_tile_bytes(rx, ry) > (size_t)kTapMaxSmem) return TBPM_OK;
  const int rs = 2 * (kTapTX + 2 * rx);
  std::unique_ptr<TapTable> tab(new TapTable());
  int cols = 0, steps = 0;
  for (auto& kv : runs) {
    const int lo = kv.second.begin()->first, n = kv.second.rbegin()->first - lo + 1;
    if (cols == kTapMaxCols || steps + n > kTapMaxSteps) return TBPM_OK;
    tab->col[cols++] = make_int4(lo * rs + kv.first.second * (rs / 2) + kv.first.first, n, steps, 0);
    for (int dy = lo; dy < lo + n; ++dy) {
      auto it = kv.second.find(dy);
      const float2 w = it == kv.second.end() ? make_float2(0.f, 0.f) : it->second;
      tab->w[steps++] = make_float4(w.x, w.x, w.y, w.y);
    }
  }
  tab->n_cols = cols;
  tab->rx = rx;
  tab->ry = ry;
  lat->taps = std::move(tab);
  return TBPM_OK;
}

}  // namespace tbpm

TBPM_DEBUG_UNIT(taps)
