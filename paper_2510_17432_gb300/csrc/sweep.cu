// Register-resident row sweep: K Chebyshev steps per pass over HBM on the honeycomb and square
// stencils, complex64 state pairs or single states, clean, disordered or with vacant sites, with the
// moment inner products of every step fused in.
//
// The recurrence phi_{n+1} = 2 H~ phi_n - phi_{n-1} (App. B) on the honeycomb couples
//   A(x,y) <- B(x,y), B(x-1,y), B(x,y-1)        B(x,y) <- A(x,y), A(x+1,y), A(x,y+1)
// so a thread that owns one cell (both sites) and one state pair finds every neighbour in its
// own registers except B(x-1,y) and A(x+1,y), which belong to the threads of the adjacent cells
// of the same row.  A CTA owns a band of CW cells (K/2 halo cells on each side) and a segment of
// rows (K/2 halo rows below and above) and sweeps it upwards as a wavefront: at sweep position r
// level L = 1..K forms phi_{n+L} at row r - (L-1) from
//   * level L-1 at rows r-L, r-L+1, r-L+2 of the same cell: registers (the thread formed them in
//     this and the two previous positions),
//   * level L-1 at row r-L+1 of the adjacent cells: a shared-memory exchange row written in the
//     previous position (double-buffered, so one barrier per position suffices),
//   * level L-2 at row r-L+1 of the same cell: registers.
// Level 0 (phi_n) and phi_{n-1} arrive row by row through 1-D TMA bulk copies (cp.async.bulk,
// one elected thread, an mbarrier per ring slot) into a ring NSLOT rows deep; a band row is
// contiguous in the [N][S] layout, so one copy per state block (two where a periodic band wraps).
// Levels K-1 and K go to HBM, so per K steps each state block crosses HBM four times: read
// phi_{n-1}, phi_n, write phi_{n+K-1}, phi_{n+K}.
//
// The same sweep serves (measured per four-step pass or per request, before -> now):
//   * the square lattice, whose cells are two neighbouring sites of a row: 2.1M sites, 8 padded
//     states, disorder: 99.5 us per one-step pass -> 160 us per four steps;
//   * one state per site (a 16-byte unit is a cell) and vacancy lattices in the full layout, D_i = NaN
//     marking vacant sites: 8.3M-site vacancy graphene, four plain steps through the index lists 211 us
//     -> one window pass 77 us;
//   * disorder: D of a row is loaded two positions ahead of its use; one position ahead, its latency
//     was the first stall (134M sites, 4 states: 4237 -> 3330 us per pass, 62 -> 78 % of the copy peak).
// What bounds a pass: HBM on large clean lattices, the per-position barrier and issue (12 warps per
// SM, shared memory and registers both full) elsewhere.
//
// Moments (cost halving of Eq. cheby_prod): for every level, <phi_{n+L-1}|phi_{n+L-1}> and
// <phi_{n+L}|phi_{n+L-1}> over the segment's interior, summed in FP32 over at most 32 units per
// thread, then FP32 lane trees per state pair, FP64 warp slots, FP64 block partials and a
// fixed-order FP64 sum by the last CTA: deterministic for a given launch shape.
//
// Every mbarrier wait is bounded by a wall-clock budget; on expiry the CTA records an error code
// in the caller's status word, stops sweeping, waits (bounded) for its copies in flight and still
// takes part in the grid reduction so that the completion counter stays consistent.
#include <cuda_runtime.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "tbpm_internal.cuh"

namespace tbpm {
namespace sweep {

constexpr uint64_t kWaitNs = 2000000000ull;  // 2 s per mbarrier wait

// Source of the bulk copies for rows that hold no data (outside an open lattice, beyond the rows
// a segment needs): two state-block rows of 2 NT units for NT <= 256.  Zero-initialised when the
// module loads and never written, so every ring read is a plain shared load.
static __device__ __align__(16) float4 g_zero_rows[2 * 256];

// SGL: one state per site (a 16-byte unit is a cell: A and B); otherwise state pairs (a unit is one
// site of one pair).
template <int NT_, int K_, int NSLOT_, bool SGL_>
struct Cfg {
  static constexpr int NT = NT_, K = K_, H = K_ / 2, NSLOT = NSLOT_;
  static constexpr int VL = SGL_ ? 2 : 4;   // sums per level: {|a|^2, Re<n|a>} per state of the unit
  static constexpr int NV = VL * K;
  static constexpr int RU = SGL_ ? NT : 2 * NT;  // units of one state block's row in the ring
  static constexpr int FOLD = 16;      // positions per FP32 partial (32 unit terms per thread)
  static constexpr int MINB = SGL_ ? 5 : NT <= 128 ? 3 : NT <= 192 ? 2 : 1;
  static constexpr int BAR_BYTES = ((NSLOT * 8 + 15) / 16) * 16;
  // ring slot: [P zero][phi_n row: RU units][P zero][phi_{n-1} row: RU units], padded to a
  // multiple of 8 units (128 bytes) so that every slot starts on the same bank
  __host__ __device__ static int slot_units(int P) { return (2 * RU + 2 * P + 7) & ~7; }
  // exchange row: [A plane: NT][P zero][B plane: NT] (float4 per pair, float2 per single state)
  __host__ __device__ static int xrow_units(int P) { return 2 * NT + P; }
  // + disordered lattices: a thread-private ring of 2 D for the last 4 rows ([4][NT] float2)
  static size_t smem(int P, bool diag) {
    return (size_t)BAR_BYTES + 16 * (size_t)NSLOT * slot_units(P) +
           (SGL_ ? 8 : 16) * (size_t)2 * (K - 1) * xrow_units(P) + 8 * (size_t)(NT / 32) * P * NV +
           (diag ? (size_t)8 * 4 * NT : 0);
  }
};

struct Args {
  const float4* prev_in;  // phi_{n-1}
  const float4* cur_in;   // phi_n
  float4* prev_out;       // phi_{n+K-1}
  float4* cur_out;        // phi_{n+K}
  const float* diag;      // rescaled D_i per site (NaN marks a vacant site) or null
  float dc2, th2;         // 2 D (clean lattice), 2 t/|H|
  float s1;               // scale of level 1: 1, or 1/2 in the first pass (phi_1 = H~ phi_0)
  int first;              // 1: phi_n = phi_0 and there is no phi_{n-1}
  int store;              // 0: the moments are the pass's only result
  int nk;                 // steps whose moments are wanted (the last pass may need fewer than K)
  int64_t Ly;
  int64_t RS;             // sites per row: 2 Lx on the honeycomb, Lx on the square lattice
  int pbc_x, pbc_y;
  int P, logP, S;
  int CW, BX, SY;         // band cells, interior cells, rows per segment
  int nbx, nsy;
  double* partials;       // [grid][P][NV]
  unsigned* counter;
  double* mu;
  int M;
  int step0;
  int* status;            // host-visible status word: nonzero = a bounded wait expired
  float4* win[4];         // window mode: phi_{n+1} .. phi_{n+4}, one buffer each (null: not wanted)
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_arrive_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0;
}

// Bounded wait for the phase of the given parity: false once budget_ns of wall-clock time has
// passed without the phase completing.
__device__ __forceinline__ bool mbar_wait_ns(uint32_t bar, uint32_t parity, uint64_t budget_ns) {
  if (mbar_try(bar, parity)) return true;
  const uint64_t t0 = globaltimer();
  while (!mbar_try(bar, parity))
    if (globaltimer() - t0 > budget_ns) return false;
  return true;
}

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  return mbar_wait_ns(bar, parity, kWaitNs);
}

// 1-D bulk copy global -> shared, completion counted in bytes on the mbarrier.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// d own + th (n1 + n2 + n3 [+ n4]) - pv as packed f32x2 halves (one state each)
__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }
template <bool SQ>
__device__ __forceinline__ float2 level_update(float d, float2 own, float th, float2 n1, float2 n2, float2 n3,
                                               float2 n4, float2 pv) {
  const float2 h = SQ ? __fadd2_rn(__fadd2_rn(n1, n2), __fadd2_rn(n3, n4)) : __fadd2_rn(__fadd2_rn(n1, n2), n3);
  return __ffma2_rn(make_float2(d, d), own, __ffma2_rn(make_float2(th, th), h, make_float2(-pv.x, -pv.y)));
}
template <bool SQ>
__device__ __forceinline__ float4 level_update(float d, float4 own, float th, float4 n1, float4 n2, float4 n3,
                                               float4 n4, float4 pv) {
  const float2 l = level_update<SQ>(d, lo2(own), th, lo2(n1), lo2(n2), lo2(n3), lo2(n4), lo2(pv));
  const float2 h = level_update<SQ>(d, hi2(own), th, hi2(n1), hi2(n2), hi2(n3), hi2(n4), hi2(pv));
  return make_float4(l.x, l.y, h.x, h.y);
}

// Moment terms of one level for the two states of a pair, a = phi_j and n = phi_{j+1}:
// <phi_j|phi_j> and Re<phi_{j+1}|phi_j> as packed (re, im) halves, summed at the fold.  For a
// Hermitian H~, <phi_{j+1}|phi_j> = <psi|T_{j+1}(H~) T_j(H~)|psi> is real (the two polynomials
// commute and are Hermitian), so its imaginary part is not accumulated.
// acc2[0] = |a_0|^2, acc2[1] = |a_1|^2, acc2[2] = Re n_0^* a_0, acc2[3] = Re n_1^* a_1 (halves)
__device__ __forceinline__ void moment_terms(float2* acc2, float4 a, float4 n) {
  acc2[0] = __ffma2_rn(lo2(a), lo2(a), acc2[0]);
  acc2[1] = __ffma2_rn(hi2(a), hi2(a), acc2[1]);
  acc2[2] = __ffma2_rn(lo2(n), lo2(a), acc2[2]);
  acc2[3] = __ffma2_rn(hi2(n), hi2(a), acc2[3]);
}
__device__ __forceinline__ void moment_terms(float2* acc2, float2 a, float2 n) {
  acc2[0] = __ffma2_rn(a, a, acc2[0]);
  acc2[1] = __ffma2_rn(n, a, acc2[1]);
}
__device__ __forceinline__ void set_zero(float4& v) { v = make_float4(0.f, 0.f, 0.f, 0.f); }
__device__ __forceinline__ void set_zero(float2& v) { v = make_float2(0.f, 0.f); }

enum { DIAG_NONE = 0, DIAG_SITE = 1, DIAG_MASKED = 2 };
enum { PASS_MOM = 0, PASS_EDGE = 1, PASS_WIN = 2 };

// SQ: square lattice, whose cells are two neighbouring sites of a row (x = 2c and 2c + 1) --
//   A <- B, B(c-1), A(y+1), A(y-1)      B <- A, A(c+1), B(y+1), B(y-1)
// so a step reaches one row where the honeycomb needs two steps per row: K halo rows instead of
// K/2.  A row of an odd number of sites ends in half a cell, whose B is neither stored nor summed.
// DIAG: none (clean), D_i per site, or D_i with NaN at vacant sites, whose amplitude stays zero.
// MODE: PASS_MOM -- levels K-1 and K go to prev_out, cur_out, with the moments of every step;
// PASS_EDGE -- the same for the first pass (phi_0 alone) and the last one (fewer steps, no states
// stored), whose checks cost the clean honeycomb pass 7 % (450 against 420 us on 67M site-states)
// when every pass carries them; PASS_WIN -- window mode for the time blocks: every level goes to
// its own buffer (a.win[L-1]) and no moment is summed.
template <int NT_, int K_, int NSLOT_, bool SQ, bool SGL, int DIAG, bool OPEN, int MODE>
__global__ void __launch_bounds__(NT_, Cfg<NT_, K_, NSLOT_, SGL>::MINB) k_sweep_moments(Args a) {
  using C = Cfg<NT_, K_, NSLOT_, SGL>;
  using V = std::conditional_t<SGL, float2, float4>;
  constexpr int NT = C::NT, K = C::K, H = C::H, NSLOT = C::NSLOT, NV = C::NV, VL = C::VL, RU = C::RU;
  constexpr int HY = SQ ? K : K / 2;  // halo rows
  constexpr bool HAS_DIAG = DIAG != DIAG_NONE, WIN = MODE == PASS_WIN, EDGE = MODE != PASS_MOM;
  // level-0 rows r and r-1 of the own cell: carried in registers, or read from the ring again where
  // the registers go to the diagonal's prefetch or to the square lattice's fourth neighbour
  constexpr bool RING0 = !SGL && (HAS_DIAG || SQ);
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ unsigned ticket;
  const int P = SGL ? 1 : a.P, logP = SGL ? 0 : a.logP, CW = SGL ? NT : a.CW;
  const int SU = C::slot_units(P), XU = C::xrow_units(P);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smraw);
  float4* ring = reinterpret_cast<float4*>(smraw + C::BAR_BYTES);  // [NSLOT][SU]
  V* xb = reinterpret_cast<V*>(ring + NSLOT * SU);                  // [K-1][2][XU]
  double* red = reinterpret_cast<double*>(xb + 2 * (K - 1) * XU);   // [warps][P][NV]
  float2* dring = reinterpret_cast<float2*>(red + (NT / 32) * P * NV);  // [4][NT] (disorder only)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
  V zero;
  set_zero(zero);

  for (int i = tid; i < NSLOT * SU; i += NT) ring[i] = zero4;
  for (int i = tid; i < 2 * (K - 1) * XU; i += NT) xb[i] = zero;
  for (int i = tid; i < (NT / 32) * P * NV; i += NT) red[i] = 0.0;
  if (tid == 0) {
    for (int s = 0; s < NSLOT; ++s) mbar_init(smem_u32(bars + s), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the zero pads written through the generic proxy must be ordered before the bulk copies
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();

  const int bx = blockIdx.x % a.nbx, sy = blockIdx.x / a.nbx;
  const int64_t RS = a.RS;
  const int64_t xs = 2 * ((int64_t)bx * a.BX - H);  // first site of the band (may lie outside the row)
  const int64_t ys = (int64_t)sy * a.SY;
  const int64_t ye = ys + a.SY < a.Ly ? ys + a.SY : a.Ly;
  const int64_t r0 = ys - HY;         // first sweep position = first level-0 row
  const int64_t rlast = ye + HY - 1;  // last level-0 row any exact value needs
  const int ny = (int)(ye - ys);
  const int npos = ny + K - 1 + HY;   // positions r0 .. ye + K - 2 (level K reaches row ye - 1)
  const int64_t row_units = SGL ? RS / 2 : RS * P;
  const int site_bytes = SGL ? 8 : 16 * P;
  // level-0 rows that hold data, as local indices i = row - r0: [v_lo, v_hi]
  const bool open_y = OPEN && !a.pbc_y;
  const int v_lo = (open_y && r0 < 0) ? (int)(-r0) : 0;
  const int v_hi = (int)(((open_y && rlast > a.Ly - 1) ? a.Ly - 1 : rlast) - r0);

  // this thread's cell and pair.  The band [xs, xs + 2 CW) and the rows r0 .. r_end lie within one
  // period of the lattice on either side (the host requires RS >= 2 CW and enough rows), so a
  // single wrap brings any coordinate back into it.
  const int c = tid >> logP, p = tid & (P - 1);
  int64_t xA = xs + 2 * c, xB = xA + 1;
  bool ghA = false, ghB = false;
  auto place = [&](int64_t& x, bool& gh) {
    if (x < 0 || x >= RS) {
      if (OPEN && !a.pbc_x) gh = true;
      else x = x < 0 ? x + RS : x - RS;
    }
  };
  const bool inx = c >= H && c < CW - H;
  const bool intA = inx && xA < RS, intB = inx && xB < RS;
  const int64_t colA = SGL ? xA / 2 : xA * P + p;  // of an interior cell (never wrapped); B at + P
  place(xA, ghA);
  place(xB, ghB);
  const int uA = SGL ? c : 2 * (c << logP) + p;  // unit of A(c, pair p) in a ring row; B is + P
  const int wA = tid, wB = NT + P + tid;
  // Ring rows of pairs interleave A and B per cell, so the A units of the cells of a quarter-warp
  // share banks.  Threads with bit 2 of tid set take each pair of level-0 loads in the opposite
  // order, which puts the two halves of a quarter-warp on different banks for any P.
  const bool swp = !SGL && ((tid >> 2) & 1);
  const int o_pvA = RU + P + uA, o_pvB = o_pvA + P;      // phi_{n-1} A, B of row r (R0)
  const int o_bxm = uA - P, o_axp = uA + 2 * P;          // B(x-1, r), A(x+1, r) (R0)
  const int o_p1 = swp ? o_pvB : o_pvA, o_p2 = swp ? o_pvA : o_pvB;
  const int o_n1 = swp ? o_axp : o_bxm, o_n2 = swp ? o_bxm : o_axp;
  const int o_c1 = swp ? uA + P : uA, o_c2 = swp ? uA : uA + P;  // A, B of a row

  // row index in the lattice of local row i, or -1 where the row holds no data
  auto grow = [&](int i) -> int64_t {
    if (i < v_lo || i > v_hi) return -1;
    const int64_t r = r0 + i;
    if (r >= 0 && r < a.Ly) return r;
    return r < 0 ? r + a.Ly : r - a.Ly;
  };

  // producer (thread 0): the band's pieces inside the lattice are the same for every row (at
  // most two: one wrap when periodic), in sites; rows are issued in order, slot after slot; a row
  // without data is filled with zeros from g_zero_rows
  int pc0 = 0, pn0 = 0, pc1 = 0, pn1 = 0;
  int64_t pg0 = 0, pg1 = 0;
  if (!a.pbc_x) {
    const int64_t lo = -xs > 0 ? -xs : 0;
    const int64_t hi = RS - xs < 2 * CW ? RS - xs : 2 * CW;
    if (lo < hi) {
      pc0 = (int)lo;
      pg0 = xs + lo;
      pn0 = (int)(hi - lo);
    }
  } else {
    pg0 = xs < 0 ? xs + RS : xs;
    pn0 = (int)(RS - pg0 < 2 * CW ? RS - pg0 : 2 * CW);
    pc1 = pn0;
    pg1 = 0;
    pn1 = 2 * CW - pn0;
  }
  if (SGL) pg0 >>= 1, pg1 >>= 1;  // first units of the pieces in a row
  else pg0 *= P, pg1 *= P;
  pc0 *= site_bytes;  // byte offsets of the pieces in a ring row
  pc1 *= site_bytes;
  const uint32_t piece_bytes0 = (uint32_t)(pn0 * site_bytes);
  const uint32_t piece_bytes1 = (uint32_t)(pn1 * site_bytes);
  const uint32_t zero_bytes = (uint32_t)RU * 16u;
  int next_row = 0;  // local index of the next row to issue
  int next_slot = 0;
  // rows 0 .. npos are read (row r+1 at the last position); none beyond is issued, so no copy is
  // in flight when the CTA finishes its sweep
  auto issue_next = [&]() {
    if (next_row > npos) return;
    const int j = next_row;
    const int slot = next_slot;
    ++next_row;
    next_slot = next_slot + 1 == NSLOT ? 0 : next_slot + 1;
    const uint32_t bar = smem_u32(bars + slot);
    const uint32_t sn = smem_u32(ring + slot * SU + P);
    const uint32_t sp = smem_u32(ring + slot * SU + RU + 2 * P);
    const int64_t gy = grow(j);
    if (gy < 0) {
      mbar_arrive_tx(bar, 2u * zero_bytes);
      bulk_g2s(sn, g_zero_rows, zero_bytes, bar);
      bulk_g2s(sp, g_zero_rows, zero_bytes, bar);
      return;
    }
    const int64_t src0 = gy * row_units + pg0;
    const int64_t src1 = gy * row_units + pg1;
    if (!TBPM_DBG_OK(src0 + (int64_t)(piece_bytes0 / 16) - 1, a.Ly * row_units, TBPM_DBG_SWEEP_ROW) ||
        (pn1 > 0 && !TBPM_DBG_OK(src1 + (int64_t)(piece_bytes1 / 16) - 1, a.Ly * row_units, TBPM_DBG_SWEEP_ROW))) {
      mbar_arrive(bar);  // debug build: the row is not copied (the kernel's results are void)
      return;
    }
    mbar_arrive_tx(bar, piece_bytes0 + piece_bytes1 + (EDGE && a.first ? zero_bytes : piece_bytes0 + piece_bytes1));
    const bool both = !(EDGE && a.first);  // the first pass has no phi_{n-1}
    if (!both) bulk_g2s(sp, g_zero_rows, zero_bytes, bar);
    bulk_g2s(sn + (uint32_t)pc0, a.cur_in + src0, piece_bytes0, bar);
    if (both) bulk_g2s(sp + (uint32_t)pc0, a.prev_in + src0, piece_bytes0, bar);
    if (pn1 > 0) {
      bulk_g2s(sn + (uint32_t)pc1, a.cur_in + src1, piece_bytes1, bar);
      if (both) bulk_g2s(sp + (uint32_t)pc1, a.prev_in + src1, piece_bytes1, bar);
    }
  };
  if (tid == 0)
    for (int k = 0; k < NSLOT; ++k) issue_next();

  // D of the cell's two sites in local row i (NaN: vacant)
  auto diag_row = [&](int i) -> float2 {
    if (!HAS_DIAG) return make_float2(a.dc2, a.dc2);
    const int64_t gy = grow(i);
    if (gy < 0 || (ghA && ghB)) return make_float2(0.f, 0.f);
    const float* row = a.diag + gy * RS;
    float2 d;
    if (!SQ) d = __ldg(reinterpret_cast<const float2*>(row + xA));
    else d = make_float2(ghA ? 0.f : __ldg(row + xA), ghB ? 0.f : __ldg(row + xB));
    return d;
  };

  // registers: level l = 1 .. K-1 at the rows formed in the last three positions (slot =
  // position % 3); level 0 (phi_n) is read from the ring, which keeps row j until position j + 1
  V RA[K][3], RB[K][3];
#pragma unroll
  for (int l = 0; l < K; ++l)
#pragma unroll
    for (int s = 0; s < 3; ++s) RA[l][s] = RB[l][s] = zero;
  float2 acc2[NV];  // packed halves of the NV sums (level L: [VL (L-1), VL L))
#pragma unroll
  for (int v = 0; v < NV; ++v) acc2[v] = make_float2(0.f, 0.f);
  int folded = 0;
  // every FOLD positions: the FP32 partials of the lanes of each state pair (lane = p + P m) are
  // reduce-scattered across the lanes (each exchange halves the values a lane keeps), so that a
  // lane ends with NV / (32 / P) fully summed values and adds only those into the warp's FP64
  // slots: the FP64 work is spread over the whole warp instead of P lanes
  static_assert(K == 4, "the fold splits 16 (pairs) or 8 (single states) values");
  auto half = [&](const float* in, float* out, int n, int off) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (k < n / 2) {
        const float keep = up ? in[n / 2 + k] : in[k];
        const float send = up ? in[k] : in[n / 2 + k];
        out[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
      }
    }
  };
  auto fold = [&]() {
    const int pp = lane & (P - 1);
    double* slot = red + (warp * P + pp) * NV;
    float v16[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      v16[v] = acc2[v].x + acc2[v].y;
      acc2[v] = make_float2(0.f, 0.f);
    }
    if constexpr (SGL) {
      float v4[4], v2[2], v1[1];
      half(v16, v4, 8, 16);
      half(v4, v2, 4, 8);
      half(v2, v1, 2, 4);
      v1[0] += __shfl_xor_sync(0xffffffffu, v1[0], 2);
      v1[0] += __shfl_xor_sync(0xffffffffu, v1[0], 1);
      if ((lane & 3) == 0) slot[((lane & 16) ? 4 : 0) + ((lane & 8) ? 2 : 0) + ((lane & 4) ? 1 : 0)] += (double)v1[0];
    } else {
      float v8[8];
      half(v16, v8, 16, 16);
      const int b16 = (lane & 16) ? 8 : 0;
      if (P == 16) {
#pragma unroll
        for (int k = 0; k < 8; ++k) slot[b16 + k] += (double)v8[k];
        return;
      }
      float v4[4];
      half(v8, v4, 8, 8);
      const int b8 = b16 + ((lane & 8) ? 4 : 0);
      if (P == 8) {
#pragma unroll
        for (int k = 0; k < 4; ++k) slot[b8 + k] += (double)v4[k];
        return;
      }
      float v2[2];
      half(v4, v2, 4, 4);
      const int b4 = b8 + ((lane & 4) ? 2 : 0);
      if (P == 4) {
#pragma unroll
        for (int k = 0; k < 2; ++k) slot[b4 + k] += (double)v2[k];
        return;
      }
      float v1[1];
      half(v2, v1, 2, 2);
      const int b2 = b4 + ((lane & 2) ? 1 : 0);
      // P = 2: every lane holds one sum; P = 1: lanes 2k and 2k+1 hold halves of the same one
      if (P == 1) v1[0] += __shfl_xor_sync(0xffffffffu, v1[0], 1);
      if (P == 2 || (lane & 1) == 0) slot[b2] += (double)v1[0];
    }
  };
  // outputs of levels K-1 and K at the rows they form at the current position
  float4* out_km1 = a.prev_out + (r0 - (K - 2)) * row_units + colA;
  float4* out_k = a.cur_out + (r0 - (K - 1)) * row_units + colA;
  int64_t off_r = r0 * row_units + colA;  // window mode: offset of row r in every level's buffer
  auto put = [&](float4* dst, const V& vA, const V& vB) {
    if constexpr (SGL) {
      __stcs(dst, make_float4(vA.x, vA.y, vB.x, vB.y));
    } else {
      __stcs(dst, vA);
      if (!SQ || intB) __stcs(dst + P, vB);
    }
  };
  // ring slots of level-0 rows r and r+1 (a slot's phi_{n-1} row follows at + RU + P)
  int slot_m1 = 0, slot_0 = 0, slot_p1 = 1 % NSLOT;  // row r0 - 1 stands in as row r0
  uint32_t wait_par = NSLOT == 1 ? 1u : 0u;  // phase parity of row r+1's slot

  // disordered lattices: D of rows r and r+1 in flight, stored into the ring at their positions (one
  // row ahead was not enough: the load's latency was the sweep's first stall)
  float2 dq0 = diag_row(0), dq1 = diag_row(1);
  bool timed_out = !mbar_wait(smem_u32(bars + 0), 0);  // this thread's waits; OR-reduced per position
  // level-0 values carried from position to position: rows r and r-1 of this thread's own cell;
  // row r0 - 1 stands in as row r0
  V c0A, c0B, cmA, cmB;
  if constexpr (SGL) {
    const float4 q = ring[P + uA];
    c0A = lo2(q);
    c0B = hi2(q);
  } else {
    c0A = ring[P + uA];
    c0B = ring[P + uA + P];
  }
  cmA = c0A;
  cmB = c0B;
  const float th = a.th2;
  bool aborted = false;
  int i_done = -1;  // last position completed

  for (int ib = 0; ib < npos && !aborted; ib += 3) {
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      const int i = ib + u;
      if (i >= npos || aborted) break;
      const int s0 = u, s1 = (u + 2) % 3, s2 = (u + 1) % 3;  // ages 0, 1, 2
      if (!mbar_wait(smem_u32(bars + slot_p1), wait_par)) timed_out = true;  // level-0 row r+1
      const float4* R0 = ring + slot_0 * SU + P;
      const float4* Rp = ring + slot_p1 * SU + P;
      const float4* Rm_ = ring + slot_m1 * SU + P;  // row r-1 (RING0)
      // x-neighbours of levels 1 .. K-1 written at the previous position, loaded before this
      // position writes the exchange row of the level before (the compiler cannot tell the two
      // parities apart): level 1's right away, the others once level 1 has been stored
      V xbm[K], xap[K];
      const V* Xprev = xb + ((i - 1) & 1) * XU;  // level l at + 2 (l - 1) XU
      xbm[1] = Xprev[wB - P];
      xap[1] = Xprev[wA + P];
      const V prevA = cmA, prevB = cmB;  // level-0 row r-1 of this cell
      if (HAS_DIAG) {
        dring[(i & 3) * NT + tid] = make_float2(2.f * dq0.x, 2.f * dq0.y);
        dq0 = dq1;
        dq1 = diag_row(i + 2);
      }
#pragma unroll
      for (int L = 1; L <= K; ++L) {
        const int iq = i - (L - 1);  // local row of this level
        V ownA, ownB, lB, rA, upA, upB, dnA, dnB, pvA, pvB;  // left B, right A, rows above and below
        if (L == 1) {
          if constexpr (SGL) {
            const float4 qp = Rp[uA], qv = R0[o_pvA];
            const float4 ql = R0[uA - 1], qr = R0[uA + 1];
            ownA = c0A;
            ownB = c0B;
            upA = lo2(qp);
            upB = hi2(qp);
            lB = hi2(ql);
            rA = lo2(qr);
            pvA = lo2(qv);
            pvB = hi2(qv);
            dnA = prevA;
            dnB = prevB;
            cmA = ownA;
            cmB = ownB;
            c0A = upA;
            c0B = upB;
          } else {
            // pairs of loads, each issued in the thread's bank order
            float4 q1, q2;
            if (SQ) {
              q1 = Rp[o_c1];
              q2 = Rp[o_c2];
            } else {
              const float4 *qa = Rp + uA, *qb = R0 + (uA + P);
              q1 = *(swp ? qa : qb);
              q2 = *(swp ? qb : qa);
            }
            const float4 n1 = R0[o_n1], n2 = R0[o_n2];
            const float4 p1 = R0[o_p1], p2 = R0[o_p2];
            lB = swp ? n2 : n1;
            rA = swp ? n1 : n2;
            pvA = swp ? p2 : p1;
            pvB = swp ? p1 : p2;
            if (SQ) {
              const float4 w1 = R0[o_c1], w2 = R0[o_c2], z1 = Rm_[o_c1], z2 = Rm_[o_c2];
              upA = swp ? q2 : q1;
              upB = swp ? q1 : q2;
              ownA = swp ? w2 : w1;
              ownB = swp ? w1 : w2;
              dnA = swp ? z2 : z1;
              dnB = swp ? z1 : z2;
            } else {
              // disordered lattices: level-0 values of rows r and r-1 from the ring
              ownA = RING0 ? R0[uA] : c0A;
              ownB = swp ? q2 : q1;
              upA = swp ? q1 : q2;
              dnB = RING0 ? Rm_[uA + P] : prevB;
              dnA = upB = zero;
              cmA = ownA;  // carried to the next position: row r becomes row r-1, A(r+1) becomes A(r)
              cmB = ownB;
              c0A = upA;
            }
          }
        } else {
          ownA = RA[L - 1][s1];
          ownB = RB[L - 1][s1];
          lB = xbm[L - 1];
          rA = xap[L - 1];
          dnA = RA[L - 1][s2];
          dnB = RB[L - 1][s2];
          upA = RA[L - 1][s0];
          upB = RB[L - 1][s0];
          if (L == 2) {
            if constexpr (RING0) {
              const float4 z1 = Rm_[o_c1], z2 = Rm_[o_c2];
              pvA = swp ? z2 : z1;
              pvB = swp ? z1 : z2;
            } else {
              pvA = prevA;
              pvB = prevB;
            }
          } else {
            pvA = RA[L - 2][s2];
            pvB = RB[L - 2][s2];
          }
        }
        // disordered lattices: 2 D of this level's row from the thread's own ring
        float2 dl = HAS_DIAG ? dring[(iq & 3) * NT + tid] : make_float2(a.dc2, a.dc2);
        float thA = th, thB = th;
        if (EDGE && L == 1) {
          dl.x *= a.s1;
          dl.y *= a.s1;
          thA = thB = th * a.s1;
        }
        if (DIAG == DIAG_MASKED) {  // a vacant site keeps the zero it starts with
          if (dl.x != dl.x) dl.x = thA = 0.f;
          if (dl.y != dl.y) dl.y = thB = 0.f;
        }
        V nA, nB;
        if (SQ) {
          nA = level_update<true>(dl.x, ownA, thA, ownB, lB, upA, dnA, pvA);
          nB = level_update<true>(dl.y, ownB, thB, ownA, rA, upB, dnB, pvB);
        } else {
          nA = level_update<false>(dl.x, ownA, thA, ownB, lB, dnB, zero, pvA);
          nB = level_update<false>(dl.y, ownB, thB, ownA, rA, upA, zero, pvB);
        }
        if (OPEN) {
          const bool out = iq < v_lo || iq > v_hi;
          if (ghA || out) nA = zero;
          if (ghB || out) nB = zero;
        }
        if (L < K) {
          RA[L][s0] = nA;
          RB[L][s0] = nB;
          V* Xout = xb + ((L - 1) * 2 + (i & 1)) * XU;
          Xout[wA] = nA;
          Xout[wB] = nB;
        }
        if (L == 1) {
#pragma unroll
          for (int l = 2; l < K; ++l) {
            xbm[l] = Xprev[2 * (l - 1) * XU + wB - P];
            xap[l] = Xprev[2 * (l - 1) * XU + wA + P];
          }
        }
        if (intA && (unsigned)(iq - HY) < (unsigned)ny &&
            TBPM_DBG_OK(off_r - (int64_t)(L - 1) * row_units, a.Ly * row_units, TBPM_DBG_SWEEP_STORE)) {
          if (WIN) {
            if (a.win[L - 1]) put(a.win[L - 1] + (off_r - (int64_t)(L - 1) * row_units), nA, nB);
          } else {
            if (!EDGE || a.store) {
              if (L == K - 1) put(out_km1, nA, nB);
              else if (L == K) put(out_k, nA, nB);
            }
            moment_terms(acc2 + (L - 1) * VL, ownA, nA);
            if (!SQ || intB) moment_terms(acc2 + (L - 1) * VL, ownB, nB);
          }
        }
      }
      off_r += row_units;
      if (!WIN) {
        out_km1 += row_units;
        out_k += row_units;
        if (++folded == C::FOLD) {
          folded = 0;
          fold();
        }
      }
      // one barrier per position; it also tells every thread whether any wait expired
      if (__syncthreads_or(timed_out ? 1 : 0)) {
        aborted = true;
        break;
      }
      i_done = i;
      // row r-1 has been read for the last time: refill its slot with row r - 1 + NSLOT
      if (tid == 0 && i >= 1) issue_next();
      slot_m1 = slot_0;
      slot_0 = slot_p1;
      slot_p1 = slot_p1 + 1 == NSLOT ? 0 : slot_p1 + 1;
      if (slot_p1 == 0) wait_par ^= 1u;
    }
  }
  if (aborted && tid == 0) {
    // copies in flight into this CTA's shared memory must land before it exits: rows
    // i_done + 2 .. next_row - 1 were issued and never waited for (bounded waits)
    bool err_wait = false;
    for (int j = i_done + 2 > 0 ? i_done + 2 : 0; j < next_row; ++j)
      if (!mbar_wait(smem_u32(bars + j % NSLOT), (uint32_t)((j / NSLOT) & 1))) err_wait = true;
    atomicExch(a.status, err_wait ? 2 : 1);
  }
  if (WIN) return;
  fold();
  __syncthreads();
  for (int qv = tid; qv < P * NV; qv += NT) {  // warps in order
    const int pp = qv / NV, v = qv - pp * NV;
    double t = 0.0;
    for (int w = 0; w < NT / 32; ++w) t += red[(w * P + pp) * NV + v];
    a.partials[(size_t)blockIdx.x * P * NV + qv] = t;
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) ticket = atomicAdd(a.counter, 1u);
  __syncthreads();
  if (ticket != gridDim.x - 1) return;
  __threadfence();
  // the last CTA: value v = (s * 2 + comp) * K + k, comp 0 = <phi_j|phi_j>, 1 = Re <phi_{j+1}|phi_j>
  const int nval = K * a.S * 2;
  for (int v = warp; v < nval; v += NT / 32) {
    const int k = v % K, comp = (v / K) & 1, s = v / (2 * K);
    const int pr = SGL ? 0 : s >> 1, sub = SGL ? 0 : s & 1;
    const int idx = k * VL + (SGL ? comp : comp * 2 + sub);
    double sum = 0.0;
    for (int t = lane; t < (int)gridDim.x; t += 32) sum += __ldcg(a.partials + ((size_t)t * P + pr) * NV + idx);
    for (int off = 16; off >= 1; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    if (lane == 0) red[v] = sum;  // nval <= P NV values: the warps' slots are free again
  }
  __syncthreads();
  for (int v = tid; v < nval; v += NT) {
    const int k = v % K, comp = (v / K) & 1, s = v / (2 * K), j = a.step0 + k;
    if (EDGE && k >= a.nk) continue;
    double* ms = a.mu + (size_t)s * a.M * 2 + 4 * (size_t)j + 2 * comp;
    if (EDGE && a.first && k == 0) {  // m_0 and m_1 themselves
      ms[0] = red[v];
      ms[1] = 0.0;
    } else {  // m_{2j} = 2 <phi_j|phi_j> - m_0 and m_{2j+1} = 2 <phi_{j+1}|phi_j> - m_1, real inner products
      const double* m0 = a.mu + (size_t)s * a.M * 2 + 2 * comp;
      ms[0] = 2.0 * red[v] - (EDGE && a.first ? red[v - k] : m0[0]);
      ms[1] = EDGE && a.first ? 0.0 : -m0[1];
    }
  }
  if (tid == 0) *a.counter = 0u;
}

// Expiry check of the bounded wait above: one warp waits on an mbarrier of its own that expects
// one arrival.  With `arrive`, thread 0 arrives first and the phase completes; without it nothing
// ever arrives, no copy is in flight, and every thread's wait gives up after budget_ns.  An
// expired wait is reported as the sweep reports one: code 1 in the caller's status word.
__global__ void __launch_bounds__(32) k_wait_probe(int* status, uint64_t budget_ns, int arrive) {
  __shared__ __align__(8) uint64_t bar;
  const uint32_t b = smem_u32(&bar);
  if (threadIdx.x == 0) {
    mbar_init(b, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (arrive && threadIdx.x == 0) mbar_arrive(b);
  const bool done = mbar_wait_ns(b, 0, budget_ns);
  if (__syncthreads_or(done ? 0 : 1) && threadIdx.x == 0) atomicExch(status, 1);
}

}  // namespace sweep

// One kernel variant: its shared-memory limit is raised once, its resident CTAs per SM are looked up
// once per number of state pairs.  Internal linkage: the counts are per loaded library.
namespace {
template <int NT, int K, int NSLOT, bool SQ, bool SGL, int DIAG, bool OPEN, int MODE>
struct SweepKernel {
  using Cf = sweep::Cfg<NT, K, NSLOT, SGL>;
  static int resident(int logP) {
    static std::mutex mu;
    static int per_sm[6] = {0, 0, 0, 0, 0, 0};
    std::lock_guard<std::mutex> lock(mu);
    if (per_sm[logP] == 0) {
      auto fn = sweep::k_sweep_moments<NT, K, NSLOT, SQ, SGL, DIAG, OPEN, MODE>;
      const size_t sm = Cf::smem(1 << logP, DIAG != sweep::DIAG_NONE);
      if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)Cf::smem(16, true)) != cudaSuccess ||
          cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm[logP], fn, NT, sm) != cudaSuccess ||
          per_sm[logP] < 1) {
        cudaGetLastError();
        per_sm[logP] = 0;
        return 0;
      }
    }
    return per_sm[logP];
  }
  static void launch(const sweep::Args& a, cudaStream_t st) {
    sweep::k_sweep_moments<NT, K, NSLOT, SQ, SGL, DIAG, OPEN, MODE>
        <<<(unsigned)(a.nbx * a.nsy), NT, Cf::smem(a.P, DIAG != sweep::DIAG_NONE), st>>>(a);
  }
};
}  // namespace

template <int NT, int K, int NSLOT, bool SQ, bool SGL, int DIAG, bool OPEN, int MODE>
static int launch_sweep_variant(tbpm_ctx* ctx, sweep::Args& a) {
  using Kn = SweepKernel<NT, K, NSLOT, SQ, SGL, DIAG, OPEN, MODE>;
  const int per_sm = Kn::resident(a.logP);
  if (per_sm < 1) {
    set_error("fused sweep: the kernel does not fit an SM");
    return TBPM_ECUDA;
  }
  // segments per band: the count whose CTAs fill the resident slots best over whole waves, weighed
  // by the sweep positions each segment adds (halo rows below and above, K - 1 to drain)
  const int extra = K - 1 + (SQ ? K : K / 2) + (SQ ? 0 : 3);
  const int64_t slots = (int64_t)ctx->num_sms * per_sm;
  const int64_t max_nsy = std::max<int64_t>(1, std::min<int64_t>(a.Ly / 4, 8 * slots / a.nbx + 1));
  int64_t nsy = 1;
  double best = -1.0;
  for (int64_t k = 1; k <= max_nsy; ++k) {
    const int64_t sy = (a.Ly + k - 1) / k;
    const int64_t ctas = a.nbx * ((a.Ly + sy - 1) / sy);
    const int64_t waves = (ctas + slots - 1) / slots;
    const double eff = (double)ctas / (double)(waves * slots) * (double)sy / (double)(sy + extra);
    if (eff > best + 1e-9) {
      best = eff;
      nsy = k;
    }
  }
  a.SY = (int)((a.Ly + nsy - 1) / nsy);
  a.nsy = (int)((a.Ly + a.SY - 1) / a.SY);
  const int64_t grid = (int64_t)a.nbx * a.nsy;
  if (MODE != sweep::PASS_WIN) {
    TBPM_TRY(ensure(ctx, ctx->ws_fused_partials, sizeof(double) * Kn::Cf::NV * (size_t)a.P * (size_t)grid));
    a.partials = (double*)ctx->ws_fused_partials.p;
  }
  Kn::launch(a, ctx->stream);
  TBPM_CK_LAUNCH(ctx);
  return TBPM_OK;
}

template <int NT, int NSLOT, bool SQ, bool SGL, int DIAG, int MODE>
static int launch_sweep_open(tbpm_ctx* ctx, sweep::Args& a) {
  return a.pbc_x && a.pbc_y ? launch_sweep_variant<NT, 4, NSLOT, SQ, SGL, DIAG, false, MODE>(ctx, a)
                            : launch_sweep_variant<NT, 4, NSLOT, SQ, SGL, DIAG, true, MODE>(ctx, a);
}

template <int NT, int NSLOT, bool SQ, bool SGL, int DIAG>
static int launch_sweep_shape(tbpm_ctx* ctx, sweep::Args& a, bool win) {
  if (win) return launch_sweep_open<NT, NSLOT, SQ, SGL, DIAG, sweep::PASS_WIN>(ctx, a);
  if (a.first || !a.store || a.nk < 4) return launch_sweep_open<NT, NSLOT, SQ, SGL, DIAG, sweep::PASS_EDGE>(ctx, a);
  return launch_sweep_open<NT, NSLOT, SQ, SGL, DIAG, sweep::PASS_MOM>(ctx, a);
}

template <int NT, int NSLOT, bool SQ, bool SGL>
static int launch_sweep_diag(tbpm_ctx* ctx, sweep::Args& a, bool win, bool masked) {
  if (masked) return launch_sweep_shape<NT, NSLOT, SQ, SGL, sweep::DIAG_MASKED>(ctx, a, win);
  if (a.diag) return launch_sweep_shape<NT, NSLOT, SQ, SGL, sweep::DIAG_SITE>(ctx, a, win);
  return launch_sweep_shape<NT, NSLOT, SQ, SGL, sweep::DIAG_NONE>(ctx, a, win);
}

// The arguments every sweep takes; nt: threads per CTA.
static int sweep_args(tbpm_ctx* ctx, const tbpm_lattice* lat, const RecurrenceArgs& ra, const void* prev_in,
                      const void* cur_in, bool first, int nt, sweep::Args* ap) {
  sweep::Args& a = *ap;
  memset(&a, 0, sizeof(a));
  if (ctx->pinned_cap < 256) {
    set_error("context has no pinned status word");
    return TBPM_ECUDA;
  }
  a.prev_in = (const float4*)prev_in;
  a.cur_in = (const float4*)cur_in;
  a.diag = (const float*)ra.diag;
  a.dc2 = ra.dc2f;
  a.th2 = ra.th2f;
  a.s1 = first ? 0.5f : 1.f;
  a.first = first ? 1 : 0;
  a.Ly = lat->geom.Ly;
  a.RS = lat->geom.row_sites;
  a.pbc_x = lat->geom.pbc_x;
  a.pbc_y = lat->geom.pbc_y;
  a.S = ra.S;
  a.P = ra.S >= 2 ? ra.S / 2 : 1;
  a.logP = 0;
  while ((1 << a.logP) < a.P) ++a.logP;
  a.CW = nt / a.P;
  a.BX = a.CW - 4;  // two halo cells on each side (K = 4)
  a.nbx = (int)(((a.RS + 1) / 2 + a.BX - 1) / a.BX);
  a.mu = ra.mu;
  a.M = ra.M;
  a.counter = ra.counter;
  a.status = reinterpret_cast<int*>(ctx->pinned + kSweepStatusSlot);
  return TBPM_OK;
}

static int launch_sweep_128(tbpm_ctx* ctx, const tbpm_lattice* lat, const RecurrenceArgs& ra, sweep::Args& a, bool win) {
  const bool sq = lat->geom.kind == TBPM_SQUARE, masked = ra.masked != 0;
  if (ra.S == 1)
    return sq ? launch_sweep_diag<128, 5, true, true>(ctx, a, win, masked)
              : launch_sweep_diag<128, 5, false, true>(ctx, a, win, masked);
  return sq ? launch_sweep_diag<128, 5, true, false>(ctx, a, win, masked)
            : launch_sweep_diag<128, 5, false, false>(ctx, a, win, masked);
}

// Whether the 128-thread register sweep takes this lattice's stencil for Spad states: one band of
// 128 / P cells (P = Spad / 2 pairs, or one state) fits a row, rows enough for the halo to wrap once,
// and, for one state, whole 16-byte cells in every row.
bool sweep_shape_ok(const tbpm_lattice* lat, int precision, int Spad) {
  const Geom& g = lat->geom;
  if (precision != TBPM_C64 || g.kind == TBPM_CUBIC || !lat->tap_t.empty()) return false;
  const int64_t band = 2 * (128 / (Spad >= 2 ? Spad / 2 : 1));
  if (g.kind == TBPM_HONEYCOMB) {
    if (Spad >= 2 && !(g.Lx >= kSweepMinCells && g.Ly >= kSweepMinRows)) return false;
    return g.row_sites >= band && g.Ly >= kSweepMinRows;
  }
  return g.row_sites >= std::max<int64_t>(band, kSweepMinSquare) && g.Ly >= kSweepMinSquare &&
         (Spad >= 2 || g.row_sites % 2 == 0);
}

// Window pass of the time blocks: phi_{n+1} .. phi_{n+4} from (prev_in = phi_{n-1}, cur_in = phi_n)
// into win[0..3] (null: not wanted) by the 128-thread register sweep; first: cur_in = phi_0, prev_in not read.
int launch_sweep_window(tbpm_ctx* ctx, const tbpm_lattice* lat, const RecurrenceArgs& ra, const void* prev_in,
                        const void* cur_in, void* const win[4], bool first) {
  sweep::Args a;
  TBPM_TRY(sweep_args(ctx, lat, ra, prev_in, cur_in, first, 128, &a));
  for (int l = 0; l < 4; ++l) a.win[l] = (float4*)win[l];
  return launch_sweep_128(ctx, lat, ra, a, true);
}

// One register-resident sweep pass: steps step0 .. step0+3 from (prev_in, cur_in) into (prev_out,
// cur_out), null when only the moments of the first nk steps are wanted.  step0 = 0: cur_in = phi_0.
// Variant 8: 128 threads; 9: 192 threads; 10: 256 threads (honeycomb pairs).
int launch_sweep_pass(tbpm_ctx* ctx, const tbpm_lattice* lat, const RecurrenceArgs& ra, const void* prev_in,
                      const void* cur_in, void* prev_out, void* cur_out, int step0, int nk, int variant) {
  const bool wide = (variant == 9 || variant == 10) && lat->geom.kind == TBPM_HONEYCOMB && ra.S >= 2 && !ra.masked;
  sweep::Args a;
  TBPM_TRY(sweep_args(ctx, lat, ra, prev_in, cur_in, step0 == 0, wide ? (variant == 9 ? 192 : 256) : 128, &a));
  a.prev_out = (float4*)prev_out;
  a.cur_out = (float4*)cur_out;
  a.store = prev_out != nullptr;
  a.nk = nk;
  a.step0 = step0;
  if (!wide) return launch_sweep_128(ctx, lat, ra, a, false);
  const bool edge = a.first || !a.store || a.nk < 4;
  auto pick = [&](auto nt) -> int {
    constexpr int NT = decltype(nt)::value;
    if (a.diag)
      return edge ? launch_sweep_open<NT, 4, false, false, sweep::DIAG_SITE, sweep::PASS_EDGE>(ctx, a)
                  : launch_sweep_open<NT, 4, false, false, sweep::DIAG_SITE, sweep::PASS_MOM>(ctx, a);
    return edge ? launch_sweep_open<NT, 4, false, false, sweep::DIAG_NONE, sweep::PASS_EDGE>(ctx, a)
                : launch_sweep_open<NT, 4, false, false, sweep::DIAG_NONE, sweep::PASS_MOM>(ctx, a);
  };
  return variant == 9 ? pick(std::integral_constant<int, 192>()) : pick(std::integral_constant<int, 256>());
}

int sweep_status(tbpm_ctx* ctx) {
  int* st = reinterpret_cast<int*>(ctx->pinned + kSweepStatusSlot);
  const int v = *st;
  if (v != 0) {
    *st = 0;
    set_error("moment recurrence: a bounded wait expired (code %d: 1, 2 a row copy of the sweep, 3 a neighbour's step)", v);
    return TBPM_ETIMEOUT;
  }
  return TBPM_OK;
}

}  // namespace tbpm

TBPM_DEBUG_UNIT(sweep)

using namespace tbpm;

// One-warp run of the register sweep's bounded mbarrier wait, reported through the sweep's status
// word and sweep_status(): TBPM_ETIMEOUT when the wait expired.
extern "C" int tbpm_wait_probe(tbpm_ctx* ctx, int arrive, double budget_s) {
  clear_error();
  if (!ctx) {
    set_error("tbpm_wait_probe: NULL context");
    return TBPM_EINVAL;
  }
  if (!(budget_s > 0.0 && budget_s <= 2.0)) {
    set_error("tbpm_wait_probe: budget %g s outside (0, 2]", budget_s);
    return TBPM_EINVAL;
  }
  if (ctx->pinned_cap < 256) {
    set_error("context has no pinned status word");
    return TBPM_ECUDA;
  }
  TBPM_CK(cudaSetDevice(ctx->device));
  int* status = reinterpret_cast<int*>(ctx->pinned + kSweepStatusSlot);
  const uint64_t budget_ns = (uint64_t)(budget_s * 1e9);
  sweep::k_wait_probe<<<1, 32, 0, ctx->stream>>>(status, budget_ns, arrive ? 1 : 0);
  TBPM_CK_LAUNCH(ctx);
  TBPM_CK(cudaStreamSynchronize(ctx->stream));
  return sweep_status(ctx);
}
