// Electronic (DC) conductivity, Sec. V: the current operator, the block inner products
// <A_a|B_b> between two families of state blocks, and the reconstruction of the EC
// correlation function and of sigma(E) (Eq. DC).
//
//  * Current operator (Sec. V): J_alpha = i[H, P_alpha] with P_alpha = -sum_i r_alpha,i |i><i|,
//    so every bond i-j carries (J_alpha)_ij = -i H_ij (r_j - r_i)_alpha (hbar = e = 1).  Bond
//    vectors are those of the library's lattices: unit-spaced square and cubic lattices; graphene
//    with C-C distance 1, A -> B bonds (1,0), (-1/2,-sqrt3/2), (-1/2,sqrt3/2) in the fixed
//    neighbour order, B -> A their negatives.  Periodic bonds use the nearest image.  On
//    long-range lattices every tap carries its own bond vector (negated on the B sublattice).
//  * Block inner products: out[s][a][b] = sum_i conj(A_a[i][s]) B_b[i][s] for nA x nB pairs of
//    state blocks in one pass; each CTA owns a TA x TB tile of pairs and walks chunks of the
//    site range, FP32 products (complex64 states) summed over 16 units per thread, folded into
//    FP64 per chunk in a fixed warp order; chunk groups are summed in order by a second kernel.
//    Deterministic for fixed sizes.  This one primitive gives <psi|Psi(E)>, the moment-form
//    m_n(E) = <J psi|T_n(H~)|J Psi(E)> (Eq. dc_mom, nA = 1) and, for a time block of b states
//    psi_1(t_j), all b x N_E correlation values at once (the state-based form).
//  * Moment form (Eq. dc_mom and the sum after it):
//        C(t_j, E) = e^{i H0 t_j} sum_{n < N(j tau~)} c_n^*(j tau~) m_n(E) / |<psi|Psi(E)>|,
//    c_n^* = a_n i^n, a_0 = J_0, a_n = 2 J_n; the phase e^{i H0 t} undoes the spectral shift.
//  * sigma(E) = D(E)/A int_0^{t_tot} Re[e^{-iEt} C(t,E)] dt (Eq. DC) with D(E) = N Re<psi|Psi(E)>
//    and A = N x (area per site), weights (2 - delta_j0)/2 on t_j = j tau.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "stencil.cuh"
#include "tbpm_internal.cuh"

namespace tbpm {

namespace {

constexpr int kXIter = 16;                       // units per thread per chunk
constexpr int kXChunk = kXIter * kThreads;       // units per chunk

struct CurArgs {
  Geom g;
  int path;
  const int32_t* ell;
  const int64_t* full_of;
  const float* masked;  // full layout: NaN at vacant sites, whose amplitude stays zero (else null)
  int64_t n_sites;
  int P, logP;
  double kw[2][6];  // t (r_j - r_i)_alpha per sublattice and neighbour slot
  float kwf[2][6];  // the same in FP32 (a conversion per bond would go through the FP64 pipe)
  const double* kwl;  // long-range lattices: the same per slot on the device, [2][z] (else null)
};

template <typename R, typename Args>
__device__ __forceinline__ R bond_weight(const Args& a, int sub, int d) {
  if constexpr (sizeof(R) == 4) return a.kwf[sub][d];
  else return a.kw[sub][d];
}

// y = J_alpha x for one block of states [n_sites][S].  Bound: HBM; 64-bit divisions per neighbour had made it
// issue-bound (36.6 us on 2.1M sites of the full layout, now 26.9 us).
template <typename R, int SPT>
__global__ void __launch_bounds__(kThreads) k_current(CurArgs c, const void* xv, void* yv) {
  using PK = Pack<R, SPT>;
  const PK* X = reinterpret_cast<const PK*>(xv);
  PK* Y = reinterpret_cast<PK*>(yv);
  const int64_t n_units = c.n_sites * c.P;
  const bool csr = c.path == TBPM_PATH_CSR;
  for (int64_t u = (int64_t)blockIdx.x * kThreads + threadIdx.x; u < n_units; u += (int64_t)gridDim.x * kThreads) {
    const int64_t i = u >> c.logP;
    const int p = (int)(u & (c.P - 1));
    int sub = 0;
    SiteAt at{};
    if (!csr) {
      at = site_at(c.g, i);
      sub = at.s;
    } else if (c.g.kind == TBPM_HONEYCOMB) {
      sub = (int)(c.full_of[i] & 1);
    }
    PK o;
#pragma unroll
    for (int k = 0; k < 2 * SPT; ++k) o.v[k] = R(0);
    const bool vacant = c.masked && isnan(__ldg(c.masked + i));
#pragma unroll 3
    for (int d = 0; d < c.g.z && !vacant; ++d) {
      const R w0 = c.kwl ? R(0) : bond_weight<R>(c, sub, d);
      if (!c.kwl && w0 == R(0)) continue;  // bonds across the direction
      const int64_t j = csr ? (int64_t)c.ell[i * c.g.z + d] : site_neighbour(c.g, at, d);
      if (j < 0) continue;
      const R w = c.kwl ? (R)__ldg(c.kwl + sub * c.g.z + d) : w0;
      const PK x = ld(X + j * c.P + p);
#pragma unroll
      for (int k = 0; k < SPT; ++k) {  // -i w (xr + i xi) = w xi - i w xr
        o.v[2 * k] += w * x.v[2 * k + 1];
        o.v[2 * k + 1] -= w * x.v[2 * k];
      }
    }
    st(Y + u, o);
  }
}

struct XdotArgs {
  const void* A;
  int64_t a_stride;  // packs between blocks of A
  int nA;
  const void* B;
  int64_t b_stride;
  int nB;
  int64_t n_units;
  int P;
  int S;             // padded states per block
  int64_t n_chunks;
  double* partials;  // [gridDim.y][nA][nB][S][2]
};

// complex64 block inner products.  A warp owns a tile of TA x TB pairs of blocks (32 sums: two per pair and
// state of the unit), its lanes walk 16 units each; the CTA's eight warps take neighbouring tiles of the
// same units, so that L1 serves the blocks the tiles share, and split the units when there are fewer tiles.
// A product conj(a) b is two packed f32x2 FMAs, (ar, ai) (br, bi) and (ar, ai) (bi, -br), whose halves are
// added at the fold.  Every 16 units the 32 sums are reduce-scattered over the lanes of a state pair
// (31 shuffles instead of 160 for a tree per sum) and each lane adds the ones it keeps in FP64.
// Bound: the latency of the 8- and 16-byte loads at 16 warps an SM for many pairs (long scoreboard 11.7 cycles per
// instruction, L1 at 21 %, FMA pipe at 26 %), HBM for one block against a few.  On 2.1M sites 16 x 64 blocks
// took 3320 us with a shuffle tree per sum and scalar FMAs, now 1206 us.
struct XTile {
  int at, bt;   // tiles along A and B
  int wa, wb;   // tiles of one CTA along A and B (wa wb divides 8)
};

template <int SPT, int TA, int TB, int LOGP>
__global__ void __launch_bounds__(kThreads, 2) k_xdot_c64(XdotArgs x, XTile tl) {
  using PK = Pack<float, SPT>;
  constexpr int V = TA * TB * SPT * 2, P = 1 << LOGP;
  static_assert(V == 32, "one sum per lane");
  const PK* A = reinterpret_cast<const PK*>(x.A);
  const PK* B = reinterpret_cast<const PK*>(x.B);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nt = tl.wa * tl.wb, share = kWarps / nt;  // warps per tile
  const int sub = warp / nt, t = warp - sub * nt;
  const int ga = (tl.at + tl.wa - 1) / tl.wa;
  const int a0 = ((blockIdx.x % ga) * tl.wa + t % tl.wa) * TA, b0 = ((blockIdx.x / ga) * tl.wb + t / tl.wa) * TB;
  const int64_t group = (int64_t)blockIdx.y * share + sub, groups = (int64_t)gridDim.y * share;
  const bool active = a0 < x.nA && b0 < x.nB;
  const PK* pa[TA];
  const PK* pb[TB];
#pragma unroll
  for (int k = 0; k < TA; ++k) pa[k] = A + (int64_t)min(a0 + k, x.nA - 1) * x.a_stride;
#pragma unroll
  for (int l = 0; l < TB; ++l) pb[l] = B + (int64_t)min(b0 + l, x.nB - 1) * x.b_stride;
  __shared__ double slots[kWarps][P][32];  // this lane's P sums
  double(&tot)[P][32] = slots[warp];
#pragma unroll
  for (int k = 0; k < P; ++k) tot[k][lane] = 0.0;
  int base = 0;  // index of this lane's first sum after the reduce-scatter
  {
    int n = V;
    for (int off = 16; off >= P; off >>= 1) {
      n >>= 1;
      if (lane & off) base += n;
    }
  }
  constexpr int kSpan = 32 * kXIter;  // units per warp and chunk
  for (int64_t chunk = group; active && chunk * kSpan < x.n_units; chunk += groups) {
    float2 re[TA][TB][SPT], im[TA][TB][SPT];
#pragma unroll
    for (int k = 0; k < TA; ++k)
#pragma unroll
      for (int l = 0; l < TB; ++l)
#pragma unroll
        for (int s = 0; s < SPT; ++s) re[k][l][s] = im[k][l][s] = make_float2(0.f, 0.f);
    const int64_t u0 = chunk * kSpan + lane;
#pragma unroll (TA == 1 ? 1 : 2)
    for (int it = 0; it < kXIter; ++it) {
      const int64_t u = u0 + it * 32;
      if (u >= x.n_units) break;
      PK a[TA], b[TB];
#pragma unroll
      for (int k = 0; k < TA; ++k) a[k] = ld(pa[k] + u);
#pragma unroll
      for (int l = 0; l < TB; ++l) b[l] = ld(pb[l] + u);
#pragma unroll
      for (int l = 0; l < TB; ++l)
#pragma unroll
        for (int s = 0; s < SPT; ++s) {
          const float2 bv = make_float2(b[l].v[2 * s], b[l].v[2 * s + 1]);
          const float2 bw = make_float2(bv.y, -bv.x);
#pragma unroll
          for (int k = 0; k < TA; ++k) {
            const float2 av = make_float2(a[k].v[2 * s], a[k].v[2 * s + 1]);
            re[k][l][s] = __ffma2_rn(av, bv, re[k][l][s]);
            im[k][l][s] = __ffma2_rn(av, bw, im[k][l][s]);  // ar bi - ai br
          }
        }
    }
    float v[V];
#pragma unroll
    for (int k = 0; k < TA; ++k)
#pragma unroll
      for (int l = 0; l < TB; ++l)
#pragma unroll
        for (int s = 0; s < SPT; ++s) {
          v[((k * TB + l) * SPT + s) * 2] = re[k][l][s].x + re[k][l][s].y;
          v[((k * TB + l) * SPT + s) * 2 + 1] = im[k][l][s].x + im[k][l][s].y;
        }
#pragma unroll
    for (int lev = 0; lev < 5 - LOGP; ++lev) {
      const int off = 16 >> lev;
      const bool up = (lane & off) != 0;
#pragma unroll
      for (int k = 0; k < (V >> (lev + 1)); ++k) {
        const float lo = v[k], hi = v[k + (V >> (lev + 1))];
        v[k] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, off);
      }
    }
#pragma unroll
    for (int k = 0; k < P; ++k) tot[k][lane] += (double)v[k];
  }
  // the warps that share a tile, in order
  __syncthreads();
  if (!active || sub != 0) return;
#pragma unroll
  for (int q = 0; q < P; ++q) {
    double sum = 0.0;
    for (int w = t; w < kWarps; w += nt) sum += slots[w][q][lane];
    const int v = base + q, c = v & 1, s = (v >> 1) % SPT, kl = (v >> 1) / SPT;
    const int ia = a0 + kl / TB, ib = b0 + kl % TB;
    if (ia < x.nA && ib < x.nB)
      x.partials[((((int64_t)blockIdx.y * x.nA + ia) * x.nB + ib) * x.S + (lane & (P - 1)) * SPT + s) * 2 + c] = sum;
  }
}

// complex128 (FP64 issue bound): grid (a_tiles * b_tiles, chunk groups); 256 threads.
template <typename R, int SPT, int TA, int TB>
__global__ void __launch_bounds__(kThreads, 2) k_xdot(XdotArgs x) {
  using PK = Pack<R, SPT>;
  using T = R;
  constexpr int V = TA * TB * SPT * 2;
  __shared__ double tot[32 * TA * TB * 2];
  const PK* A = reinterpret_cast<const PK*>(x.A);
  const PK* B = reinterpret_cast<const PK*>(x.B);
  const int b_tiles = (x.nB + TB - 1) / TB;
  const int at = blockIdx.x / b_tiles, bt = blockIdx.x - at * b_tiles;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int PV = x.P * V;
  for (int q = threadIdx.x; q < PV; q += kThreads) tot[q] = 0.0;
  const PK* pa[TA];
  const PK* pb[TB];
#pragma unroll
  for (int k = 0; k < TA; ++k) pa[k] = A + (int64_t)min(at * TA + k, x.nA - 1) * x.a_stride;
#pragma unroll
  for (int l = 0; l < TB; ++l) pb[l] = B + (int64_t)min(bt * TB + l, x.nB - 1) * x.b_stride;
  __syncthreads();

  for (int64_t chunk = blockIdx.y; chunk < x.n_chunks; chunk += gridDim.y) {
    T acc[V];
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = T(0);
    const int64_t u0 = chunk * kXChunk + threadIdx.x;
#pragma unroll 2
    for (int it = 0; it < kXIter; ++it) {
      const int64_t u = u0 + (int64_t)it * kThreads;
      if (u >= x.n_units) break;
      PK a[TA], b[TB];
#pragma unroll
      for (int k = 0; k < TA; ++k) a[k] = ld(pa[k] + u);
#pragma unroll
      for (int l = 0; l < TB; ++l) b[l] = ld(pb[l] + u);
#pragma unroll
      for (int k = 0; k < TA; ++k)
#pragma unroll
        for (int l = 0; l < TB; ++l)
#pragma unroll
          for (int s = 0; s < SPT; ++s) {
            const T ar = a[k].v[2 * s], ai = a[k].v[2 * s + 1];
            const T br = b[l].v[2 * s], bi = b[l].v[2 * s + 1];
            T* o = acc + ((k * TB + l) * SPT + s) * 2;
            o[0] += ar * br + ai * bi;
            o[1] += ar * bi - ai * br;
          }
    }
    // lanes with the same state group p = lane % P
#pragma unroll
    for (int v = 0; v < V; ++v)
      for (int off = 16; off >= x.P; off >>= 1) acc[v] += __shfl_xor_sync(0xffffffffu, acc[v], off);
    for (int w = 0; w < kThreads / 32; ++w) {
      if (warp == w && lane < x.P) {
#pragma unroll
        for (int v = 0; v < V; ++v) tot[lane * V + v] += (double)acc[v];
      }
      __syncthreads();
    }
  }
  for (int q = threadIdx.x; q < PV; q += kThreads) {
    const int p = q / V, v = q - p * V;
    const int c = v & 1, s = (v >> 1) % SPT, kl = (v >> 1) / SPT;
    const int k = kl / TB, l = kl - k * TB;
    const int ia = at * TA + k, ib = bt * TB + l;
    if (ia < x.nA && ib < x.nB)
      x.partials[((((int64_t)blockIdx.y * x.nA + ia) * x.nB + ib) * x.S + p * SPT + s) * 2 + c] = tot[q];
  }
}

// out[(s*os + a*oa + b*ob + off)*2 + c] = sum over chunk groups in a fixed order: a CTA takes 32 outputs
// (lanes) and splits the groups over its 32 warps.
__global__ void __launch_bounds__(1024) k_xdot_reduce(const double* partials, int G, int nA, int nB, int S, double* out,
                                                      int64_t os, int64_t oa, int64_t ob, int64_t off) {
  __shared__ double sh[32][33];
  const int64_t per = (int64_t)nA * nB * S * 2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t q = (int64_t)blockIdx.x * 32 + lane;
  double acc = 0.0;
  if (q < per)
    for (int g = warp; g < G; g += 32) acc += partials[(int64_t)g * per + q];
  sh[warp][lane] = acc;
  __syncthreads();
  if (warp != 0 || q >= per) return;
  acc = 0.0;
  for (int w = 0; w < 32; ++w) acc += sh[w][lane];
  const int c = (int)(q & 1);
  const int64_t r = q >> 1;
  const int s = (int)(r % S);
  const int64_t ab = r / S;
  const int b = (int)(ab % nB), a = (int)(ab / nB);
  out[(s * os + a * oa + b * ob + off) * 2 + c] = acc;
}

__device__ __forceinline__ double block_sum256(double v, double* sh) {
  for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < 8; ++w) r += sh[w];
  return r;  // valid in thread 0
}

// grid (n_steps+1, ceil(rows/8)).  m [rows][Nn][2]; C [rows][n_steps+1][2] (not yet normalised).
constexpr int kEcRows = 8;
__global__ void __launch_bounds__(256) k_ec_corr_m(const double* table, const int* n_per_step, int n_steps,
                                                   const double* m, int rows, int Nn, double shift, double tau,
                                                   double* C) {
  __shared__ double sh[8];
  const int j = blockIdx.x, r0 = blockIdx.y * kEcRows;
  const int64_t width = n_steps + 1;
  const int nj = min(n_per_step[j], Nn);
  double re[kEcRows], im[kEcRows];
#pragma unroll
  for (int q = 0; q < kEcRows; ++q) re[q] = im[q] = 0.0;
  for (int n = threadIdx.x; n < nj; n += blockDim.x) {
    const double Jn = table[(int64_t)n * width + j];
    const double a = (n == 0) ? Jn : 2.0 * Jn;
    double cr, ci;  // c_n^* = a i^n
    switch (n & 3) {
      case 0: cr = a; ci = 0.0; break;
      case 1: cr = 0.0; ci = a; break;
      case 2: cr = -a; ci = 0.0; break;
      default: cr = 0.0; ci = -a; break;
    }
#pragma unroll
    for (int q = 0; q < kEcRows; ++q) {
      if (r0 + q < rows) {
        const double* mr = m + ((int64_t)(r0 + q) * Nn + n) * 2;
        re[q] += cr * mr[0] - ci * mr[1];
        im[q] += cr * mr[1] + ci * mr[0];
      }
    }
  }
  double sn, cs;
  sincos(shift * (double)j * tau, &sn, &cs);  // e^{+i H0 t_j}
  for (int q = 0; q < kEcRows && r0 + q < rows; ++q) {
    const double R = block_sum256(re[q], sh);
    const double I = block_sum256(im[q], sh);
    if (threadIdx.x == 0) {
      C[((int64_t)(r0 + q) * width + j) * 2] = cs * R - sn * I;
      C[((int64_t)(r0 + q) * width + j) * 2 + 1] = cs * I + sn * R;
    }
  }
}

// One block per row = s*nE + k: C /= |<psi|Psi(E_k)>| and sigma from Eq. DC.
__global__ void __launch_bounds__(256) k_ec_finish(double* C, const double* nrm, const double* energies, int nE,
                                                   int n_steps, double tphys, double area, double* sigma) {
  __shared__ double sh[8];
  const int row = blockIdx.x, k = row % nE;
  const int64_t width = n_steps + 1;
  const double nr = nrm[2 * row], ni = nrm[2 * row + 1];
  const double mag = hypot(nr, ni);
  const double inv = mag > 0.0 ? 1.0 / mag : 0.0;
  const double E = energies[k];
  double* Cr = C + (int64_t)row * width * 2;
  double acc = 0.0;
  for (int j = threadIdx.x; j <= n_steps; j += blockDim.x) {
    const double cr = Cr[2 * j] * inv, ci = Cr[2 * j + 1] * inv;
    Cr[2 * j] = cr;
    Cr[2 * j + 1] = ci;
    double sn, cs;
    sincos(-E * (double)j * tphys, &sn, &cs);
    acc += (j == 0 ? 0.5 : 1.0) * (cs * cr - sn * ci);
  }
  const double tot = block_sum256(acc, sh);
  if (threadIdx.x == 0) sigma[row] = mag > 0.0 ? nr / area * tphys * tot : 0.0;
}

// <psi|Psi(E_k)> = tau / 2 pi sum_{|j| <= n_steps} e^{i E_k t_j} C(t_j) with C(-t) = C(t)^*: one block per row s*nE + k.
__global__ void __launch_bounds__(256) k_ec_overlap(const double* corr, const double* energies, int nE, int n_steps,
                                                    double tphys, double* nrm) {
  __shared__ double sh[8];
  const int row = blockIdx.x, k = row % nE;
  const double* c = corr + (int64_t)(row / nE) * (n_steps + 1) * 2;
  const double E = energies[k];
  double acc = 0.0;
  for (int j = threadIdx.x; j <= n_steps; j += blockDim.x) {
    double sn, cs;
    sincos(E * (double)j * tphys, &sn, &cs);
    acc += (j == 0 ? 1.0 : 2.0) * (cs * c[2 * j] - sn * c[2 * j + 1]);
  }
  const double tot = block_sum256(acc, sh);
  if (threadIdx.x == 0) {
    nrm[2 * row] = tphys / (2.0 * M_PI) * tot;
    nrm[2 * row + 1] = 0.0;
  }
}

int spt_for(int precision, int S) { return (precision == TBPM_C64 && S >= 2) ? 2 : 1; }

template <typename R, int SPT, int TA, int TB>
int xdot_launch(tbpm_ctx* ctx, const XdotArgs& xa0, int G) {
  XdotArgs xa = xa0;
  const int pairs = ((xa.nA + TA - 1) / TA) * ((xa.nB + TB - 1) / TB);
  k_xdot<R, SPT, TA, TB><<<dim3(pairs, G), kThreads, 0, ctx->stream>>>(xa);
  TBPM_CK_LAUNCH(ctx);
  return TBPM_OK;
}

template <int SPT, int TA, int TB>
int xdot_c64_launch(tbpm_ctx* ctx, const XdotArgs& xa, const XTile& tl, dim3 grid) {
  cudaStream_t st = ctx->stream;
  if constexpr (SPT == 1) {
    k_xdot_c64<1, TA, TB, 0><<<grid, kThreads, 0, st>>>(xa, tl);
  } else {
    switch (xa.P) {
      case 1: k_xdot_c64<2, TA, TB, 0><<<grid, kThreads, 0, st>>>(xa, tl); break;
      case 2: k_xdot_c64<2, TA, TB, 1><<<grid, kThreads, 0, st>>>(xa, tl); break;
      case 4: k_xdot_c64<2, TA, TB, 2><<<grid, kThreads, 0, st>>>(xa, tl); break;
      case 8: k_xdot_c64<2, TA, TB, 3><<<grid, kThreads, 0, st>>>(xa, tl); break;
      default: k_xdot_c64<2, TA, TB, 4><<<grid, kThreads, 0, st>>>(xa, tl); break;
    }
  }
  TBPM_CK_LAUNCH(ctx);
  return TBPM_OK;
}

}  // namespace

// Bond-vector components (r_j - r_i)_alpha per sublattice and neighbour slot, times t.
void current_weights(int kind, int direction, double t, double kw[2][6]) {
  for (int s = 0; s < 2; ++s)
    for (int d = 0; d < 6; ++d) kw[s][d] = 0.0;
  if (kind == TBPM_HONEYCOMB) {
    const double h = sqrt(3.0) / 2.0;
    const double vx[3] = {1.0, -0.5, -0.5}, vy[3] = {0.0, -h, h};
    for (int d = 0; d < 3; ++d) {
      const double c = direction == 0 ? vx[d] : direction == 1 ? vy[d] : 0.0;
      kw[0][d] = t * c;
      kw[1][d] = -t * c;
    }
  } else {
    // slots +x, -x, +y, -y, +z, -z
    for (int d = 0; d < 6; ++d) {
      const double c = (d / 2 == direction) ? ((d & 1) ? -1.0 : 1.0) : 0.0;
      kw[0][d] = kw[1][d] = t * c;
    }
  }
}

int launch_current(tbpm_ctx* ctx, const tbpm_lattice* lat, int precision, int S, int direction, const void* x,
                   void* y, bool full) {
  CurArgs c;
  c.g = lat->geom;
  c.path = full ? TBPM_PATH_STENCIL : lat->path;
  c.masked = full ? lat->dfull : nullptr;
  c.ell = lat->ell;
  c.full_of = lat->full_of;
  c.n_sites = full ? lat->geom.n_full : lat->n_sites;
  const int spt = spt_for(precision, S);
  c.P = S / spt;
  c.logP = 0;
  while ((1 << c.logP) < c.P) ++c.logP;
  current_weights(lat->desc.kind, direction, lat->desc.t, c.kw);
  for (int k = 0; k < 12; ++k) (&c.kwf[0][0])[k] = (float)(&c.kw[0][0])[k];
  c.kwl = lat->jw ? lat->jw + (size_t)direction * 2 * lat->geom.z : nullptr;
  if (c.path == TBPM_PATH_CSR && !c.ell) {
    set_error("current operator: ELL lists missing");
    return TBPM_EINVAL;
  }
  const int64_t n_units = c.n_sites * c.P;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((n_units + kThreads - 1) / kThreads,
                                                               (int64_t)ctx->num_sms * 8));
  if (precision == TBPM_C128)
    k_current<double, 1><<<grid, kThreads, 0, ctx->stream>>>(c, x, y);
  else if (spt == 2)
    k_current<float, 2><<<grid, kThreads, 0, ctx->stream>>>(c, x, y);
  else
    k_current<float, 1><<<grid, kThreads, 0, ctx->stream>>>(c, x, y);
  TBPM_CK_LAUNCH(ctx);
  return TBPM_OK;
}

// out[(s*os + a*oa + b*ob + off)] (complex) = <A_a|B_b> for state s; blocks are [n_sites][S].
int launch_xdot(tbpm_ctx* ctx, int precision, int S, int64_t n_sites, const void* A, int nA, const void* B, int nB,
                double* out, int64_t os, int64_t oa, int64_t ob, int64_t off) {
  if (nA < 1 || nB < 1) return TBPM_OK;
  const int spt = spt_for(precision, S);
  XdotArgs xa;
  xa.A = A;
  xa.B = B;
  xa.nA = nA;
  xa.nB = nB;
  xa.P = S / spt;
  xa.S = S;
  xa.n_units = n_sites * xa.P;
  xa.a_stride = xa.n_units;
  xa.b_stride = xa.n_units;
  xa.n_chunks = (xa.n_units + kXChunk - 1) / kXChunk;
  const bool single = nA == 1;
  const bool c128 = precision == TBPM_C128;
  const int TA = single ? 1 : (spt == 2 ? 2 : 4), TB = c128 ? (single ? 8 : 4) : (single ? (spt == 2 ? 8 : 16) : 4);
  const int at = (nA + TA - 1) / TA, bt = (nB + TB - 1) / TB;
  const int64_t per = (int64_t)nA * nB * S * 2;
  const int64_t cap = std::max<int64_t>(1, (64LL << 20) / (int64_t)(per * sizeof(double)));  // partials of 64 MiB
  if ((int64_t)at * bt > 2147483647LL) {
    set_error("too many state-block pairs");
    return TBPM_EUNSUPPORTED;
  }
  if (c128) {
    // enough CTAs for ~4 waves of 2 per SM
    int64_t G = std::max<int64_t>(1, ((int64_t)ctx->num_sms * 8 + (int64_t)at * bt - 1) / ((int64_t)at * bt));
    G = std::min<int64_t>(std::min<int64_t>(G, xa.n_chunks), std::min<int64_t>(cap, 65535));
    TBPM_TRY(ensure(ctx, ctx->ws_xdot, sizeof(double) * (size_t)(per * G)));
    xa.partials = (double*)ctx->ws_xdot.p;
    TBPM_TRY((single ? xdot_launch<double, 1, 1, 8>(ctx, xa, (int)G) : xdot_launch<double, 1, 4, 4>(ctx, xa, (int)G)));
    return launch_partial_reduce(ctx, xa.partials, (int)G, nA, nB, S, out, os, oa, ob, off);
  }
  // tiles per CTA: up to four along A (they share the B blocks), then along B, a power of two up to 8
  XTile tl{at, bt, 1, 1};
  while (tl.wa < 4 && tl.wa < at) tl.wa *= 2;
  while (tl.wa * tl.wb < kWarps && tl.wb < bt) tl.wb *= 2;
  const int share = kWarps / (tl.wa * tl.wb);
  const int64_t ctas = (int64_t)((at + tl.wa - 1) / tl.wa) * ((bt + tl.wb - 1) / tl.wb);
  const int64_t spans = (xa.n_units + 32 * kXIter - 1) / (32 * kXIter);  // chunks a warp can take
  int64_t G = std::max<int64_t>(1, ((int64_t)ctx->num_sms * 4 + ctas - 1) / ctas);
  G = std::min<int64_t>(G, (spans + share - 1) / share);
  G = std::max<int64_t>(1, std::min<int64_t>(G, std::min<int64_t>(cap, 65535)));
  TBPM_TRY(ensure(ctx, ctx->ws_xdot, sizeof(double) * (size_t)(per * G)));
  xa.partials = (double*)ctx->ws_xdot.p;
  const dim3 grid((unsigned)ctas, (unsigned)G);
  int r;
  if (spt == 2) r = single ? xdot_c64_launch<2, 1, 8>(ctx, xa, tl, grid) : xdot_c64_launch<2, 2, 4>(ctx, xa, tl, grid);
  else r = single ? xdot_c64_launch<1, 1, 16>(ctx, xa, tl, grid) : xdot_c64_launch<1, 4, 4>(ctx, xa, tl, grid);
  TBPM_TRY(r);
  return launch_partial_reduce(ctx, xa.partials, (int)G, nA, nB, S, out, os, oa, ob, off);
}

int launch_partial_reduce(tbpm_ctx* ctx, const double* partials, int G, int nA, int nB, int S, double* out,
                          int64_t os, int64_t oa, int64_t ob, int64_t off) {
  const int64_t per = (int64_t)nA * nB * S * 2;
  k_xdot_reduce<<<(unsigned)((per + 31) / 32), 1024, 0, ctx->stream>>>(partials, G, nA, nB, S, out, os, oa, ob, off);
  TBPM_CK_LAUNCH(ctx);
  return TBPM_OK;
}

int launch_ec_corr_from_moments(tbpm_ctx* ctx, const double* table, const int* n_per_step, int n_steps,
                                const double* m, int rows, int Nn, double shift, double tau, double* C) {
  k_ec_corr_m<<<dim3(n_steps + 1, (rows + kEcRows - 1) / kEcRows), 256, 0, ctx->stream>>>(
      table, n_per_step, n_steps, m, rows, Nn, shift, tau, C);
  TBPM_CK_LAUNCH(ctx);
  return TBPM_OK;
}

int launch_ec_overlap(tbpm_ctx* ctx, const double* corr, const double* energies, int nE, int rows, int n_steps,
                      double tphys, double* nrm) {
  k_ec_overlap<<<rows, 256, 0, ctx->stream>>>(corr, energies, nE, n_steps, tphys, nrm);
  TBPM_CK_LAUNCH(ctx);
  return TBPM_OK;
}

int launch_ec_finish(tbpm_ctx* ctx, double* C, const double* nrm, const double* energies, int nE, int rows,
                     int n_steps, double tphys, double area, double* sigma) {
  k_ec_finish<<<rows, 256, 0, ctx->stream>>>(C, nrm, energies, nE, n_steps, tphys, area, sigma);
  TBPM_CK_LAUNCH(ctx);
  return TBPM_OK;
}

}  // namespace tbpm
