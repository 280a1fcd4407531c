// Resident moment recurrence: every Chebyshev step of a request in one cooperative launch, for lattices
// whose two state blocks fit in the SMs' shared memory (up to about 15 MB a block, 2M complex64 site-states;
// use_resident says which of them).
//
// One launch per step costs 6 to 8 us on a small lattice (launch, cold L1, the grid reduction's tail),
// whatever its size.  Here a CTA owns a run of lattice lines (x-lines of the [row][site][state] layout) for
// the whole request and keeps phi_n and phi_{n-1} of its lines, and their on-site terms, in shared memory.
// Units of a line with a neighbour line in another CTA are also published in global memory as packets of
// 16 bytes, two 64-bit halves of a data word and a tag that names the step, in one of two buffers by the parity
// of n; a step's thread reads its remote neighbours by polling their packets until both tags are those of phi_n.  So data and flag travel together: no fence, no
// barrier between CTAs, one L2 round trip per step (flags with release and acquire and a read of the data
// after them took 2.7 us per step on 64 x 64 complex128 sites, packets take 2.0).  A buffer is safe to reuse: the thread that
// overwrites its packet of phi_n with phi_{n+2} has read the phi_{n+1} of every thread that reads the packet
// (neighbours are mutual), and those were formed from phi_n.  Tags are never used twice (a counter in the
// context).  All CTAs are resident (cooperative launch), so every wait ends; each is bounded all the same.  A
// thread whose wait expired waits no more, its CTA ends with the step, the CTAs that wait for it follow within
// their own two seconds, and the status word reports it.
//
// Moments: <phi_n|phi_n> and Re <phi_{n+1}|phi_n> (real for a Hermitian H~), summed per thread (at most 32
// units), reduce-scattered over the lanes of a state pair -- FP32 values as compensated
// pairs, so no precision is lost in the tree -- and added in FP64 over the warps in a fixed order; the
// per-CTA sums of every step are added in CTA order by a second kernel.  Deterministic.
//
// Bound: the exchange latency per step (a packet's way through L2 to the polling thread) for small lattices; shared-memory
// bandwidth (complex64) or FP64 issue (complex128) when the blocks are large.  Measured, us per step, one
// launch per step -> resident: 64 x 64 square, complex128, one state 6.6 -> 2.1; 45 x 47 honeycomb, 4 states
// 8.1 -> 2.0; 40^3 cubic, 8 states 23.8 -> 7.5.
#include <cuda_runtime.h>
#include <string.h>

#include <algorithm>
#include <mutex>

#include "stencil.cuh"
#include "tbpm_internal.cuh"

namespace tbpm {
namespace {

constexpr int kResThreads = 512;     // at most; fewer where a CTA owns fewer units
constexpr int kResBatch = 8;         // steps whose warp sums are added and stored together
constexpr int kResMaxCtas = 256;
constexpr int kResMaxUnits = 32;     // units of a thread, summed in FP32
constexpr uint64_t kResWaitNs = 2000000000ull;  // 2 s per packet

struct ResArgs {
  Geom g;
  const void* diag;   // per-site D_i or null
  double diag_const, thop;
  float th1f, dc1f;
  const void* x0;     // phi_0
  ulonglong2* packets;     // [2][units][packets per unit]
  int64_t n_units;
  unsigned tag;       // phi_n is published with tag + n
  int P, logP, S;
  int lines, upr;     // lines per CTA, units per line
  uint32_t magic;     // ceil(2^32 / upr): unit / upr for units below 2^16
  int steps;
  double* partials;   // [steps][S * 2][gridDim.x]
  int* status;
};

__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// A packet: two 64-bit words, each a data word below its tag; 64-bit accesses are single-copy atomic, so a
// word whose tag is right carries the right data.
template <typename R, int SPT>
struct Packets {
  static constexpr int N = sizeof(Pack<R, SPT>) / 8;  // packets of a unit
};
template <typename R, int SPT>
__device__ __forceinline__ void publish(ulonglong2* p, const Pack<R, SPT>& v, unsigned tag) {
  unsigned w[sizeof(Pack<R, SPT>) / 4];
  memcpy(w, &v, sizeof(v));
  const uint64_t t = (uint64_t)tag << 32;
#pragma unroll
  for (int k = 0; k < Packets<R, SPT>::N; ++k)
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p + k), "l"(t | w[2 * k]), "l"(t | w[2 * k + 1])
                 : "memory");
}
// The unit once it carries the tag; false when budget_ns pass without it.
template <typename R, int SPT>
__device__ __forceinline__ bool receive(const ulonglong2* p, unsigned tag, uint64_t budget_ns, Pack<R, SPT>& v) {
  constexpr int N = Packets<R, SPT>::N;
  uint64_t q[2 * N], t0 = 0;
  for (int spin = 0;; ++spin) {
    bool here = true;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(q[2 * k]), "=l"(q[2 * k + 1]) : "l"(p + k) : "memory");
      here = here && (unsigned)(q[2 * k] >> 32) == tag && (unsigned)(q[2 * k + 1] >> 32) == tag;
    }
    if (here) break;
    if ((spin & 255) == 255) {
      const uint64_t t = now_ns();
      if (t0 == 0) t0 = t;
      else if (t - t0 > budget_ns) return false;
    }
  }
  unsigned w[2 * N];
#pragma unroll
  for (int k = 0; k < 2 * N; ++k) w[k] = (unsigned)q[k];
  memcpy(&v, w, sizeof(v));
  return true;
}

// The same for a thread that has many to wait for: zero once one of its waits has expired (failed).
template <typename R, int SPT>
__device__ __forceinline__ Pack<R, SPT> receive_or_zero(const ulonglong2* p, unsigned tag, uint64_t budget_ns,
                                                        bool& failed) {
  Pack<R, SPT> v{};
  if (!failed) failed = !receive<R, SPT>(p, tag, budget_ns, v);
  return v;
}

// Neighbour lines of a line, in the neighbour order of the stencil: y + 1, y - 1, z + 1, z - 1 (-1: none).
template <int KIND>
__device__ __forceinline__ void line_neighbours(const Geom& g, int64_t row, int64_t (&nb)[4]) {
  const LineBases b = line_bases<KIND>(g, row, 1);  // bases in lines
  nb[0] = b.up;
  nb[1] = b.dn;
  nb[2] = b.zup;
  nb[3] = b.zdn;
}

// MAXT: threads at most.  512 threads with the registers they would like (78 to 84) fill an SM's register file, and
// requests of two contexts took turns: with two CTAs to an SM (48 registers, no spills) 100 x 100 honeycomb cells
// with 8 states from eight contexts went from 1086 to 2355 requests a second and one context's from 1026 to 970.
// Smaller CTAs leave room as they are.
template <int KIND, typename R, int SPT, int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT == kResThreads ? 2 : 1) k_resident(ResArgs a) {
  using PK = Pack<R, SPT>;
  constexpr int NL = KIND == TBPM_CUBIC ? 4 : 2;  // neighbour lines
  constexpr int NV = 2 * SPT;                     // sums per thread: A and B of each state of the unit
  extern __shared__ __align__(16) unsigned char smraw[];
  const Geom g = a.g;
  const int P = a.P, logP = a.logP, upr = a.upr, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int NT = blockDim.x, warps = NT >> 5;
  const int64_t l0 = (int64_t)blockIdx.x * a.lines;
  const int nl = (int)(l0 + a.lines < g.n_rows ? a.lines : g.n_rows - l0);
  const int nu = nl * upr, cap = a.lines * upr;  // units owned, units of a full CTA
  PK* sA = reinterpret_cast<PK*>(smraw);
  PK* sB = sA + cap;
  double* red = reinterpret_cast<double*>(sB + cap + (cap & 1));  // [kResBatch][warps][P * NV]
  int64_t* tab = reinterpret_cast<int64_t*>(red + kResBatch * warps * P * NV);  // [lines][NL]
  unsigned char* pub = reinterpret_cast<unsigned char*>(tab + (size_t)a.lines * NL);  // [lines], padded
  R* sD = reinterpret_cast<R*>(pub + ((a.lines + 15) & ~15));
  const bool has_diag = a.diag != nullptr;

  // tables: where a line's neighbour lines are (>= 0: unit offset in shared memory, -1: nowhere,
  // <= -2: -(unit offset in the lattice) - 2, in another CTA), and which lines others read
  for (int li = tid; li < nl; li += NT) {
    int64_t nb[4];
    line_neighbours<KIND>(g, l0 + li, nb);
    bool out = false;
#pragma unroll
    for (int d = 0; d < NL; ++d) {
      const int64_t r = nb[d];
      int64_t v = -1;
      if (r >= 0) {
        if (r >= l0 && r < l0 + nl) {
          v = (r - l0) * upr;
        } else {
          v = -(r * upr) - 2;
          out = true;
        }
      }
      tab[li * NL + d] = v;
    }
    pub[li] = out;
  }
  const PK* x0 = reinterpret_cast<const PK*>(a.x0) + l0 * upr;
  for (int u = tid; u < nu; u += NT)
    if (TBPM_DBG_OK(l0 * upr + u, a.n_units, TBPM_DBG_RESIDENT)) sA[u] = x0[u];
  if (has_diag)
    for (int i = tid; i < (nu >> logP); i += NT)
      if (TBPM_DBG_OK((l0 * upr >> logP) + i, g.n_full, TBPM_DBG_RESIDENT))
        sD[i] = reinterpret_cast<const R*>(a.diag)[(l0 * upr >> logP) + i];
  __syncthreads();
  PK* cur = sA;
  PK* prv = sB;
  const int p = tid & (P - 1);
  const int Lx = (int)g.Lx;
  const R D0 = sizeof(R) == 4 ? (R)a.dc1f : (R)a.diag_const;
  const R T0 = sizeof(R) == 4 ? (R)a.th1f : (R)a.thop;
  bool failed = false;
  for (int n = 0; n < a.steps; ++n) {
    const bool first = n == 0;
    const R th = first ? T0 : T0 + T0, dc = first ? D0 : D0 + D0;
    constexpr int NP = Packets<R, SPT>::N;
    const ulonglong2* pr_in = a.packets + (n & 1) * a.n_units * NP;
    ulonglong2* pr_out = a.packets + (((n + 1) & 1) * a.n_units + l0 * upr) * NP;
    const unsigned tag = a.tag + (unsigned)n;
    R s[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) s[k] = R(0);
#pragma unroll 2
    for (int u = tid; u < nu; u += NT) {
      const int li = (int)(((uint64_t)(uint32_t)u * a.magic) >> 32);
      const int q = u - li * upr;  // unit in the line
      const PK ph = cur[u];
      PK h;
      bool any = false;
      auto take = [&](const PK& t) {
#pragma unroll
        for (int w = 0; w < 2 * SPT; ++w) h.v[w] = any ? h.v[w] + t.v[w] : t.v[w];
        any = true;
      };
      auto line = [&](int d, int off) {  // unit `off` of neighbour line d
        const int64_t t = tab[li * NL + d];
        if (t >= 0) take(cur[(int)t + off]);
        else if (t != -1) {
          const int64_t r = -(t + 2) + off;
          if (!TBPM_DBG_OK(r, a.n_units, TBPM_DBG_RESIDENT)) return;
          if (first) take(reinterpret_cast<const PK*>(a.x0)[r]);
          else take(receive_or_zero<R, SPT>(pr_in + r * NP, tag, kResWaitNs, failed));
        }
      };
#pragma unroll
      for (int w = 0; w < 2 * SPT; ++w) h.v[w] = R(0);
      if constexpr (KIND == TBPM_HONEYCOMB) {
        const int sir = q >> logP, sub = sir & 1, xc = sir >> 1;
        take(cur[u ^ P]);
        if (sub) {
          if (xc < Lx - 1) take(cur[u + P]);
          else if (g.pbc_x) take(cur[li * upr + p]);
          line(0, q - P);
        } else {
          if (xc > 0) take(cur[u - P]);
          else if (g.pbc_x) take(cur[u - P + upr]);
          line(1, q + P);
        }
      } else {
        const int xc = q >> logP;
        if (xc < Lx - 1) take(cur[u + P]);
        else if (g.pbc_x) take(cur[li * upr + p]);
        if (xc > 0) take(cur[u - P]);
        else if (g.pbc_x) take(cur[u - P + upr]);
#pragma unroll
        for (int d = 0; d < NL; ++d) line(d, q);
      }
      R d = dc;
      if (has_diag) {
        const R dd = sD[u >> logP];
        d = first ? dd : dd + dd;
      }
      PK o;
      if (first) {
#pragma unroll
        for (int w = 0; w < 2 * SPT; ++w) o.v[w] = fma(d, ph.v[w], th * h.v[w]);
      } else {
        const PK pv = prv[u];
#pragma unroll
        for (int w = 0; w < 2 * SPT; ++w) o.v[w] = fma(d, ph.v[w], fma(th, h.v[w], -pv.v[w]));
      }
      prv[u] = o;
      if (pub[li] && TBPM_DBG_OK(l0 * upr + u, a.n_units, TBPM_DBG_RESIDENT))
        publish<R, SPT>(pr_out + (int64_t)u * NP, o, tag + 1);
#pragma unroll
      for (int k = 0; k < SPT; ++k) {
        const R pr = ph.v[2 * k], pi = ph.v[2 * k + 1];
        s[2 * k] = fma(pr, pr, fma(pi, pi, s[2 * k]));
        s[2 * k + 1] = fma(o.v[2 * k], pr, fma(o.v[2 * k + 1], pi, s[2 * k + 1]));
      }
    }
    if (__syncthreads_or(failed ? 1 : 0)) {
      if (tid == 0) atomicExch(a.status, 3);
      return;
    }
    // warp sums of this step
    {
      using SumT = decltype(sum_of(R(0)));
      SumT v[NV];
#pragma unroll
      for (int k = 0; k < NV; ++k) v[k] = sum_of(s[k]);
      double* slot = red + ((size_t)(n & (kResBatch - 1)) * warps + warp) * P * NV + (lane & (P - 1)) * NV;
      reduce_lanes<NV>(v, P, logP, lane, [&](int k, double t) { slot[k] = t; });
    }
    if ((n & (kResBatch - 1)) == kResBatch - 1 || n == a.steps - 1) {
      const int n0 = n & ~(kResBatch - 1), have = n - n0 + 1;
      __syncthreads();
      for (int i = tid; i < have * P * NV; i += NT) {
        const int j = i / (P * NV), q = i - j * (P * NV);
        double t = 0.0;
        for (int w = 0; w < warps; ++w) t += red[((size_t)j * warps + w) * P * NV + q];
        a.partials[((size_t)(n0 + j) * P * NV + q) * gridDim.x + blockIdx.x] = t;
      }
      __syncthreads();
    }
    PK* t = cur;
    cur = prv;
    prv = t;
  }
}

// Moments from the per-CTA sums: one block per step; value q = (2 s + c), c = 0: <phi_n|phi_n>, 1: Re <phi_{n+1}|phi_n>.
__global__ void __launch_bounds__(256) k_resident_moments(const double* partials, int ctas, int S, double* mu, int M) {
  const int n = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto total = [&](int step, int q) {
    const double* p = partials + ((size_t)step * 2 * S + q) * ctas;
    double t = 0.0;
    for (int i = lane; i < ctas; i += 32) t += p[i];
    for (int off = 16; off >= 1; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    return t;
  };
  for (int q = warp; q < 2 * S; q += 8) {
    const double first = total(0, q), t = n == 0 ? first : total(n, q);
    if (lane == 0) {
      double* m = mu + ((size_t)(q >> 1) * M + 2 * n + (q & 1)) * 2;
      m[0] = n == 0 ? t : 2.0 * t - first;
      m[1] = 0.0;
    }
  }
}

template <typename R, int SPT, int MAXT>
void* resident_kind(int kind) {
  return kind == TBPM_SQUARE      ? (void*)k_resident<TBPM_SQUARE, R, SPT, MAXT>
         : kind == TBPM_HONEYCOMB ? (void*)k_resident<TBPM_HONEYCOMB, R, SPT, MAXT>
                                  : (void*)k_resident<TBPM_CUBIC, R, SPT, MAXT>;
}

template <typename R, int SPT>
void* resident_fn(int kind, int threads) {
  return threads <= kResThreads / 2 ? resident_kind<R, SPT, kResThreads / 2>(kind) : resident_kind<R, SPT, kResThreads>(kind);
}

// Lines per CTA and shared memory of a request; false when it does not fit.
struct ResPlan {
  int lines, ctas, upr, threads;
  size_t smem;
};
bool plan_resident(tbpm_ctx* ctx, const Geom& g, int precision, int Spad, bool diag, ResPlan* r) {
  const int spt = precision == TBPM_C64 && Spad >= 2 ? 2 : 1, P = Spad / spt;
  const size_t unit = precision == TBPM_C64 ? 8 * (size_t)spt : 16, real = precision == TBPM_C64 ? 4 : 8;
  const int64_t upr = g.row_sites * P, most = std::min(ctx->num_sms, kResMaxCtas);
  const int64_t lines = (g.n_rows + most - 1) / most;
  // a thread's share of FP32 sums (220 KB hold at most 28 units a thread), within the range of the division
  // by multiplication
  if (lines * upr > kResMaxUnits * kResThreads || upr < 2) return false;
  const size_t cap = (size_t)(lines * upr);
  r->lines = (int)lines;
  r->ctas = (int)((g.n_rows + lines - 1) / lines);
  r->upr = (int)upr;
  r->threads = (int)std::min<size_t>(kResThreads, std::max<size_t>(64, (cap + 31) / 32 * 32));
  r->smem = 2 * cap * unit + (cap & 1) * unit + sizeof(double) * kResBatch * (r->threads / 32) * P * 2 * spt +
            sizeof(int64_t) * (size_t)lines * (g.kind == TBPM_CUBIC ? 4 : 2) + ((lines + 15) & ~15) +
            (diag ? cap / P * real : 0);
  return r->smem <= 220 * 1024;
}

}  // namespace

// Whether a request's recurrence runs resident: a stencil lattice whose two blocks fit in shared memory.
bool resident_applicable(tbpm_ctx* ctx, const tbpm_lattice* lat, int precision, int Spad, int64_t steps) {
  ResPlan r;
  if (lat->path != TBPM_PATH_STENCIL || steps < 2) return false;
  if (!plan_resident(ctx, lat->geom, precision, Spad, lat->has_v, &r)) return false;
  return (size_t)steps * 2 * Spad * r.ctas * sizeof(double) <= (512u << 20);  // per-CTA sums of every step
}

// All `steps` steps from phi_0 in x0.  TBPM_EUNSUPPORTED where the grid cannot be resident as a whole (fewer SMs
// for this process than the device has, no cooperative launches): the caller takes another pass.
int launch_resident(tbpm_ctx* ctx, const tbpm_lattice* lat, const RecurrenceArgs& ra, int precision, const void* x0,
                    int64_t steps) {
  ResPlan r;
  if (!plan_resident(ctx, lat->geom, precision, ra.S, ra.diag != nullptr, &r)) {
    set_error("resident recurrence: the lattice does not fit");
    return TBPM_EUNSUPPORTED;
  }
  const int spt = precision == TBPM_C64 && ra.S >= 2 ? 2 : 1;
  const int kind = lat->geom.kind;
  void* fn = precision == TBPM_C128 ? resident_fn<double, 1>(kind, r.threads)
             : spt == 2 ? resident_fn<float, 2>(kind, r.threads) : resident_fn<float, 1>(kind, r.threads);
  TBPM_CK(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
  TBPM_TRY(ensure(ctx, ctx->ws_fused_partials, sizeof(double) * (size_t)steps * 2 * ra.S * r.ctas));
  // packets: their tags must never meet an earlier launch's, so the buffer starts at zero and the tags count on
  const int64_t n_units = lat->geom.n_rows * (int64_t)r.upr;
  const size_t packet_bytes = (size_t)n_units * 2 * (precision == TBPM_C64 ? 16 * spt : 32);
  const void* old = ctx->ws_packets.p;
  TBPM_TRY(ensure(ctx, ctx->ws_packets, packet_bytes));
  if (ctx->ws_packets.p != old || ctx->packet_cap != ctx->ws_packets.cap || ctx->packet_tag + steps > 0xfffffff0ll) {
    TBPM_CK(cudaMemsetAsync(ctx->ws_packets.p, 0, ctx->ws_packets.cap, ctx->stream));
    ctx->packet_cap = ctx->ws_packets.cap;
    ctx->packet_tag = 0;
  }
  ResArgs a;
  memset(&a, 0, sizeof(a));
  a.g = lat->geom;
  a.diag = ra.diag;
  a.diag_const = ra.diag_const;
  a.thop = ra.thop;
  a.th1f = ra.th1f;
  a.dc1f = ra.dc1f;
  a.x0 = x0;
  a.packets = (ulonglong2*)ctx->ws_packets.p;
  a.n_units = n_units;
  a.tag = (unsigned)ctx->packet_tag;  // phi_1 is the first to be published: tags tag + 1 .. tag + steps
  ctx->packet_tag += steps;
  a.P = ra.P;
  a.logP = ra.logP;
  a.S = ra.S;
  a.lines = r.lines;
  a.upr = r.upr;
  a.magic = (uint32_t)(((1ull << 32) + r.upr - 1) / r.upr);
  a.steps = (int)steps;
  a.partials = (double*)ctx->ws_fused_partials.p;
  a.status = reinterpret_cast<int*>(ctx->pinned + kSweepStatusSlot);
  void* args[] = {&a};
  const cudaError_t e = cudaLaunchCooperativeKernel(fn, dim3(r.ctas), dim3(r.threads), args, r.smem, ctx->stream);
  if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
    cudaGetLastError();
    set_error("resident recurrence: %s", cudaGetErrorString(e));
    return TBPM_EUNSUPPORTED;
  }
  TBPM_CK(e);
  ctx->launches++;
  k_resident_moments<<<(unsigned)steps, 256, 0, ctx->stream>>>(a.partials, r.ctas, ra.S, ra.mu, ra.M);
  TBPM_CK_LAUNCH(ctx);
  return TBPM_OK;
}

}  // namespace tbpm

TBPM_DEBUG_UNIT(resident)
