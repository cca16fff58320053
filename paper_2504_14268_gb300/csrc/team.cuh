// Team solver: one system solved by a team of CTAs whose scalars travel in one hop.
//
// What bounds a small or middle-sized solve is not bandwidth but the chain of one iteration:
// product -> nu -> alpha -> residual -> rho, sigma -> beta, action -> direction -> product.
// cg_persistent pays for each of the three team steps an arrival counter, a reduction by the
// last CTA, a scalar step on state in global memory and a release that the others poll, about
// 10 us each. Here
//   * every CTA keeps its own copy of the system's state, descriptor and Q-table
//     in shared memory and runs the scalar step itself on the same sums in the same order, so
//     the copies stay equal bit for bit and nothing has to be broadcast;
//   * a step's partial sums go from each CTA to every other in one message that carries data
//     and signal together: in a cluster, st.async into the peers' shared memory completing on
//     their mbarriers; over the whole grid, one 16-byte word {value, epoch} per CTA that the
//     others poll;
//   * r, p, x and q (then z) of a CTA's rows live in its shared memory (32 bytes per row; in
//     global memory when they do not fit), so phases B and C touch no global memory but p's
//     copy that the next product gathers.
// Three exchanges per iteration remain: nu, (||r||^2, sigma), and the release of p.
#pragma once
#define MPCG_STEP __noinline__
#include "solver.cuh"

namespace mpcg {
namespace {

constexpr int kTT = kTeamThreads;
constexpr int kIcBars = kTeamIcBars;
constexpr int kTW = kTT / 32;
constexpr int kXV = 4;            // values per exchange at most
constexpr int kMidRow = 32;       // longer rows are summed by a warp
constexpr int kShortRow = 8;      // matrices of rows up to this load a row at once
constexpr int kLongBatch = 16;    // rows summed by the CTA between two barriers
constexpr int kLongRowTeam = 512; // ... and longer ones by the CTA (fp32: kLongRow, see team_product)

// A CTA's rows and where their vectors live (index row - r0).
struct TeamVec {
  int r0, n;
  double *r, *p, *x, *q;
};

struct TeamSmem {
  Smem sm;
  SysState st;
  DevSys S;
  TeamVec V;
  int rank, size;
  int base;           // clusters: the team's first CTA in the cluster
  uint4* gslot;       // whole-grid teams: [2][size][kXV] words {value, epoch}
  double* xs;         // ... polled values [kXV][size] (shared memory)
  double red[kXV][kTW];
  double slot[2][kTeamMaxCluster][kXV];
  double sum[kXV];
  unsigned long long xbar[2], pbar[2];
  double lpart[kLongBatch][kTW];  // long rows: the warps' partial accumulations
  float2 lcorr[kLongBatch][kTW];
  int lrow[kLongBatch];
  int nq, nl;  // queued rows (zero between products)
  unsigned char* tile;            // the warps' tiles of the product, or nullptr
  const int *rp, *ci;             // the row bounds and columns, the matrix's or the CTA's own copy, ...
  int rbase, ebase;               // ... whose first elements are these rows and entries
  int queue[kTT];
  float* icW;                     // IC(0): the substitutions' vector (used in the team's first CTA)
  unsigned char* icring;          // ... and the ring of level blocks
  unsigned long long icbar[kIcBars];
  unsigned icuse;                 // ... blocks so far, modulo 2 kIcBars (the barriers' parity)
  unsigned icissued;              // ... blocks of this application whose copies have been issued
  int icstop[2];                  // ... a wait gave up
  int icdone;                     // ... levels consumed in this application
  // the short scalar step (team_step_b): squared thresholds ([0]: the tolerance) as bit patterns
  long long thr2[32];
  long long margin;   // distance of bit patterns below which the full step decides
  double rr;          // ||r||^2 of the last iteration when st.rho is not formed from it yet
  int stale;          // ... 1 then
  int fast, slow;     // the launch admits the short step; this iteration takes the full one
  int bad;
  int nact;  // warps that hold rows
  int ntop;  // half the next power of two of nact
};

// What a thread counts: exchanges and releases of p so far (the same in every thread).
struct Team {
  unsigned ep, pph;
};


__device__ __forceinline__ unsigned cluster_map(unsigned addr, int rank) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_async64(unsigned addr, double v, unsigned bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(addr),
               "l"(__double_as_longlong(v)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(unsigned long long* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, "
      "p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void st_word(uint4* p, double v, unsigned ep) {
  asm volatile("{\n .reg .b128 w;\n mov.b128 w, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], w;\n}\n" ::"l"(p),
               "l"(__double_as_longlong(v)), "l"((unsigned long long)ep)
               : "memory");
}
__device__ __forceinline__ void ld_word(const uint4* p, double& v, unsigned& ep) {
  long long a;
  unsigned long long e;
  asm volatile("{\n .reg .b128 w;\n ld.relaxed.gpu.global.b128 w, [%2];\n mov.b128 {%0, %1}, w;\n}\n"
               : "=l"(a), "=l"(e)
               : "l"(p)
               : "memory");
  v = __longlong_as_double(a);
  ep = (unsigned)e;
}

// Shared memory by 32-bit address.
__device__ __forceinline__ float lds_f32(unsigned a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ unsigned lds_u16(unsigned a) {
  unsigned short v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ int2 lds_v2(unsigned a) {
  int2 v;
  asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ int4 lds_v4(unsigned a) {
  int4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(a)
               : "memory");
  return v;
}
__device__ __forceinline__ int lds_acquire(unsigned a) {
  int v;
  asm volatile("ld.acquire.cta.shared.b32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts_release(unsigned a, int v) {
  asm volatile("st.release.cta.shared.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_f32(unsigned a, float v) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster_f32(unsigned addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ float ld_cluster_f32(unsigned addr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// A dot accumulator summed over the warp (the pair by an xor butterfly of TwoSum steps), in fp64.
__device__ __forceinline__ double warp_dot(DotAcc a, bool low) {
  if (!low) return warp_sum(a.d);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float s2 = __shfl_xor_sync(kFull, a.s, o), c2 = __shfl_xor_sync(kFull, a.c, o);
    float t;
    two_sum(a.s, s2, a.s, t);
    a.c = __fadd_rn(__fadd_rn(a.c, c2), t);
  }
  return (double)a.s + (double)a.c;
}

// A wait that exceeded the launch's limit, or another CTA's error: the CTA's threads see t.bad
// after their next barrier and leave together (solve_team returns false).
__device__ __forceinline__ bool wait_over(const Launch& L, TeamSmem& t, long long t0, unsigned spins) {
  if ((spins & 63u) != 0u) return false;
  if (!err_set(L)) {
    if (clock64() - t0 <= L.timeout_cycles) return false;
    atomicCAS(L.err, 0u, (unsigned)DERR_TIMEOUT);
  }
  t.bad = 1;
  return true;
}

// Sums v[0..nv) (values per warp, every lane the warp's own) over the team, each in the order
// warps, then CTAs by fixed trees, so that all CTAs get the same bits. The sums are in t.sum for
// thread 0 (for the others after the next CTA barrier). Contains CTA barriers. Only the warps
// that hold rows (the first t.nact) have values: an fp64 addition takes 64 cycles and the SM
// 19 cycles per warp, so an idle warp's part of the trees is worth leaving out.
template <bool CL, int NV>
__device__ __forceinline__ void team_exchange(const Launch& L, TeamSmem& t, Team& T, const double (&v)[NV], int nv = NV) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
#pragma unroll
    for (int j = 0; j < NV; ++j) t.red[j][w] = v[j];
  }
  __syncthreads();
  const int nact = t.nact;
  auto cta_value = [&](int j) {
    double s = lane < nact ? t.red[j][lane] : 0.0;
    for (int o = t.ntop; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
    return __shfl_sync(kFull, s, 0);
  };
  if (t.size == 1) {
    if (w < nv) {
      const double s = cta_value(w);
      if (lane == 0) t.sum[w] = s;
    }
    if (nv > 1) __syncthreads();
    return;
  }
  const unsigned ep = ++T.ep;
  const int par = (int)(ep & 1u);
  if constexpr (CL) {
    // the peers' slots of this parity were last read two exchanges ago, before those CTAs sent
    // the message of the exchange in between that this CTA has since received
    if (w < nv) {
      const double s = cta_value(w);
      if (lane < t.size)
        st_async64(cluster_map(smem_u32(&t.slot[par][t.rank][w]), t.base + lane), s,
                   cluster_map(smem_u32(&t.xbar[par]), t.base + lane));
    }
    if (w == 0) {
      if (lane == 0) mbar_expect_tx(&t.xbar[par], (unsigned)(t.size * nv * 8));
      __syncwarp();
      const unsigned want = ((ep - 1u) >> 1) & 1u;
      const long long t0 = clock64();
      unsigned spins = 0;
      while (!mbar_try_wait(&t.xbar[par], want))
        if (wait_over(L, t, t0, ++spins)) break;
      // lanes 0..15 sum value 0, lanes 16..31 value 1
      double s = 0.0;
      if ((lane & 15) < t.size && (lane >> 4) < nv) s = t.slot[par][lane & 15][lane >> 4];
      double s2 = NV > 2 && nv > 2 && lane < t.size ? t.slot[par][lane][2] : 0.0;
      for (int o = t.size >> 1; o > 0; o >>= 1) {
        s += __shfl_xor_sync(kFull, s, o);
        if (NV > 2) s2 += __shfl_xor_sync(kFull, s2, o);
      }
      if ((lane & 15) == 0) t.sum[lane >> 4] = s;
      if (NV > 2 && lane == 0) t.sum[2] = s2;
      __syncwarp();
    }
  } else {
    uint4* buf = t.gslot + (long long)par * t.size * kXV;
    if (w < nv) {
      const double s = cta_value(w);
      if (lane == 0) st_word(buf + (long long)t.rank * kXV + w, s, ep);
    }
    for (int i = threadIdx.x; i < t.size * nv; i += kTT) {
      const int c = i / nv, j = i - c * nv;
      double x;
      unsigned e;
      const long long t0 = clock64();
      unsigned spins = 0;
      ld_word(buf + (long long)c * kXV + j, x, e);
      while (e != ep) {
        if (wait_over(L, t, t0, ++spins)) break;
        ld_word(buf + (long long)c * kXV + j, x, e);
      }
      t.xs[j * t.size + c] = x;
    }
    __syncthreads();
    if (w < nv) {
      double s = 0.0;
      for (int c = lane; c < t.size; c += 32) s += t.xs[w * t.size + c];
      s = warp_sum(s);
      if (lane == 0) t.sum[w] = s;
    }
    if (nv > 1) __syncthreads();
  }
}

// Makes this CTA's global stores (p's copy, or x) visible to the team and waits for the
// others'. Starts and ends with a CTA barrier or an equivalent wait of every thread.
template <bool CL>
__device__ __forceinline__ void team_publish(const Launch& L, TeamSmem& t, Team& T) {
  __syncthreads();
  if (t.size == 1) return;
  if constexpr (CL) {
    if (threadIdx.x < t.size)
      asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(
                       cluster_map(smem_u32(&t.pbar[T.pph & 1u]), t.base + (int)threadIdx.x))
                   : "memory");
    // (two barriers in turn: a peer that is ahead by one release may arrive for it before another
    // peer's arrival for this one is here)
    unsigned long long* bar = &t.pbar[T.pph & 1u];
    const unsigned par = (T.pph >> 1) & 1u;
    ++T.pph;
    const long long t0 = clock64();
    unsigned spins = 0;
    while (!mbar_try_wait_cluster(bar, par))
      if (wait_over(L, t, t0, ++spins)) break;
  } else {
    const unsigned ep = ++T.ep;
    uint4* buf = t.gslot + (long long)(ep & 1u) * t.size * kXV;
    if (threadIdx.x == 0) {
      __threadfence();
      st_word(buf + (long long)t.rank * kXV, 0.0, ep);
    }
    if (threadIdx.x < t.size) {
      double x;
      unsigned e;
      const long long t0 = clock64();
      unsigned spins = 0;
      ld_word(buf + (long long)threadIdx.x * kXV, x, e);
      while (e != ep) {
        if (wait_over(L, t, t0, ++spins)) break;
        ld_word(buf + (long long)threadIdx.x * kXV, x, e);
      }
      __threadfence();
    }
    __syncthreads();
  }
}

// First row r with rp[r] + 4 r >= target (rows [0, n]), by the whole warp: 33-ary search.
__device__ __forceinline__ int warp_row_at(const int* __restrict__ rp, int n, long long target) {
  int lo = 0, hi = n;  // the answer lies in [lo, hi]
  const int lane = threadIdx.x & 31;
  while (lo < hi) {
    const int step = (hi - lo + 31) / 32;
    const int at = lo + step * (lane + 1) - 1;  // probes lo + step - 1, lo + 2 step - 1, ...
    const bool below = at < hi && (long long)__ldg(rp + at) + 4LL * at < target;
    const int k = __popc(__ballot_sync(kFull, below));  // monotone: the first k probes are below
    const int nlo = lo + step * k;
    hi = min(hi, lo + step * (k + 1) - 1);
    lo = min(nlo, n);
    if (lo > hi) hi = lo;
  }
  return lo;
}

// q = fl_p1(A x) over the CTA's rows, as fp64 with the row scale applied. Each row's sum runs in
// the order of its schedule (one thread: columns in order; K lanes: strided, butterfly), except
// that the fp64 and the compensated sums of rows over kMidRow nonzeros are spread over a warp and
// over kLongRowTeam over the CTA: a thread walks four columns per memory round trip, 0.6 us, so
// that one row of 1000 held the whole team for 150 us (160k-node graph, fp64: 188 us a product
// before). The fp32 sums keep their order, whose rounding shows in the result. The rows of a
// chunk that are left for a warp or the CTA are queued in shared memory (a chunk never holds
// more than the queue), so which way a row is summed depends on the matrix alone.
// A finished row to q: rounded onto p1, with the row scale. (The exact fp64 sum for a rounding
// that the error bound leaves open, essentially never, is out of line.)
template <typename VT>
__device__ __noinline__ float team_row_exact(const DevSys& S, const VT* vals, const VT* xin, int row, int p1) {
  double acc = 0.0;
  for (int e = __ldg(S.A.rp + row); e < __ldg(S.A.rp + row + 1); ++e)
    acc = fma(f2d(to_acc(ldg_val(vals + e))), f2d(to_acc(xin[__ldg(S.A.ci + e)])), acc);
  return RowAcc<VT, true>::slow_round(p1, acc);
}
template <typename VT, bool COMP>
__device__ __forceinline__ void team_finish(const TeamSmem& t, const VT* vals, const VT* xin, int p1, double* q, int row,
                                            int len, const RowAcc<VT, COMP>& acc) {
  const DevSys& S = t.S;
  double v;
  if constexpr (sizeof(VT) == 8) {
    v = acc.s;
  } else {
    float f;
    if constexpr (COMP) f = acc.rounded(p1, len, [&] { return 0.0; }, [&] { return team_row_exact<VT>(S, vals, xin, row, p1); });
    else f = acc.s;
    v = f2d(f);
    if (row_scaled(p1)) v = scale2(v, __ldg(S.A.rexp + row));
  }
  q[row - t.V.r0] = v;
}

// The rows that a chunk of team_product has queued: t.nq for a warp each (from the front of the
// queue), t.nl for the CTA (from the back). Contains CTA barriers.
template <typename VT, bool COMP>
__device__ __noinline__ void team_queued(TeamSmem& t, const VT* __restrict__ vals, const VT* xin, int p1, double* q) {
  constexpr bool kOrdered = sizeof(VT) == 4 && !COMP;
  const int* __restrict__ rp = t.S.A.rp;
  const int* __restrict__ ci = t.S.A.ci;
  __builtin_assume(__isGlobal(xin));
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  const int nq = t.nq, nl = t.nl;
  for (int i = w; i < nq; i += kTW) {
    const int qr = t.queue[i];
    const int e0 = __ldg(rp + qr), e1 = __ldg(rp + qr + 1);
    RowAcc<VT, COMP> acc;
#pragma unroll 4
    for (int e = e0 + lane; e < e1; e += 32) acc.add(ldg_val(vals + e), xin[__ldg(ci + e)]);
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) acc.step(kFull, o);
    if (lane == 0) team_finish<VT, COMP>(t, vals, xin, p1, q, qr, e1 - e0, acc);
  }
  // rows for the whole CTA: every warp takes its strided part of up to kLongBatch rows before
  // one barrier, then warp i merges the parts of the i-th row
  constexpr int NL = kOrdered ? kThreads : kTT;  // threads of a long row
  for (int i = 0; i < nl;) {
    int nb = 0;
    for (; i < nl && nb < kLongBatch; ++i, ++nb) {
      const int qr = t.queue[kTT - 1 - i];
      const int e0 = __ldg(rp + qr), e1 = __ldg(rp + qr + 1);
      if (threadIdx.x == 0) t.lrow[nb] = qr;
      if (threadIdx.x < NL) {
        RowAcc<VT, COMP> acc;
#pragma unroll 4
        for (int e = e0 + threadIdx.x; e < e1; e += NL) acc.add(ldg_val(vals + e), xin[__ldg(ci + e)]);
#pragma unroll 1
        for (int o = 16; o > 0; o >>= 1) acc.step(kFull, o);
        if (lane == 0) {
          t.lpart[nb][w] = acc.s;
          t.lcorr[nb][w] = make_float2((float)acc.c, (float)acc.a);
        }
      }
    }
    __syncthreads();
    if (w < nb) {
      RowAcc<VT, COMP> acc;
      if constexpr (kOrdered) {  // the warps' sums in warp order
        acc.s = (float)t.lpart[w][0];
        for (int u = 1; u < NL / 32; ++u) acc.merge(t.lpart[w][u], 0.0, 0.0);
      } else {
        if (lane < kTW) {
          acc.s = t.lpart[w][lane];
          acc.c = t.lcorr[w][lane].x;
          acc.a = t.lcorr[w][lane].y;
        }
#pragma unroll 1
        for (int o = 16; o > 0; o >>= 1) acc.step(kFull, o);
      }
      const int qr = t.lrow[w];
      if (lane == 0) team_finish<VT, COMP>(t, vals, xin, p1, q, qr, __ldg(rp + qr + 1) - __ldg(rp + qr), acc);
    }
    __syncthreads();
  }
  __syncthreads();
  if (threadIdx.x == 0) t.nq = t.nl = 0;
  __syncthreads();
}

// The product from warp tiles (spmv_tile's scheme), the tile being 32 rows of values of up to four
// bytes; fp64 rows, whose sum has no order to keep, come 16 to a tile with two lanes each. (64^3
// 27-point system on the whole grid, tf32: 23 us a product from direct loads.)
template <typename VT, bool COMP>
__device__ __forceinline__ void team_tiles(TeamSmem& t, const VT* __restrict__ vals, const VT* xin, int p1, double* q) {
  constexpr int PER = 16 / (int)sizeof(VT);
  constexpr int LPR = sizeof(VT) == 8 ? 2 : 1;  // lanes per row
  constexpr int TR = 32 / LPR;
  constexpr int CAP = sizeof(VT) == 8 ? 592 : 896;
  constexpr int U = sizeof(VT) == 8 ? 7 : 14;
  static_assert(4 * (CAP + 8) + (int)sizeof(VT) * (CAP + PER) <= kTeamTileWarp, "a tile exceeds its place");
  const int* __restrict__ ci = t.S.A.ci;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int* sc = reinterpret_cast<int*>(t.tile + (size_t)w * kTeamTileWarp);
  VT* sv = reinterpret_cast<VT*>(reinterpret_cast<unsigned char*>(sc) + 4 * (CAP + 8));
  const unsigned sc32 = smem_u32(sc), sv32 = smem_u32(sv);
  const int r0 = t.V.r0, r1 = r0 + t.V.n, rb = t.rbase;
  const int* rp = t.rp;
  for (int base = r0 + TR * w; base < r1; base += TR * kTW) {
    const int row = base + lane / LPR;
    const int e0 = rp[min(row, r1) - rb], e1 = rp[min(row + 1, r1) - rb];
    const int E0 = __shfl_sync(kFull, e0, 0), E1 = __shfl_sync(kFull, e1, 31);
    const int cb = E0 & ~3, vb = E0 & ~(PER - 1);
    const bool staged = E1 - E0 <= CAP;
    if (staged) {
      for (int i = lane; 4 * i < E1 - cb; i += 32) cp_async16(sc32 + 16u * i, ci + cb + 4 * i);
      for (int i = lane; PER * i < E1 - vb; i += 32) cp_async16(sv32 + 16u * i, vals + vb + PER * i);
      asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
      __syncwarp();
    }
    RowAcc<VT, COMP> acc;
    const int len = e1 - e0, k0 = lane & (LPR - 1);
    const int* c = staged ? sc + (e0 - cb) : ci + e0;
    const VT* v = staged ? sv + (e0 - vb) : vals + e0;
    int k = k0;
    for (; k + LPR * (U - 1) < len; k += LPR * U) {
      VT x[U];
#pragma unroll
      for (int j = 0; j < U; ++j) x[j] = xin[c[k + LPR * j]];
#pragma unroll
      for (int j = 0; j < U; ++j) acc.add(v[k + LPR * j], x[j]);
    }
    if (k < len) {
      VT x[U];
#pragma unroll
      for (int j = 0; j < U - 1; ++j)
        if (k + LPR * j < len) x[j] = xin[c[k + LPR * j]];
#pragma unroll
      for (int j = 0; j < U - 1; ++j)
        if (k + LPR * j < len) acc.add(v[k + LPR * j], x[j]);
    }
    if constexpr (LPR == 2) acc.step(kFull, 1);
    if (row < r1 && k0 == 0) team_finish<VT, COMP>(t, vals, xin, p1, q, row, len, acc);
    __syncwarp();  // the tile is read before the next one replaces it
  }
  if (LPR > 1) __syncthreads();  // rows finished by other threads than their own
}

template <typename VT, bool COMP>
__device__ __forceinline__ void team_product(TeamSmem& t, const VT* __restrict__ vals, const VT* xin, int p1, double* q) {
  const DevSys& S = t.S;
  if (t.tile && S.A.sched[p1] == SCHED_VLOAD) {
    team_tiles<VT, COMP>(t, vals, xin, p1, q);
    return;
  }
  const int* rp = t.rp;  // in shared memory when they fit
  const int* ci = t.ci;
  const int rbase = t.rbase, ebase = t.ebase;
  __builtin_assume(__isGlobal(xin));
  constexpr bool kOrdered = sizeof(VT) == 4 && !COMP;
  constexpr int kLong = kOrdered ? kLongRow : kLongRowTeam;
  const int r0 = t.V.r0, r1 = r0 + t.V.n;
  const bool vload = S.A.sched[p1] == SCHED_VLOAD;
  const int K = vload ? 1 : S.A.lanes[p1];
  const int mid = vload && !kOrdered ? kMidRow : kLong;  // longer rows are queued
  const bool queueing = S.A.max_row > mid;               // the same for the whole team
  const bool shortrows = vload && S.A.max_row <= kShortRow;
  const int chunk = kTT / K;
  for (int base = r0; base < r1; base += chunk) {
    const int row = base + (int)threadIdx.x / K;
    if (row < r1) {
      const int e0 = rp[row - rbase], e1 = rp[row - rbase + 1];
      RowAcc<VT, COMP> acc;
      if (e1 - e0 > mid) {
        if ((threadIdx.x & (K - 1)) == 0) {  // for a warp: from the front; for the CTA: from the back
          if (e1 - e0 > kLong) t.queue[kTT - 1 - atomicAdd(&t.nl, 1)] = row;
          else t.queue[atomicAdd(&t.nq, 1)] = row;
        }
      } else if (sizeof(VT) >= 4 && shortrows) {
        // all loads of the row at once: from 16-byte groups a row of five doubles is two or three
        // round trips to L2, one after the other
        const int len = e1 - e0;
        const int* c = ci + (e0 - ebase);
        VT v[kShortRow], x[kShortRow];
#pragma unroll
        for (int j = 0; j < kShortRow; ++j)
          v[j] = x[j] = VT();
#pragma unroll
        for (int j = 0; j < kShortRow; ++j)
          if (j < len) {
            v[j] = ldg_val(vals + e0 + j);
            x[j] = xin[c[j]];
          }
#pragma unroll
        for (int j = 0; j < kShortRow; ++j)
          if (j < len) acc.add(v[j], x[j]);
        team_finish<VT, COMP>(t, vals, xin, p1, q, row, len, acc);
      } else if (vload) {
        constexpr int G = sizeof(VT) <= 2 ? 8 : 4;
        constexpr int NV = G * (int)sizeof(VT) / 16;
        for (int g = e0 & ~(G - 1); g < e1; g += G) {
          int c[G];
          VT v[G];
#pragma unroll
          for (int h = 0; h < G / 4; ++h) {
            const int4 cc = *(reinterpret_cast<const int4*>(ci + (g - ebase)) + h);
            c[4 * h] = cc.x;
            c[4 * h + 1] = cc.y;
            c[4 * h + 2] = cc.z;
            c[4 * h + 3] = cc.w;
          }
          if constexpr (NV == 0) {
            const int2 v2 = __ldg(reinterpret_cast<const int2*>(vals + g));
            const int4 vv = make_int4(v2.x, v2.y, 0, 0);
#pragma unroll
            for (int k = 0; k < G; ++k) v[k] = lane_of<VT>(vv, k);
          }
#pragma unroll
          for (int h = 0; h < NV; ++h) {
            const int4 vv = __ldg(reinterpret_cast<const int4*>(vals + g) + h);
            constexpr int PER = 16 / (int)sizeof(VT);
#pragma unroll
            for (int k = 0; k < PER; ++k) v[h * PER + k] = lane_of<VT>(vv, k);
          }
          VT xv[G];
#pragma unroll
          for (int j = 0; j < G; ++j)
            if (g + j >= e0 && g + j < e1) xv[j] = xin[c[j]];
#pragma unroll
          for (int j = 0; j < G; ++j)
            if (g + j >= e0 && g + j < e1) acc.add(v[j], xv[j]);
        }
        team_finish<VT, COMP>(t, vals, xin, p1, q, row, e1 - e0, acc);
      } else {
        const int kl = threadIdx.x & (K - 1);
        const unsigned kmask = K == 32 ? kFull : (((1u << K) - 1u) << ((threadIdx.x & 31) & ~(K - 1)));
#pragma unroll 4
        for (int e = e0 + kl; e < e1; e += K) acc.add(ldg_val(vals + e), xin[ci[e - ebase]]);
#pragma unroll 1
        for (int o = K / 2; o > 0; o >>= 1) acc.step(kmask, o);
        if (kl == 0) team_finish<VT, COMP>(t, vals, xin, p1, q, row, e1 - e0, acc);
      }
    }
    if (queueing) team_queued<VT, COMP>(t, vals, xin, p1, q);
  }
  // a row was finished by another thread than the one that owns it in the vector phases
  if (K > 1) __syncthreads();
}

// Product in format p1 of the global vector that p's copy went to (fp64: x64 itself).
__device__ __forceinline__ void team_spmv(TeamSmem& t, int p1, const double* x64, double* q) {
  const DevSys& S = t.S;
  switch (p1) {
    case F64: team_product<double, false>(t, S.A.v64, x64, F64, q); break;
    case F32: team_product<float, false>(t, S.A.v32, (const float*)S.plow, F32, q); break;
    case TF32: team_product<float, true>(t, S.A.vtf, (const float*)S.plow, TF32, q); break;
    case F16: team_product<__half, true>(t, S.A.v16, (const __half*)S.plow, F16, q); break;
    case BF16: team_product<__nv_bfloat16, true>(t, S.A.vbf, (const __nv_bfloat16*)S.plow, BF16, q); break;
    case F16R: team_product<__half, true>(t, S.A.v16r, (const __half*)S.plow, F16R, q); break;
    case Q52: team_product<q52_t, true>(t, S.A.v8, (const q52_t*)S.plow, Q52, q); break;
    default: team_product<__nv_bfloat16, true>(t, S.A.vbfr, (const __nv_bfloat16*)S.plow, BF16R, q); break;
  }
}

// ---- IC(0): w = M^-1 fl32(r) ------------------------------------------------------------
//
// The substitutions are a chain of levels (2N - 1 of them on an N^2 five-point grid, 7N on an N^3
// 27-point grid, each way), so what counts is the time from one level to the next. The team's
// first CTA runs them alone: the vector lives in its shared memory (the other CTAs write their
// rows' fl32(r) there and read w back through the cluster), the factor comes as one block per
// level in the order of use (header; row and diagonal per position; 16-bit columns and values in
// quads, transposed over the lanes), streamed through a ring up to kIcBars levels ahead by bulk
// copies that a warp of its own issues (a copy takes some 2 us to arrive: four blocks in flight
// left the levels waiting), and a level ends with a barrier of the warps the widest level needs. A level costs a wait, two shared
// loads, the row's chain and a division instead of polls of words in L2: 8-10 us before (28^3
// 27-point system: 2.1 ms an application). Rows are summed in column order with one division,
// every operation a rounded fp32 one, as in the sequential substitution, bit for bit.
// Q quads of a lane's entries: s -= v_k W[c_k] in order. All columns and values are loaded, then
// all elements of W, then the chain runs (loading quad by quad took 300 cycles each). Padding
// entries are 0 times a cell that holds 0.
template <int Q>
__device__ __forceinline__ void ic_quads(unsigned W, unsigned ac, unsigned av, float& s) {
  int2 c[Q];
  int4 v[Q];
  float x[4 * Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    c[q] = lds_v2(ac + 256u * q);
    v[q] = lds_v4(av + 512u * q);
  }
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    x[4 * q] = lds_f32(W + 4u * (c[q].x & 0xffff));
    x[4 * q + 1] = lds_f32(W + 4u * ((unsigned)c[q].x >> 16));
    x[4 * q + 2] = lds_f32(W + 4u * (c[q].y & 0xffff));
    x[4 * q + 3] = lds_f32(W + 4u * ((unsigned)c[q].y >> 16));
  }
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    s = __fsub_rn(s, __fmul_rn(__int_as_float(v[q].x), x[4 * q]));
    s = __fsub_rn(s, __fmul_rn(__int_as_float(v[q].y), x[4 * q + 1]));
    s = __fsub_rn(s, __fmul_rn(__int_as_float(v[q].z), x[4 * q + 2]));
    s = __fsub_rn(s, __fmul_rn(__int_as_float(v[q].w), x[4 * q + 3]));
  }
}

__device__ __noinline__ void ic_levels_team(const Launch& L, TeamSmem& t) {
  const DevSys& S = t.S;
  const int nw = S.A.icwarps;  // at most kTW - 2: one warp waits, the last one issues the copies
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nl = S.A.nlevf + S.A.nlevb;
  const unsigned use0 = t.icuse;
  if (w == kTW - 1) {
    // per level: place and size in the blob and place in the ring (16-byte units), and the number of
    // levels that must have been consumed before the block may be written; 32 at a time, the next 32
    // on their way (one load per level held every copy up by its latency)
    const int4* __restrict__ desc = S.A.icdesc;
    const unsigned ring = smem_u32(t.icring), bars = smem_u32(t.icbar), done = smem_u32(&t.icdone);
    int4 dn = __ldg(desc + min(lane, nl - 1));
    for (int l0 = 0; l0 < nl; l0 += 32) {
      const int4 d = dn;
      dn = __ldg(desc + min(l0 + 32 + lane, nl - 1));
      for (int j = 0; j < 32 && l0 + j < nl; ++j) {
        const int from = __shfl_sync(kFull, d.x, j), size = __shfl_sync(kFull, d.y, j);
        const int to = __shfl_sync(kFull, d.z, j), need = __shfl_sync(kFull, d.w, j);
        if (lane == 0) {
          int have = lds_acquire(done);
          const long long t0 = clock64();
          unsigned spins = 0;
          while (have < need && !wait_over(L, t, t0, ++spins)) have = lds_acquire(done);
          if (have >= need) {
            const unsigned bar = bars + 8u * ((use0 + (unsigned)(l0 + j)) % kIcBars);
            t.icissued = (unsigned)(l0 + j + 1);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(size * 16) : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                             ring + 16u * (unsigned)to),
                         "l"(S.A.icblob + (size_t)from * 16), "r"(size * 16), "r"(bar)
                         : "memory");
          }
        }
        __syncwarp();
        if (*(volatile int*)&t.bad) return;
      }
    }
    return;
  }
  if (w > nw) return;
  const unsigned ring = smem_u32(t.icring);
  if (w == nw) {  // a warp that only waits for the next block while the others sum, then joins their barrier
    for (int l = 0; l <= nl; ++l) {
      if (lane == 0 && l < nl) {
        const unsigned use = use0 + (unsigned)l, par = (use / kIcBars) & 1u;
        unsigned long long* bar = &t.icbar[use % kIcBars];
        const long long t0 = clock64();
        unsigned spins = 0;
        while (!mbar_try_wait(bar, par))
          if (wait_over(L, t, t0, ++spins)) break;
      }
      // whether to go on is decided here and read by all after the barrier (two cells in turn)
      if (lane == 0) t.icstop[l & 1] = *(volatile int*)&t.bad;
      __syncwarp();
      asm volatile("bar.sync 1, %0;" ::"r"(nw * 32 + 32) : "memory");
      if (*(volatile int*)&t.icstop[l & 1]) return;
      if (lane == 0) sts_release(smem_u32(&t.icdone), l);
    }
    if (lane == 0) {
      t.icuse = (use0 + (unsigned)nl) % (2u * kIcBars);
      t.icissued = 0;
      sts_release(smem_u32(&t.icdone), 0);  // (the producer has issued the last block)
    }
    return;
  }
  // 32-bit shared addresses: the loop is bound by the latencies and instructions of one level
  const unsigned W = smem_u32(t.icW);
  asm volatile("bar.sync 1, %0;" ::"r"(nw * 32 + 32) : "memory");
  unsigned blk = ring;
  for (int l = 0; l < nl && !*(volatile int*)&t.icstop[l & 1]; ++l) {
    const int4 h = lds_v4(blk);  // groups, quads of entries, next block's place, bytes of a group
    for (int g = w; g < h.x; g += nw) {
      const unsigned a = blk + 16u + (unsigned)(g * h.w) + 8u * lane;
      const int2 m = lds_v2(a);  // row, diagonal
      if (m.x != 0xffff) {
        const unsigned ar = W + 4u * (unsigned)m.x;
        float s = lds_f32(ar);
        unsigned ac = a + 256u, av = a + 256u + 256u * (unsigned)h.y + 8u * lane;
        if (h.y == 1) {
          ic_quads<1>(W, ac, av, s);
        } else if (h.y == 2) {
          ic_quads<2>(W, ac, av, s);
        } else {
          for (int k = 0; k < h.y; k += 4, ac += 1024u, av += 2048u) ic_quads<4>(W, ac, av, s);
        }
        sts_f32(ar, __fdiv_rn(s, __int_as_float(m.y)));
      }
    }
    asm volatile("bar.sync 1, %0;" ::"r"(nw * 32 + 32) : "memory");
    blk = ring + 16u * (unsigned)h.z;
  }
}

// After a wait that gave up: waits for the block copies still in flight, so that none lands in shared
// memory that has passed to another CTA. A barrier of the ring was last used by one of the last kIcBars
// blocks issued. (A copy needs nothing of the other CTAs; the limit is far beyond what it takes.)
__device__ __noinline__ void ic_drain(TeamSmem& t) {
  if (threadIdx.x != 0) return;
  const unsigned n = t.icissued;
  for (unsigned l = n > (unsigned)kIcBars ? n - kIcBars : 0u; l < n; ++l) {
    const unsigned use = t.icuse + l;
    const long long t0 = clock64();
    while (!mbar_try_wait(&t.icbar[use % kIcBars], (use / kIcBars) & 1u))
      if (clock64() - t0 > 100000000ll) return;
  }
}

// w = M^-1 fl32(r), r the CTA's rows; afterwards team_minv reads it. Contains team barriers.
template <bool CL>
__device__ __noinline__ Team team_apply_ic(const Launch& L, TeamSmem& t, Team T) {
  const TeamVec V = t.V;
  const unsigned dst = cluster_map(smem_u32(t.icW), t.base) + 4u * (unsigned)V.r0;
  for (int i = threadIdx.x; i < V.n; i += kTT) st_cluster_f32(dst + 4u * (unsigned)i, __double2float_rn(V.r[i]));
  team_publish<CL>(L, t, T);
  if (t.rank == 0) ic_levels_team(L, t);
  team_publish<CL>(L, t, T);
  return T;
}

// (M^-1 r)_i of the CTA's i-th row: the last IC(0) application, Jacobi, or r itself. (The kernels
// without IC(0) are instantiations of their own: its code cost them 1.5 us an iteration in
// registers and instruction fetches.)
template <bool IC>
struct TeamMinv {
  unsigned ic;          // IC(0): cluster address of the first row's w
  const double* dinv;   // the first row's reciprocal diagonal, or nullptr
  __device__ __forceinline__ double operator()(int i, double ri) const {
    if constexpr (IC) return (double)ld_cluster_f32(ic + 4u * (unsigned)i);
    return dinv ? ri * __ldg(dinv + i) : ri;
  }
};
template <bool IC>
__device__ __forceinline__ TeamMinv<IC> team_minv(const TeamSmem& t) {
  TeamMinv<IC> m;
  m.ic = IC ? cluster_map(smem_u32(t.icW), t.base) + 4u * (unsigned)t.V.r0 : 0u;
  m.dinv = t.S.A.dinv ? t.S.A.dinv + t.V.r0 : nullptr;
  return m;
}

// r = b - A x in fp64 (x from global memory, released before); returns the thread's part of r.r.
__device__ __noinline__ double team_true_res(TeamSmem& t) {
  team_product<double, false>(t, t.S.A.v64, t.S.x, F64, t.V.q);
  const TeamVec V = t.V;
  double rr = 0.0;
  for (int i = threadIdx.x; i < V.n; i += kTT) {
    const double ri = __ldg(t.S.b + V.r0 + i) - V.q[i];
    V.r[i] = ri;
    rr = fma(ri, ri, rr);
  }
  return rr;
}

// With r known: with copy_p the direction p = M^-1 r and r.p in fp64, with p2 >= 0 the sigma
// terms of z = fl_p2(M^-1 r).
struct TeamDot {
  Team T;
  DotAcc sg;
};
template <bool CL, bool IC>
__device__ __noinline__ TeamDot team_use_r(const Launch& L, TeamSmem& t, Team T, int p2, int p4, bool copy_p) {
  if constexpr (IC) T = team_apply_ic<CL>(L, t, T);
  const TeamVec V = t.V;
  const TeamMinv<IC> minv = team_minv<IC>(t);
  DotAcc acc{0.0, 0.f, 0.f};
  for (int i = threadIdx.x; i < V.n; i += kTT) {
    const double ri = V.r[i], wi = minv(i, ri);
    if (copy_p) {
      V.p[i] = wi;
      acc.d = fma(ri, wi, acc.d);
    }
    if (p2 >= 0) sigma_term(ri, wi, p2, p4, acc);
  }
  return TeamDot{T, acc};
}

// p of the CTA's rows in the next product's format where that product gathers it.
__device__ __forceinline__ void team_copy_p(const TeamSmem& t, int p1) {
  const DevSys& S = t.S;
  const TeamVec V = t.V;
  for (int i = threadIdx.x; i < V.n; i += kTT) {
    if (p1 == F64) S.p[V.r0 + i] = V.p[i];
    else store_low(S.plow, V.r0 + i, V.p[i], p1);
  }
}

__device__ __forceinline__ DotAcc team_phase_nu(const TeamSmem& t, int p3) {
  const TeamVec V = t.V;
  DotAcc nu{0.0, 0.f, 0.f};
  if (p3 == F64) {
    for (int i = threadIdx.x; i < V.n; i += kTT) nu.d = fma(V.p[i], V.q[i], nu.d);
  } else {
    for (int i = threadIdx.x; i < V.n; i += kTT) dot_low(nu, round_d2f(V.p[i], p3), round_d2f(V.q[i], p3), p3);
  }
  return nu;
}

// Phase B: r -= alpha q, ||r||^2, the sigma terms; z = fl_p2(M^-1 r) takes q's place. With IC(0)
// in two passes around the application (part 1: r, part 2: z and sigma), else in one (part 0).
template <bool IC>
__device__ __forceinline__ void team_phase_b(const TeamSmem& t, int part, double alpha, int p2, int p4,
                                          bool sig_rr, double& rr, DotAcc& sg) {
  const TeamVec V = t.V;
  const TeamMinv<IC> minv = team_minv<IC>(t);
  double sum = rr;
  DotAcc acc = sg;
  for (int i = threadIdx.x; i < V.n; i += kTT) {
    double ri;
    if (IC && part == 2) {
      ri = V.r[i];
    } else {
      ri = fma(-alpha, V.q[i], V.r[i]);
      V.r[i] = ri;
      sum = fma(ri, ri, sum);
      if (IC && part == 1) continue;
    }
    const double wi = minv(i, ri);
    if (!sig_rr) sigma_term(ri, wi, p2, p4, acc);
    V.q[i] = p2 == F64 ? wi : f2d(round_d2f(wi, p2));
  }
  rr = sum;
  sg = acc;
}

// Phase C: x += alpha p; p = z + beta p; p's copy in the next product's format.
__device__ __forceinline__ void team_phase_c(const TeamSmem& t, double alpha, double beta, int p1n) {
  const DevSys& S = t.S;
  const TeamVec V = t.V;
  const bool low = p1n != F64;
  for (int i = threadIdx.x; i < V.n; i += kTT) {
    const double po = V.p[i];
    V.x[i] = fma(alpha, po, V.x[i]);
    const double pn = fma(beta, po, V.q[i]);
    V.p[i] = pn;
    if (low) store_low(S.plow, V.r0 + i, pn, p1n);
    else S.p[V.r0 + i] = pn;
  }
}

// x of the CTA's rows to global memory (for the residual's gathers, and the result).
__device__ __forceinline__ void team_store_x(const TeamSmem& t) {
  const TeamVec V = t.V;
  for (int i = threadIdx.x; i < V.n; i += kTT) t.S.x[V.r0 + i] = V.x[i];
}

// ---- The scalar steps of an ordinary iteration --------------------------------------------
//
// One warp's straight-line code runs at about five cycles an instruction here (it is fetched
// anew every iteration), an fp64 division takes 560 cycles, a square root 600, a comparison 64.
// The full steps (step_A, step_B: records, stopping, breakdowns, features, any policy)
// took 1,300 and 6,800 cycles of an iteration; an ordinary iteration of an inference solve needs
// of them alpha, beta, the residual bin and the four formats. These come here from one warp: the bin
// and the stopping test by comparing ||r||^2 with the squared thresholds as integers, rho itself
// only when something asks for it (team_rho). Whenever a comparison is too close for the squares
// to decide, the residual is below the tolerance, a value is not finite or the last iteration is
// due, the full step runs instead; so decisions and results are those of the full step.

__device__ __forceinline__ bool finite_bits(double v) {
  return (__double_as_longlong(v) & 0x7fffffffffffffffll) < 0x7ff0000000000000ll;
}

// st.rho of the last iteration, formed now if the short steps left it out (thread 0).
__device__ __forceinline__ void team_rho(TeamSmem& t) {
  if (t.stale) {
    t.st.rho = sqrt(t.rr) / t.st.bnorm;
    t.st.rho_hist[0] = t.st.rho;
    t.stale = 0;
  }
}

// After the initialisation: whether the short steps apply, and their thresholds (threads 0..31).
__device__ __forceinline__ void team_fast_setup(const Launch& L, TeamSmem& t) {
  const OptView& o = L.opt;
  const int m = threadIdx.x;
  if (m >= 32) return;
  const double thr = m == 0 ? t.S.tol : m < o.r_bins ? o.thr[m] : 0.0;
  const double e = thr * t.st.bnorm;
  t.thr2[m] = __double_as_longlong(e * e);
  if (m == 0) {
    t.fast = !t.S.hist && o.true_every <= 0 &&
             (L.pol.kind <= 1 || (L.pol.kind == 2 && !o.joint)) && o.edge_tol < 0.1;
    // 2^21 units in the last place: far more than the squares' rounding; with a table also the
    // neighbourhood of an edge that near_edge_count counts
    const long long edge = (long long)(2.2 * o.edge_tol * 0x1.0p53);
    t.margin = L.pol.kind == 2 && edge > (1ll << 21) ? edge : (1ll << 21);
    t.stale = 0;
    t.slow = 0;
  }
}

// After phase A (thread 0).
__device__ __forceinline__ void team_step_a(const Launch& L, TeamSmem& t) {
  if (threadIdx.x != 0) return;
  SysState& st = t.st;
  const double nu_sum = t.sum[0];
  if (t.fast) {
    const int p3 = st.fmt[2];
    const double nu = p3 == F64 ? nu_sum : round_fmt(nu_sum, p3);
    const double alpha = st.sigma / nu;
    if (__double_as_longlong(nu) > 0 && finite_bits(nu) && finite_bits(alpha)) {
      st.nu = nu;
      st.alpha = alpha;
      st.mode = M_CONT;  // (M_RESTART after a residual replacement)
      return;
    }
    team_rho(t);
  }
  step_A(L, t.S, &st, nu_sum);
}

// After phase B: all threads; ends without a barrier. sig: the sum that is sigma.
__device__ __forceinline__ void team_step_b(const Launch& L, TeamSmem& t, int sig) {
  SysState& st = t.st;
  if (t.fast) {
    if (threadIdx.x < 32) {
      const int lane = threadIdx.x;
      const OptView& o = L.opt;
      const PolicyView& P = L.pol;
      __syncwarp();
      const double rr = t.sum[0], sg = t.sum[sig];
      const int p4 = st.fmt[3], k1 = st.k + 1, z = st.fmt[1];
      const double sn = p4 == F64 ? sg : round_fmt(sg, p4);
      const double beta = sn / st.sigma;
      const long long dist = __double_as_longlong(rr) - t.thr2[lane];
      const bool valid = lane < o.r_bins;
      const unsigned below = __ballot_sync(kFull, valid && dist <= 0);
      const unsigned close = __ballot_sync(kFull, valid && (dist < 0 ? -dist : dist) < t.margin);
      const bool slow = close || (below & 1u) || !finite_bits(rr) || !finite_bits(sn) || !finite_bits(beta) ||
                        k1 >= t.S.max_iter || st.fp64_lock;
      __syncwarp();
      if (slow) {
        if (lane == 0) t.slow = 1;
      } else {
        if (lane < 4) {
          int f;
          if (P.kind == 0) {
            f = P.fixed[lane];
          } else if (P.kind == 1) {
            f = P.sched[(k1 < P.sched_len ? k1 : P.sched_len - 1) * 4 + lane];
          } else {
            const int bin = min(k1 / o.t_width, o.b_bins - 1), S = o.b_bins * o.r_bins;
            const int s = lane * S + bin * o.r_bins + __popc(below);  // (bit 0 is clear)
            const double* Q = t.S.vtab ? t.S.Qpriv : P.Q;
            const int* vis = t.S.vtab ? t.S.vtab : P.visits;
            const unsigned mask = (unsigned)o.op_mask[lane];
            int act = row_argmax(Q + (long long)s * o.nprec, o.nprec, mask);
            if (vis && o.fallback_fmt >= 0 && o.fallback_idx >= 0 && ((mask >> o.fallback_idx) & 1u) && vis[s] == 0)
              act = o.fallback_idx;
            f = o.precs[act];
          }
          st.fmt[lane] = f;
          st.counts[lane][f & 7] += 1;
        }
        if (lane == 0) {
          st.sigma = sn;
          st.beta = beta;
          st.zfmt = z;
          st.k = k1;
          t.rr = rr;
          t.stale = 1;
        }
      }
    }
    __syncthreads();
    if (!t.slow) return;
    __syncthreads();
    if (threadIdx.x == 0) {
      t.slow = 0;
      team_rho(t);
    }
  }
  step_B(L, t.S, &st, t.sum[0], t.sum[sig], t.sm);
}

// The CTA barrier that ends a scalar step; false when a wait has given up. (A release of p
// that gave up is seen here after the next exchange; the columns gathered meanwhile are valid.)
__device__ __forceinline__ bool team_ok(const TeamSmem& t) {
  __syncthreads();
  return t.bad == 0;
}

// fp64 restart after a breakdown: r = b - A x and p = M^-1 r, then step_restart.
struct TeamOk {
  Team T;
  bool ok;
};
template <bool CL, bool IC>
__device__ __noinline__ TeamOk team_restart64(const Launch& L, TeamSmem& t, Team T) {
  team_store_x(t);
  team_publish<CL>(L, t, T);
  const double rr = team_true_res(t);
  const TeamDot u = team_use_r<CL, IC>(L, t, T, -1, -1, true);
  T = u.T;
  const DotAcc sg = u.sg;
  const double v[2] = {warp_sum(rr), warp_dot(sg, false)};
  team_exchange<CL, 2>(L, t, T, v);
  if (threadIdx.x == 0) t.stale = 0;
  step_restart(L, t.S, &t.st, t.sum[0], t.sum[1], t.sm);
  if (!team_ok(t)) return TeamOk{T, false};
  team_copy_p(t, t.st.fmt[0]);
  team_publish<CL>(L, t, T);
  return TeamOk{T, true};
}

constexpr size_t kTeamFixed = (sizeof(TeamSmem) + 127) / 128 * 128;

// One system solved by the team (the phases and transitions of solve_system). All CTAs of the
// team take the same branches: their states are equal.
template <bool CL, bool IC>
__device__ bool solve_team(const Launch& L, TeamSmem& t, int sid) {
  Team T{0u, 0u};
  const DevSys& S = t.S;
  const TeamVec V = t.V;
  SysState* st = &t.st;
  Smem& sm = t.sm;
  const OptView& o = L.opt;
  const bool active = (int)(threadIdx.x >> 5) < t.nact;

  // ---- initialisation ----
  {
    double bb = 0.0, rr = 0.0;
    for (int i = threadIdx.x; i < V.n; i += kTT) {
      const double bi = __ldg(S.b + V.r0 + i);
      bb = fma(bi, bi, bb);
      if (!o.warm_start) {
        V.x[i] = 0.0;
        V.r[i] = bi;
      } else {
        V.x[i] = S.x[V.r0 + i];
      }
    }
    if (o.warm_start) rr = team_true_res(t);
    else rr = bb;
    const TeamDot u = team_use_r<CL, IC>(L, t, T, -1, -1, true);
    T = u.T;
    const DotAcc sg = u.sg;
    const double v[3] = {warp_sum(bb), warp_sum(rr), warp_dot(sg, false)};
    team_exchange<CL, 3>(L, t, T, v);
    step_init(L, S, st, t.sum[0], t.sum[1], t.sum[2], sm);
    if (!team_ok(t)) return false;
    team_fast_setup(L, t);
  }

  if (st->mode == M_CONT) {
    team_copy_p(t, st->fmt[0]);
    team_publish<CL>(L, t, T);
    while (true) {
      // ---- phase A ----
      {
        const int p1 = st->fmt[0], p3 = st->fmt[2];
        team_spmv(t, p1, S.p, V.q);
        const DotAcc nu = team_phase_nu(t, p3);
        const double v[1] = {active ? warp_dot(nu, p3 != F64) : 0.0};
        team_exchange<CL, 1>(L, t, T, v);
        team_step_a(L, t);
        if (!team_ok(t)) return false;
        if (st->mode == M_RESTART64) {
          const TeamOk ro = team_restart64<CL, IC>(L, t, T);
          T = ro.T;
          if (!ro.ok) return false;
          if (st->mode != M_CONT) break;
          continue;
        }
        if (st->mode != M_CONT) break;
      }
      // ---- phase B ----
      {
        const double alpha = st->alpha;
        const int p2 = st->fmt[1], p4 = st->fmt[3];
        const bool sig_rr = (p2 == F64 && p4 == F64 && !S.A.dinv && !IC);
        double rr = 0.0;
        DotAcc sg{0.0, 0.f, 0.f};
        team_phase_b<IC>(t, IC ? 1 : 0, alpha, p2, p4, sig_rr, rr, sg);
        if constexpr (IC) {
          T = team_apply_ic<CL>(L, t, T);
          team_phase_b<IC>(t, 2, alpha, p2, p4, false, rr, sg);
        }
        if (active) rr = warp_sum(rr);
        const double v[2] = {rr, active && !sig_rr ? warp_dot(sg, p4 != F64) : 0.0};
        team_exchange<CL, 2>(L, t, T, v, sig_rr ? 1 : 2);
        team_step_b(L, t, sig_rr ? 0 : 1);
        if (!team_ok(t)) return false;
      }
      const int mode = st->mode;
      const double alpha = st->alpha;
      if (mode == M_CONT) {
        // ---- phase C ----
        team_phase_c(t, alpha, st->beta, st->fmt[0]);
        const int k = st->k;
        team_publish<CL>(L, t, T);
        stamp_c(S, st);
        if (k >= S.max_iter) break;
        continue;
      }
      if (mode == M_DONE) break;
      // ---- phase X ----
      for (int i = threadIdx.x; i < V.n; i += kTT) V.x[i] = fma(alpha, V.p[i], V.x[i]);
      if (mode == M_X_THEN_DONE) break;
      if (mode == M_X_THEN_RESTART64) {
        const TeamOk ro = team_restart64<CL, IC>(L, t, T);
        T = ro.T;
        if (!ro.ok) return false;
        if (st->mode != M_CONT) break;
        continue;
      }
      // ---- phase T ----
      {
        const int p2 = st->fmt[1], p4 = st->fmt[3];
        team_store_x(t);
        team_publish<CL>(L, t, T);
        const double rr = team_true_res(t);
        const TeamDot u = team_use_r<CL, IC>(L, t, T, p2, p4, false);
        T = u.T;
        const DotAcc sg = u.sg;
        const double v[2] = {warp_sum(rr), warp_dot(sg, p4 != F64)};
        team_exchange<CL, 2>(L, t, T, v);
        step_T(L, S, st, t.sum[0], t.sum[1], sm);
        if (!team_ok(t)) return false;
      }
      if (st->mode == M_RESTART64) {
        const TeamOk ro = team_restart64<CL, IC>(L, t, T);
        T = ro.T;
        if (!ro.ok) return false;
        if (st->mode != M_CONT) break;
        continue;
      }
      if (st->mode == M_RESTART) {
        const int p2 = st->zfmt, p1n = st->fmt[0], k = st->k;
        const TeamMinv<IC> minv = team_minv<IC>(t);  // (IC(0): the application of phase T)
        for (int i = threadIdx.x; i < V.n; i += kTT) V.p[i] = z_of(minv(i, V.r[i]), p2);
        team_copy_p(t, p1n);
        team_publish<CL>(L, t, T);
        if (k >= S.max_iter) break;
        continue;
      }
      break;
    }
  }

  // ---- x, and ||b - A x|| in fp64 unless already known ----
  team_store_x(t);
  if (threadIdx.x == 0) team_rho(t);
  double rr = 0.0;
  if (!st->true_known) {
    team_publish<CL>(L, t, T);
    rr = team_true_res(t);
  }
  const double v[1] = {warp_sum(rr)};
  team_exchange<CL, 1>(L, t, T, v);
  if (t.rank == 0) {
    step_final(L, S, st, sid, t.sum[0]);
    __syncthreads();
    const int words = (int)(sizeof(SysState) / 4);
    for (int i = threadIdx.x; i < words; i += kTT) ((unsigned*)(L.st + sid))[i] = ((const unsigned*)st)[i];
  }
  return team_ok(t);
}

// Clusters: team_cta gives every CTA its system (-1: none), rank, team size and the team's first
// CTA in the cluster; a cluster holds one team or several smaller ones, and the hardware starts
// the next cluster where one has finished. Whole grid: all CTAs are one team on system 0.
template <bool CL, bool IC>
__global__ void __launch_bounds__(kTT, 1) cg_team(const __grid_constant__ Launch L) {
  extern __shared__ __align__(128) unsigned char dyn[];
  TeamSmem& t = *reinterpret_cast<TeamSmem*>(dyn);
  double* heap = reinterpret_cast<double*>(dyn + kTeamFixed);
  int sid = 0, rank = blockIdx.x, size = gridDim.x, base = 0;
  if constexpr (CL) {
    const int4 a = L.team_cta[blockIdx.x];
    sid = a.x;
    rank = a.y;
    size = a.z;
    base = a.w;
    if (sid < 0) {  // a place of the cluster that no system needs
      cluster_sync_all();
      cluster_sync_all();
      return;
    }
  }
  for (int i = threadIdx.x; i < (int)(sizeof(DevSys) / 4); i += kTT)
    ((unsigned*)&t.S)[i] = ((const unsigned*)(L.sys + sid))[i];
  for (int i = threadIdx.x; i < (int)(sizeof(SysState) / 4); i += kTT) ((unsigned*)&t.st)[i] = 0u;
  if (threadIdx.x == 0) {
    t.rank = rank;
    t.size = size;
    t.base = base;
    t.gslot = L.xch;
    t.xs = heap;
    t.bad = 0;
    t.nq = t.nl = 0;
    mbar_init(t.xbar + 0, 1);
    mbar_init(t.xbar + 1, 1);
    mbar_init(t.pbar + 0, (unsigned)size);
    mbar_init(t.pbar + 1, (unsigned)size);
    for (int i = 0; i < kIcBars; ++i) mbar_init(&t.icbar[i], 1);
    t.icuse = 0;
    t.icissued = 0;
    t.icdone = 0;
    mbar_fence_init();
  }
  __syncthreads();
  if constexpr (CL) cluster_sync_all();
  long long room = (long long)L.team_heap / 8;  // fp64 values of shared memory left
  if constexpr (!CL) {
    const long long used = (long long)kXV * t.size;
    heap += used;
    room -= used;
  }
  if (L.team_q) {  // a copy of the table (its reads are on the chain)
    for (int i = threadIdx.x; i < L.team_q; i += kTT) heap[i] = L.pol.Q[i];
    int* vis = (int*)(heap + L.team_q);
    const int nv = L.pol.visits ? L.team_v : 0;
    for (int i = threadIdx.x; i < nv; i += kTT) vis[i] = L.pol.visits[i];
    __syncthreads();
    if (threadIdx.x == 0) {
      t.S.Qpriv = heap;
      t.S.vtab = nv ? vis : nullptr;
    }
    const int used = (L.team_q + (L.team_v + 1) / 2 + 1) & ~1;  // (16-byte alignment)
    heap += used;
    room -= used;
  }
  if constexpr (IC) {
    if (threadIdx.x == 0) {
      t.icring = (unsigned char*)heap;  // (first: the block copies need 16-byte alignment)
      t.icW = (float*)(heap + t.S.A.icring / 8);
      t.icW[t.S.A.n] = 0.f;  // the padding entries' cell
    }
    const long long used = t.S.A.icring / 8 + (t.S.A.n + 2) / 2;
    heap += used;
    room -= used;
  }
  if (threadIdx.x < 32) {
    const long long W = t.S.A.nnz + 4LL * t.S.A.n;
    const int a = t.rank == 0 ? 0 : warp_row_at(t.S.A.rp, t.S.A.n, W * t.rank / t.size);
    const int b = t.rank + 1 == t.size ? t.S.A.n : warp_row_at(t.S.A.rp, t.S.A.n, W * (t.rank + 1) / t.size);
    if (threadIdx.x == 0) {
      t.sm.r0 = a;
      t.sm.r1 = b;
      if (t.rank != 0) t.S.hist = nullptr;  // one CTA of the team writes the records
    }
  }
  double* const heap0 = heap;
  if (threadIdx.x == 0) {
    TeamVec& V = t.V;
    V.r0 = t.sm.r0;
    V.n = t.sm.r1 - t.sm.r0;
    t.nact = V.n >= kTT ? kTW : (V.n + 31) / 32;
    t.ntop = t.nact > 1 ? 1 << (31 - __clz(t.nact - 1)) : 0;
    if (4LL * V.n <= room) {
      V.r = heap;
      V.p = V.r + V.n;
      V.x = V.p + V.n;
      V.q = V.x + V.n;
    } else {
      V.r = t.S.r + V.r0;
      V.p = t.S.p + V.r0;
      V.x = t.S.x + V.r0;
      V.q = (double*)t.S.q + V.r0;
    }
  }
  __syncthreads();
  // The warps' product tiles, then (without tiles) the row bounds and columns to shared memory when
  // there is room: the product's chain of dependent loads then has one step outside it (the values
  // and the gathers, issued together) instead of three.
  {
    const int n = t.V.n, r0 = t.V.r0;
    const long long room0 = room - 4LL * n;
    const bool shared = t.V.r == heap0;
    double* const after = shared ? heap0 + 4LL * n : heap0;
    const bool tiles = t.S.A.tile && L.tile && (long long)kTeamTileWarp * kTW / 8 + 2 <= (shared ? room0 : room);
    const int ea = n > 0 ? __ldg(t.S.A.rp + r0) & ~7 : 0, eb = n > 0 ? (__ldg(t.S.A.rp + r0 + n) + 7) & ~7 : 0;
    const long long words = (long long)(eb - ea) + n + 8;
    const bool fits = shared && !tiles && words / 2 + 2 <= room0;
    int* cs = reinterpret_cast<int*>(reinterpret_cast<unsigned long long>(heap0 + 4LL * n + 1) & ~15ull);
    int* rs = cs + (eb - ea);
    if (fits) {
      for (int i = threadIdx.x; i < eb - ea; i += kTT) cs[i] = __ldg(t.S.A.ci + ea + i);
      for (int i = threadIdx.x; i <= n && n > 0; i += kTT) rs[i] = __ldg(t.S.A.rp + r0 + i);
    }
    if (threadIdx.x == 0) {
      t.tile = tiles ? reinterpret_cast<unsigned char*>((reinterpret_cast<unsigned long long>(after + 1)) & ~15ull) : nullptr;
      // (no pointer is moved below its array: shared addresses are 32 bits wide)
      t.rp = fits ? rs : t.S.A.rp;
      t.ci = fits ? cs : t.S.A.ci;
      t.rbase = fits ? r0 : 0;
      t.ebase = fits ? ea : 0;
    }
    __syncthreads();
  }
  const bool ok = solve_team<CL, IC>(L, t, sid);
  if constexpr (IC) {
    if (!ok) ic_drain(t);
  }
  // no CTA of a cluster leaves while a peer may still write into its shared memory; after a wait that gave
  // up, messages that nobody waits for any more (a microsecond each) get time to land
  if constexpr (CL) {
    cluster_sync_all();
    if (!ok)
      for (int i = 0; i < 100; ++i) __nanosleep(1000);
  }
}

// Launches a cluster form of the kernel.
inline cudaError_t team_launch_cluster(void (*kernel)(const Launch), const Launch& L, int cluster, int grid, size_t smem,
                                       cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cluster;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kTT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, L);
}

}  // namespace
}  // namespace mpcg
