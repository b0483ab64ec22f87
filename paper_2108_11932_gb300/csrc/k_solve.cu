// TLR triangular solves (Algorithm 7 and its transpose), and the vector kernels of preconditioned CG.
//
// One persistent kernel does both solves of a group of right-hand sides, left-looking:
//   forward, k = 0 .. nb-1:   X_k -= Urow_k T_k;  Z_k = L_kk^-1 X_k;  T_ik = V_ik^T Z_k (all i > k)
//   (L D L^T)                 W_k = D_k^-1 Z_k
//   backward, k = nb-1 .. 0:  W_k -= Vcol_k S_k;  X_k = L_kk^-T W_k;  S_kj = U_kj^T X_k (all j < k)
// where T_k (S_k) stacks the T_kj (S_ik) in the order of the block row's (column's) contiguous panel.  That is
// a chain of 6 nb dependent steps of a few microseconds of FP64 work for the whole GPU at N = 131072, and
// less below.  Launched one by one (a captured graph) a step cost 10 us at N = 131072 and 4 us at N = 4096.
// Here the CTAs stay resident (cooperative launch, one per SM), a step ends with a grid barrier, and what a
// step costs beyond its FP64 work is kept to one L2 round trip: the factor entries that a thread multiplies
// first are loaded into registers before the barrier (they do not depend on the solution), and the step
// after next is prefetched into L2.  Two kinds of step:
//   rows  y(m) = sum_k A(m, k) x(k): units of 4 to 16 rows, the 8 warps of a CTA sharing k
//   cols  y(c) = sum_k A(k, c) x(k): one warp per column
// (right-looking updates of all remaining tiles, tried first, took 25 us a step: a tile's rank varies from
// 0 to ten times the mean, and the deepest tile's chain of loads set the pace).
//
// (One cluster of 16 CTAs with the hardware's cluster barrier, tried for small problems, gains 5% at N = 2048,
// b = 256, one column, and loses from N = 4096 on: 334 against 343 us.)
//
// Right-hand sides go in groups of NR <= 8 columns held in registers, without padding to a tile; the
// vector a step multiplies is staged in shared memory.  Bound: the FP64 unit (one DFMA per entry and
// column) plus the barriers.  Sums run in a fixed order: results do not depend on timing.
//
// Measured, graph of launches -> now: 2D N = 131072 (b = 1024, eps = 1e-6), 1 column 7.7 -> 4.5 ms (1.1 ms of it
// FP64 work, the rest 763 steps of about 4.5 us: 1.0 barrier, 0.6 staging, 0.8 sums and stores); N = 4096
// (b = 256) 395 -> 338 us; 3D N = 20011 L D L^T, 32 columns 14.7 -> 9.1 ms (4.6 ms of FP64 work).
//
// Every wait is bounded: a barrier that runs out sets a flag in host-visible memory, the CTAs leave the
// kernel, the result is overwritten with NaN and the context's next solve reports TLR_ERR_TIMEOUT.
#include <algorithm>
#include <cstring>

#include "internal.h"
#include "warpsum.cuh"

namespace tlr {

namespace {

constexpr int SV_T = 256, SV_W = SV_T / 32;
constexpr int SV_NRHS = 32;        // right-hand sides per launch
constexpr int SV_RB = 16;          // most rows of a unit
constexpr int SV_U = 32;           // factor entries a thread holds in flight
constexpr int SV_RLD = SV_W + 1;   // padded row of warp partials
constexpr int SV_XS = 16384;       // staged vector entries (128 KB)
constexpr unsigned long long SV_WAIT_NS = 2000000000ull;

// A step.  Rows: y = A x over the n columns of A (b rows; kind 1: column k has rows m >= k); kind 0
// X_k -= y with x = T_k, 1 Z_k = y and W_k = D_k^-1 y, 2 W_k -= y with x = S_k.  Cols: y = A^T x for the n
// columns of A; kind 3 x = Z_k into T, 4 x = W_k (rows m >= c) into X_k, 5 x = X_k into S.
struct __align__(16) SvStep {
  const double* A;
  const int* map;  // kinds 3, 5: row of T or S for each column
  int kind, k, n;
  int t0;          // kinds 0, 2: first row of T_k or S_k
};
struct SvTab {
  const SvStep* steps;
  const double* dvec;  // L D L^T, else null
  int nsteps, b;
};
struct SvVec {
  double *X, *Z, *W, *TS;  // column-major, ng NR columns; X, Z, W with leading dimension np; T and S share TS (ld ldt)
  int64_t np, ldt;
  int ng, xs;              // xs: staged vector entries per column
  unsigned* bar;           // {grid barrier arrivals, a wait ran out}, zero at launch
  volatile int* timeout;   // the latter, host-visible
};

__device__ __forceinline__ unsigned sv_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long sv_clock() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Prefetch into L2 of the whole 16-byte words of [p, p + bytes).
__device__ __forceinline__ void sv_prefetch(const void* p, int64_t bytes) {
  uintptr_t a = reinterpret_cast<uintptr_t>(p);
  const uintptr_t e = (a + bytes) & ~uintptr_t(15);
  a = (a + 15) & ~uintptr_t(15);
  if (a < e)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"((unsigned)(e - a)) : "memory");
}

template <int NR>
__host__ __device__ constexpr int sv_pow2() { return NR == 3 ? 4 : NR == 6 ? 8 : NR; }


template <int NR>
__global__ void __launch_bounds__(SV_T, 1) k_solve(SvTab T, SvVec v) {
  extern __shared__ __align__(16) double sm[];
  double* red = sm;                       // SV_RB NR x SV_RLD
  double* xs = sm + SV_RLD * NR * SV_RB;  // NR x v.xs: the step's vector, column-major
  __shared__ int go;
  __shared__ SvStep ring[4];
  const int b = T.b, G = (int)gridDim.x, bid = (int)blockIdx.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned arrivals = 0;

  // The barrier in two halves: what a CTA does between them (loads that do not depend on the solution)
  // is neither ordered by the release nor in the way of the other CTAs.
  auto arrive = [&]() {
    __syncthreads();
    arrivals += G;
    if (tid == 0) {
      __threadfence();
      atomicAdd(v.bar, 1u);
    }
  };
  auto wait = [&]() -> bool {
    if (tid == 0) {
      int good = 1;
      if (sv_acquire(v.bar) < arrivals) {
        const unsigned long long t0 = sv_clock();
        for (unsigned it = 0; sv_acquire(v.bar) < arrivals; ++it)
          if ((it & 63u) == 63u && (sv_acquire(v.bar + 1) || sv_clock() - t0 > SV_WAIT_NS || it > (1u << 28))) {
            atomicExch(v.bar + 1, 1u);
            *v.timeout = 1;
            good = 0;
            break;
          }
      }
      __threadfence();
      go = good;
    }
    __syncthreads();
    return go != 0;
  };

  // rows r0 .. r0 + len - 1 of group g's columns of x (leading dimension ldx) into shared memory
  auto stage = [&](const double* x, int64_t ldx, int g, int64_t r0, int len) {
    constexpr int SU = NR >= 4 ? 2 : 8 / NR;  // SU NR loads in flight per thread
    const double* p = x + (int64_t)g * NR * ldx + r0;
    for (int k0 = tid; k0 < len; k0 += SU * SV_T) {
      double t[SU][NR];
#pragma unroll
      for (int u = 0; u < SU; ++u)
#pragma unroll
        for (int n = 0; n < NR; ++n)
          if (k0 + u * SV_T < len) t[u][n] = __ldcg(p + n * ldx + k0 + u * SV_T);
#pragma unroll
      for (int u = 0; u < SU; ++u)
#pragma unroll
        for (int n = 0; n < NR; ++n)
          if (k0 + u * SV_T < len) xs[n * v.xs + k0 + u * SV_T] = t[u][n];
    }
  };

  // ---- rows steps: unit = RB = 2^rsh rows of one group; units (longest first for a triangle) dealt out
  // forth and back over the CTAs.  Lane (row, sub) of warp w takes k = slot + u 2^lsh, slot = w subs + sub.
  int rsh = 2;
  while (rsh < 4 && ((b + (1 << rsh) - 1) >> rsh) * v.ng > G) ++rsh;
  const int RB = 1 << rsh, lsh = 8 - rsh, slots = 1 << lsh, slot = (warp << (5 - rsh)) + (lane >> rsh);
  const int nu = (b + RB - 1) >> rsh, units = nu * v.ng;
  static_assert(SV_T == 256 && SV_RB == 16, "slots of a unit");
  auto unit_at = [&](int t) { return (t & 1) ? (t + 1) * G - 1 - bid : t * G + bid; };
  auto unit_r0 = [&](int id) { return (nu - 1 - id / v.ng) << rsh; };
  auto unit_len = [&](const SvStep& s, int id) { return s.kind == 1 ? min(b, unit_r0(id) + RB) : s.n; };
  // entries k0 + slot + u slots < len of this lane's row
  auto rows_load = [&](const SvStep& s, int id, int k0, int len, double (&a)[SV_U]) {
    const int m = unit_r0(id) + (lane & (RB - 1));
    const int lim = m < b ? (s.kind == 1 ? min(len, m + 1) : len) : 0;
    const int n = (lim - k0 - slot + slots - 1) >> lsh;  // <= 0: none
    const double* p = s.A + m + (size_t)(k0 + slot) * b;
    const size_t st = (size_t)b << lsh;
#pragma unroll
    for (int u = 0; u < SV_U; ++u) {
      a[u] = u < n ? __ldg(p) : 0.0;
      p += st;
    }
  };
  auto rows_run = [&](const SvStep& s, double (&a)[SV_U]) {
    const double* x = s.kind == 1 ? v.X + (size_t)s.k * b : v.TS + s.t0;
    const int64_t ldx = s.kind == 1 ? v.np : v.ldt;
    for (int t = 0; t * G < units; ++t) {
      const int id = unit_at(t);
      if (id >= units) continue;
      const int g = id % v.ng, r0 = unit_r0(id), len = unit_len(s, id);
      if (t > 0) rows_load(s, id, 0, len, a);
      double acc[NR];
#pragma unroll
      for (int n = 0; n < NR; ++n) acc[n] = 0.0;
      for (int c0 = 0; c0 < len; c0 += v.xs) {  // staged pieces of x
        const int cn = min(v.xs, len - c0);
        __syncthreads();
        stage(x, ldx, g, c0, cn);
        __syncthreads();
        for (int k0 = 0; k0 < cn; k0 += SV_U * slots) {
          if (c0 + k0 > 0) rows_load(s, id, c0 + k0, c0 + cn, a);
          const int nl = (cn - k0 - slot + slots - 1) >> lsh;                        // this lane's entries
          const int nw = (cn - k0 - (warp << (5 - rsh)) + slots - 1) >> lsh;         // the warp's most
          const double* xp = xs + k0 + slot;
#pragma unroll
          for (int u = 0; u < SV_U; ++u) {
            if (u >= nw) break;
#pragma unroll
            for (int n = 0; n < NR; ++n) acc[n] = fma(a[u], u < nl ? xp[n * v.xs + u * slots] : 0.0, acc[n]);
          }
        }
      }
#pragma unroll
      for (int n = 0; n < NR; ++n) {
        for (int o = RB; o < 32; o *= 2) acc[n] += __shfl_xor_sync(0xffffffffu, acc[n], o);
        if (lane < RB) red[((n << rsh) + lane) * SV_RLD + warp] = acc[n];
      }
      __syncthreads();
      // warp partials: four lanes per output
      for (int o = tid >> 2; o < RB * NR; o += SV_T / 4) {
        const double* r = red + o * SV_RLD + (tid & 3) * (SV_W / 4);
        const int row = r0 + (o & (RB - 1));
        const bool out = (tid & 3) == 0 && row < b;
        const int64_t at = (int64_t)(g * NR + (o >> rsh)) * v.np + (size_t)s.k * b + row;
        double old = 0.0;
        if (out && s.kind == 0) old = __ldcg(v.X + at);
        if (out && s.kind == 2) old = __ldcg(v.W + at);
        if (out && s.kind == 1 && T.dvec) old = 1.0 / __ldg(T.dvec + (size_t)s.k * b + row);
        double z = r[0];
#pragma unroll
        for (int w = 1; w < SV_W / 4; ++w) z += r[w];
        const unsigned mask = __activemask();  // whole groups of four
        z += __shfl_xor_sync(mask, z, 1);
        z += __shfl_xor_sync(mask, z, 2);
        if (out) {
          if (s.kind == 0) {
            v.X[at] = old - z;
          } else if (s.kind == 2) {
            v.W[at] = old - z;
          } else {
            v.Z[at] = z;
            if (T.dvec) v.W[at] = z * old;
          }
        }
      }
    }
  };

  // ---- cols steps: one warp per column and group; consecutive columns go to different CTAs
  const bool cols_staged = b <= v.xs;
  auto cols_load = [&](const SvStep& s, int c, int k0, double (&a)[SV_U]) {
    const double* p = s.A + (size_t)c * b + k0 + lane;
    const int n = (b - k0 - lane + 31) >> 5;
#pragma unroll
    for (int u = 0; u < SV_U; ++u) a[u] = u < n ? __ldg(p + 32 * u) : 0.0;
    if (s.kind == 4 && k0 + lane < c) a[0] = 0.0;  // k0 <= c: the rows above the diagonal are in the first load
  };
  auto cols_first = [&](const SvStep& s, int c) { return s.kind == 4 ? c & ~31 : 0; };
  // position p (of cpc G per group) -> column
  auto col_of = [&](int p, int cpc) { return (p % cpc) * G + p / cpc; };
  auto cols_run = [&](const SvStep& s, double (&a)[SV_U]) {
    constexpr int P = sv_pow2<NR>();
    const double* x = (s.kind == 3 ? v.Z : s.kind == 4 ? v.W : v.X) + (size_t)s.k * b;
    const int cpc = (s.n + G - 1) / G, per = cpc * G, q0 = bid * cpc * v.ng, q1 = q0 + cpc * v.ng;
    for (int q = q0; q < q1;) {
      const int g = q / per, qe = min(q1, (g + 1) * per);
      if (cols_staged) {
        __syncthreads();
        stage(x, v.np, g, 0, b);
        __syncthreads();
      }
      for (int p = q + warp; p < qe; p += SV_W) {
        const int c = col_of(p - g * per, cpc);
        if (c >= s.n) continue;
        const int row = s.kind == 4 ? 0 : __ldg(s.map + c);
        double acc[P];
#pragma unroll
        for (int n = 0; n < P; ++n) acc[n] = 0.0;
        const int kb = cols_first(s, c);
        for (int k0 = kb; k0 < b; k0 += 32 * SV_U) {
          if (p != q0 + warp || k0 != kb) cols_load(s, c, k0, a);
          const int nl = (b - k0 - lane + 31) >> 5, nw = (b - k0 + 31) >> 5;
          if (cols_staged) {
            const double* xp = xs + k0 + lane;
#pragma unroll
            for (int u = 0; u < SV_U; ++u) {
              if (u >= nw) break;
#pragma unroll
              for (int n = 0; n < NR; ++n) acc[n] = fma(a[u], u < nl ? xp[n * v.xs + 32 * u] : 0.0, acc[n]);
            }
          } else {
            const double* xp = x + (int64_t)g * NR * v.np + k0 + lane;
#pragma unroll
            for (int u = 0; u < SV_U; ++u) {
              if (u >= nw) break;
#pragma unroll
              for (int n = 0; n < NR; ++n) acc[n] = fma(a[u], u < nl ? __ldcg(xp + n * v.np + 32 * u) : 0.0, acc[n]);
            }
          }
        }
        const double y = warp_sums<P>(acc, lane);
        const int n = lane / (32 / P);
        if (lane % (32 / P) == 0 && n < NR) {
          if (s.kind == 4) v.X[(int64_t)(g * NR + n) * v.np + (size_t)s.k * b + c] = y;
          else v.TS[(int64_t)(g * NR + n) * v.ldt + row] = y;
        }
      }
      q = qe;
    }
  };

  // the factor entries a thread multiplies first in a step
  auto load_first = [&](const SvStep& s, double (&a)[SV_U]) {
    if (s.kind < 3) {
      const int id = unit_at(0);
      if (id < units) rows_load(s, id, 0, min(unit_len(s, id), v.xs), a);
    } else {
      const int cpc = (s.n + G - 1) / G, p = bid * cpc * v.ng + warp, per = cpc * G;
      if (p < (bid + 1) * cpc * v.ng) {
        const int c = col_of(p % per, cpc);
        if (c < s.n) cols_load(s, c, cols_first(s, c), a);
      }
    }
  };

  // L2 prefetch of a step's factor data, dealt out over the CTAs (one warp)
  auto prefetch = [&](const SvStep& s) {
    if (s.kind == 1 || s.kind == 4) {
      for (int c = bid * 32 + lane; c < b; c += G * 32) sv_prefetch(s.A + c + (size_t)c * b, sizeof(double) * (b - c));
    } else {
      constexpr int64_t CH = 1024;  // 8 KB pieces
      const int64_t n = (int64_t)b * s.n;
      for (int64_t c = (int64_t)(lane * G + bid) * CH; c < n; c += (int64_t)G * 32 * CH)
        sv_prefetch(s.A + c, sizeof(double) * min(CH, n - c));
    }
  };
  // Steps i .. i + 3 in a ring in shared memory, copied asynchronously two steps before they are first read
  // (the list ends with three copies of its last step, so that the look-ahead needs no test).
  auto fetch = [&](int i) {
    if (tid < (int)(sizeof(SvStep) / 16)) {
      const unsigned d = (unsigned)__cvta_generic_to_shared(reinterpret_cast<char*>(ring + (i & 3)) + 16 * tid);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d),
                   "l"(reinterpret_cast<const char*>(T.steps + i) + 16 * tid)
                   : "memory");
    }
  };
  auto landed = [&]() { asm volatile("cp.async.wait_all;" ::: "memory"); };

  double a[SV_U];
  fetch(0);
  fetch(1);
  fetch(2);
  landed();
  __syncthreads();
  load_first(ring[0], a);
  for (int i = 0;;) {
    const SvStep& s = ring[i & 3];
    if (s.kind < 3) rows_run(s, a);
    else cols_run(s, a);
    landed();
    if (++i == T.nsteps) break;
    arrive();
    load_first(ring[i & 3], a);
    fetch(i + 2);  // into the slot of step i - 2
    if (warp == SV_W - 1) prefetch(ring[(i + 1) & 3]);
    if (!wait()) break;
  }
  landed();
}

// gather: X[p, c] = B[perm[p], c] (rows past N zero), and the barrier words cleared; scatter: the reverse,
// NaN after a wait that ran out
__global__ void k_solve_gather(int64_t N, int64_t np, int nrhs, const int64_t* __restrict__ perm,
                               const double* __restrict__ B, int64_t ldb, double* __restrict__ X, unsigned* bar) {
  if (blockIdx.x == 0 && threadIdx.x < 2) bar[threadIdx.x] = 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < np * nrhs; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = e % np, c = e / np;
    X[e] = p < N ? B[perm[p] + c * ldb] : 0.0;
  }
}
__global__ void k_solve_scatter(int64_t N, int64_t np, int nrhs, const int64_t* __restrict__ perm,
                                const double* __restrict__ X, double* __restrict__ B, int64_t ldb,
                                const unsigned* __restrict__ bar) {
  const bool bad = bar[1] != 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < N * nrhs; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = e % N, c = e / N;
    B[perm[p] + c * ldb] = bad ? nan("") : X[p + c * np];
  }
}

unsigned sv_blocks(int64_t n) { return (unsigned)std::min<int64_t>((n + 255) / 256, 8192); }

}  // namespace

// A factor's tables for the solve kernel (panel pointers and offsets; device) and its work vectors, kept
// until the factor's storage changes.  The vectors grow with the widest solve seen (<= 32 columns).
struct SolvePlan {
  char* tab = nullptr;
  double* vec = nullptr;
  SvTab T{};
  int64_t np = 0, ldt = 0, len = 0;  // len: longest panel (columns)
  int cols = 0;        // columns the vectors hold
};

void plan_destroy(tlr_ctx* ctx, SolvePlan* P) {
  if (!P) return;
  dfree(ctx, P->tab);
  dfree(ctx, P->vec);
  delete P;
}

static SolvePlan* plan_build(tlr_ctx* ctx, const tlr_mat* F) {
  const int nb = F->nb, b = F->b;
  std::vector<int64_t> tr0(nb + 1, 0), sc0(nb + 1, 0);
  int64_t len = 1;
  for (int i = 0; i < nb; ++i) {
    tr0[i + 1] = tr0[i] + F->ulen[i];
    sc0[i + 1] = sc0[i] + F->vlen[i];
    len = std::max<int64_t>({len, F->ulen[i], F->vlen[i]});
  }
  const int64_t R = tr0[nb];
  TLR_REQUIRE(R < (1LL << 31), TLR_ERR_LIMIT, "solve: too many factor columns");
  // maps between the V panels' columns (S's rows) and the U panels' columns (T's rows), then the steps
  std::vector<int> map(2 * (size_t)R);
  int *v2u = map.data(), *u2v = v2u + R;
  for (int i = 0; i < nb; ++i)
    for (int j = 0; j < i; ++j) {
      const int64_t uc = tr0[i] + F->uoff[ix(F, i, j)], vc = sc0[j] + F->voff[ix(F, i, j)];
      for (int a = 0; a < F->rank[ix(F, i, j)]; ++a) {
        v2u[vc + a] = (int)(uc + a);
        u2v[uc + a] = (int)(vc + a);
      }
    }
  const size_t bm = sizeof(int) * map.size(), bs = sizeof(SvStep) * (6 * (size_t)nb + 3), os = (bm + 15) / 16 * 16;
  auto* P = new SolvePlan();
  P->np = (int64_t)nb * b;
  P->ldt = std::max<int64_t>(R, 1);
  P->len = len;
  try {
    P->tab = static_cast<char*>(dalloc(ctx, os + bs));
    const int* dv2u = reinterpret_cast<const int*>(P->tab);
    const int* du2v = dv2u + R;
    std::vector<SvStep> st;
    auto dk = [&](int k) { return F->dinv + (size_t)k * b * b; };
    for (int k = 0; k < nb; ++k) {
      const int ul = (int)F->ulen[k], vl = (int)F->vlen[k];
      if (ul > 0) st.push_back(SvStep{F->Urow[k], nullptr, 0, k, ul, (int)tr0[k]});
      st.push_back(SvStep{dk(k), nullptr, 1, k, b, 0});
      if (vl > 0) st.push_back(SvStep{F->Vcol[k], dv2u + sc0[k], 3, k, vl, 0});
    }
    for (int k = nb - 1; k >= 0; --k) {
      const int ul = (int)F->ulen[k], vl = (int)F->vlen[k];
      if (vl > 0) st.push_back(SvStep{F->Vcol[k], nullptr, 2, k, vl, (int)sc0[k]});
      st.push_back(SvStep{dk(k), nullptr, 4, k, b, 0});
      if (ul > 0) st.push_back(SvStep{F->Urow[k], du2v + tr0[k], 5, k, ul, 0});
    }
    P->T = SvTab{reinterpret_cast<const SvStep*>(P->tab + os), F->state == 2 ? F->dvec : nullptr, (int)st.size(), b};
    for (int q = 0; q < 3; ++q) st.push_back(st.back());
    const size_t chunk = (size_t)16 << 20;  // through the pinned upload ring (no host synchronization)
    auto put = [&](char* dst, const void* src, size_t bytes) {
      for (size_t o = 0; o < bytes; o += chunk) {
        const size_t n = std::min(chunk, bytes - o);
        TLR_CUDA(cudaMemcpyAsync(dst + o, upload(ctx, static_cast<const char*>(src) + o, n), n, cudaMemcpyDeviceToDevice,
                                 ctx->stream));
      }
    };
    put(P->tab, map.data(), bm);
    put(P->tab + os, st.data(), sizeof(SvStep) * st.size());
  } catch (...) {
    plan_destroy(ctx, P);
    throw;
  }
  return P;
}

template <int NR>
static void solve_launch(tlr_ctx* ctx, const SolvePlan* P, SvVec v) {
  const int b = P->T.b;
  v.xs = (int)std::min<int64_t>(SV_XS / NR, std::max<int64_t>(b, P->len));
  const size_t smem = sizeof(double) * ((size_t)SV_RLD * NR * SV_RB + (size_t)NR * v.xs);
  cudaLaunchConfig_t cf{};
  cudaLaunchAttribute at{};
  cf.blockDim = dim3(SV_T);
  cf.dynamicSmemBytes = smem;
  cf.stream = ctx->stream;
  cf.attrs = &at;
  cf.numAttrs = 1;
  auto kern = k_solve<NR>;
  TLR_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  at.id = cudaLaunchAttributeCooperative;  // the CTAs wait for one another: all resident, or none
  at.val.cooperative = 1;
  cf.gridDim = dim3((unsigned)ctx->sm_count);
  TLR_SITE_PRE(ctx);
  TLR_CUDA(cudaLaunchKernelEx(&cf, kern, P->T, v));
  TLR_LAUNCH_CHECK(ctx);
}

void tlr_solve_factor(tlr_ctx* ctx, tlr_mat* F, int nrhs, double* B, int64_t ldb) {
  if (*ctx->wait_out) {
    *ctx->wait_out = 0;
    throw Error(TLR_ERR_TIMEOUT, "solve: a bounded device wait of an earlier solve ran out");
  }
  if (!F->plan) F->plan = plan_build(ctx, F);
  SolvePlan* P = F->plan;
  const int ng32 = (nrhs + SV_NRHS - 1) / SV_NRHS;
  for (int h = 0; h < ng32; ++h) {  // equal launches of at most 32 columns, each in equal groups of at most 8
    const int c0 = (int)((int64_t)nrhs * h / ng32), nc = (int)((int64_t)nrhs * (h + 1) / ng32) - c0;
    const int ng = (nc + 7) / 8, w = (nc + ng - 1) / ng, nr = w <= 4 ? w : w <= 6 ? 6 : 8, cols = ng * nr;
    const size_t one = 3 * (size_t)P->np + (size_t)P->ldt;
    if (cols > P->cols) {
      dfree(ctx, P->vec);
      P->vec = nullptr;
      P->cols = 0;
      P->vec = static_cast<double*>(dalloc(ctx, sizeof(double) * (one * cols + 32)));
      P->cols = cols;
    }
    SvVec v{};
    v.np = P->np;
    v.ldt = P->ldt;
    v.ng = ng;
    v.bar = reinterpret_cast<unsigned*>(P->vec);
    v.X = P->vec + 32;
    v.Z = v.X + (size_t)P->np * cols;
    v.W = P->T.dvec ? v.Z + (size_t)P->np * cols : v.Z;
    v.TS = v.Z + 2 * (size_t)P->np * cols;
    v.timeout = ctx->wait_out;
    double* Bc = B + (size_t)c0 * ldb;
    TLR_SITE_PRE(ctx);
    k_solve_gather<<<sv_blocks(P->np * nc), 256, 0, ctx->stream>>>(F->N, P->np, nc, F->dperm, Bc, ldb, v.X, v.bar);
    TLR_LAUNCH_CHECK(ctx);
    if (cols > nc)  // padding columns of the last group
      TLR_CUDA(cudaMemsetAsync(v.X + (size_t)P->np * nc, 0, sizeof(double) * (size_t)P->np * (cols - nc), ctx->stream));
    if (nr == 1) solve_launch<1>(ctx, P, v);
    else if (nr == 2) solve_launch<2>(ctx, P, v);
    else if (nr == 3) solve_launch<3>(ctx, P, v);
    else if (nr == 4) solve_launch<4>(ctx, P, v);
    else if (nr == 6) solve_launch<6>(ctx, P, v);
    else solve_launch<8>(ctx, P, v);
    TLR_SITE_PRE(ctx);
    k_solve_scatter<<<sv_blocks(F->N * nc), 256, 0, ctx->stream>>>(F->N, P->np, nc, F->dperm, v.X, Bc, ldb, v.bar);
    TLR_LAUNCH_CHECK(ctx);
  }
}

// ------------------------------------------------------------------ preconditioned CG vectors
// out[c] = sum_i X(i, c) Y(i, c): one CTA per column, strided partial sums, then a fixed-order tree.
__global__ void __launch_bounds__(256) k_coldot(int64_t n, const double* __restrict__ X, int64_t ldx,
                                                const double* __restrict__ Y, int64_t ldy, double* __restrict__ out) {
  __shared__ double sh[256];
  const int c = blockIdx.x;
  const double* x = X + (size_t)c * ldx;
  const double* y = Y + (size_t)c * ldy;
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += 256) s = fma(x[i], y[i], s);
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[c] = sh[0];
}

void coldot(tlr_ctx* ctx, int64_t n, int ncols, const double* X, int64_t ldx, const double* Y, int64_t ldy,
            double* out) {
  if (ncols <= 0) return;
  TLR_SITE_PRE(ctx);
  k_coldot<<<(unsigned)ncols, 256, 0, ctx->stream>>>(n, X, ldx, Y, ldy, out);
  TLR_LAUNCH_CHECK(ctx);
}

// Active columns c (active[c] != 0): x += a p, r -= a q with a = num[c] / den[c].
__global__ void k_pcg_xr(int64_t n, const double* __restrict__ num, const double* __restrict__ den,
                         const int* __restrict__ active, double* __restrict__ x, int64_t ldx,
                         const double* __restrict__ p, double* __restrict__ r, const double* __restrict__ q,
                         int64_t ld) {
  const int c = blockIdx.y;
  if (!active[c]) return;
  const double a = num[c] / den[c];
  const size_t o = (size_t)c * ld;
  double* xc = x + (size_t)c * ldx;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    xc[i] = fma(a, p[o + i], xc[i]);
    r[o + i] = fma(-a, q[o + i], r[o + i]);
  }
}

// Active columns: p = z + b p with b = num[c] / den[c].
__global__ void k_pcg_p(int64_t n, const double* __restrict__ num, const double* __restrict__ den,
                        const int* __restrict__ active, const double* __restrict__ z, double* __restrict__ p,
                        int64_t ld) {
  const int c = blockIdx.y;
  if (!active[c]) return;
  const double bt = num[c] / den[c];
  const size_t o = (size_t)c * ld;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    p[o + i] = fma(bt, p[o + i], z[o + i]);
}

void pcg_update_xr(tlr_ctx* ctx, int64_t n, int ncols, const double* num, const double* den, const int* active,
                   double* x, int64_t ldx, const double* p, double* r, const double* q, int64_t ld) {
  if (ncols <= 0 || n <= 0) return;
  const unsigned gx = (unsigned)std::min<int64_t>((n + 255) / 256, 1024);
  TLR_SITE_PRE(ctx);
  k_pcg_xr<<<dim3(gx, (unsigned)ncols), 256, 0, ctx->stream>>>(n, num, den, active, x, ldx, p, r, q, ld);
  TLR_LAUNCH_CHECK(ctx);
}

void pcg_update_p(tlr_ctx* ctx, int64_t n, int ncols, const double* num, const double* den, const int* active,
                  const double* z, double* p, int64_t ld) {
  if (ncols <= 0 || n <= 0) return;
  const unsigned gx = (unsigned)std::min<int64_t>((n + 255) / 256, 1024);
  TLR_SITE_PRE(ctx);
  k_pcg_p<<<dim3(gx, (unsigned)ncols), 256, 0, ctx->stream>>>(n, num, den, active, z, p, ld);
  TLR_LAUNCH_CHECK(ctx);
}

}  // namespace tlr
