// TLR triangular solves (Algorithm 7 and its transpose), and the vector kernels of preconditioned CG.
//
// One persistent kernel does both solves of a group of right-hand sides, left-looking:
//   forward, k = 0 .. nb-1:   X_k -= Urow_k T_k;  Z_k = L_kk^-1 X_k;  T_ik = V_ik^T Z_k (all i > k)
//   (L D L^T)                 W_k = D_k^-1 Z_k
//   backward, k = nb-1 .. 0:  W_k -= Vcol_k S_k;  X_k = L_kk^-T W_k;  S_kj = U_kj^T X_k (all j < k)
// where T_k (S_k) stacks the T_kj (S_ik) in the order of the block row's (column's) contiguous panel.  That is
// a chain of 6 nb dependent steps of a few microseconds of FP64 work for the whole GPU at N = 131072, and
// less below.  Launched one by one (a captured graph) a step cost 10 us at N = 131072 and 4 us at N = 4096.
// Here the CTAs stay resident (cooperative launch, one per SM), and the steps are joined by the data alone: every
// vector entry is written once per solve, into memory that first holds a NaN that stands for "not yet", and a CTA that
// stages its step's vector reads the entries until they are there.  No barrier and no fence: an entry is an 8-byte
// access that is whole by itself, and it is on its way to the readers as soon as it is stored.  (A grid barrier per
// step, tried first, cost its fence, an atomic and two more round trips to L2: 336 us at N = 4096, 4.48 ms at 131072.)
// Two kinds of step:
//   rows  y(m) = sum_k A(m, k) x(k): units of 4 to 16 rows, the 8 warps of a CTA sharing k
//   cols  y(c) = sum_k A(k, c) x(k): one warp per column
// A step's first factor entries are copied to shared memory (cp.async) before its wait, and the step after next is
// prefetched into L2: neither depends on the solution.  (Right-looking updates of all remaining tiles took 25 us a
// step: a tile's rank varies from 0 to ten times the mean, and the deepest tile's chain of loads set the pace.  One
// cluster of 16 CTAs for small problems gains 5% at N = 2048, b = 256, one column, and loses from N = 4096 on.)
//
// Right-hand sides go in groups of NR <= 8 columns held in registers, without padding to a tile; the vector a step
// multiplies is staged in shared memory.  Groups do not depend on one another: each has a team of CTAs of its own.
// Bound: the FP64 unit (one DFMA per entry and column) and the steps' latency: a store reaches the readers'
// registers after about 1100 cycles, the sums of a step's last products take 500 to 1000.  Sums run in a fixed order:
// results do not depend on timing.
//
// Measured, graph of launches -> now: 2D N = 131072 (b = 1024, eps = 1e-6), 1 column 7.6 -> 3.9 ms (763 steps of
// 5.1 us; 1.1 ms of FP64 work); N = 4096 (b = 256) 393 -> 225 us; 3D N = 20011 L D L^T, 32 columns 14.7 -> 8.0 ms
// (4.6 ms of FP64 work); preconditioned CG, 2D N = 32768, 12 iterations 51 -> 7.8 ms.
//
// Every wait is bounded: a wait that runs out sets a flag in device and host-visible memory that ends all others, the
// result is overwritten with NaN and the context's next solve reports TLR_ERR_TIMEOUT.
#include <algorithm>
#include <cstring>

#include "internal.h"
#include "warpsum.cuh"

namespace tlr {

namespace {

constexpr int SV_T = 256, SV_W = SV_T / 32;
constexpr int SV_NRHS = 32;        // right-hand sides per launch
constexpr int SV_RB = 16;          // most rows of a unit
constexpr int SV_C = 16, SV_NC = 3;  // factor entries of a thread per chunk, chunks in flight
constexpr int SV_RLD = SV_W + 1;   // padded row of warp partials
constexpr int SV_XS = 14336;       // staged vector entries (112 KB)
constexpr unsigned long long SV_WAIT_NS = 2000000000ull;

// A step.  Rows: y = A x over the n columns of A (b rows; kind 1: column k has rows m >= k); kind 0
// X_k -= y with x = T_k, 1 Z_k = y and W_k = D_k^-1 y, 2 W_k -= y with x = S_k.  Cols: y = A^T x for the n
// columns of A; kind 3 x = Z_k into T, 4 x = W_k (rows m >= c) into X_k, 5 x = X_k into S.
// Every array is written once per solve: X_k and W_k before and after their update are arrays of their own
// (B and X1, W and W1), and so are T and S.
struct __align__(16) SvStep {
  const double* A;
  const int* map;  // kinds 3, 5: row of T or S for each column
  int kind, k, n;
  int t0;          // kinds 0, 2: first row of T_k or S_k; 1, 4: X_k (W_k) has been updated
};
struct SvTab {
  const SvStep* steps;
  const double* dvec;  // L D L^T, else null
  const double* any;   // readable memory
  int nsteps, b;
};
struct SvVec {
  // column-major, ng NR columns: right-hand side, X1, Z, W (Z itself for L L^T), W1, solution (ld np); T, S (ld ldt)
  double *B, *X1, *Z, *W, *W1, *X, *T, *S;
  int64_t np, ldt;
  int ng, xs;              // xs: staged vector entries per column
  unsigned* out;           // a wait ran out, zero at launch
  volatile int* timeout;   // the same, host-visible
};

// "Not written yet": a NaN that is never stored as a value (sv_value).
constexpr unsigned long long SV_EMPTY = 0x7ff85a3c96e10f2dull;
__device__ __forceinline__ double sv_value(double x) {
  return __double_as_longlong(x) == (long long)SV_EMPTY ? __longlong_as_double(0x7ff8000000000000ll) : x;
}
__device__ __forceinline__ bool sv_empty(double x) { return __double_as_longlong(x) == (long long)SV_EMPTY; }
// Entries of the vectors, read and written at L2 by 8-byte accesses that are whole by themselves: no other data
// hangs on an entry, so nothing has to be ordered.
__device__ __forceinline__ double sv_ld(const double* p) {
  double x;
  asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(x) : "l"(p) : "memory");
  return x;
}
__device__ __forceinline__ void sv_st(double* p, double x) {
  asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(sv_value(x)) : "memory");
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
  double* ab = sm + SV_RLD * NR * SV_RB;      // factor entries: chunk, entry, thread
  double* xs = ab + SV_NC * SV_C * SV_T;      // NR x v.xs: the step's vector, column-major
  __shared__ SvStep ring[4];
  const int b = T.b;
  // groups of columns are independent: a team of G CTAs for each
  const int G = (int)gridDim.x / v.ng, team = (int)blockIdx.x / G, bid = (int)blockIdx.x % G;
  if (team >= v.ng) return;
  for (double** p : {&v.B, &v.X1, &v.Z, &v.W, &v.W1, &v.X}) *p += (int64_t)team * NR * v.np;
  v.T += (int64_t)team * NR * v.ldt;
  v.S += (int64_t)team * NR * v.ldt;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // Wait of a thread for entries: again() is called until it returns false (all there) or the wait has run out, here or
  // elsewhere; entries that are still missing are then taken as they are (NaN), and so are all later ones.
  auto wait_for = [&](auto again) {
    unsigned long long t0 = 0;
#pragma unroll 1
    for (unsigned it = 1; again(); ++it) {
      if (it & 31u) continue;
      const unsigned long long t = sv_clock();
      if (!t0) t0 = t;
      if (*(volatile unsigned*)v.out) return;
      if (t - t0 > SV_WAIT_NS || it > (1u << 28)) {
        atomicExch(v.out, 1u);
        *v.timeout = 1;
        return;
      }
    }
  };

  // rows r0 .. r0 + len - 1 of the columns of x (leading dimension ldx) into shared memory, zeros up to a multiple of 64
  auto stage = [&](const double* x, int64_t ldx, int64_t r0, int len) {
    constexpr int SU = NR >= 4 ? 1 : 4 / NR;  // SU NR loads in flight per thread
    const double* p = x + r0;
    const int lp = (len + 63) & ~63;
#pragma unroll 1
    for (int k0 = tid; k0 < lp; k0 += SU * SV_T) {
      double t[SU][NR];
#pragma unroll
      for (int u = 0; u < SU; ++u)
#pragma unroll
        for (int n = 0; n < NR; ++n) t[u][n] = k0 + u * SV_T < len ? sv_ld(p + n * ldx + k0 + u * SV_T) : 0.0;
      wait_for([&]() {
        bool miss = false;
#pragma unroll
        for (int u = 0; u < SU; ++u)
#pragma unroll
          for (int n = 0; n < NR; ++n)
            if (sv_empty(t[u][n])) {
              t[u][n] = sv_ld(p + n * ldx + k0 + u * SV_T);
              miss = true;
            }
        return miss;
      });
      __syncwarp();  // lanes leave the wait at different times
#pragma unroll
      for (int u = 0; u < SU; ++u)
#pragma unroll
        for (int n = 0; n < NR; ++n)
          if (k0 + u * SV_T < lp) xs[n * v.xs + k0 + u * SV_T] = t[u][n];
    }
  };

  // Factor entries travel in chunks of SV_C per thread, each thread copying its own into its slots of a ring of
  // SV_NC chunks (no barrier); a step's first chunks are on their way before the wait for its vector.
  auto put = [&](int buf, int u, const double* p, bool ok) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(ab + (buf * SV_C + u) * SV_T + tid)),
                 "l"(ok ? p : T.any), "r"(ok ? 8 : 0)
                 : "memory");
  };
  auto commit = [&]() { asm volatile("cp.async.commit_group;" ::: "memory"); };
  auto chunk_here = [&]() { asm volatile("cp.async.wait_group %0;" ::"n"(SV_NC - 1) : "memory"); };
  struct Cur {  // next chunk to copy: unit id (the t-th of this CTA) or column id, first index k0
    int t, id, k0;
  };

  // ---- rows steps: unit = RB = 2^rsh rows; units (longest first for a triangle) dealt out
  // forth and back over the CTAs.  Lane (row, sub) of warp w takes k = slot + u 2^lsh, slot = w subs + sub.
  int rsh = 2;
  while (rsh < 4 && ((b + (1 << rsh) - 1) >> rsh) > G) ++rsh;
  const int RB = 1 << rsh, lsh = 8 - rsh, slots = 1 << lsh, slot = (warp << (5 - rsh)) + (lane >> rsh);
  const int nu = (b + RB - 1) >> rsh;
  static_assert(SV_T == 256 && SV_RB == 16, "slots of a unit");
  auto unit_r0 = [&](int id) { return (nu - 1 - id) << rsh; };
  auto unit_len = [&](const SvStep& s, int id) { return s.kind == 1 ? min(b, unit_r0(id) + RB) : s.n; };
  auto unit_at = [&](int t) { return (t & 1) ? (t + 1) * G - 1 - bid : t * G + bid; };  // nu and more: none
  auto rows_copy = [&](const SvStep& s, Cur& c, int buf) {
    if (c.id < nu) {
      const int m = unit_r0(c.id) + (lane & (RB - 1)), len = unit_len(s, c.id);
      const int lim = m < b ? (s.kind == 1 ? min(len, m + 1) : len) : 0;
      const int n = (lim - c.k0 - slot + slots - 1) >> lsh, nc = min(SV_C, (len - c.k0 + slots - 1) >> lsh);
      const double* p = s.A + m + (size_t)(c.k0 + slot) * b;
      const size_t st = (size_t)b << lsh;
#pragma unroll 4
      for (int u = 0; u < nc; ++u, p += st) put(buf, u, p, u < n);
      c.k0 += SV_C << lsh;
      if (c.k0 >= len) {
        c.k0 = 0;
        c.id = unit_at(++c.t);
      }
    }
    commit();
  };
  auto rows_run = [&](const SvStep& s, Cur& next) {
    const double* x = s.kind == 1 ? (s.t0 ? v.X1 : v.B) + (size_t)s.k * b : (s.kind == 0 ? v.T : v.S) + s.t0;
    const int64_t ldx = s.kind == 1 ? v.np : v.ldt;
    int buf = 0;
#pragma unroll 1
    for (int t = 0, id; (id = unit_at(t)) < nu; ++t) {
      const int r0 = unit_r0(id), len = unit_len(s, id);
      // what an output is subtracted from (or scaled by): of this thread's first output already here
      auto at = [&](int o) { return (int64_t)(o >> rsh) * v.np + (size_t)s.k * b + r0 + (o & (RB - 1)); };
      auto is_out = [&](int o) { return (tid & 3) == 0 && r0 + (o & (RB - 1)) < b; };
      auto before = [&](int o) {
        if (s.kind == 1) return T.dvec ? 1.0 / sv_ld(T.dvec + (size_t)s.k * b + r0 + (o & (RB - 1))) : 0.0;
        return sv_ld((s.kind == 0 ? v.B : v.W) + at(o));
      };
      const double old0 = (tid >> 2) < RB * NR && is_out(tid >> 2) ? before(tid >> 2) : 0.0;
      double acc[NR];
#pragma unroll
      for (int n = 0; n < NR; ++n) acc[n] = 0.0;
#pragma unroll 1
      for (int c0 = 0; c0 < len; c0 += v.xs) {  // staged pieces of x, whole chunks
        const int cn = min(v.xs, len - c0);
        if (t > 0 || c0 > 0) __syncthreads();
        stage(x, ldx, c0, cn);
        __syncthreads();
#pragma unroll 1
        for (int k0 = 0; k0 < cn; k0 += SV_C << lsh) {
          chunk_here();
          const int nw = min(SV_C, (cn - k0 - (warp << (5 - rsh)) + slots - 1) >> lsh);  // the warp's most
          const double *xp = xs + k0 + slot, *ap = ab + buf * SV_C * SV_T + tid;
#pragma unroll (NR >= 4 ? 2 : 4)
          for (int u = 0; u < nw; ++u) {
            const double e = ap[u * SV_T];
#pragma unroll
            for (int n = 0; n < NR; ++n) acc[n] = fma(e, xp[n * v.xs + (u << lsh)], acc[n]);
          }
          rows_copy(s, next, buf);
          buf = buf + 1 == SV_NC ? 0 : buf + 1;
        }
      }
#pragma unroll
      for (int n = 0; n < NR; ++n) {
#pragma unroll 1
        for (int o = RB; o < 32; o *= 2) acc[n] += __shfl_xor_sync(0xffffffffu, acc[n], o);
        if (lane < RB) red[((n << rsh) + lane) * SV_RLD + warp] = acc[n];
      }
      __syncthreads();
      // warp partials: four lanes per output, whole warps (the lanes leave the waits below at different times)
#pragma unroll 1
      for (int o0 = warp * 8; o0 < RB * NR; o0 += SV_T / 4) {
        const int o = o0 + (lane >> 2);
        const bool live = o < RB * NR, out = live && is_out(o);
        const double* r = red + (live ? o : 0) * SV_RLD + (tid & 3) * (SV_W / 4);
        double old = old0;
        if (out && o >= SV_T / 4) old = before(o);
        double z = r[0];
#pragma unroll
        for (int w = 1; w < SV_W / 4; ++w) z += r[w];
        z += __shfl_xor_sync(0xffffffffu, z, 1);
        z += __shfl_xor_sync(0xffffffffu, z, 2);
        if (out) {
          if (s.kind == 1) {
            sv_st(v.Z + at(o), z);
            if (T.dvec) sv_st(v.W + at(o), z * old);
          } else {
            if (s.kind == 2)
              wait_for([&]() {
                const bool miss = sv_empty(old);
                if (miss) old = sv_ld(v.W + at(o));
                return miss;
              });
            sv_st((s.kind == 0 ? v.X1 : v.W1) + at(o), old - z);
          }
        }
      }
    }
  };

  // ---- cols steps: one warp per column; consecutive columns go to different CTAs
  const bool cols_staged = b <= v.xs;
  auto cols_first = [&](const SvStep& s, int c) { return s.kind == 4 ? c & ~31 : 0; };
  auto cols_copy = [&](const SvStep& s, Cur& c, int buf) {
    if (c.id < s.n) {
      const double* p = s.A + (size_t)c.id * b + c.k0 + lane;
      const int n = (b - c.k0 - lane + 31) >> 5, nc = min(SV_C, (b - c.k0 + 31) >> 5);
      const int first = s.kind == 4 && c.k0 + lane < c.id;  // above the diagonal
#pragma unroll 4
      for (int u = 0; u < nc; ++u) put(buf, u, p + 32 * u, u < n && u >= first);
      c.k0 += 32 * SV_C;
      if (c.k0 >= b) {
        c.id += SV_W * G;
        c.k0 = cols_first(s, c.id);
      }
    }
    commit();
  };
  auto cols_run = [&](const SvStep& s, Cur& next) {
    constexpr int P = sv_pow2<NR>();
    const double* x = (s.kind == 3 ? v.Z : s.kind == 5 ? v.X : s.t0 ? v.W1 : v.W) + (size_t)s.k * b;
    int buf = 0, c = bid + warp * G, row = s.kind != 4 && c < s.n ? __ldg(s.map + c) : 0;
    if (bid >= s.n) return;  // no column for this CTA
#pragma unroll 1
    for (int k0 = 0; k0 < b; k0 += v.xs) stage(x, v.np, k0, min(v.xs, b - k0));  // too long: waited for in pieces, read from L2
    __syncthreads();
#pragma unroll 1
    while (c < s.n) {
      double acc[P];
#pragma unroll
      for (int n = 0; n < P; ++n) acc[n] = 0.0;
#pragma unroll 1
      for (int k0 = cols_first(s, c); k0 < b; k0 += 32 * SV_C) {
        chunk_here();
        const double* ap = ab + buf * SV_C * SV_T + tid;
        const int nw = min(SV_C, (b - k0 + 31) >> 5);
        if (cols_staged) {
          const double* xp = xs + k0 + lane;
#pragma unroll (NR >= 4 ? 2 : 4)
          for (int u = 0; u < nw; ++u) {
            const double e = ap[u * SV_T];
#pragma unroll
            for (int n = 0; n < NR; ++n) acc[n] = fma(e, xp[n * v.xs + 32 * u], acc[n]);
          }
        } else {
#pragma unroll 1
          for (int u = 0; u < nw; ++u) {
            const double e = ap[u * SV_T];
            const int k = min(k0 + lane + 32 * u, b - 1);  // e is zero past the last
#pragma unroll
            for (int n = 0; n < NR; ++n) acc[n] = fma(e, __ldcg(x + n * v.np + k), acc[n]);
          }
        }
        cols_copy(s, next, buf);
        buf = buf + 1 == SV_NC ? 0 : buf + 1;
      }
      const double y = warp_sums<P>(acc, lane);
      const int n = lane / (32 / P);
      if (lane % (32 / P) == 0 && n < NR) {
        if (s.kind == 4) sv_st(v.X + (int64_t)n * v.np + (size_t)s.k * b + c, y);
        else sv_st((s.kind == 3 ? v.T : v.S) + (int64_t)n * v.ldt + row, y);
      }
      c += SV_W * G;
      if (s.kind != 4 && c < s.n) row = __ldg(s.map + c);
    }
  };

  // the first chunks of a step
  auto load_first = [&](const SvStep& s, Cur& next) {
    next = s.kind < 3 ? Cur{0, unit_at(0), 0} : Cur{0, bid + warp * G, cols_first(s, bid + warp * G)};
#pragma unroll 1
    for (int q = 0; q < SV_NC; ++q) {
      if (s.kind < 3) rows_copy(s, next, q);
      else cols_copy(s, next, q);
    }
  };

  // L2 prefetch of a step's factor data, dealt out over the CTAs (one warp)
  auto prefetch = [&](const SvStep& s) {
    const int bid = (int)blockIdx.x, G = (int)gridDim.x;
    if (s.kind == 1 || s.kind == 4) {
#pragma unroll 1
      for (int c = bid * 32 + lane; c < b; c += G * 32) sv_prefetch(s.A + c + (size_t)c * b, sizeof(double) * (b - c));
    } else {
      constexpr int64_t CH = 1024;  // 8 KB pieces
      const int64_t n = (int64_t)b * s.n;
#pragma unroll 1
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

  Cur next;
  fetch(0);
  fetch(1);
  fetch(2);
  landed();
  __syncthreads();
  load_first(ring[0], next);
  for (int i = 0;;) {
    const SvStep& s = ring[i & 3];
    if (s.kind < 3) rows_run(s, next);
    else cols_run(s, next);
    landed();
    if (++i == T.nsteps) break;
    __syncthreads();  // shared memory is free, the fetched steps are there
    load_first(ring[i & 3], next);
    fetch(i + 2);  // into the slot of step i - 2
    if (warp == SV_W - 1) prefetch(ring[(i + 1) & 3]);
  }
  landed();
}

// gather: V[p, c] = B[perm[p], c] (rows past N and columns past nrhs zero) in the first np cols entries, the rest of
// the vectors empty, the flag cleared; scatter: the reverse, NaN after a wait that ran out
__global__ void k_solve_gather(int64_t N, int64_t np, int nrhs, int cols, int64_t total, const int64_t* __restrict__ perm,
                               const double* __restrict__ B, int64_t ldb, double* __restrict__ V, unsigned* out) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *out = 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    double x = __longlong_as_double((long long)SV_EMPTY);
    if (e < np * cols) {
      const int64_t p = e % np, c = e / np;
      x = p < N && c < nrhs ? sv_value(B[perm[p] + c * ldb]) : 0.0;
    }
    V[e] = x;
  }
}
__global__ void k_solve_scatter(int64_t N, int64_t np, int nrhs, const int64_t* __restrict__ perm,
                                const double* __restrict__ X, double* __restrict__ B, int64_t ldb,
                                const unsigned* __restrict__ out) {
  const bool bad = *out != 0;
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
      st.push_back(SvStep{dk(k), nullptr, 1, k, b, ul > 0});
      if (vl > 0) st.push_back(SvStep{F->Vcol[k], dv2u + sc0[k], 3, k, vl, 0});
    }
    for (int k = nb - 1; k >= 0; --k) {
      const int ul = (int)F->ulen[k], vl = (int)F->vlen[k];
      if (vl > 0) st.push_back(SvStep{F->Vcol[k], nullptr, 2, k, vl, (int)sc0[k]});
      st.push_back(SvStep{dk(k), nullptr, 4, k, b, vl > 0});
      if (ul > 0) st.push_back(SvStep{F->Urow[k], du2v + tr0[k], 5, k, ul, 0});
    }
    P->T = SvTab{reinterpret_cast<const SvStep*>(P->tab + os), F->state == 2 ? F->dvec : nullptr, F->dinv, (int)st.size(), b};
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
static constexpr size_t solve_smem(int xs) {
  return sizeof(double) * ((size_t)SV_RLD * NR * SV_RB + SV_NC * SV_C * SV_T + (size_t)NR * xs);
}

template <int NR>
static void solve_launch(tlr_ctx* ctx, const SolvePlan* P, SvVec v) {
  const int b = P->T.b;
  // whole chunks of a rows step, or all of the vector with zeros to a multiple of 64
  constexpr int most = SV_XS / NR / 1024 * 1024;
  v.xs = (int)std::min<int64_t>(most, (std::max<int64_t>(b, P->len) + 63) / 64 * 64);
  const size_t smem = solve_smem<NR>(v.xs);
  cudaLaunchConfig_t cf{};
  cudaLaunchAttribute at{};
  cf.blockDim = dim3(SV_T);
  cf.dynamicSmemBytes = smem;
  cf.stream = ctx->stream;
  cf.attrs = &at;
  cf.numAttrs = 1;
  auto kern = k_solve<NR>;
  // the limit is the kernel's, for all contexts and threads: always the largest launch's, never this one's
  TLR_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)solve_smem<NR>(most)));
  at.id = cudaLaunchAttributeCooperative;  // the CTAs wait for one another: all resident, or none
  at.val.cooperative = 1;
  cf.gridDim = dim3((unsigned)ctx->sm_count);
  TLR_SITE_PRE(ctx);
  TLR_CUDA(cudaLaunchKernelEx(&cf, kern, P->T, v));
  TLR_LAUNCH_CHECK(ctx);
}

// Right-hand sides go in equal launches of at most 32 columns, each in equal groups of at most 8: launches, the groups of
// a launch of nc columns, and the columns that a group is computed in
static int solve_launches(int nrhs) { return (nrhs + SV_NRHS - 1) / SV_NRHS; }
static int solve_groups(int nc) { return (nc + 7) / 8; }
static int solve_width(int nc) {
  const int w = (nc + solve_groups(nc) - 1) / solve_groups(nc);
  return w <= 4 ? w : w <= 6 ? 6 : 8;
}
static size_t solve_vectors(int64_t np, int64_t ldt, bool ldl) { return (ldl ? 6 : 5) * (size_t)np + 2 * (size_t)ldt; }

size_t solve_doubles(int64_t np, int64_t R, bool ldl, int nrhs) {
  if (nrhs <= 0) return 0;
  const int nc = (nrhs + solve_launches(nrhs) - 1) / solve_launches(nrhs);  // the widest launch
  return solve_vectors(np, std::max<int64_t>(R, 1), ldl) * solve_groups(nc) * solve_width(nc) + 32;
}

bool solve_timeout_flag(tlr_ctx* ctx) {
  volatile int* out = ctx->wait_out;
  if (!*out) return false;
  *out = 0;
  return true;
}

void tlr_solve_factor(tlr_ctx* ctx, tlr_mat* F, int nrhs, double* B, int64_t ldb) {
  TLR_REQUIRE(!solve_timeout_flag(ctx), TLR_ERR_TIMEOUT, "solve: a bounded device wait of an earlier solve ran out");
  if (!F->plan) F->plan = plan_build(ctx, F);
  SolvePlan* P = F->plan;
  const int ng32 = solve_launches(nrhs);
  for (int h = 0; h < ng32; ++h) {
    const int c0 = (int)((int64_t)nrhs * h / ng32), nc = (int)((int64_t)nrhs * (h + 1) / ng32) - c0;
    const int ng = solve_groups(nc), nr = solve_width(nc), cols = ng * nr;
    const size_t one = solve_vectors(P->np, P->ldt, P->T.dvec != nullptr);
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
    v.out = reinterpret_cast<unsigned*>(P->vec);
    const size_t npc = (size_t)P->np * cols;
    v.B = P->vec + 32;
    v.X1 = v.B + npc;
    v.Z = v.X1 + npc;
    v.W1 = v.Z + npc;
    v.X = v.W1 + npc;
    v.T = v.X + npc;
    v.S = v.T + (size_t)P->ldt * cols;
    v.W = P->T.dvec ? v.S + (size_t)P->ldt * cols : v.Z;
    v.timeout = ctx->wait_out;
    double* Bc = B + (size_t)c0 * ldb;
    TLR_SITE_PRE(ctx);
    k_solve_gather<<<sv_blocks(one * cols), 256, 0, ctx->stream>>>(F->N, P->np, nc, cols, (int64_t)(one * cols), F->dperm, Bc,
                                                                  ldb, v.B, v.out);
    TLR_LAUNCH_CHECK(ctx);
    if (nr == 1) solve_launch<1>(ctx, P, v);
    else if (nr == 2) solve_launch<2>(ctx, P, v);
    else if (nr == 3) solve_launch<3>(ctx, P, v);
    else if (nr == 4) solve_launch<4>(ctx, P, v);
    else if (nr == 6) solve_launch<6>(ctx, P, v);
    else solve_launch<8>(ctx, P, v);
    TLR_SITE_PRE(ctx);
    k_solve_scatter<<<sv_blocks(F->N * nc), 256, 0, ctx->stream>>>(F->N, P->np, nc, F->dperm, v.X, Bc, ldb, v.out);
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

// The word that a solve's bounded waits set, for tests that set it from the host (not part of the C API).
extern "C" int* tlr_solve_wait_word(tlr_ctx* ctx) { return ctx->wait_out; }
