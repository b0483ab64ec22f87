// Products with a whole TLR matrix or factor: Y = A X, L X, L^T X and L (D) L^T X (Section 4.4).
//
// A product with U_ij V_ij^T is two skinny contractions: T_ij = V_ij^T X_j, then Y_i += U_ij T_ij (and
// for the symmetric half S_ij = U_ij^T X_i, Y_j += V_ij S_ij).  No tile's first half depends on another
// tile's second half, so a whole product is two launches, whatever the number of tiles:
//   k_apply_tn  every column of every V panel (and U panel, and for L^T every column of every diagonal
//               tile) times its block of X: T and S for all tiles, one warp per four columns;
//   k_apply_nn  every row block of Y: [D_i | Urow_i | Vcol_i] [X_i; T_i; S_i] as one long contraction
//               over the block row's contiguous panels, one CTA per 64 rows, its eight warps sharing the
//               contraction index; where the matrix has too few row blocks for the GPU, a cluster of up
//               to eight CTAs shares it and adds its parts through distributed shared memory.
// T_ij is written at U_ij's place in block row i's coefficient vector and S_ij at V_ij's place in block
// column j's, found by a search in the panel's offset table.
//
// Bound: the FP64 unit (2 DFMA per clock and SM, 0.63 T/s): one DFMA per 8-byte entry and right-hand
// side is 5.0 TB/s of factor entries at one column, below HBM's 6.8, so the number of DFMAs is what
// counts: right-hand sides are not padded to a tile (up to 8 columns per pass, 1, 2, 3, 4, 6 or 8
// accumulator columns), the warp sums are halving exchanges (about one addition per output instead of
// five), and every load is 16 bytes per lane.  Four GEMM launches per block column with 32 x 16 output
// tiles, which this replaces, did 16 columns' work for one and left the GPU nearly empty in each launch.
// Measured before -> now: A X, 2D, eps = 1e-6, N = 4096 (b = 256), 1 column 952 -> 60 us; N = 131072
// (b = 1024), 8 columns 25.2 -> 9.15 ms (0.94 of the DFMA rate); L D L^T X, 3D N = 20011, b = 512,
// eps = 1e-4, 1 column 6.50 -> 0.32 ms.  Several columns of a large matrix go to the tensor cores (below): the
// 8 columns of N = 131072 9.15 -> 2.26 ms.
//
// Sums run in a fixed order: results do not depend on timing.
#include <cooperative_groups.h>

#include <cstring>

#include "internal.h"
#include "tcdigits.cuh"
#include "warpsum.cuh"

namespace cg = cooperative_groups;

namespace tlr {

namespace {

constexpr int AP_T = 256, AP_W = AP_T / 32;
constexpr int AP_CW = 4;  // panel columns per warp in k_apply_tn

struct ApPanel {  // columns of one panel: kind 0 V panel (-> T), 1 U panel (-> S), 2 diagonal tile (-> YD)
  const double* A;
  int ncols, blk, kind, cta0;
};
struct ApRow {  // block row i: D_i, its U panel and its V panel, with the rows of T and S they multiply
  const double *D, *U, *V;
  int64_t tr0, sc0;
  int ulen, vlen;
};
struct ApTab {
  const ApPanel* pan;
  const ApRow* row;
  const int* voff;  // [j (nb + 1) + i]: first column of tile i in V panel j
  const int* uoff;  // [i (nb + 1) + j]: first column of tile j in U panel i
  int npan, nb, b, unit;
  int64_t N;
  // if set: the kernel (of FP64 products) runs only if *gate is not zero, and those CTAs (of k_apply_tn, row blocks of
  // k_apply_nn) whose entry of redo is not
  const int *gate, *redo;
};

// coefficient vectors are row-major with this many doubles per row (16-byte rows past one column)
template <int NR>
__host__ __device__ constexpr int ap_ld() { return NR == 1 ? 1 : (NR + 1) & ~1; }

template <int NR>
__device__ __forceinline__ void ap_row(const double* p, double (&x)[NR]) {
  if constexpr (NR == 1) {
    x[0] = __ldg(p);
  } else {
#pragma unroll
    for (int n = 0; n < NR; n += 2) {
      const double2 v = __ldg(reinterpret_cast<const double2*>(p + n));
      x[n] = v.x;
      if (n + 1 < NR) x[n + 1] = v.y;
    }
  }
}

template <int VEC>
__device__ __forceinline__ void ap_ld_a(const double* p, double (&a)[VEC]) {
  if constexpr (VEC == 2) {
    const double2 v = __ldg(reinterpret_cast<const double2*>(p));
    a[0] = v.x;
    a[1] = v.y;
  } else {
    a[0] = __ldg(p);
  }
}

// X (original order) -> Xp (KD order, padded with zeros, row-major)
__global__ void k_apply_gather(int64_t N, int64_t np, int nr, int ld, const int64_t* __restrict__ perm,
                               const double* __restrict__ X, int64_t ldx, double* __restrict__ Xp, int* flags,
                               int64_t nflags) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nflags; e += (int64_t)gridDim.x * blockDim.x) flags[e] = 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < np * ld; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = e / ld;
    const int c = (int)(e % ld);
    Xp[e] = p < N && c < nr ? X[perm[p] + (int64_t)c * ldx] : 0.0;
  }
}

// the panel of CTA c of a list
__device__ __forceinline__ int ap_panel(const ApTab& T, int c) {
  int lo = 0, hi = T.npan - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (T.pan[mid].cta0 <= c) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

template <int NR, int VEC>
__global__ void __launch_bounds__(AP_T) k_apply_tn(ApTab T, const double* __restrict__ X, double* __restrict__ TR,
                                                   double* __restrict__ SC, double* __restrict__ YD) {
  constexpr int LD = ap_ld<NR>(), UN = NR <= 4 ? 2 : 1, STEP = 32 * VEC;
  constexpr int P = AP_CW * (NR == 3 ? 4 : NR == 6 ? 8 : NR), LANES = 32 / P;  // lanes that share a sum
  __shared__ int panel;
  if (T.gate && *T.gate == 0 && T.redo[blockIdx.x] == 0) return;
  if (threadIdx.x == 0) panel = ap_panel(T, (int)blockIdx.x);
  __syncthreads();
  const ApPanel pn = T.pan[panel];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, b = T.b;
  const int c0 = (((int)blockIdx.x - pn.cta0) * AP_W + warp) * AP_CW;
  if (c0 >= pn.ncols) return;
  const int nc = min(AP_CW, pn.ncols - c0);
  // output of this lane: column c0 + oc, right-hand side on, at row `dst` of the coefficient vector
  const int ov = lane / LANES, oc = ov / (P / AP_CW), on = ov % (P / AP_CW);
  const bool out = lane % LANES == 0 && oc < nc && on < NR;
  double* O = nullptr;
  if (out) {
    const int c = c0 + oc, j = pn.blk;
    int64_t dst;
    if (pn.kind == 2) {
      O = YD;
      dst = (int64_t)j * b + c;
    } else {
      // tile t of the panel with off[t] <= c < off[t + 1] (tiles of rank 0 are empty ranges)
      const int* off = (pn.kind == 0 ? T.voff : T.uoff) + (size_t)j * (T.nb + 1);
      int lo = 0, hi = T.nb - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= c) lo = mid;
        else hi = mid - 1;
      }
      const int a = c - off[lo];
      if (pn.kind == 0) {
        O = TR;
        dst = T.row[lo].tr0 + T.uoff[(size_t)lo * (T.nb + 1) + j] + a;
      } else {
        O = SC;
        dst = T.row[lo].sc0 + T.voff[(size_t)lo * (T.nb + 1) + j] + a;
      }
    }
    O += dst * LD + on;
  }
  const double* A = pn.A + (size_t)c0 * b;
  const double* x = X + (size_t)pn.blk * b * LD;
  const bool tri = pn.kind == 2;
  double acc[AP_CW][NR];
#pragma unroll
  for (int c = 0; c < AP_CW; ++c)
#pragma unroll
    for (int n = 0; n < NR; ++n) acc[c][n] = 0.0;
  for (int k0 = (tri ? c0 / STEP * STEP : 0) + lane * VEC; k0 < b; k0 += STEP * UN) {
    double a[UN][AP_CW][VEC];
#pragma unroll
    for (int u = 0; u < UN; ++u)
#pragma unroll
      for (int c = 0; c < AP_CW; ++c) {
        const int k = k0 + u * STEP;
        if (k < b && c < nc) {
          ap_ld_a<VEC>(A + (size_t)c * b + k, a[u][c]);
        } else {
#pragma unroll
          for (int e = 0; e < VEC; ++e) a[u][c][e] = 0.0;
        }
      }
    if (tri) {  // lower triangle of the tile, unit diagonal for L D L^T
#pragma unroll
      for (int u = 0; u < UN; ++u)
#pragma unroll
        for (int c = 0; c < AP_CW; ++c)
#pragma unroll
          for (int e = 0; e < VEC; ++e) {
            const int k = k0 + u * STEP + e;
            if (k < c0 + c) a[u][c][e] = 0.0;
            else if (k == c0 + c && T.unit) a[u][c][e] = 1.0;
          }
    }
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      const int k = k0 + u * STEP;
      if (k >= b) break;
#pragma unroll
      for (int e = 0; e < VEC; ++e) {
        double xv[NR];
        ap_row<NR>(x + (size_t)(k + e) * LD, xv);
#pragma unroll
        for (int c = 0; c < AP_CW; ++c)
#pragma unroll
          for (int n = 0; n < NR; ++n) acc[c][n] = fma(a[u][c][e], xv[n], acc[c][n]);
      }
    }
  }
  double v[P];
#pragma unroll
  for (int i = 0; i < P; ++i) v[i] = i % (P / AP_CW) < NR ? acc[i / (P / AP_CW)][(i % (P / AP_CW)) % NR] : 0.0;
  const double s = warp_sums<P>(v, lane);
  if (out) *O = s;
}

struct ApOut {
  const double* add;    // added to every row (the diagonal tiles' part of L^T X), or null
  const double* scale;  // rows scaled by this (D of L D L^T), or null
  double* Z;            // KD order, row-major, or:
  double* Y;            // original order, column-major, through perm
  const int64_t* perm;
  int64_t ldy, N;
  int nr;  // columns of Y
};

// dmode: 0 no diagonal tiles, 1 full tiles, 2 lower triangles (unit diagonal for L D L^T)
template <int NR, int VEC>
__global__ void __launch_bounds__(AP_T) k_apply_nn(ApTab T, int dmode, int use_u, int use_v, int S,
                                                   const double* __restrict__ X, const double* __restrict__ TR,
                                                   const double* __restrict__ SC, ApOut out) {
  constexpr int LD = ap_ld<NR>(), RB = 32 * VEC, UN = 4;
  __shared__ double red[AP_W * NR * RB];
  __shared__ double part[NR * RB];
  const int b = T.b, rbs = (b + RB - 1) / RB;
  const int rank = (int)blockIdx.x % S, rb = (int)blockIdx.x / S;
  if (T.gate && *T.gate == 0 && T.redo[rb] == 0) return;  // the whole cluster
  const int i = rb / rbs, r0 = (rb % rbs) * RB;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r = r0 + lane * VEC;
  const ApRow row = T.row[i];
  const bool ok = r < b;
  double acc[VEC][NR];
#pragma unroll
  for (int e = 0; e < VEC; ++e)
#pragma unroll
    for (int n = 0; n < NR; ++n) acc[e][n] = 0.0;
  // the contraction index runs over the three segments; this CTA takes [s0, s1), warp w every eighth
  const int l0 = dmode == 0 ? 0 : dmode == 1 ? b : min(b, r0 + RB), l1 = use_u ? row.ulen : 0, l2 = use_v ? row.vlen : 0;
  const int64_t K = (int64_t)l0 + l1 + l2;
  const int64_t s0 = K * rank / S, s1 = K * (rank + 1) / S;
  auto segment = [&](const double* A, int64_t base, int len, const double* coef, bool tri) {
    const int k1 = (int)min((int64_t)len, s1 - base);
    int k = (int)max((int64_t)0, s0 - base) + warp;
    for (; k < k1; k += AP_W * UN) {
      double a[UN][VEC];
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const int ku = k + u * AP_W;
        if (ok && ku < k1) {
          ap_ld_a<VEC>(A + r + (size_t)ku * b, a[u]);
        } else {
#pragma unroll
          for (int e = 0; e < VEC; ++e) a[u][e] = 0.0;
        }
        if (tri && ku < k1) {
#pragma unroll
          for (int e = 0; e < VEC; ++e) {
            if (r + e < ku) a[u][e] = 0.0;
            else if (r + e == ku && T.unit) a[u][e] = 1.0;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const int ku = k + u * AP_W;
        if (ku >= k1) break;
        double xv[NR];
        ap_row<NR>(coef + (size_t)ku * LD, xv);
#pragma unroll
        for (int e = 0; e < VEC; ++e)
#pragma unroll
          for (int n = 0; n < NR; ++n) acc[e][n] = fma(a[u][e], xv[n], acc[e][n]);
      }
    }
  };
  if (l0) segment(row.D, 0, l0, X + (size_t)i * b * LD, dmode == 2);
  if (l1) segment(row.U, l0, l1, TR + row.tr0 * LD, false);
  if (l2) segment(row.V, (int64_t)l0 + l1, l2, SC + row.sc0 * LD, false);
#pragma unroll
  for (int n = 0; n < NR; ++n)
#pragma unroll
    for (int e = 0; e < VEC; ++e) red[(warp * NR + n) * RB + lane * VEC + e] = acc[e][n];
  __syncthreads();
  auto store = [&](int o, double v) {
    const int m = r0 + o % RB, n = o / RB;
    if (m >= b || (!out.Z && n >= out.nr)) return;
    const int64_t g = (int64_t)i * b + m;
    if (out.add) v += out.add[g * LD + n];
    if (out.scale) v *= out.scale[g];
    if (out.Z) out.Z[g * LD + n] = v;
    else if (g < out.N) out.Y[out.perm[g] + n * out.ldy] = v;
  };
  for (int o = threadIdx.x; o < NR * RB; o += AP_T) {
    double v = red[o];
#pragma unroll
    for (int w = 1; w < AP_W; ++w) v += red[w * NR * RB + o];
    if (S == 1) store(o, v);
    else part[o] = v;
  }
  if (S == 1) return;
  cg::cluster_group cl = cg::this_cluster();
  cl.sync();
  // the cluster's parts in rank order; each CTA finishes its share of the outputs
  for (int o = rank * AP_T + threadIdx.x; o < NR * RB; o += S * AP_T) {
    double v = 0.0;
    for (int q = 0; q < S; ++q) v += cl.map_shared_rank(part, q)[o];
    store(o, v);
  }
  cl.sync();  // no CTA leaves while its part is still read
}

// ------------------------------------------------------------------ several columns: tensor cores
// With two or more right-hand sides the DFMAs (one per entry and column, 2 per clock and SM) take several times
// HBM's time.  The same contractions then run as exact integer products on the 16-bit tensor cores
// (mma.sync.m16n8k16, FP16 in, FP32 accumulate: the eight columns are its N, and a fragment's FP64 entries
// are split in the registers that loaded them, so that the factor is read as it lies; tcgen05 wants its
// operands in shared or tensor memory and 128 rows, which a panel of a few columns does not fill).  The
// splitting is that of tcdigits.cuh, seven digits below a bound 2^e of the operand's column: a panel column's own
// bound for the factor, the block's for each right-hand side.  Pairs with i + j <= 9 are kept (34 products a step;
// the dropped ones are 2^-66 of the bounds); a group of equal i + j sums below 13 2^14 4 16 < 2^24 over four steps,
// exact in FP32, and moves to 64-bit integers then; one rounding at the end.
// Where the contraction index is the panel's column (Y_i += U_ij T_ij), the column's bound 2^e moves to the
// coefficient: (A(m, k) 2^-e_k) (2^e_k T(k)).
// Error: 2^-58 of the bounds per entry and factor, whatever the size of a result's own terms, where FP64 has 2^-53 of
// the running sum per term.  So the sum of the terms' sizes is estimated too (one product more a step, of the leading
// digits), and where it is small against the bounds (tcdigits.cuh; the first rows of a triangle, the far rows of a unit
// vector's product, right-hand sides with small entries beside large ones) the FP64 kernel that follows each
// contraction computes the 32 columns or 64 rows that the result is among, decided on the device.  Of A X, L X, L^T X
// and L (D) L^T X in 2D and 3D, N = 6000 and 8192, normal, positive and smooth right-hand sides, unit vectors and values
// over eight decades, against extended precision: in norm 0.2 to 1.0 of the DFMA kernels' error; row by row, over
// u |A| |X|, the mean square at most theirs and the largest at most 1.15 of it.  (Truncating F instead of rounding, two
// instructions less, would make it up to twice theirs.)
// Bound: the integer instructions that split (about 18 per entry, at half rate; the ALU is busy 57 % of the
// time, the tensor pipe 32 %, 16 warps per SM at 128 registers).  35 products of 16 x 8 x 16 per 256 entries.
// Latency: each lane copies its own fragments of the next steps into shared memory (cp.async, no barrier).
// The estimates and what follows from them cost 3 % of A X (N = 131072, 8 columns 2.19 -> 2.26 ms).
constexpr int TC_KS = 16;    // k per step
constexpr int TC_STG = 3;    // steps in flight per warp
constexpr int TC_SPC = 8;    // CTAs (a cluster) per block in k_apply_split
constexpr int TC_FRAG = 64;  // uint4 per step of a split right-hand side: [2][lane], tc_digits' words, the sign on top
constexpr int TC_ZERO = -100000;  // exponent of a column of zeros
constexpr int TC_W = 4, TC_T = 32 * TC_W;  // warps of k_apply_tn_tc and k_apply_nn_tc
constexpr int TC_SMEM = TC_W * TC_STG * 32 * (64 + 32 + 16);

__device__ __forceinline__ void tc_mma(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// One step (CHECK: notes entries outside their bounds): the tile's fragments x[row half][k half][2] (rows g, g + 8;
// k 2t, 2t + 1, 2t + 8, 2t + 9 of the lane g = lane / 4, t = lane % 4) with shifts e, times the split right-hand side's
// step (column g; the same k)
template <bool CHECK>
__device__ __forceinline__ void tc_step(const double (&x)[2][2][2], const int (&e)[2][2][2], uint4 f0, uint4 f1, TcAcc& acc) {
  int bad = 0;
  unsigned d[2][2][TC_P], b0[TC_P], b1[TC_P];
  tc_pairs(make_uint2(f0.x, f0.y & 0x7fffffffu), make_uint2(f0.z, f0.w & 0x7fffffffu), f0.y, f0.w, b0);
  tc_pairs(make_uint2(f1.x, f1.y & 0x7fffffffu), make_uint2(f1.z, f1.w & 0x7fffffffu), f1.y, f1.w, b1);
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      tc_pairs(tc_digits(x[r][h][0], e[r][h][0], bad), tc_digits(x[r][h][1], e[r][h][1], bad),
               (unsigned)__double2hiint(x[r][h][0]), (unsigned)__double2hiint(x[r][h][1]), d[r][h]);
#pragma unroll
  for (int i = 0; i < TC_P; ++i) {
    const unsigned a[4] = {d[0][0][i], d[1][0][i], d[0][1][i], d[1][1][i]};
#pragma unroll
    for (int j = 0; j < TC_P; ++j)
      if (i + j <= 7) tc_mma(acc.f[i + j], a, b0[j], b1[j]);
  }
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f16.f16.f16.f16 {%0,%1}, {%2,%3,%4,%5}, {%6,%7}, {%0,%1};"
               : "+r"(acc.est[0]), "+r"(acc.est[1])
               : "r"(tc_abs2(d[0][0][0])), "r"(tc_abs2(d[1][0][0])), "r"(tc_abs2(d[0][1][0])), "r"(tc_abs2(d[1][1][0])),
                 "r"(tc_abs2s(b0[0])), "r"(tc_abs2s(b1[0])));
  if (CHECK) acc.bad |= bad;
  if (++acc.win == TC_WIN) tc_drain(acc);
}
// The warps' totals through shared memory: thread `threadIdx.x` < 128 gets entry (lane / 4 + 8 (c / 2), 2 (lane % 4) + c % 2)
// of the fragment, lane = threadIdx.x / 4, c = threadIdx.x % 4
// (est: the same of the estimates)
__device__ __forceinline__ void tc_total(TcAcc& acc, long long* part, long long& h, long long& l, float& est) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* pest = reinterpret_cast<float*>(part + TC_W * 32 * 8);
  static_assert(TC_W * 32 * (8 * sizeof(long long) + 4 * sizeof(float)) <= TC_SMEM, "the totals fit the buffers");
  tc_drain(acc);
  __syncthreads();  // the copies' buffers are free
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    part[(warp * 32 + lane) * 8 + c] = acc.hi[c];
    part[(warp * 32 + lane) * 8 + 4 + c] = acc.lo[c];
    pest[(warp * 32 + lane) * 4 + c] = tc_half(acc.est[c >> 1], c & 1);
  }
  __syncthreads();
  h = l = 0;
  est = 0.f;
  if (threadIdx.x >= TC_T) return;
#pragma unroll
  for (int w = 0; w < TC_W; ++w) {
    h += part[(w * 32 + (threadIdx.x >> 2)) * 8 + (threadIdx.x & 3)];
    l += part[(w * 32 + (threadIdx.x >> 2)) * 8 + 4 + (threadIdx.x & 3)];
    est += pest[(w * 32 + (threadIdx.x >> 2)) * 4 + (threadIdx.x & 3)];
  }
}
// copies of a lane's own bytes to shared memory, zeros if !ok (src must be readable memory all the same)
__device__ __forceinline__ void tc_cp16(void* dst, const void* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(ok ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void tc_cp8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
struct TcLane {  // a lane's slots of a warp's ring
  char* base;
  __device__ __forceinline__ TcLane(char* smem) : base(smem + (threadIdx.x >> 5) * (TC_STG * 32 * 112)) {}
  __device__ __forceinline__ double2* x(int st, int q) const {
    return reinterpret_cast<double2*>(base + st * 32 * 112) + q * 32 + (threadIdx.x & 31);
  }
  __device__ __forceinline__ uint4* f(int st, int q) const {
    return reinterpret_cast<uint4*>(base + st * 32 * 112 + 2048) + q * 32 + (threadIdx.x & 31);
  }
  __device__ __forceinline__ int2* e(int st, int q) const {
    return reinterpret_cast<int2*>(base + st * 32 * 112 + 3072) + q * 32 + (threadIdx.x & 31);
  }
};
// steps first, first + TC_W, ... < end of a warp: issue(step, stage) copies, use(step, stage) computes
template <class I>
__device__ __forceinline__ void tc_ring_begin(int first, int end, I issue) {
#pragma unroll
  for (int q = 0; q < TC_STG - 1; ++q) {
    if (first + q * TC_W < end) issue(first + q * TC_W, q);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
}
template <class I, class C>
__device__ __forceinline__ void tc_ring(int first, int end, I issue, C use) {
  int next = first + (TC_STG - 1) * TC_W, st = 0, sn = TC_STG - 1;
  for (int s = first; s < end; s += TC_W) {
    asm volatile("cp.async.wait_group %0;" ::"n"(TC_STG - 2) : "memory");
    if (next < end) issue(next, sn);
    next += TC_W;
    asm volatile("cp.async.commit_group;" ::: "memory");
    use(s, st);
    st = st + 1 == TC_STG ? 0 : st + 1;
    sn = sn + 1 == TC_STG ? 0 : sn + 1;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

struct TcSeg {  // a split right-hand side: a block's rows in up to three segments, each padded to whole steps
  int64_t ks0;  // first step
  int n0, n1, n2;
};

// Splits the right-hand sides of block blockIdx.x / TC_SPC: rows of X (SEG = 1: the block's b rows), or
// [X_i; T_i; S_i] scaled by the panels' column bounds (SEG = 3; the bounds' shifts, by step, to ek).
// Fragments to frag, the columns' exponents to ef.  A cluster per block finds the bounds together.
// SEG = 3: a coefficient whose row is below 4^-d of the columns' bounds goes up by 2^d and its panel column down, so that
// their roundings, 2^-58 of the bounds each, weigh the same in a product: a term's error falls with the root of its size
// (T and S fall off by orders of magnitude).  least: what an estimate has to
// reach (tcdigits.cuh), with the bounds themselves for the entries, 4 tc_least(sum 4^-d).
template <int SEG>
__global__ void __cluster_dims__(TC_SPC, 1, 1) __launch_bounds__(256)
    k_apply_split(const TcSeg* __restrict__ segs, const ApRow* __restrict__ rows, int b, const double* __restrict__ X,
                  const double* __restrict__ TR, const double* __restrict__ SC, const int* __restrict__ eD,
                  const int* __restrict__ eU, const int* __restrict__ eV, uint4* __restrict__ frag, int* __restrict__ ek_out,
                  int* __restrict__ ef, float* __restrict__ least, int* bad_out) {
  cg::cluster_group cl = cg::this_cluster();
  const int i = blockIdx.x / TC_SPC, rank = blockIdx.x % TC_SPC, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const TcSeg sg = segs[i];
  const int s0 = (sg.n0 + TC_KS - 1) / TC_KS, s1 = SEG > 1 ? (sg.n1 + TC_KS - 1) / TC_KS : 0,
            s2 = SEG > 1 ? (sg.n2 + TC_KS - 1) / TC_KS : 0, steps = s0 + s1 + s2;
  __shared__ int part[8], emax[8];
  __shared__ float wsum[SEG > 1 ? 8 : 1];
  if (tid < 8) part[tid] = TC_ZERO;
  __syncthreads();
  // row k of step s: its coefficients and the exponent of its panel column
  auto entry = [&](int s, int k, int& ek) -> const double* {
    ek = SEG > 1 ? 1 : 0;
    if (s < s0) {
      k += s * TC_KS;
      if (k >= sg.n0) return nullptr;
      if (SEG > 1) ek = eD[(int64_t)i * b + k];
      return X + ((int64_t)i * b + k) * 8;
    }
    if (s < s0 + s1) {
      k += (s - s0) * TC_KS;
      if (k >= sg.n1) return nullptr;
      ek = eU[rows[i].tr0 + k];
      return TR + (rows[i].tr0 + k) * 8;
    }
    k += (s - s0 - s1) * TC_KS;
    if (k >= sg.n2) return nullptr;
    ek = eV[rows[i].sc0 + k];
    return SC + (rows[i].sc0 + k) * 8;
  };
  int m = TC_ZERO;  // of column tid % 8
  for (int o = rank * 256 + tid; o < steps * 128; o += TC_SPC * 256) {
    int ek;
    const double* p = entry(o >> 7, (o >> 3) & 15, ek);
    const unsigned hw = p ? (unsigned)__double2hiint(p[o & 7]) & 0x7fffffffu : 0u;
    if (hw) m = max(m, tc_exp(hw) + ek);
  }
  atomicMax(&part[tid & 7], m);
  cl.sync();
  if (tid < 8) {
    int v = TC_ZERO;
#pragma unroll
    for (int q = 0; q < TC_SPC; ++q) v = max(v, cl.map_shared_rank(part, q)[tid]);
    if (rank == 0) ef[i * 8 + tid] = v;  // TC_ZERO for a column of zeros
    if (v == TC_ZERO) v = 1;
    else if (tc_odd(v)) *bad_out = 1;
    emax[tid] = v;
  }
  cl.sync();
  const int n = lane >> 2, t = lane & 3, en = emax[n];
  float w = 0.f;
  for (int s = rank * 8 + warp; s < steps; s += TC_SPC * 8) {
    uint2 q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      int ek;
      const int k = 2 * t + (u & 1) + (u >> 1) * 8;
      const double* p = entry(s, k, ek);
      const double x = p ? p[n] : 0.0;
      if constexpr (SEG > 1) {
        int g = x == 0.0 ? -48 : max(-48, tc_exp((unsigned)__double2hiint(x) & 0x7fffffffu) + ek - en);
#pragma unroll
        for (int o = 4; o < 32; o *= 2) g = max(g, __shfl_xor_sync(0xffffffffu, g, o));
        const int d = max(0, -g / 2);
        ek += d;
        if (n == 0) {
          ek_out[(sg.ks0 + s) * TC_KS + k] = tc_shift(ek);
          if (p) w += exp2f(-2.f * (float)d);
        }
      }
      const int e = x == 0.0 ? 1 : en - ek;
      if (tc_odd(e)) *bad_out = 1;
      int bad = 0;  // |x| < 2^e by its making
      q[u] = tc_digits(x, tc_shift(e), bad);
      q[u].y |= (unsigned)__double2hiint(x) & 0x80000000u;
    }
    uint4* out = frag + (sg.ks0 + s) * TC_FRAG + lane;
    out[0] = make_uint4(q[0].x, q[0].y, q[1].x, q[1].y);
    out[32] = make_uint4(q[2].x, q[2].y, q[3].x, q[3].y);
  }
  if constexpr (SEG > 1) {
    for (int o = 16; o; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
    if (lane == 0) wsum[warp] = w;
    cl.sync();
    if (rank == 0 && tid == 0) {
      float v = 0.f;
      for (int q = 0; q < TC_SPC; ++q)
        for (int u = 0; u < 8; ++u) v += cl.map_shared_rank(wsum, q)[u];
      least[i] = 4.f * tc_least(v);
    }
    cl.sync();  // no CTA leaves while its sums are still read
  }
}

// place of a panel column's exponent
__device__ __forceinline__ int* tc_expof(const ApTab& T, const ApPanel& pn, int c, int* eU, int* eV, int* eD) {
  return pn.kind == 0 ? eV + T.row[pn.blk].sc0 + c : pn.kind == 1 ? eU + T.row[pn.blk].tr0 + c : eD + (int64_t)pn.blk * T.b + c;
}

// the last q in [0, n) with at(q) <= c (at(0) <= c, at monotone), by a whole warp, 32 places at a time
template <class F>
__device__ __forceinline__ int tc_search(int c, int n, F at) {
  const int lane = threadIdx.x & 31;
  int lo = 0;
  while (n > 1) {
    const int step = (n + 31) / 32, q = lane * step;
    const unsigned m = __ballot_sync(0xffffffffu, q < n && at(lo + q) <= c);
    const int k = 31 - __clz(m);
    lo += k * step;
    n = min(step, n - k * step);
  }
  return lo;
}

// k_apply_tn on the tensor cores: 16 columns of a panel per CTA, its warps sharing the b rows.  The columns'
// bounds are found first (the second pass over the 16 columns comes from the caches) and kept for k_apply_nn_tc.
__global__ void __launch_bounds__(TC_T, 4) k_apply_tn_tc(ApTab T, const TcSeg* __restrict__ segs, const uint4* __restrict__ frag,
                                                         const int* __restrict__ ef, double* __restrict__ TR,
                                                         double* __restrict__ SC, double* __restrict__ YD,
                                                         int* __restrict__ eU, int* __restrict__ eV, int* __restrict__ eD,
                                                         float least, int* bad_out, int* __restrict__ redo) {
  extern __shared__ __align__(16) char tc_smem[];
  __shared__ int64_t dst[16];  // row of a column's coefficients
  __shared__ unsigned cmax[TC_W][16];
  const ApPanel pn = T.pan[tc_search((int)blockIdx.x / 2, T.npan, [&](int q) { return __ldg(&T.pan[q].cta0); })];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, b = T.b;
  const int c0 = ((int)blockIdx.x - 2 * pn.cta0) * 16, steps = (b + TC_KS - 1) / TC_KS;
  if (c0 >= pn.ncols) return;
  const bool tri = pn.kind == 2;
  const double* A[2];
  bool live[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    live[r] = c0 + g + 8 * r < pn.ncols;
    A[r] = pn.A + (size_t)(live[r] ? c0 + g + 8 * r : c0) * b;
  }
  for (int q = warp; q < 16 && c0 + q < pn.ncols; q += TC_W) {
    const int c = c0 + q, j = pn.blk;
    int64_t d = (int64_t)j * b + c;
    if (!tri) {  // tile a of the panel with off[a] <= c < off[a + 1] (tiles of rank 0 are empty ranges)
      const int* off = (pn.kind == 0 ? T.voff : T.uoff) + (size_t)j * (T.nb + 1);
      const int a = tc_search(c, T.nb, [&](int k) { return __ldg(off + k); });
      const int at = c - off[a];
      d = pn.kind == 0 ? T.row[a].tr0 + T.uoff[(size_t)a * (T.nb + 1) + j] + at : T.row[a].sc0 + T.voff[(size_t)a * (T.nb + 1) + j] + at;
    }
    if (lane == 0) dst[q] = d;
  }
  // lower triangle of a tile, unit diagonal for L D L^T
  auto mask = [&](int r, int k, double2& v) {
    const int c = c0 + g + 8 * r;
    if (k < c) v.x = 0.0;
    else if (k == c && T.unit) v.x = 1.0;
    if (k + 1 < c) v.y = 0.0;
    else if (k + 1 == c && T.unit) v.y = 1.0;
  };
  const int first = (tri ? c0 / TC_KS : 0) + warp;  // steps before the diagonal are zero
  const uint4* fr = frag + segs[pn.blk].ks0 * TC_FRAG + lane;
  const TcLane ring(tc_smem);
  auto issue = [&](int s, int st) {
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k = s * TC_KS + 2 * t + 8 * h;
        tc_cp16(ring.x(st, 2 * r + h), A[r] + (k < b ? k : 0), live[r] && k < b);
      }
    tc_cp16(ring.f(st, 0), fr + (int64_t)s * TC_FRAG, true);
    tc_cp16(ring.f(st, 1), fr + (int64_t)s * TC_FRAG + 32, true);
  };
  tc_ring_begin(first, steps, issue);
  unsigned m[2] = {0, 0};
#pragma unroll 4
  for (int s = first; s < steps; s += TC_W) {
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k = s * TC_KS + 2 * t + 8 * h;
        double2 v = make_double2(0.0, 0.0);
        if (live[r] && k < b) v = __ldg(reinterpret_cast<const double2*>(A[r] + k));  // b is even
        if (tri) mask(r, k, v);
        m[r] = max(m[r], max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu));
      }
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    m[r] = max(m[r], __shfl_xor_sync(0xffffffffu, m[r], 1));
    m[r] = max(m[r], __shfl_xor_sync(0xffffffffu, m[r], 2));
    if (t == 0) cmax[warp][g + 8 * r] = m[r];
  }
  __syncthreads();
  auto bound = [&](int c) {
    unsigned v = 0;
#pragma unroll
    for (int w = 0; w < TC_W; ++w) v = max(v, cmax[w][c]);
    return tc_exp(v);
  };
  int ec[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    ec[r] = bound(g + 8 * r);
    if (warp == 0 && t == 0 && live[r]) {
      *tc_expof(T, pn, c0 + g + 8 * r, eU, eV, eD) = ec[r];
      if (tc_odd(ec[r])) *bad_out = 1;
    }
  }
  const int h0 = tc_shift(ec[0]), h1 = tc_shift(ec[1]), e[2][2][2] = {{{h0, h0}, {h0, h0}}, {{h1, h1}, {h1, h1}}};
  TcAcc acc;
  tc_init(acc);
  tc_ring(
      first, steps, issue,
      [&](int s, int st) {
        double x[2][2][2];
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            double2 v = *ring.x(st, 2 * r + h);
            if (tri) mask(r, s * TC_KS + 2 * t + 8 * h, v);
            x[r][h][0] = v.x;
            x[r][h][1] = v.y;
          }
        tc_step<false>(x, e, *ring.f(st, 0), *ring.f(st, 1), acc);
      });
  long long h, l;
  float est;
  tc_total(acc, reinterpret_cast<long long*>(tc_smem), h, l, est);
  const int ol = threadIdx.x >> 2, oc = threadIdx.x & 3, or_ = (ol >> 2) + 8 * (oc >> 1), cc = c0 + or_, n = 2 * (ol & 3) + (oc & 1);
  if (cc >= pn.ncols) return;
  const int en = ef[pn.blk * 8 + n];
  if (est < least && en != TC_ZERO && !(tri && (int64_t)pn.blk * b + cc >= T.N)) redo[blockIdx.x / 2] = 1;
  const double y = tc_value(h, l, bound(or_) + en);
  (tri ? YD : pn.kind == 0 ? TR : SC)[dst[or_] * 8 + n] = y;
}

// k_apply_nn on the tensor cores: 16 rows of a block row per CTA, its warps sharing the steps of
// [D_i | Urow_i | Vcol_i] [X_i; T_i; S_i].  Rows 2 g and 2 g + 1 are the fragment's rows g and g + 8 (16-byte loads).
__global__ void __launch_bounds__(TC_T, 4) k_apply_nn_tc(ApTab T, int dmode, const TcSeg* __restrict__ segs,
                                                         const uint4* __restrict__ frag, const int* __restrict__ ek,
                                                         const int* __restrict__ ef, const float* __restrict__ least,
                                                         ApOut out, int* bad_out,
                                                         int* __restrict__ redo) {
  extern __shared__ __align__(16) char tc_smem[];
  const int b = T.b, rbs = (b + 15) / 16, i = (int)blockIdx.x / rbs, r0 = ((int)blockIdx.x % rbs) * 16;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const ApRow row = T.row[i];
  const TcSeg sg = segs[i];
  const int s0 = (sg.n0 + TC_KS - 1) / TC_KS, s1 = (sg.n1 + TC_KS - 1) / TC_KS, s2 = (sg.n2 + TC_KS - 1) / TC_KS;
  const int d0 = dmode == 2 ? min(s0, r0 / TC_KS + 1) : s0;  // steps past the diagonal are zero
  const int mr = r0 + 2 * g;
  TcAcc acc;
  tc_init(acc);
  const uint4* fr = frag + sg.ks0 * TC_FRAG + lane;
  const int* er = ek + sg.ks0 * TC_KS + 2 * t;
  const TcLane ring(tc_smem);
  auto issue = [&](int v, int st) {
    const int s = v < d0 ? v : v - d0 + s0;
    const double* P = s < s0 ? row.D : s < s0 + s1 ? row.U : row.V;
    const int kb = (s < s0 ? s : s < s0 + s1 ? s - s0 : s - s0 - s1) * TC_KS, len = s < s0 ? sg.n0 : s < s0 + s1 ? sg.n1 : sg.n2;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = kb + 2 * t + (q & 1) + 8 * (q >> 1);
      const bool ok = k < len && mr < b;
      tc_cp16(ring.x(st, q), ok ? P + mr + (size_t)k * b : P, ok);
    }
    tc_cp16(ring.f(st, 0), fr + (int64_t)s * TC_FRAG, true);
    tc_cp16(ring.f(st, 1), fr + (int64_t)s * TC_FRAG + 32, true);
    tc_cp8(ring.e(st, 0), er + (int64_t)s * TC_KS);
    tc_cp8(ring.e(st, 1), er + (int64_t)s * TC_KS + 8);
  };
  tc_ring_begin(warp, d0 + s1 + s2, issue);
  tc_ring(
      warp, d0 + s1 + s2, issue,
      [&](int v, int st) {
        double x[2][2][2];
        int e[2][2][2];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          double2 a = *ring.x(st, q);
          if (dmode == 2 && v < d0) {
            const int k = v * TC_KS + 2 * t + (q & 1) + 8 * (q >> 1);
            if (mr < k) a.x = 0.0;
            else if (mr == k && T.unit) a.x = 1.0;
            if (mr + 1 < k) a.y = 0.0;
            else if (mr + 1 == k && T.unit) a.y = 1.0;
          }
          x[0][q >> 1][q & 1] = a.x;
          x[1][q >> 1][q & 1] = a.y;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int2 ev = *ring.e(st, h);
          e[0][h][0] = e[1][h][0] = ev.x;  // shifts
          e[0][h][1] = e[1][h][1] = ev.y;
        }
        if (dmode == 1) tc_step<true>(x, e, *ring.f(st, 0), *ring.f(st, 1), acc);
        else tc_step<false>(x, e, *ring.f(st, 0), *ring.f(st, 1), acc);
      });
  if (acc.bad < 0) *bad_out = 1;
  long long h, l;
  float est;
  tc_total(acc, reinterpret_cast<long long*>(tc_smem), h, l, est);
  const int ol = threadIdx.x >> 2, oc = threadIdx.x & 3, m = r0 + 2 * (ol >> 2) + (oc >> 1), n = 2 * (ol & 3) + (oc & 1);
  if (m >= b || (!out.Z && n >= out.nr)) return;
  const int en = ef[i * 8 + n];
  double v = tc_value(h, l, en);
  const int64_t gr = (int64_t)i * b + m;
  if (out.add) {
    const double a = out.add[gr * 8 + n];
    if (en != TC_ZERO) est += (float)fmin(ldexp(fabs(a), 11 - en), 65504.0);  // a term like the others
    v += a;
  }
  if (est < least[i] && en != TC_ZERO && gr < T.N) redo[i * ((b + 63) / 64) + m / 64] = 1;
  if (out.scale) v *= out.scale[gr];
  if (out.Z) out.Z[gr * 8 + n] = v;
  else if (gr < out.N) out.Y[out.perm[gr] + n * out.ldy] = v;
}

// exponents of the columns of a list's panels that k_apply_nn_tc reads and k_apply_tn_tc has not: a warp per column
__global__ void __launch_bounds__(AP_T) k_apply_colexp(ApTab T, int* __restrict__ eU, int* __restrict__ eV,
                                                       int* __restrict__ eD, int* bad_out) {
  const ApPanel pn = T.pan[ap_panel(T, (int)blockIdx.x)];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, b = T.b;
  for (int q = 0; q < AP_CW; ++q) {
    const int c = ((int)blockIdx.x - pn.cta0) * AP_W * AP_CW + q * AP_W + warp;
    if (c >= pn.ncols) return;
    const double* A = pn.A + (size_t)c * b;
    unsigned m = pn.kind == 2 && T.unit ? 0x3ff00000u : 0u;
    const int first = pn.kind == 2 ? c + (T.unit ? 1 : 0) : 0;
#pragma unroll 4
    for (int k = 2 * lane; k < b; k += 64) {
      const double2 v = __ldg(reinterpret_cast<const double2*>(A + k));
      if (k >= first) m = max(m, (unsigned)__double2hiint(v.x) & 0x7fffffffu);
      if (k + 1 >= first) m = max(m, (unsigned)__double2hiint(v.y) & 0x7fffffffu);
    }
    for (int o = 16; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) {
      *tc_expof(T, pn, c, eU, eV, eD) = tc_exp(m);
      if (tc_odd(tc_exp(m))) *bad_out = 1;
    }
  }
}
__global__ void k_apply_fill(int64_t n, int e, int* __restrict__ eD) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) eD[i] = e;
}

unsigned blocks(int64_t n, int t) { return (unsigned)std::min<int64_t>((n + t - 1) / t, 8192); }

template <int NR, int VEC>
void run_tn(tlr_ctx* ctx, const ApTab& T, int ctas, const double* X, double* TR, double* SC, double* YD) {
  if (ctas <= 0) return;
  TLR_SITE_PRE(ctx);
  k_apply_tn<NR, VEC><<<(unsigned)ctas, AP_T, 0, ctx->stream>>>(T, X, TR, SC, YD);
  TLR_LAUNCH_CHECK(ctx);
}

template <int NR, int VEC>
void run_nn(tlr_ctx* ctx, const ApTab& T, int dmode, int use_u, int use_v, int64_t ktot, const double* X,
            const double* TR, const double* SC, const ApOut& out) {
  constexpr int RB = 32 * VEC;
  const int64_t rbs = (int64_t)T.nb * ((T.b + RB - 1) / RB);
  // CTAs sharing a row block: until the launch holds four CTAs per SM, while each still has 64 steps of
  // the (mean) contraction length
  int S = 1;
  while (S < 8 && rbs * S < 4 * (int64_t)ctx->sm_count && ktot / T.nb / (2 * S) >= 64) S *= 2;
  cudaLaunchConfig_t cf{};
  cf.gridDim = dim3((unsigned)(rbs * S));
  cf.blockDim = dim3(AP_T);
  cf.stream = ctx->stream;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)S;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cf.attrs = &at;
  cf.numAttrs = 1;
  TLR_SITE_PRE(ctx);
  TLR_CUDA(cudaLaunchKernelEx(&cf, k_apply_nn<NR, VEC>, T, dmode, use_u, use_v, S, X, TR, SC, out));
  TLR_LAUNCH_CHECK(ctx);
}

struct ApPlan {  // host side of one matrix's tables
  ApTab T;       // pan set per list
  const ApPanel* lists[3];  // of the contractions, and the columns whose exponents they don't find
  int npan[3], ctas[3];
  int64_t R, np;
  // tensor-core path: the blocks' right-hand sides (X; what follows for L^T X: S; then [X; T; S] or [Z; T]) and their steps
  bool tc;
  const TcSeg* segs[3];
  int64_t steps[3];
};

template <int NR, int VEC>
void apply_group(tlr_ctx* ctx, const tlr_mat* M, int op, const ApPlan& pl, int nr, const double* X, int64_t ldx, double* Y,
                 int64_t ldy, Buf& work) {
  constexpr int LD = ap_ld<NR>();
  const int64_t np = pl.np, R = std::max<int64_t>(pl.R, 1);
  double* Xp = work.need<double>((size_t)(3 * np + 2 * R) * LD);
  double *YD = Xp + np * LD, *Z = YD + np * LD, *TR = Z + np * LD, *SC = TR + R * LD;
  TLR_SITE_PRE(ctx);
  k_apply_gather<<<blocks(np * LD, 256), 256, 0, ctx->stream>>>(M->N, np, nr, LD, M->dperm, X, ldx, Xp, nullptr, 0);
  TLR_LAUNCH_CHECK(ctx);
  const int64_t kd = (int64_t)M->nb * M->b;
  const ApTab& T = pl.T;
  auto tn = [&](int l, const double* x) {
    ApTab Tl = T;
    Tl.pan = pl.lists[l];
    Tl.npan = pl.npan[l];
    run_tn<NR, VEC>(ctx, Tl, pl.ctas[l], x, TR, SC, YD);
  };
  ApOut fin{nullptr, nullptr, nullptr, Y, M->dperm, ldy, M->N, nr};
  tn(0, Xp);
  if (op == TLR_OP_A) {
    run_nn<NR, VEC>(ctx, T, 1, 1, 1, kd + 2 * pl.R, Xp, TR, SC, fin);
  } else if (op == TLR_OP_L) {
    run_nn<NR, VEC>(ctx, T, 2, 1, 0, kd / 2 + pl.R, Xp, TR, SC, fin);
  } else if (op == TLR_OP_LT) {
    fin.add = YD;
    run_nn<NR, VEC>(ctx, T, 0, 0, 1, pl.R, Xp, TR, SC, fin);
  } else {  // L (D) (L^T X)
    ApOut mid{YD, M->state == 2 ? M->dvec : nullptr, Z, nullptr, nullptr, 0, 0, nr};
    run_nn<NR, VEC>(ctx, T, 0, 0, 1, pl.R, Xp, TR, SC, mid);
    tn(1, Z);
    run_nn<NR, VEC>(ctx, T, 2, 1, 0, kd / 2 + pl.R, Z, TR, SC, fin);
  }
}

// The same on the tensor cores (8 columns, zero past nr).  After each contraction the FP64 kernel computes what would have
// fewer digits (redo), or all of it if numbers are outside what the digits hold (bad: not finite, or a column's largest
// below 2^-900 or above 2^900).
void apply_group_tc(tlr_ctx* ctx, const tlr_mat* M, int op, const ApPlan& pl, int nr, const double* X, int64_t ldx, double* Y,
                    int64_t ldy, Buf& work) {
  const int64_t np = pl.np, R = std::max<int64_t>(pl.R, 1), kd = np;
  const int64_t steps = std::max({pl.steps[0], pl.steps[1], pl.steps[2]});
  const int nb = M->nb, b = M->b;
  // flags: bad, then redo of the contractions of list 0 and 1 (k_apply_tn's CTAs) and of the middle and the final rows
  const int64_t rbs = (int64_t)nb * ((b + 63) / 64), nflags = 1 + pl.ctas[0] + pl.ctas[1] + 2 * rbs;
  // doubles: Xp, YD, Z (np x 8), T, S (R x 8); fragments (16 bytes); ints: exponents by step, of U, V
  // and tile columns, of the blocks' right-hand sides, the least estimates, the flags
  const size_t nd = (size_t)(3 * np + 2 * R) * 8, nf = 2 * (size_t)steps * TC_FRAG,
               ni = (size_t)(steps * TC_KS + 2 * R + np + 9 * (int64_t)nb + nflags);
  double* Xp = work.need<double>(nd + nf + (ni + 1) / 2);
  double *YD = Xp + np * 8, *Z = YD + np * 8, *TR = Z + np * 8, *SC = TR + R * 8;
  uint4* frag = reinterpret_cast<uint4*>(Xp + nd);
  int* ek = reinterpret_cast<int*>(Xp + nd + nf);
  int *eU = ek + steps * TC_KS, *eV = eU + R, *eD = eV + R, *ef = eD + np, *bad = ef + 9 * (int64_t)nb;
  float* least = reinterpret_cast<float*>(ef + 8 * (int64_t)nb);
  int *redo_tn[2] = {bad + 1, bad + 1 + pl.ctas[0]}, *redo_nn[2] = {redo_tn[1] + pl.ctas[1], redo_tn[1] + pl.ctas[1] + rbs};
  TLR_SITE_PRE(ctx);
  k_apply_gather<<<blocks(np * 8, 256), 256, 0, ctx->stream>>>(M->N, np, nr, 8, M->dperm, X, ldx, Xp, bad, nflags);
  TLR_LAUNCH_CHECK(ctx);
  for (const void* f : {(const void*)k_apply_tn_tc, (const void*)k_apply_nn_tc})
    TLR_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM));
  ApTab T = pl.T;
  T.gate = bad;
  auto tn = [&](int l, const double* x) {
    TLR_SITE_PRE(ctx);
    k_apply_split<1><<<(unsigned)nb * TC_SPC, 256, 0, ctx->stream>>>(pl.segs[0], T.row, b, x, TR, SC, eD, eU, eV, frag, ek, ef,
                                                                     least, bad);
    TLR_LAUNCH_CHECK(ctx);
    if (pl.ctas[l] <= 0) return;
    T.pan = pl.lists[l];
    T.npan = pl.npan[l];
    T.redo = redo_tn[l];
    TLR_SITE_PRE(ctx);
    k_apply_tn_tc<<<2 * (unsigned)pl.ctas[l], TC_T, TC_SMEM, ctx->stream>>>(T, pl.segs[0], frag, ef, TR, SC, YD, eU, eV, eD,
                                                                            tc_least((float)b), bad, redo_tn[l]);
    TLR_LAUNCH_CHECK(ctx);
    run_tn<8, 2>(ctx, T, pl.ctas[l], x, TR, SC, YD);
  };
  // rows [D | U | V] (dmode, use_u, use_v) of the q-th segment list; f: the final rows
  auto nn = [&](int q, int dmode, int use_u, int use_v, int64_t ktot, const double* x, const ApOut& o, int f) {
    TLR_SITE_PRE(ctx);
    k_apply_split<3><<<(unsigned)nb * TC_SPC, 256, 0, ctx->stream>>>(pl.segs[q], T.row, b, x, TR, SC, eD, eU, eV, frag, ek, ef,
                                                                     least, bad);
    TLR_LAUNCH_CHECK(ctx);
    T.redo = redo_nn[f];
    TLR_SITE_PRE(ctx);
    k_apply_nn_tc<<<(unsigned)((int64_t)nb * ((b + 15) / 16)), TC_T, TC_SMEM, ctx->stream>>>(T, dmode, pl.segs[q], frag, ek,
                                                                                          ef, least, o, bad, redo_nn[f]);
    TLR_LAUNCH_CHECK(ctx);
    run_nn<8, 2>(ctx, T, dmode, use_u, use_v, ktot, x, TR, SC, o);
  };
  if (op == TLR_OP_A) {  // kernel entries are at most 1, the diagonal's 1 + nugget
    TLR_SITE_PRE(ctx);
    k_apply_fill<<<blocks(np, 256), 256, 0, ctx->stream>>>(np, ilogb(std::max(1.0, 1.0 + M->kern.nugget)) + 1, eD);
    TLR_LAUNCH_CHECK(ctx);
  } else if (pl.ctas[2] > 0) {
    T.pan = pl.lists[2];
    T.npan = pl.npan[2];
    TLR_SITE_PRE(ctx);
    k_apply_colexp<<<(unsigned)pl.ctas[2], AP_T, 0, ctx->stream>>>(T, eU, eV, eD, bad);
    TLR_LAUNCH_CHECK(ctx);
  }
  ApOut fin{nullptr, nullptr, nullptr, Y, M->dperm, ldy, M->N, nr};
  tn(0, Xp);
  if (op == TLR_OP_A) {
    nn(2, 1, 1, 1, kd + 2 * pl.R, Xp, fin, 1);
  } else if (op == TLR_OP_L) {
    nn(2, 2, 1, 0, kd / 2 + pl.R, Xp, fin, 1);
  } else if (op == TLR_OP_LT) {
    fin.add = YD;
    nn(1, 0, 0, 1, pl.R, Xp, fin, 1);
  } else {  // L (D) (L^T X); the first contraction has left the exponents of U's and the tiles' columns
    ApOut mid{YD, M->state == 2 ? M->dvec : nullptr, Z, nullptr, nullptr, 0, 0, nr};
    nn(1, 0, 0, 1, pl.R, Xp, mid, 0);
    tn(1, Z);
    nn(2, 2, 1, 0, kd / 2 + pl.R, Z, fin, 1);
  }
}

template <int VEC>
void apply_width(tlr_ctx* ctx, const tlr_mat* M, int op, const ApPlan& pl, int nr, const double* X, int64_t ldx,
                 double* Y, int64_t ldy, Buf& work) {
  if (nr == 1) apply_group<1, VEC>(ctx, M, op, pl, nr, X, ldx, Y, ldy, work);
  else if (nr == 2) apply_group<2, VEC>(ctx, M, op, pl, nr, X, ldx, Y, ldy, work);
  else if (nr == 3) apply_group<3, VEC>(ctx, M, op, pl, nr, X, ldx, Y, ldy, work);
  else if (nr == 4) apply_group<4, VEC>(ctx, M, op, pl, nr, X, ldx, Y, ldy, work);
  else if (nr <= 6) apply_group<6, VEC>(ctx, M, op, pl, nr, X, ldx, Y, ldy, work);
  else apply_group<8, VEC>(ctx, M, op, pl, nr, X, ldx, Y, ldy, work);
}

}  // namespace

void tlr_apply(tlr_ctx* ctx, const tlr_mat* M, int op, int nrhs, const double* X, int64_t ldx, double* Y, int64_t ldy) {
  const int nb = M->nb, b = M->b;
  // Tables, made for each call from the matrix's ranks (O(nb^2) integers): nothing is kept.
  const size_t tabn = (size_t)nb * (nb + 1);
  std::vector<int> off(2 * tabn);
  int* vo = off.data();
  int* uo = vo + tabn;
  std::vector<ApRow> rows(nb);
  ApPlan pl{};
  bool aligned = b % 2 == 0;
  auto al = [&](const double* p) { aligned &= reinterpret_cast<uintptr_t>(p) % 16 == 0; };
  al(M->diag);
  int64_t tr = 0, sc = 0;
  for (int i = 0; i < nb; ++i) {
    // monotone offsets: a tile of rank 0 starts where the next one does
    int* v = vo + (size_t)i * (nb + 1);
    v[nb] = (int)M->vlen[i];
    for (int t = nb - 1; t > i; --t) v[t] = M->rank[ix(M, t, i)] > 0 ? (int)M->voff[ix(M, t, i)] : v[t + 1];
    for (int t = 0; t <= i; ++t) v[t] = 0;
    int* u = uo + (size_t)i * (nb + 1);
    for (int t = i; t <= nb; ++t) u[t] = (int)M->ulen[i];
    for (int t = i - 1; t >= 0; --t) u[t] = M->rank[ix(M, i, t)] > 0 ? (int)M->uoff[ix(M, i, t)] : u[t + 1];
    rows[i] = ApRow{M->diag + (size_t)i * b * b, M->Urow[i], M->Vcol[i], tr, sc, (int)M->ulen[i], (int)M->vlen[i]};
    tr += M->ulen[i];
    sc += M->vlen[i];
    al(M->Urow[i]);
    al(M->Vcol[i]);
  }
  // Tensor cores where the DFMAs (1.67 ps per entry and accumulator column) take longer than the tensor cores' passes
  // (3.2 ps per entry for up to eight columns), the DFMAs of eight columns for the share of the entries whose results
  // are computed again, and their further launches.  That share is none for A and, for the factors' triangles of the
  // covariance problems (normal right-hand sides), about 0.6 of L, 0.55 of L^T, 0.5 of both.  Measured, DFMA / tensor
  // cores, us: A, 6.7e8 entries 2412 / 2260 (2 columns), 9103 / 2266 (8); 3.6e7 213 / 241 (2), 284 / 241 (3), 608 / 240
  // (8); 4.8e6 108 / 121 (4), 155 / 124 (8).  8 columns, L, 3.7e8 entries 4548 / 3973; 5.4e7 932 / 907; 1.3e7 287 / 319;
  // L^T 4439 / 3486, 880 / 840, 280 / 300; L (D) L^T, 7.3e8 entries 8899 / 5587; 1.1e8 1753 / 1693; 2.5e7 517 / 507;
  // 4 columns 4570 / 5328, 949 / 1572, 312 / 495.
  const int ng = (nrhs + 7) / 8;  // right-hand sides in equal groups of at most eight
  const int nr = (nrhs + ng - 1) / ng, cols = nr <= 4 ? nr : nr <= 6 ? 6 : 8;
  const double lower = 2.0 * b * (double)tr + 0.5 * nb * b * b;
  const double entries = op == TLR_OP_L || op == TLR_OP_LT ? lower : 2.0 * lower;
  const double again = op == TLR_OP_A ? 0.0 : op == TLR_OP_L ? 0.6 : op == TLR_OP_LT ? 0.55 : 0.5;
  const double launches = op == TLR_OP_A ? 45e6 : op == TLR_OP_LLT ? 100e6 : 60e6;
  pl.tc = aligned && entries * (1.67 * cols - 3.2 - 1.67 * 8 * again) > launches;
  std::vector<ApPanel> pans;
  int n0[4] = {0, 0, 0, 0};
  auto list = [&](int l, bool v, bool u, bool dg) {
    int cta = 0;
    auto add = [&](const double* A, int64_t ncols, int blk, int kind) {
      if (ncols <= 0) return;
      pans.push_back(ApPanel{A, (int)ncols, blk, kind, cta});
      cta += (int)((ncols + AP_W * AP_CW - 1) / (AP_W * AP_CW));
    };
    for (int i = 0; i < nb; ++i) {
      if (dg) add(M->diag + (size_t)i * b * b, b, i, 2);
      if (v) add(M->Vcol[i], M->vlen[i], i, 0);
      if (u) add(M->Urow[i], M->ulen[i], i, 1);
    }
    n0[l + 1] = (int)pans.size();
    pl.npan[l] = n0[l + 1] - n0[l];
    pl.ctas[l] = cta;
  };
  if (op == TLR_OP_A) list(0, true, true, false);
  else if (op == TLR_OP_L) list(0, true, false, false);
  else list(0, false, true, true);
  list(1, op == TLR_OP_LLT, false, false);
  list(2, pl.tc && (op == TLR_OP_LT || op == TLR_OP_LLT), pl.tc && op == TLR_OP_L, pl.tc && op == TLR_OP_L);
  // one table on the device: rows, panels, offsets
  std::vector<TcSeg> segs;
  for (int q = 0; pl.tc && q < 3; ++q) {
    int64_t ks = 0;
    for (int i = 0; i < nb; ++i) {
      TcSeg g{ks, 0, 0, 0};
      if (q == 0) g.n0 = b;                          // X
      else if (q == 1) g.n2 = (int)M->vlen[i];       // S
      else {                                         // [X; T; S] of A, [X; T] of L
        g.n0 = b;
        g.n1 = (int)M->ulen[i];
        g.n2 = op == TLR_OP_A ? (int)M->vlen[i] : 0;
      }
      for (int n : {g.n0, g.n1, g.n2}) ks += (n + TC_KS - 1) / TC_KS;
      segs.push_back(g);
    }
    pl.steps[q] = ks;
  }
  const size_t br = sizeof(ApRow) * nb, bp = sizeof(ApPanel) * pans.size(), bg = sizeof(TcSeg) * segs.size(),
               bo = sizeof(int) * off.size();
  std::vector<char> tab(br + bp + bg + bo);
  memcpy(tab.data(), rows.data(), br);
  if (bp) memcpy(tab.data() + br, pans.data(), bp);
  if (bg) memcpy(tab.data() + br + bp, segs.data(), bg);
  memcpy(tab.data() + br + bp + bg, off.data(), bo);
  Buf btab(ctx), work(ctx);
  const char* dt;
  const size_t chunk = (size_t)16 << 20;
  if (tab.size() <= chunk) {
    dt = static_cast<const char*>(upload(ctx, tab.data(), tab.size()));
  } else {  // larger than a share of the upload ring: in pieces into an array of its own
    char* d = btab.need<char>(tab.size());
    for (size_t o = 0; o < tab.size(); o += chunk) {
      const size_t n = std::min(chunk, tab.size() - o);
      TLR_CUDA(cudaMemcpyAsync(d + o, upload(ctx, tab.data() + o, n), n, cudaMemcpyDeviceToDevice, ctx->stream));
    }
    dt = d;
  }
  pl.T.row = reinterpret_cast<const ApRow*>(dt);
  pl.lists[0] = reinterpret_cast<const ApPanel*>(dt + br);
  pl.lists[1] = pl.lists[0] + n0[1];
  pl.lists[2] = pl.lists[0] + n0[2];
  for (int q = 0; q < 3; ++q) pl.segs[q] = reinterpret_cast<const TcSeg*>(dt + br + bp) + (pl.tc ? (size_t)q * nb : 0);
  pl.T.voff = reinterpret_cast<const int*>(dt + br + bp + bg);
  pl.T.uoff = pl.T.voff + tabn;
  pl.T.nb = nb;
  pl.T.b = b;
  pl.T.unit = M->state == 2;
  pl.T.N = M->N;
  pl.R = tr;
  pl.np = (int64_t)nb * b;
  for (int g = 0; g < ng; ++g) {
    const int c0 = (int)((int64_t)nrhs * g / ng), nr = (int)((int64_t)nrhs * (g + 1) / ng) - c0;
    const double* Xg = X + (size_t)c0 * ldx;
    double* Yg = Y + (size_t)c0 * ldy;
    if (pl.tc) apply_group_tc(ctx, M, op, pl, nr, Xg, ldx, Yg, ldy, work);
    else if (aligned) apply_width<2>(ctx, M, op, pl, nr, Xg, ldx, Yg, ldy, work);
    else apply_width<1>(ctx, M, op, pl, nr, Xg, ldx, Yg, ldy, work);
  }
}

}  // namespace tlr
