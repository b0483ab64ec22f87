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
// eps = 1e-4, 1 column 6.50 -> 0.32 ms.
//
// Sums run in a fixed order: results do not depend on timing.
#include <cooperative_groups.h>

#include <cstring>

#include "internal.h"
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
                               const double* __restrict__ X, int64_t ldx, double* __restrict__ Xp) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < np * ld; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = e / ld;
    const int c = (int)(e % ld);
    Xp[e] = p < N && c < nr ? X[perm[p] + (int64_t)c * ldx] : 0.0;
  }
}

template <int NR, int VEC>
__global__ void __launch_bounds__(AP_T) k_apply_tn(ApTab T, const double* __restrict__ X, double* __restrict__ TR,
                                                   double* __restrict__ SC, double* __restrict__ YD) {
  constexpr int LD = ap_ld<NR>(), UN = NR <= 4 ? 2 : 1, STEP = 32 * VEC;
  constexpr int P = AP_CW * (NR == 3 ? 4 : NR == 6 ? 8 : NR), LANES = 32 / P;  // lanes that share a sum
  __shared__ int panel;
  if (threadIdx.x == 0) {
    int lo = 0, hi = T.npan - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (T.pan[mid].cta0 <= (int)blockIdx.x) lo = mid;
      else hi = mid - 1;
    }
    panel = lo;
  }
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
  const ApPanel* lists[2];
  int npan[2], ctas[2];
  int64_t R, np, ktot_d;
};

template <int NR, int VEC>
void apply_group(tlr_ctx* ctx, const tlr_mat* M, int op, const ApPlan& pl, int nr, const double* X, int64_t ldx, double* Y,
                 int64_t ldy, Buf& work) {
  constexpr int LD = ap_ld<NR>();
  const int64_t np = pl.np, R = std::max<int64_t>(pl.R, 1);
  double* Xp = work.need<double>((size_t)(3 * np + 2 * R) * LD);
  double *YD = Xp + np * LD, *Z = YD + np * LD, *TR = Z + np * LD, *SC = TR + R * LD;
  TLR_SITE_PRE(ctx);
  k_apply_gather<<<blocks(np * LD, 256), 256, 0, ctx->stream>>>(M->N, np, nr, LD, M->dperm, X, ldx, Xp);
  TLR_LAUNCH_CHECK(ctx);
  ApTab T = pl.T;
  auto tn = [&](int l, const double* x) {
    T.pan = pl.lists[l];
    T.npan = pl.npan[l];
    run_tn<NR, VEC>(ctx, T, pl.ctas[l], x, TR, SC, YD);
  };
  ApOut fin{nullptr, nullptr, nullptr, Y, M->dperm, ldy, M->N, nr};
  const int64_t kd = (int64_t)M->nb * M->b;
  if (op == TLR_OP_A) {
    tn(0, Xp);
    run_nn<NR, VEC>(ctx, T, 1, 1, 1, kd + 2 * pl.R, Xp, TR, SC, fin);
  } else if (op == TLR_OP_L) {
    tn(0, Xp);
    run_nn<NR, VEC>(ctx, T, 2, 1, 0, kd / 2 + pl.R, Xp, TR, SC, fin);
  } else if (op == TLR_OP_LT) {
    tn(0, Xp);
    fin.add = YD;
    run_nn<NR, VEC>(ctx, T, 0, 0, 1, pl.R, Xp, TR, SC, fin);
  } else {  // L (D) (L^T X)
    tn(0, Xp);
    ApOut mid{YD, M->state == 2 ? M->dvec : nullptr, Z, nullptr, nullptr, 0, 0, nr};
    run_nn<NR, VEC>(ctx, T, 0, 0, 1, pl.R, Xp, TR, SC, mid);
    tn(1, Z);
    run_nn<NR, VEC>(ctx, T, 2, 1, 0, kd / 2 + pl.R, Z, TR, SC, fin);
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
  std::vector<ApPanel> pans;
  int n0[3] = {0, 0, 0};
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
  if (op == TLR_OP_LLT) list(1, true, false, false);
  // one table on the device: rows, panels, offsets
  const size_t br = sizeof(ApRow) * nb, bp = sizeof(ApPanel) * pans.size(), bo = sizeof(int) * off.size();
  std::vector<char> tab(br + bp + bo);
  memcpy(tab.data(), rows.data(), br);
  if (bp) memcpy(tab.data() + br, pans.data(), bp);
  memcpy(tab.data() + br + bp, off.data(), bo);
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
  pl.T.voff = reinterpret_cast<const int*>(dt + br + bp);
  pl.T.uoff = pl.T.voff + tabn;
  pl.T.nb = nb;
  pl.T.b = b;
  pl.T.unit = M->state == 2;
  pl.R = tr;
  pl.np = (int64_t)nb * b;
  // right-hand sides in equal groups of at most eight
  const int ng = (nrhs + 7) / 8;
  for (int g = 0; g < ng; ++g) {
    const int c0 = (int)((int64_t)nrhs * g / ng), nr = (int)((int64_t)nrhs * (g + 1) / ng) - c0;
    const double* Xg = X + (size_t)c0 * ldx;
    double* Yg = Y + (size_t)c0 * ldy;
    if (aligned) apply_width<2>(ctx, M, op, pl, nr, Xg, ldx, Yg, ldy, work);
    else apply_width<1>(ctx, M, op, pl, nr, Xg, ldx, Yg, ldy, work);
  }
}

}  // namespace tlr
