// ARA -> SVD rank trimming of low-rank tiles (Section 6: the post-processing step that applies the SVD
// to each low-rank tile to bring its rank down to the minimum).
//
// A tile Q B^T with orthonormal Q (b x r) has the singular values of B.  One CTA, or a cluster of four or eight, per
// tile: a Householder QR of B (B = H R, the reflectors applied to the trailing columns in place, in a working
// copy in global memory), then one-sided Jacobi (Hestenes) on X = R^T: plane rotations of column pairs in the
// parallel round-robin order (r/2 disjoint pairs per round, r - 1 rounds per sweep) until no pair is rotated,
// giving X J = Y with orthogonal columns whose norms are the singular values sigma of R (and of B), and
// Y / sigma the right singular vectors Z of B (R = J S (Y S^-1)^T).  Jacobi on R^T rather than R takes
// about a third of the sweeps on these matrices.  The columns with sigma > eps, in descending order,
// form Z_r (r x r'); Q' = Q Z_r and B' = B Z_r = W_r S_r are two batched GEMMs.  Every reduction has a
// fixed order, so the result depends on the tile only.
//
// The FP64 unit is the bound: a sweep is 5 r^3 / 2 lane operations (one product for the pair's inner product,
// four for the rotation; the squared norms are updated by the rotation, a' = a - t g, b' = b + t g, and
// recomputed once per sweep) plus a square root, a reciprocal and a reciprocal square root per pair.  So
//   * several lanes share a pair, as many as keep the CTA's threads busy, and the pairs' rotation angles are
//     computed together, one thread per pair, so that the scalar work fills its warps;
//   * the tiles of the highest ranks are each spread over a cluster, the columns dealt out over the CTAs' shared memory
//     and reached through distributed shared memory: the few tiles of high rank next to the diagonal are what a
//     matrix's trimming waits for;
//   * the tiles of low rank run beside them on the side stream.
// Measured, one thread per pair and rank classes one after another -> now: trimming a matrix of N = 16384, b = 512
// (ranks up to 142, mean 27) 109 -> 12.9 ms; 12 tiles of rank 140 61 -> 9.5 ms; 57 of rank 64 12.9 -> 3.7; 400 of
// rank 16 1.36 -> 1.01; 4 of rank 300 (b = 1024) 723 -> 60.
#include <cooperative_groups.h>
#include <math.h>

#include <functional>
#include <map>

#include "internal.h"

namespace cg = cooperative_groups;

namespace tlr {

namespace {

constexpr int TR_T = 256, TR_W = TR_T / 32;
constexpr int TR_SWEEPS = 60;  // a bound only: the tiles converge in about 10
constexpr int TR_SOLO = 48;    // tiles up to this rank always take one CTA

struct TrimDev {
  const double* B;  // b x r, leading dimension b
  double* W;        // working copy (b x r)
  double* X;        // R^T (r x r) and the squared norms (r) when they do not fit in shared memory
  double* Zs;       // out: Z_r (r x r', leading dimension r)
  int* rank;        // out: r'
  int r;
};

// warp sum, the lane-0 value broadcast so that every lane holds the same bits
__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return __shfl_sync(0xffffffffu, v, 0);
}

__device__ double block_sum(double v, double* red) {
  v = warp_sum(v);
  __syncthreads();  // red is free
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  for (int i = 0; i < TR_W; ++i) s += red[i];
  return s;
}

// 1 / v by two Newton steps, v normal.  (Any tangent makes an orthogonal rotation; one that is off by a few ulps is
// corrected by later rotations.)
__device__ __forceinline__ double recip_approx(double v) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(v));
  y = fma(y, fma(-v, y, 1.0), y);
  return fma(y, fma(-v, y, 1.0), y);
}

// Whether columns with squared norms a, b and inner product g are to be rotated (g^2 > tol2 a b), and the tangent of
// the rotation, 2 g / (d + sign(d) sqrt(d^2 + 4 g^2)) with d = b - a
__device__ __forceinline__ bool rotation_in_range(double a, double b, double g, double tol2, double& t) {
  const double d = b - a, g2 = 2.0 * g, h = fma(d, d, g2 * g2);
  if (!(g * g > tol2 * (a * b))) return false;
  const double hs = h * rsqrt(h);
  t = (d >= 0.0 ? g2 : -g2) * recip_approx(fabs(d) + hs);
  return true;
}
__device__ __forceinline__ int exp_field(double x) { return (int)((unsigned)__double2hiint(x) >> 20 & 0x7ffu); }
// 2^(1023 - f) for a biased exponent f in 1 .. 2045
__device__ __forceinline__ double pow2_inv(int f) { return __hiloint2double((2046 - f) << 20, 0); }
// The squares of a, b and g leave FP64's range (norms beyond about 2^+-225): the same on numbers scaled by powers of
// two, a and b to order one each for the test and to the larger of them for the angle
__device__ __noinline__ bool rotation_scaled(double a, double b, double g, double tol2, double& t) {
  const int fa = min(max(exp_field(a), 1), 2045), fb = min(max(exp_field(b), 1), 2045), odd = (fa ^ fb) & 1;
  const double gn = g * pow2_inv((fa + fb + odd) / 2), an = a * pow2_inv(fa), bn = b * pow2_inv(min(fb + odd, 2045));
  if (!(gn * gn > tol2 * (an * bn))) return false;
  const double sc = pow2_inv(max(fa, fb));
  t = 0.0;
  return rotation_in_range(a * sc, b * sc, g * sc, -1.0, t);
}
__device__ __forceinline__ bool rotation(double a, double b, double g, double tol2, double& t) {
  const unsigned fa = exp_field(a) - 573, fb = exp_field(b) - 573;  // 2^-450 .. 2^450
  if (max(fa, fb) <= 900u) return rotation_in_range(a, b, g, tol2, t);
  return rotation_scaled(a, b, g, tol2, t);
}

// Lane gl's share, of L lanes, of the inner product of two columns of r entries, to be added up over the lanes by
// halving exchanges (o = L / 2, .., 1).  The sum is that of 32 chains, chain c of the rows c, c + 32, .., added in
// halves whatever L is: lane gl holds the chains gl, gl + L, ..
template <int L, class LD>
__device__ __forceinline__ double pair_dot(const double* x, const double* y, int r, int gl, LD ld) {
  constexpr int C = 32 / L;
  double a[C];
#pragma unroll
  for (int u = 0; u < C; ++u) a[u] = 0.0;
  int m = gl;
#pragma unroll(C < 4 ? 4 / C : 1)
  for (; m + (C - 1) * L < r; m += 32)
#pragma unroll
    for (int u = 0; u < C; ++u) a[u] = fma(ld(x + m + u * L), ld(y + m + u * L), a[u]);
#pragma unroll
  for (int u = 0; u < C - 1; ++u)
    if (m + u * L < r) a[u] = fma(ld(x + m + u * L), ld(y + m + u * L), a[u]);
#pragma unroll
  for (int h = C / 2; h; h /= 2)
#pragma unroll
    for (int u = 0; u < h; ++u) a[u] += a[u + h];
  return a[0];
}

// CS: CTAs of the tile's cluster.  SM: X and the norms live in shared memory, column c in CTA c % CS at place
// c / CS; otherwise in global memory.  Registers for the CTAs that share an SM: five single ones when ranks are low (2000
// tiles of rank 16, b = 1024: 5.2 ms; 6.0 with three), two of clusters of four (57 tiles of rank 80: 6.5 ms; 9.8 with one,
// 6.6 with four), one of clusters of eight, which are few.
template <int CS, bool SM>
__global__ void __launch_bounds__(TR_T, CS == 1 ? 5 : CS == 4 ? 2 : 1) k_trim(const TrimDev* __restrict__ jobs, int b, double eps) {
  const TrimDev J = jobs[blockIdx.x / CS];
  const int rank = (int)(blockIdx.x % CS);
  const int r = J.r, tid = threadIdx.x, w = tid >> 5, l = tid & 31;
  extern __shared__ double sm[];
  __shared__ double cc[TR_T], sn[TR_T], gs[TR_T];  // rotations of a pass's pairs
  __shared__ double red[TR_W];
  __shared__ int rot, keep;
  const int rp = r | 1, nc = (r + CS - 1) / CS;  // leading dimension of X (odd: no bank conflicts), columns per CTA
  double* v = sm;                                // b: the current reflector
  double* beta = v + b;                          // r: the diagonal of R, later the singular values
  double* nrm_s = beta + r;                      // nc: squared norms of this CTA's columns
  double* X_s = nrm_s + (SM ? nc : 0);           // nc columns
  int* pos = reinterpret_cast<int*>(X_s + (SM ? (size_t)nc * rp : 0));  // r
  auto csync = [&]() {
    if (CS == 1) __syncthreads();
    else cg::this_cluster().sync();
  };
  auto peer = [&](double* p, int q) { return CS == 1 ? p : cg::this_cluster().map_shared_rank(p, q); };
  auto col = [&](int c) { return SM ? peer(X_s, c % CS) + (size_t)(c / CS) * rp : J.X + (size_t)c * rp; };
  auto nrm = [&](int c) { return SM ? peer(nrm_s, c % CS) + c / CS : J.X + (size_t)r * rp + c; };
  auto ld = [](const double* p) { return SM ? *p : __ldcg(p); };  // other CTAs write X
  if (r == 0) {  // the whole cluster
    if (tid == 0 && rank == 0) *J.rank = 0;
    return;
  }
  double* W = J.W;
  for (int c = rank; c < r; c += CS)
    for (int m = tid; m < b; m += TR_T) W[m + (size_t)c * b] = J.B[m + (size_t)c * b];
  // ---- Householder QR: R's strict upper triangle in W's first rows, its diagonal in beta.  Every CTA forms the
  // reflector; column c of the trailing part is CTA c % CS's.
  for (int j = 0; j < r; ++j) {
    csync();  // column j is complete
    const double* cj = W + (size_t)j * b;
    double s = 0.0;
    for (int m = j + 1 + tid; m < b; m += TR_T) {
      const double x = __ldcg(cj + m);
      v[m] = x;
      s += x * x;
    }
    s = block_sum(s, red);
    const double alpha = __ldcg(cj + j);
    double d = alpha;
    if (s > 0.0) {  // uniform: s is the block's sum
      const double nr = sqrt(alpha * alpha + s);
      d = alpha >= 0.0 ? -nr : nr;
      const double tau = (d - alpha) / d, scal = 1.0 / (alpha - d);
      for (int m = j + 1 + tid; m < b; m += TR_T) v[m] *= scal;
      if (tid == 0) v[j] = 1.0;
      __syncthreads();
      // H = I - tau v v^T on this CTA's trailing columns, a warp each
      for (int c = j + 1 + ((rank - (j + 1)) % CS + CS) % CS + w * CS; c < r; c += TR_W * CS) {
        double* x = W + (size_t)c * b;
        double dt = 0.0;
#pragma unroll 4
        for (int m = j + l; m < b; m += 32) dt += v[m] * x[m];
        const double f = tau * warp_sum(dt);
#pragma unroll 4
        for (int m = j + l; m < b; m += 32) x[m] -= f * v[m];
      }
    }
    if (tid == 0) beta[j] = d;
  }
  csync();
  // ---- X = R^T (lower triangular)
  for (int c = rank; c < r; c += CS) {
    double* x = col(c);
    for (int m = tid; m < r; m += TR_T) x[m] = c < m ? __ldcg(W + c + (size_t)m * b) : c == m ? beta[c] : 0.0;
  }
  // ---- one-sided Jacobi on X, round-robin pairs (position 0 fixed, 1 .. n-1 rotating); pair k is CTA k % CS's
  const int n = r + (r & 1), np = n / 2, mine = (np - rank + CS - 1) / CS;
  int L = 32;  // lanes of a pair (pair_dot)
  while (L > 4 && mine * L > TR_T) L >>= 1;
  const int G = TR_T / L, grp = tid / L, gl = tid % L;
  const double tol2 = ((double)r * 0x1p-53) * ((double)r * 0x1p-53);
  auto norms = [&]() {  // squared norms of this CTA's columns
    for (int c = rank + w * CS; c < r; c += TR_W * CS) {
      const double* x = col(c);
      double s2 = 0.0;
      for (int m = l; m < r; m += 32) {
        const double y = ld(x + m);
        s2 += y * y;
      }
      s2 = warp_sum(s2);
      if (l == 0) *nrm(c) = s2;
    }
  };
  auto pair_of = [&](int k, int t, int& p, int& q) {
    p = k == 0 ? 0 : (k - 1 + t) % (n - 1) + 1;
    q = (n - 2 - k + t) % (n - 1) + 1;  // the position n - 1 - k >= 1
    if (p > q) {
      const int x = p;
      p = q;
      q = x;
    }
  };
  for (int sweep = 0; sweep < TR_SWEEPS; ++sweep) {
    csync();
    norms();
    if (tid == 0) rot = 0;
    csync();
    for (int t = 0; t < n - 1; ++t) {
      for (int k0 = 0; k0 < mine; k0 += G) {
        const int i = k0 + grp;
        int p = 0, q = r;
        if (i < mine) pair_of(rank + i * CS, t, p, q);
        const bool live = i < mine && q < r;  // q = r: the padding index of an odd r
        double *xp = nullptr, *xq = nullptr;
        double g = 0.0;
        if (live) {
          xp = col(p);
          xq = col(q);
          g = L == 32   ? pair_dot<32>(xp, xq, r, gl, ld)
              : L == 16 ? pair_dot<16>(xp, xq, r, gl, ld)
              : L == 8  ? pair_dot<8>(xp, xq, r, gl, ld)
                        : pair_dot<4>(xp, xq, r, gl, ld);
        }
        for (int o = L >> 1; o; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
        if (gl == 0) gs[grp] = g;
        __syncthreads();
        if (tid < G) {  // the pass's angles, one thread per pair
          const int i2 = k0 + tid;
          double c = 1.0, s = 0.0;
          int p2 = 0, q2 = r;
          if (i2 < mine) pair_of(rank + i2 * CS, t, p2, q2);
          if (i2 < mine && q2 < r) {
            double *ap = nrm(p2), *bp = nrm(q2);
            const double aa = ld(ap), bb = ld(bp), gg = gs[tid];
            double tt;
            if (rotation(aa, bb, gg, tol2, tt)) {
              c = rsqrt(fma(tt, tt, 1.0));
              s = c * tt;
              *ap = fma(-tt, gg, aa);
              *bp = fma(tt, gg, bb);
              rot = 1;
            }
          }
          cc[tid] = c;
          sn[tid] = s;
        }
        __syncthreads();
        const double c = cc[grp], s = sn[grp];
        if (live && s != 0.0) {
#pragma unroll 4
          for (int m = gl; m < r; m += L) {
            const double x = ld(xp + m), y = ld(xq + m);
            xp[m] = c * x - s * y;
            xq[m] = s * x + c * y;
          }
        }
      }
      csync();
    }
    int any = 0;
    for (int q = 0; q < CS; ++q) any |= CS == 1 ? rot : *cg::this_cluster().map_shared_rank(&rot, q);
    if (!any) break;  // the next sweep's first barrier comes before rot is cleared
  }
  csync();
  // ---- singular values (in every CTA), their descending order, the kept columns
  norms();
  csync();
  for (int c = tid; c < r; c += TR_T) beta[c] = sqrt(ld(nrm(c)));
  __syncthreads();
  for (int c = tid; c < r; c += TR_T) {
    const double sc = beta[c];
    int ps = 0;
    for (int d = 0; d < r; ++d) ps += (beta[d] > sc || (beta[d] == sc && d < c)) ? 1 : 0;
    pos[c] = ps;
  }
  if (tid == 0) {
    int kk = 0;
    for (int c = 0; c < r; ++c) kk += beta[c] > eps ? 1 : 0;
    keep = kk;
  }
  __syncthreads();
  for (int c = rank + w * CS; c < r; c += TR_W * CS) {
    const int ps = pos[c];
    if (ps >= keep) continue;
    const double inv = 1.0 / beta[c];
    const double* xc = col(c);
    double* zc = J.Zs + (size_t)ps * r;
    for (int m = l; m < r; m += 32) zc[m] = ld(xc + m) * inv;
  }
  if (tid == 0 && rank == 0) *J.rank = keep;
  csync();  // no CTA leaves while its columns are still read
}

size_t trim_smem(int b, int r, int cs, bool in_smem) {
  const size_t nc = (r + cs - 1) / cs;
  return sizeof(double) * ((size_t)b + r + (in_smem ? nc + nc * (r | 1) : 0)) + sizeof(int) * ((size_t)r + (r & 1));
}

constexpr size_t TRIM_SMEM_MAX = 220 * 1024;

template <int CS, bool SM>
void trim_launch(tlr_ctx* ctx, const TrimDev* dj, int cnt, size_t smem, int b, double eps) {
  auto kern = k_trim<CS, SM>;
  // the limit is the kernel's, for all contexts and threads: always the largest launch's, never this one's
  TLR_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TRIM_SMEM_MAX));
  cudaLaunchConfig_t cf{};
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = CS;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cf.gridDim = dim3((unsigned)(cnt * CS));
  cf.blockDim = dim3(TR_T);
  cf.dynamicSmemBytes = smem;
  cf.stream = ctx->stream;
  cf.attrs = &at;
  cf.numAttrs = 1;
  TLR_SITE_PRE(ctx);
  TLR_CUDA(cudaLaunchKernelEx(&cf, kern, dj, b, eps));
  TLR_LAUNCH_CHECK(ctx);
}

}  // namespace

bool trim_fits(int b) { return trim_smem(b, b, 8, false) <= TRIM_SMEM_MAX; }

void trim_tiles(tlr_ctx* ctx, int b, const std::vector<TrimTile>& tiles, double eps, std::vector<int>& rank,
                std::vector<double*>& Zs, Buf& work) {
  const int nt = (int)tiles.size();
  rank.assign(nt, 0);
  Zs.assign(nt, nullptr);
  if (nt == 0) return;
  TLR_REQUIRE(trim_fits(b), TLR_ERR_LIMIT, "rank trimming: tile size above the shared-memory limit");
  // workspace per tile: W (b r), X (r (r | 1)) and the norms (r), used when they do not fit in shared memory, Zs
  // (r^2); ranks
  int64_t tot = 0;
  std::vector<int64_t> off(nt);
  for (int t = 0; t < nt; ++t) {
    off[t] = tot;
    tot += (int64_t)tiles[t].r * (b + (tiles[t].r | 1) + 1 + (int64_t)tiles[t].r);
  }
  double* ws = work.need<double>((size_t)std::max<int64_t>(tot, 1) + (size_t)(nt + 1) / 2 + 1);
  int* dr = reinterpret_cast<int*>(ws + std::max<int64_t>(tot, 1));
  // Launch groups, highest ranks first.  The tiles of the highest ranks, as many as fill the GPU twice, take a cluster
  // of four (57 tiles of rank 80: 5.5 ms against 7.2 as single CTAs; of rank 56: 3.2 against 3.4, so not below TR_SOLO),
  // or of eight where they are too few for the GPU or four CTAs' shared memory does not hold X; where eight do not
  // either, X lives in global memory.  Further tiles fill the GPU one CTA each (152 of rank 64: 5.2 ms against 8.3 in
  // clusters) unless X does not fit one, in rank classes (so that a group's shared memory, sized by its largest
  // rank, does not hold many small tiles to one CTA per SM).
  static const int cls[] = {8, 16, 24, 32, TR_SOLO, 64, 96, 128, 1 << 30};
  std::vector<int> by_rank;
  for (const TrimTile& t : tiles) by_rank.push_back(t.r);
  std::sort(by_rank.begin(), by_rank.end(), std::greater<int>());
  const size_t most = (size_t)std::max(1, ctx->sm_count / 2);  // clusters of four
  const int top = std::max(TR_SOLO, (int)by_rank.size() > (int)most ? by_rank[most] : 0);
  auto spread = [&](int r) { return r > top || (r > TR_SOLO && trim_smem(b, r, 1, true) > TRIM_SMEM_MAX); };
  int nbig = 0;
  for (const TrimTile& t : tiles) nbig += spread(t.r);
  struct Group {
    int cs = 1;
    bool sm = true;
    int rmax = 0;
    std::vector<TrimDev> js;
  };
  std::map<int, Group> groups;  // the key orders the launches
  for (int t = 0; t < nt; ++t) {
    const int r = tiles[t].r;
    double* W = ws + off[t];
    double* X = W + (size_t)b * r;
    TrimDev d{tiles[t].B, W, X, X + (size_t)r * ((r | 1) + 1), dr + t, r};
    Zs[t] = d.Zs;
    int key, cs = 1;
    bool sm;
    if (spread(r)) {
      cs = nbig * 8 <= ctx->sm_count || trim_smem(b, r, 4, true) > TRIM_SMEM_MAX ? 8 : 4;
      sm = trim_smem(b, r, cs, true) <= TRIM_SMEM_MAX;
      key = !sm ? 0 : cs == 8 ? 1 : 2;
    } else {
      int c = 0;
      while (cls[c] < r) ++c;
      sm = trim_smem(b, r, 1, true) <= TRIM_SMEM_MAX;
      key = sm ? 20 - c : 3;
    }
    Group& g = groups[key];
    g.cs = cs;
    g.sm = sm;
    g.rmax = std::max(g.rmax, r);
    g.js.push_back(d);
  }
  // the clusters on the main stream, the single-CTA tiles beside them on the side stream
  // (joined on every way out: the side stream's launches read the workspace and the job tables)
  struct Side {
    tlr_ctx* ctx;
    cudaStream_t saved;
    bool open = false;
    void join() {
      if (!open) return;
      open = false;
      TLR_CUDA(cudaEventRecord(ctx->ev_join, ctx->side));
      TLR_CUDA(cudaStreamWaitEvent(ctx->main, ctx->ev_join, 0));
    }
    ~Side() {
      ctx->stream = saved;
      if (open && (cudaEventRecord(ctx->ev_join, ctx->side) != cudaSuccess ||
                   cudaStreamWaitEvent(ctx->main, ctx->ev_join, 0) != cudaSuccess))
        cudaStreamSynchronize(ctx->side);
    }
  } side{ctx, ctx->stream};
  if (nbig > 0 && nbig < nt && ctx->side && ctx->stream == ctx->main) {
    TLR_CUDA(cudaEventRecord(ctx->ev_fork, ctx->main));
    TLR_CUDA(cudaStreamWaitEvent(ctx->side, ctx->ev_fork, 0));
    side.open = true;
  }
  for (auto& kv : groups) {
    Group& g = kv.second;
    std::stable_sort(g.js.begin(), g.js.end(), [](const TrimDev& x, const TrimDev& y) { return x.r > y.r; });
    const size_t sm = trim_smem(b, g.rmax, g.cs, g.sm);
    ctx->stream = side.open && g.cs == 1 ? ctx->side : side.saved;
    for (size_t o = 0; o < g.js.size(); o += 65535) {
      const int cnt = (int)std::min<size_t>(65535, g.js.size() - o);
      const TrimDev* dj = static_cast<const TrimDev*>(upload(ctx, g.js.data() + o, sizeof(TrimDev) * cnt));
      if (g.cs == 8 && g.sm) trim_launch<8, true>(ctx, dj, cnt, sm, b, eps);
      else if (g.cs == 8) trim_launch<8, false>(ctx, dj, cnt, sm, b, eps);
      else if (g.cs == 4) trim_launch<4, true>(ctx, dj, cnt, sm, b, eps);
      else if (g.sm) trim_launch<1, true>(ctx, dj, cnt, sm, b, eps);
      else trim_launch<1, false>(ctx, dj, cnt, sm, b, eps);
    }
  }
  ctx->stream = side.saved;
  side.join();
  TLR_CUDA(cudaMemcpyAsync(rank.data(), dr, sizeof(int) * nt, cudaMemcpyDeviceToHost, ctx->stream));
  TLR_CUDA(cudaStreamSynchronize(ctx->stream));
}

// Every off-diagonal tile U_ij V_ij^T of M replaced by Q' B'^T: new block-row and block-column panels
// (ranks never grow), solve plans dropped (they point into the old panels).
void trim_matrix(tlr_ctx* ctx, tlr_mat* M, double eps) {
  const int nb = M->nb, b = M->b;
  std::vector<TrimTile> tl;
  std::vector<std::pair<int, int>> ij;
  for (int i = 0; i < nb; ++i)
    for (int j = 0; j < i; ++j) {
      const int r = M->rank[ix(M, i, j)];
      if (r == 0) continue;
      tl.push_back(TrimTile{Vptr(M, i, j), r});
      ij.push_back({i, j});
    }
  Buf work(ctx);
  std::vector<int> rk;
  std::vector<double*> Zs;
  trim_tiles(ctx, b, tl, eps, rk, Zs, work);
  std::vector<int> nr((size_t)nb * nb, 0);
  for (size_t t = 0; t < tl.size(); ++t) nr[ix(M, ij[t].first, ij[t].second)] = rk[t];
  std::vector<double*> Urow(nb, nullptr), Vcol(nb, nullptr);
  std::vector<int64_t> ulen(nb, 0), vlen(nb, 0), uoff((size_t)nb * nb, 0), voff((size_t)nb * nb, 0);
  for (int i = 0; i < nb; ++i)
    for (int j = 0; j < i; ++j) {
      uoff[ix(M, i, j)] = ulen[i];
      ulen[i] += nr[ix(M, i, j)];
    }
  for (int j = 0; j < nb; ++j)
    for (int i = j + 1; i < nb; ++i) {
      voff[ix(M, i, j)] = vlen[j];
      vlen[j] += nr[ix(M, i, j)];
    }
  for (int i = 0; i < nb; ++i) {
    Urow[i] = static_cast<double*>(dalloc(ctx, sizeof(double) * (size_t)std::max<int64_t>(ulen[i], 1) * b));
    Vcol[i] = static_cast<double*>(dalloc(ctx, sizeof(double) * (size_t)std::max<int64_t>(vlen[i], 1) * b));
  }
  std::vector<GemmJob<double>> jobs;
  for (size_t t = 0; t < tl.size(); ++t) {
    const int i = ij[t].first, j = ij[t].second, r = tl[t].r, q = rk[t];
    if (q == 0) continue;
    jobs.push_back(job<double>(NN, b, q, Uptr(M, i, j), b, Zs[t], r, r, Urow[i] + (size_t)b * uoff[ix(M, i, j)], b,
                               1.0, 0.0));
    jobs.push_back(job<double>(NN, b, q, Vptr(M, i, j), b, Zs[t], r, r, Vcol[j] + (size_t)b * voff[ix(M, i, j)], b,
                               1.0, 0.0));
  }
  gemm<double>(ctx, NN, jobs);
  mat_free_storage(ctx, M);  // also drops the solve plans
  M->Urow = Urow;
  M->Vcol = Vcol;
  M->rank = nr;
  M->uoff = uoff;
  M->voff = voff;
  M->ulen = ulen;
  M->vlen = vlen;
  for (int i = 0; i < nb; ++i) M->ucap[i] = std::max<int64_t>(ulen[i], 1);
}

}  // namespace tlr
