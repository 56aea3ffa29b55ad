// spe.cu -- the spectral positional encoding of Sec. 4.3 computed on the GPU (aecct_spe_table), in
// double precision (GB300 executes two double FMAs per cycle and SM, so operations are counted here):
//
//   tridiag_kernel    the Tanner-graph Laplacian L = D - A reduced to tridiagonal form by Householder
//                     reflections (4/3 T^3 operations, where Jacobi rotations take about 10 sweeps of
//                     6 T^3).  One cooperative launch; the rows stay in shared memory and a step
//                     takes one grid-wide barrier.
//   bisect_kernel     the eigenvalues of the tridiagonal matrix by bisection on Sturm counts.
//   group_kernel      clusters of equal eigenvalues (consecutive gaps <= cluster_tol x
//                     max(1, |lambda|max)).
//   invit_kernel      eigenvectors of the tridiagonal matrix by inverse iteration from random vectors
//                     (for a cluster: vectors that span its invariant subspace).
//   gram_kernel, chol_kernel, trsm_kernel
//                     an orthonormal basis of each cluster's subspace: V <- L^-1 V with V V^T = L L^T,
//                     twice (Cholesky QR, whose second round leaves the orthogonality of a Householder
//                     factorisation).
//   overlap_kernel, polish_kernel
//                     X <- X - (X X^T - I) X / 2: vectors of neighbouring eigenvalues come out of the
//                     inverse iteration orthogonal to eps |L| / gap only.
//   back_kernel       the reflections applied to the eigenvectors.
//   canonical_kernel  per cluster, the canonical basis: Gram-Schmidt of P e_0, P e_1, ... in node
//                     order, P the cluster's projector, skipping residuals of norm <= vanish_tol; in the
//                     coordinates of the cluster's basis, where P e_j is row j of it.  For a large cluster
//                     select_kernel finds the nodes whose residual does not vanish, and their rows take the
//                     same Cholesky QR.
//   basis_kernel      the canonical basis vectors in node coordinates.
//   mhsa_kernel       SPE_j = mean over rows of MHSA(Phi_j W_pe), Phi_j row i = (lambda_i, phi_i[j]):
//                     every projection of row i is lambda_i (w0 W) + phi_i[j] (w1 W) for the rows
//                     w0, w1 of W_pe, so each head's scores are a 2 x 2 bilinear form and
//                     softmax(S) V_j = (P lambda)(w0 Wv) + (P phi[j])(w1 Wv); two passes per query
//                     row (maximum, then the sums).
//
// The long code of 576 nodes (LDPC(384,192)), where Jacobi rotations (about 10 sweeps of 575 steps with
// three grid-wide barriers each) and Gram-Schmidt in node coordinates took 327 ms: tridiagonal form 3.9 ms,
// eigenvalues 0.9, inverse iteration 0.8, the clusters' bases 2.2, polishing 0.6, reflections 1.4, canonical basis 2.6;
// the attention 3.8 (41 with double operations).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <type_traits>
#include <vector>

#include "aecct_internal.h"

namespace aecct {

namespace {

constexpr int kTriThreads = 128;
constexpr int kInvitIters = 3;
constexpr int kSeqGroup = 24;         // clusters up to this size: Gram-Schmidt by one CTA
constexpr double kEps = 2.220446049250313e-16;

// block-wide sum of one double per thread (every thread gets the result)
__device__ double block_sum(double v, double *red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) s += red[w];
  __syncthreads();
  return s;
}

// The sums of a 128-thread CTA: every warp's part, then all of them (after a barrier).  A warp's double
// operation occupies its scheduler's pipe for 64 cycles, so there is one warp to a scheduler, and scalar work
// is done by one warp and handed on through shared memory.
__device__ __forceinline__ void warp_part(double v, double *red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
}
__device__ __forceinline__ double all_parts(const double *red) {
  static_assert(kTriThreads == 128, "four parts");
  return (red[0] + red[1]) + (red[2] + red[3]);
}

// Barrier of a cooperative launch: every CTA adds one to `count` and thread 0 waits until it reaches
// `target`, with `polls` left for all of a launch's barriers (its CTAs are resident together; past the
// limit `status` is set and the launch runs on to its end without waiting).
constexpr int kBarrierPolls = 1 << 25;
__device__ __forceinline__ void grid_barrier(unsigned *count, unsigned target, int &polls, int *status) {
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned seen;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(count) : "memory");
    } while (seen < target && --polls > 0);
    if (seen < target) atomicOr(status, 2);
  }
  __syncthreads();
}

// Householder tridiagonalisation of the Laplacian of H [m][n].  CTA b holds rows b, b + grid, ... in
// shared memory.  Step k: every CTA forms column k of the matrix as updated by the steps before k, its
// reflection v (v[k + 1] = 1, zeros up to k; row k of Vh) and tau, applies the update of step k - 1 to
// its rows and multiplies them by v; after the barrier every CTA forms w = tau A v - (tau/2)(tau v^T A v) v
// for the rank-2 update A - v w^T - w v^T of this step, which it applies in the next pass.  Column k comes
// from row k as it was before the update of step k - 1, which its owner left in rowbuf[k & 1].
// d and e receive the diagonal and the off-diagonal.  Bound by the latency of a step (the barrier, two
// block sums, a square root and two divisions); the vector work that every CTA repeats costs less than
// a second barrier would.
__global__ void __launch_bounds__(kTriThreads) tridiag_kernel(const uint8_t *__restrict__ H, int n, int m, double *Vh,
                                                             double *tau, double *d, double *e, double *rowbuf,
                                                             double *pbuf, unsigned *count, int *status) {
  extern __shared__ double sh[];
  __shared__ double red[2][kTriThreads / 32], s_col[2], s_scal[4];
  const int T = n + m, G = gridDim.x, b = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  double *v = sh, *w = sh + T, *vn = sh + 2 * T, *rows = sh + 3 * T;
  const int R = (T + G - 1) / G;
  unsigned target = G;
  int polls = kBarrierPolls;
  for (int rr = warp; rr < R; rr += kTriThreads / 32) {
    const int i = b + rr * G;
    if (i >= T) continue;
    double deg = 0.0;
    for (int j = lane; j < T; j += 32) {
      double a = 0.0;
      if (i < n && j >= n && H[static_cast<size_t>(j - n) * n + i]) a = -1.0;
      if (i >= n && j < n && H[static_cast<size_t>(i - n) * n + j]) a = -1.0;
      rows[static_cast<size_t>(rr) * T + j] = a;
      deg -= a;
    }
    for (int o = 16; o > 0; o >>= 1) deg += __shfl_xor_sync(0xffffffffu, deg, o);
    __syncwarp();
    if (lane == 0) rows[static_cast<size_t>(rr) * T + i] = deg;
    __syncwarp();
    if (i == 0)
      for (int j = lane; j < T; j += 32) rowbuf[j] = rows[j];
  }
  grid_barrier(count, target, polls, status);
  double wk = 0.0;  // w[k] of step k - 1 (its v[k] is 1)
  for (int k = 0; k + 2 < T; ++k) {
    const double *rb = rowbuf + static_cast<size_t>(k & 1) * T;
    double s = 0.0;
    for (int j = k + tid; j < T; j += kTriThreads) {
      double c = __ldcg(rb + j);
      if (k > 0) c = c - w[j] - wk * v[j];
      vn[j] = c;
      if (j <= k + 1) s_col[j - k] = c;
      else s = fma(c, c, s);
    }
    warp_part(s, red[0]);
    __syncthreads();
    if (warp == 0) {
      const double ss = all_parts(red[0]), alpha = s_col[1];
      double beta = alpha, tk = 0.0, sc = 0.0;
      if (ss > 0.0) {
        // tau = (beta - alpha) / beta and 1 / (alpha - beta) with one division
        beta = -copysign(sqrt(fma(alpha, alpha, ss)), alpha);
        const double diff = alpha - beta, inv = 1.0 / (beta * diff);
        tk = -diff * diff * inv;
        sc = beta * inv;
      }
      if (lane == 0) {
        s_scal[0] = tk, s_scal[1] = sc;
        if (b == 0) d[k] = s_col[0], e[k] = beta, tau[k] = tk;
      }
    }
    __syncthreads();
    const double tk = s_scal[0], sc = s_scal[1];
    for (int j = k + tid; j < T; j += kTriThreads)
      if (j > k) vn[j] = j == k + 1 ? 1.0 : vn[j] * sc;
    __syncthreads();
    for (int rr = warp; rr < R; rr += kTriThreads / 32) {
      const int i = b + rr * G;
      if (i <= k || i >= T) continue;
      double *row = rows + static_cast<size_t>(rr) * T;
      const double vi = k > 0 ? v[i] : 0.0, wi = k > 0 ? w[i] : 0.0;
      double *next = i == k + 1 ? rowbuf + static_cast<size_t>((k + 1) & 1) * T : nullptr;
      double acc = 0.0;
#pragma unroll 2
      for (int j = k + 1 + lane; j < T; j += 32) {
        double a = row[j];
        if (k > 0) row[j] = a = fma(-vi, w[j], fma(-wi, v[j], a));
        if (next) next[j] = a;
        acc = fma(a, vn[j], acc);
      }
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) pbuf[static_cast<size_t>(k & 1) * T + i] = acc;
    }
    target += G;
    grid_barrier(count, target, polls, status);
    const double *pb = pbuf + static_cast<size_t>(k & 1) * T;
    const double p1 = __ldcg(pb + k + 1);
    s = 0.0;
    for (int j = k + 1 + tid; j < T; j += kTriThreads) {
      const double pj = tk * __ldcg(pb + j);
      w[j] = pj;
      v[j] = vn[j];
      s = fma(pj, vn[j], s);
    }
    warp_part(s, red[1]);
    __syncthreads();
    if (tid == 0) s_scal[2] = -0.5 * tk * all_parts(red[1]);
    __syncthreads();
    const double kk = s_scal[2];
    for (int j = k + 1 + tid; j < T; j += kTriThreads) {
      w[j] = fma(kk, vn[j], w[j]);
      if (b == k % G) Vh[static_cast<size_t>(k) * T + j] = vn[j];
    }
    wk = tk * p1 + kk;
  }
  __syncthreads();
  // the last 2 x 2 block: row T - 2 as of the step before the last update, and the owner's row T - 1
  const int q = T - 2;
  if (b == 0 && tid == 0) {
    const double *rb = rowbuf + static_cast<size_t>(q & 1) * T;
    for (int j = q; j < T; ++j) {
      const double c = fma(-v[q], w[j], fma(-w[q], v[j], __ldcg(rb + j)));
      if (j == q) d[q] = c;
      else e[q] = c;
    }
  }
  if (b == (T - 1) % G && tid == 0)
    d[T - 1] = fma(-2.0 * v[T - 1], w[T - 1], rows[static_cast<size_t>((T - 1) / G) * T + T - 1]);
}

// Eigenvalue i (ascending) by bisection into 33 parts a round, a warp an eigenvalue: the number of
// eigenvalues below x is the number of sign changes in the Sturm sequence
// p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2} (a zero counts as the sign opposite to its predecessor's),
// rescaled by a power of two every 8 steps.  The recurrence without divisions takes three double
// operations a step; a warp's double operation occupies its scheduler's pipe for 64 cycles whatever its
// lanes do, so more parts a round on more warps (up to four to an SM) mean fewer rounds for nothing.
// e^2 is kept above (1e-18 |L|)^2, far below rounding, so that a split matrix does not end the sequence in
// zeros.
__global__ void __launch_bounds__(32) bisect_kernel(const double *__restrict__ d, const double *__restrict__ e, int T,
                                                   double *lam) {
  extern __shared__ double2 de[];  // d_i and e_{i-1}^2
  const int lane = threadIdx.x, i = blockIdx.x;
  double lo = INFINITY, hi = -INFINITY;
  for (int j = lane; j < T; j += 32) {
    const double r = (j > 0 ? fabs(e[j - 1]) : 0.0) + (j + 1 < T ? fabs(e[j]) : 0.0);
    lo = fmin(lo, d[j] - r), hi = fmax(hi, d[j] + r);
  }
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  const double nt = fmax(fabs(lo), fabs(hi));
  for (int j = lane; j < T; j += 32)
    de[j] = make_double2(d[j], j > 0 ? fmax(e[j - 1] * e[j - 1], 1e-36 * nt * nt) : 0.0);
  __syncwarp();
  lo -= 8.0 * kEps * nt * T, hi += 8.0 * kEps * nt * T;
  for (int round = 0; round < 12; ++round) {  // 33^12 > 2^60
    const double h = (hi - lo) / 33.0, x = fma(h, static_cast<double>(lane + 1), lo);
    double p0 = 1.0, p1 = de[0].x - x;
    int sign = p1 <= 0.0 ? 1 : 0, cnt = sign;  // sign of the last term: 1 negative
    auto step = [&](const double2 &c) {
      const double p2 = fma(c.x - x, p1, -c.y * p0);
      p0 = p1, p1 = p2;
      const int hw = __double2hiint(p2);
      const int now = ((hw << 1) | __double2loint(p2)) == 0 ? 1 - sign : static_cast<int>(static_cast<unsigned>(hw) >> 31);
      cnt += now ^ sign;
      sign = now;
    };
    int j = 1;
#pragma unroll 1
    for (; j + 8 <= T; j += 8) {
      double2 c[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) c[u] = de[j + u];
#pragma unroll
      for (int u = 0; u < 8; ++u) step(c[u]);
      const int ex = max(__double2hiint(p0) & 0x7FF00000, __double2hiint(p1) & 0x7FF00000);
      const double f = __hiloint2double(ex == 0 ? 0x5FF00000 : 0x7FE00000 - ex, 0);  // 2^-(exponent)
      p0 *= f, p1 *= f;
    }
    for (; j < T; ++j) step(de[j]);
    const uint32_t above = __ballot_sync(0xffffffffu, cnt > i);
    const int f = above ? __ffs(above) - 1 : 32;  // the first point with more than i eigenvalues below it
    const double base = lo;
    if (f < 32) hi = fma(h, static_cast<double>(f + 1), base);
    if (f > 0) lo = fma(h, static_cast<double>(f), base);
  }
  if (lane == 0) lam[i] = 0.5 * (lo + hi);
}

// ascending eigenvalues (equal ones can come out of the bisection a rounding apart in either order) and
// their clusters: gs[i] the first index of i's cluster, gn[i] its size
__global__ void __launch_bounds__(kSpeMaxTokens) group_kernel(double *lam, int T, double cluster_tol, int *gs, int *gn) {
  __shared__ double x[kSpeMaxTokens];
  __shared__ int first[kSpeMaxTokens + 1];
  const int i = threadIdx.x;
  if (i < T) x[i] = lam[i];
  __syncthreads();
  for (int o = 1; o < T; o <<= 1) {  // running maximum
    const double y = i < T && i >= o ? fmax(x[i], x[i - o]) : (i < T ? x[i] : 0.0);
    __syncthreads();
    if (i < T) x[i] = y;
    __syncthreads();
  }
  const double tol = cluster_tol * fmax(1.0, fmax(fabs(x[0]), fabs(x[T - 1])));
  if (i < T) {
    lam[i] = x[i];
    first[i] = i == 0 || x[i] - x[i - 1] > tol;
  }
  if (i == 0) first[T] = 1;
  __syncthreads();
  if (i >= T) return;
  int a = i, z = i + 1;
  while (!first[a]) --a;
  while (!first[z]) ++z;
  gs[i] = a;
  gn[i] = z - a;
}

// Inverse iteration on the tridiagonal matrix, a thread per eigenvector (nv to a CTA, their factors in
// shared memory): (T - s I) = P L U with row exchanges, then kInvitIters solves from a random vector.  A
// single eigenvalue is its own shift s; a cluster's shift lies 1e-10 |L| beside it, so that every vector
// of its subspace is amplified alike and the random starts stay independent.  Row i of Z is vector i.
__global__ void invit_kernel(const double *__restrict__ d, const double *__restrict__ e, const double *__restrict__ lam,
                             const int *__restrict__ gn, int T, int nv, uint32_t seed, double *Z) {
  extern __shared__ double sh[];
  const int t = threadIdx.x, vec = blockIdx.x * nv + t;
  if (t >= nv || vec >= T) return;
  double *u0 = sh, *u1 = u0 + static_cast<size_t>(T) * nv, *u2 = u1 + static_cast<size_t>(T) * nv,
         *lf = u2 + static_cast<size_t>(T) * nv, *x = lf + static_cast<size_t>(T) * nv;
  uint8_t *sw = reinterpret_cast<uint8_t *>(x + static_cast<size_t>(T) * nv);
  const double nt = fmax(fmax(fabs(lam[0]), fabs(lam[T - 1])), 1e-290);
  const double tiny = 1e-2 * kEps * nt, s = lam[vec] + (gn[vec] > 1 ? 1e-10 * nt : 0.0);
  double a = d[0] - s, b = e[0];
  for (int i = 0; i + 1 < T; ++i) {
    const double c = e[i], dn = d[i + 1] - s, en = i + 2 < T ? e[i + 1] : 0.0;
    const bool swap = fabs(c) > fabs(a);
    double piv = swap ? c : a;
    if (fabs(piv) < tiny) piv = tiny;
    const double r1 = swap ? dn : b, r2 = swap ? en : 0.0, rp = 1.0 / piv, l = (swap ? a : c) * rp;
    u0[i * nv + t] = rp, u1[i * nv + t] = r1, u2[i * nv + t] = r2, lf[i * nv + t] = l;
    sw[i * nv + t] = swap;
    a = fma(-l, r1, swap ? b : dn);
    b = fma(-l, r2, swap ? 0.0 : en);
  }
  u0[(T - 1) * nv + t] = 1.0 / (fabs(a) < tiny ? tiny : a);
  uint32_t h = seed + 2654435761u * static_cast<uint32_t>(vec + 1);
  for (int i = 0; i < T; ++i) {
    h ^= h << 13, h ^= h >> 17, h ^= h << 5;
    x[i * nv + t] = static_cast<double>(static_cast<int32_t>(h)) * 4.656612873077393e-10;
  }
  double norm = 1.0;
  for (int it = 0; it < kInvitIters; ++it) {
    double y = x[t] * norm;
    for (int i = 0; i + 1 < T; ++i) {
      const double yn = x[(i + 1) * nv + t] * norm;
      const bool swap = sw[i * nv + t] != 0;
      const double p = swap ? yn : y;
      x[i * nv + t] = p;
      y = fma(-lf[i * nv + t], p, swap ? y : yn);
    }
    double z1 = y * u0[(T - 1) * nv + t], z2 = 0.0, ss = z1 * z1;
    x[(T - 1) * nv + t] = z1;
    for (int i = T - 2; i >= 0; --i) {
      const double z = fma(-u1[i * nv + t], z1, fma(-u2[i * nv + t], z2, x[i * nv + t])) * u0[i * nv + t];
      x[i * nv + t] = z;
      ss = fma(z, z, ss);
      z2 = z1, z1 = z;
    }
    norm = 1.0 / sqrt(ss);
  }
  for (int i = 0; i < T; ++i) Z[static_cast<size_t>(vec) * T + i] = x[i * nv + t] * norm;
}

// length of the vectors of a cluster of size r: T (rows of the eigenvector array) or r (coordinates)
__device__ __forceinline__ int vec_len(int r, int T, int coords) { return coords ? r : T; }

// Gm[a][b] = row a of V . row b of V for a >= b of one cluster larger than rmin (32 x 32 tiles)
__global__ void __launch_bounds__(256) gram_kernel(const double *__restrict__ V, const int *__restrict__ gs,
                                                  const int *__restrict__ gn, int T, int rmin, int coords, double *Gm) {
  __shared__ double sa[32][33], sb[32][33];
  const int a0 = blockIdx.y * 32, b0 = blockIdx.x * 32;
  if (b0 > a0) return;
  int len = 0;
  for (int a = a0; a < min(a0 + 32, T); ++a)
    if (gn[a] > rmin && gs[a] <= min(b0 + 31, a)) len = max(len, vec_len(gn[a], T, coords));
  if (len == 0) return;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  for (int c0 = 0; c0 < len; c0 += 32) {
    for (int it = threadIdx.x; it < 1024; it += 256) {
      const int rr = it >> 5, c = c0 + (it & 31), a = a0 + rr, b = b0 + rr;
      sa[rr][it & 31] = a < T && c < vec_len(gn[a], T, coords) ? V[static_cast<size_t>(a) * T + c] : 0.0;
      sb[rr][it & 31] = b < T && c < vec_len(gn[b], T, coords) ? V[static_cast<size_t>(b) * T + c] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int c = 0; c < 32; ++c) {
      const double x0 = sa[ty][c], x1 = sa[ty + 16][c], y0 = sb[tx][c], y1 = sb[tx + 16][c];
      acc[0][0] = fma(x0, y0, acc[0][0]), acc[0][1] = fma(x0, y1, acc[0][1]);
      acc[1][0] = fma(x1, y0, acc[1][0]), acc[1][1] = fma(x1, y1, acc[1][1]);
    }
    __syncthreads();
  }
  for (int i = 0; i < 2; ++i)
    for (int j = 0; j < 2; ++j) {
      const int a = a0 + ty + 16 * i, b = b0 + tx + 16 * j;
      if (a < T && b <= a && gs[a] <= b) Gm[static_cast<size_t>(a) * T + b] = acc[i][j];
    }
}

// In place, L of Gm = L L^T of every cluster larger than rmin (one CTA each, its lower triangle in shared
// memory where it fits).  A squared pivot of at most `thr` marks the cluster in `bad`.  Columns go in
// panels of 16: one warp factors the panel's diagonal block, every thread a row of the rest of the
// panel, and the trailing triangle takes the panel's update in one pass.
constexpr int kCholThreads = 512;
constexpr int kCholPanel = 16;
// rows of a triangle in shared memory: 187,488 bytes (up to 237 would fit; larger clusters' Cholesky works in global memory
// and their node choice one by one, 690 nodes with a cluster of 230 take 54 ms, 576 with 192 take 17)
constexpr int kCholShared = 216;
constexpr size_t kCholSmem = sizeof(double) * kCholShared * (kCholShared + 1) / 2;
__global__ void __launch_bounds__(kCholThreads) chol_kernel(double *Gm, const int *__restrict__ gs,
                                                            const int *__restrict__ gn, int T, int rmin, double thr,
                                                            int *bad) {
  extern __shared__ double tri[];
  __shared__ double diag[kCholPanel][kCholPanel + 1], dinv[kCholPanel];
  const int g0 = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (gs[g0] != g0 || gn[g0] <= rmin) return;
  const int r = gn[g0];
  const bool packed = r <= kCholShared;
  auto glob = [&](int a, int b) -> double * { return Gm + static_cast<size_t>(g0 + a) * T + g0 + b; };
  auto at = [&](int a, int b) -> double * { return packed ? tri + a * (a + 1) / 2 + b : glob(a, b); };
  if (packed)
    for (int a = warp; a < r; a += kCholThreads / 32)
      for (int b = lane; b <= a; b += 32) *at(a, b) = *glob(a, b);
  __syncthreads();
  bool ok = true;
  for (int j0 = 0; j0 < r; j0 += kCholPanel) {
    const int nb = min(kCholPanel, r - j0);
    if (warp == 0) {
      // lane a holds row j0 + a of the diagonal block
      double x[kCholPanel];
#pragma unroll
      for (int c = 0; c < kCholPanel; ++c) x[c] = lane < nb && c <= lane ? *at(j0 + lane, j0 + c) : (c == lane ? 1.0 : 0.0);
#pragma unroll
      for (int c = 0; c < kCholPanel; ++c) {
        const double piv = __shfl_sync(0xffffffffu, x[c], c);
        if (c < nb && !(piv > thr)) ok = false;
        const double inv = rsqrt(fmax(piv, 1e-300)), root = fmax(piv, 1e-300) * inv;
        x[c] = lane == c ? root : x[c] * inv;
        if (lane == c) dinv[c] = inv;
#pragma unroll
        for (int k = c + 1; k < kCholPanel; ++k) {
          const double lk = __shfl_sync(0xffffffffu, x[c], k);
          if (lane >= k) x[k] = fma(-x[c], lk, x[k]);
        }
      }
#pragma unroll
      for (int c = 0; c < kCholPanel; ++c)
        if (lane < nb && c <= lane) diag[lane][c] = *at(j0 + lane, j0 + c) = x[c];
    }
    __syncthreads();
    for (int a = j0 + kCholPanel + tid; a < r; a += kCholThreads) {  // (a full panel: nb = kCholPanel)
      double x[kCholPanel];
#pragma unroll
      for (int c = 0; c < kCholPanel; ++c) x[c] = *at(a, j0 + c);
#pragma unroll
      for (int c = 0; c < kCholPanel; ++c) {
        x[c] *= dinv[c];
#pragma unroll
        for (int k = c + 1; k < kCholPanel; ++k) x[k] = fma(-x[c], diag[k][c], x[k]);
      }
#pragma unroll
      for (int c = 0; c < kCholPanel; ++c) *at(a, j0 + c) = x[c];
    }
    __syncthreads();
    for (int a = j0 + kCholPanel + warp; a < r; a += kCholThreads / 32) {
      double la[kCholPanel];
#pragma unroll
      for (int c = 0; c < kCholPanel; ++c) la[c] = *at(a, j0 + c);
      for (int b = j0 + kCholPanel + lane; b <= a; b += 32) {
        double x0 = *at(a, b), x1 = 0.0;
#pragma unroll
        for (int c = 0; c < kCholPanel; c += 2) {
          x0 = fma(-la[c], *at(b, j0 + c), x0);
          x1 = fma(-la[c + 1], *at(b, j0 + c + 1), x1);
        }
        *at(a, b) = x0 + x1;
      }
    }
    __syncthreads();
  }
  if (packed)
    for (int a = warp; a < r; a += kCholThreads / 32)
      for (int b = lane; b <= a; b += 32) *glob(a, b) = *at(a, b);
  if (tid == 0 && !ok) bad[g0] = 1;
}

// P[a][b] = sum_c X[g0 + c][a] X[g0 + c][b] of every cluster larger than rmin over its first S nodes (32 x 32
// tiles, a >= b), stored S to a row at the cluster's rows of Pm
__host__ __device__ __forceinline__ int select_nodes(int r, int T) {
  const int s = r + r / 8 + 24;
  return s < T ? (s < kCholShared ? s : kCholShared) : (T < kCholShared ? T : kCholShared);
}
__global__ void __launch_bounds__(256) proj_kernel(const double *__restrict__ X, const int *__restrict__ gs,
                                                  const int *__restrict__ gn, int T, int rmin, double *Pm) {
  const int g0 = blockIdx.z, a0 = blockIdx.y * 32, b0 = blockIdx.x * 32;
  if (gs[g0] != g0 || gn[g0] <= rmin || b0 > a0) return;
  const int r = gn[g0], S = select_nodes(r, T);
  if (r > S || S * S > r * T || a0 >= S) return;
  __shared__ double sa[32][33], sb[32][33];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  for (int c0 = 0; c0 < r; c0 += 32) {
    for (int it = threadIdx.x; it < 1024; it += 256) {
      const int c = c0 + (it >> 5), u = it & 31;
      sa[it >> 5][u] = c < r && a0 + u < S ? X[static_cast<size_t>(g0 + c) * T + a0 + u] : 0.0;
      sb[it >> 5][u] = c < r && b0 + u < S ? X[static_cast<size_t>(g0 + c) * T + b0 + u] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int c = 0; c < 32; ++c) {
      const double x0 = sa[c][ty], x1 = sa[c][ty + 16], y0 = sb[c][tx], y1 = sb[c][tx + 16];
      acc[0][0] = fma(x0, y0, acc[0][0]), acc[0][1] = fma(x0, y1, acc[0][1]);
      acc[1][0] = fma(x1, y0, acc[1][0]), acc[1][1] = fma(x1, y1, acc[1][1]);
    }
    __syncthreads();
  }
  double *P = Pm + static_cast<size_t>(g0) * T;
  for (int i = 0; i < 2; ++i)
    for (int j = 0; j < 2; ++j) {
      const int a = a0 + ty + 16 * i, b = b0 + tx + 16 * j;
      if (a < S && b <= a) P[static_cast<size_t>(a) * S + b] = acc[i][j];
    }
}

// The nodes of each cluster larger than kSeqGroup that give its canonical basis: the first r nodes, in
// order, whose P e_j is independent of those chosen before (codes have exactly dependent ones).  A
// right-looking Cholesky of P (over the nodes 0 .. S - 1) that leaves a node out where the
// squared residual is below 1e-14; one between that and 1e-8, where this arithmetic cannot tell, or too few
// nodes, mark the cluster for the one-by-one kernel.  node[g0 + a]: the a-th node chosen.
__global__ void __launch_bounds__(kCholThreads) select_kernel(const double *__restrict__ V, const double *__restrict__ Pm, const int *__restrict__ gs,
                                                              const int *__restrict__ gn, int T, int rmin, int *node,
                                                              int *bad) {
  extern __shared__ double tri[];
  __shared__ double col[kCholShared];
  const int g0 = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (gs[g0] != g0 || gn[g0] <= rmin) return;
  const int r = gn[g0], S = select_nodes(r, T);
  if (r > S) {
    if (tid == 0) bad[g0] = 1;
    return;
  }
  const bool ready = S * S <= r * T;  // proj_kernel has formed P
  if (ready) {
    const double *P = Pm + static_cast<size_t>(g0) * T;
    for (int a = warp; a < S; a += kCholThreads / 32)
      for (int b = lane; b <= a; b += 32) tri[a * (a + 1) / 2 + b] = P[static_cast<size_t>(a) * S + b];
  }
  // else here, 4 x 4 outputs a thread
  const double *X = V + static_cast<size_t>(g0) * T;
  const int nt = (S + 3) / 4, ntri = nt * (nt + 1) / 2;
  for (int t = ready ? ntri : tid; t < ntri; t += kCholThreads) {
    int ta = static_cast<int>((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
    while ((ta + 1) * (ta + 2) / 2 <= t) ++ta;
    while (ta * (ta + 1) / 2 > t) --ta;
    const int a0 = 4 * ta, b0 = 4 * (t - ta * (ta + 1) / 2);
    double acc[4][4] = {};
    for (int c = 0; c < r; ++c) {
      double xa[4], xb[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        xa[u] = a0 + u < S ? X[static_cast<size_t>(c) * T + a0 + u] : 0.0;
        xb[u] = b0 + u < S ? X[static_cast<size_t>(c) * T + b0 + u] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[u][q] = fma(xa[u], xb[q], acc[u][q]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (a0 + u < S && b0 + q <= a0 + u) tri[(a0 + u) * (a0 + u + 1) / 2 + b0 + q] = acc[u][q];
  }
  __syncthreads();
  int got = 0;
  bool ok = true;
  for (int j = 0; j < S && got < r; ++j) {
    const double piv = tri[j * (j + 1) / 2 + j];
    if (!(piv > 1e-14)) continue;
    if (!(piv > 1e-8)) ok = false;
    if (tid == 0) node[g0 + got] = j;
    ++got;
    const double inv = rsqrt(piv);
    for (int a = j + 1 + tid; a < S; a += kCholThreads) col[a] = tri[a * (a + 1) / 2 + j] * inv;
    __syncthreads();
    for (int a = j + 1 + warp; a < S; a += kCholThreads / 32) {
      const double ca = col[a];
      for (int b = j + 1 + lane; b <= a; b += 32) tri[a * (a + 1) / 2 + b] = fma(-ca, col[b], tri[a * (a + 1) / 2 + b]);
    }
    __syncthreads();
  }
  if (tid == 0 && (!ok || got < r)) bad[g0] = 1;
}

// V <- L^-1 V for the rows of every cluster larger than rmin: 16 columns of V to a CTA, in blocks of 16
// rows (the rows before the block subtracted by all threads, one row and column each, then the block's
// 16 x 16 triangle one row after another)
__global__ void __launch_bounds__(256) trsm_kernel(const double *__restrict__ Gm, double *V, const int *__restrict__ gs,
                                                  const int *__restrict__ gn, int T, int rmin, int coords) {
  __shared__ double lb[16][17], xb[16][17], rhs[16][17];
  const int g0 = blockIdx.y, i0 = blockIdx.x * 16, c = threadIdx.x & 15, a = threadIdx.x >> 4;
  if (gs[g0] != g0 || gn[g0] <= rmin) return;
  const int r = gn[g0], len = vec_len(r, T, coords);
  if (i0 >= len) return;
  const bool in = i0 + c < len;
  double *x = V + static_cast<size_t>(g0) * T + i0 + c;
  for (int a0 = 0; a0 < r; a0 += 16) {
    const bool row = a0 + a < r;
    const double *la = Gm + static_cast<size_t>(g0 + a0 + a) * T + g0;
    double s0 = row && in ? x[static_cast<size_t>(a0 + a) * T] : 0.0, s1 = 0.0;
    for (int b0 = 0; b0 < a0; b0 += 16) {
      lb[a][c] = row ? la[b0 + c] : 0.0;
      xb[a][c] = in ? x[static_cast<size_t>(b0 + a) * T] : 0.0;
      __syncthreads();
#pragma unroll
      for (int b = 0; b < 16; b += 2) {
        s0 = fma(-lb[a][b], xb[b][c], s0);
        s1 = fma(-lb[a][b + 1], xb[b + 1][c], s1);
      }
      __syncthreads();
    }
    lb[a][c] = row && a0 + c < r && c <= a ? la[a0 + c] : 0.0;
    rhs[a][c] = s0 + s1;
    __syncthreads();
    if (threadIdx.x < 16) {  // thread c: column c of the block
      double y[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) y[k] = rhs[k][c];
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        y[k] = a0 + k < r ? y[k] / lb[k][k] : 0.0;
#pragma unroll
        for (int q = k + 1; q < 16; ++q) y[q] = fma(-lb[q][k], y[k], y[q]);
      }
#pragma unroll
      for (int k = 0; k < 16; ++k) rhs[k][c] = y[k];
    }
    __syncthreads();
    if (row && in) x[static_cast<size_t>(a0 + a) * T] = rhs[a][c];
    __syncthreads();
  }
}

// E = X X^T - I (32 x 32 tiles, the lower ones computed) and, per tile, whether an entry of it exceeds kOverlapSkip.
// Inverse iteration leaves vectors of eigenvalues a gap apart with a product of about eps |L| / gap (9e-12 for
// Polar(64,32), whose closest ones are 5e-6 apart), which nothing after it removes.  `again` is set where
// an entry is so large that its square is not yet rounding; with `go` null or set the tiles are computed.
constexpr double kOverlapSkip = 4.0 * kEps, kOverlapAgain = 1e-9;
__global__ void __launch_bounds__(256) overlap_kernel(const double *__restrict__ X, int T, const int *go, double *E, int *busy,
                                                     int *again) {
  __shared__ double sa[32][33], sb[32][33];
  const int a0 = blockIdx.y * 32, b0 = blockIdx.x * 32, tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  if (b0 > a0 || (go && !*go)) return;
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  for (int c0 = 0; c0 < T; c0 += 32) {
    for (int it = threadIdx.x; it < 1024; it += 256) {
      const int rr = it >> 5, c = c0 + (it & 31);
      sa[rr][it & 31] = a0 + rr < T && c < T ? X[static_cast<size_t>(a0 + rr) * T + c] : 0.0;
      sb[rr][it & 31] = b0 + rr < T && c < T ? X[static_cast<size_t>(b0 + rr) * T + c] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int c = 0; c < 32; ++c) {
      const double x0 = sa[ty][c], x1 = sa[ty + 16][c], y0 = sb[tx][c], y1 = sb[tx + 16][c];
      acc[0][0] = fma(x0, y0, acc[0][0]), acc[0][1] = fma(x0, y1, acc[0][1]);
      acc[1][0] = fma(x1, y0, acc[1][0]), acc[1][1] = fma(x1, y1, acc[1][1]);
    }
    __syncthreads();
  }
  double top = 0.0;
  for (int i = 0; i < 2; ++i)
    for (int j = 0; j < 2; ++j) {
      const int a = a0 + ty + 16 * i, b = b0 + tx + 16 * j;
      if (a >= T || b > a) continue;
      const double e = acc[i][j] - (a == b ? 1.0 : 0.0);
      E[static_cast<size_t>(a) * T + b] = E[static_cast<size_t>(b) * T + a] = e;
      top = fmax(top, fabs(e));
    }
  const int some = __syncthreads_or(top > kOverlapSkip), much = __syncthreads_or(top > kOverlapAgain);
  if (threadIdx.x == 0) {
    busy[blockIdx.y * gridDim.x + blockIdx.x] = busy[blockIdx.x * gridDim.x + blockIdx.y] = some;
    if (much) *again = 1;
  }
}

// Y = X - E X / 2, from the tiles of E that are marked (all of them as they are with `go` unset)
__global__ void __launch_bounds__(256) polish_kernel(const double *__restrict__ X, const double *__restrict__ E,
                                                    const int *__restrict__ busy, int T, const int *go, double *Y) {
  __shared__ double se[32][33], sx[32][33];
  const int a0 = blockIdx.y * 32, c0 = blockIdx.x * 32, tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  const bool on = !go || *go;
  for (int b0 = 0; on && b0 < T; b0 += 32) {
    if (!busy[blockIdx.y * gridDim.y + b0 / 32]) continue;
    for (int it = threadIdx.x; it < 1024; it += 256) {
      const int rr = it >> 5, u = it & 31;
      se[rr][u] = a0 + rr < T && b0 + u < T ? E[static_cast<size_t>(a0 + rr) * T + b0 + u] : 0.0;
      sx[rr][u] = b0 + rr < T && c0 + u < T ? X[static_cast<size_t>(b0 + rr) * T + c0 + u] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int b = 0; b < 32; ++b) {
      const double x0 = se[ty][b], x1 = se[ty + 16][b], y0 = sx[b][tx], y1 = sx[b][tx + 16];
      acc[0][0] = fma(x0, y0, acc[0][0]), acc[0][1] = fma(x0, y1, acc[0][1]);
      acc[1][0] = fma(x1, y0, acc[1][0]), acc[1][1] = fma(x1, y1, acc[1][1]);
    }
    __syncthreads();
  }
  for (int i = 0; i < 2; ++i)
    for (int j = 0; j < 2; ++j) {
      const int a = a0 + ty + 16 * i, c = c0 + tx + 16 * j;
      if (a < T && c < T) Y[static_cast<size_t>(a) * T + c] = fma(-0.5, acc[i][j], X[static_cast<size_t>(a) * T + c]);
    }
}

// g[k] = v_k . v_{k-1} for the pairs of reflections that back_kernel applies together
__global__ void __launch_bounds__(32) pair_kernel(const double *__restrict__ Vh, int T, double *g) {
  const int k = blockIdx.x + 1;
  double s = 0.0;
  for (int j = k + 1 + threadIdx.x; j < T; j += 32)
    s = fma(Vh[static_cast<size_t>(k) * T + j], Vh[static_cast<size_t>(k - 1) * T + j], s);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (threadIdx.x == 0) g[k] = s;
}

// Z <- (H_0 H_1 ... H_{T-3}) Z for every row of Z: a warp per vector, its elements j = lane + 32 u in
// registers (NE per lane), two reflections at a time: z + t_k v_k + t_{k-1} v_{k-1} with
// t_k = -tau_k (v_k . z) and t_{k-1} = -tau_{k-1} (v_{k-1} . z + t_k g_k).  Bound by the latency of the
// sums; the vectors of the next two reflections are loaded while the current ones are applied.
template <int NE>
__global__ void __launch_bounds__(64) back_kernel(const double *__restrict__ Vh, const double *__restrict__ tau,
                                                 const double *__restrict__ g, int T, double *Z) {
  const int vec = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (vec >= T) return;
  double z[NE], va[NE], vb[NE], ta = 0.0, tb = 0.0, gg = 0.0;
#pragma unroll
  for (int u = 0; u < NE; ++u) z[u] = lane + 32 * u < T ? Z[static_cast<size_t>(vec) * T + lane + 32 * u] : 0.0;
  auto load = [&](int k) {  // reflections k and k - 1 (none below 0)
#pragma unroll
    for (int u = 0; u < NE; ++u) {
      const int j = lane + 32 * u;
      va[u] = k >= 0 && j > k && j < T ? __ldg(Vh + static_cast<size_t>(k) * T + j) : 0.0;
      vb[u] = k >= 1 && j > k - 1 && j < T ? __ldg(Vh + static_cast<size_t>(k - 1) * T + j) : 0.0;
    }
    ta = k >= 0 ? -__ldg(tau + k) : 0.0;
    tb = k >= 1 ? -__ldg(tau + k - 1) : 0.0;
    gg = k >= 1 ? __ldg(g + k) : 0.0;
  };
  load(T - 3);
  for (int k = T - 3; k >= 0; k -= 2) {
    double ca[NE], cb[NE], sa[3] = {0.0, 0.0, 0.0}, sb[3] = {0.0, 0.0, 0.0};
    const double tak = ta, tbk = tb, gk = gg;
#pragma unroll
    for (int u = 0; u < NE; ++u) ca[u] = va[u], cb[u] = vb[u];
    load(k - 2);
    const int u0 = k >> 5;  // elements up to k - 1 of both vectors are zero
#pragma unroll
    for (int u = 0; u < NE; ++u)
      if (u >= u0) sa[u % 3] = fma(ca[u], z[u], sa[u % 3]), sb[u % 3] = fma(cb[u], z[u], sb[u % 3]);
    double a = (sa[0] + sa[1]) + sa[2], c = (sb[0] + sb[1]) + sb[2];
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    const double t0 = tak * a, t1 = tbk * fma(t0, gk, c);
#pragma unroll
    for (int u = 0; u < NE; ++u)
      if (u >= u0) z[u] = fma(t1, cb[u], fma(t0, ca[u], z[u]));
  }
#pragma unroll
  for (int u = 0; u < NE; ++u)
    if (lane + 32 * u < T) Z[static_cast<size_t>(vec) * T + lane + 32 * u] = z[u];
}

// The chosen nodes' rows of a large cluster's basis, in its coordinates: Q[g0 + a][c]
__global__ void coords_kernel(const double *__restrict__ X, const int *__restrict__ gs, const int *__restrict__ gn,
                              const int *__restrict__ node, const int *__restrict__ bad, int T, int rmin, double *Q) {
  const int row = blockIdx.x;
  if (gn[row] <= rmin || bad[gs[row]]) return;
  const int g0 = gs[row], a = node[row];
  for (int c = threadIdx.x; c < gn[row]; c += blockDim.x)
    Q[static_cast<size_t>(row) * T + c] = X[static_cast<size_t>(g0 + c) * T + a];
}

// Canonical basis in coordinates, Q[g0 + a][c], of every cluster up to kSeqGroup and of the larger ones
// marked in `bad`: Gram-Schmidt of the rows P e_0, P e_1, ... one by one, each
// projected twice ("twice is enough"), skipping residuals of norm <= vanish_tol.  One CTA per cluster.
constexpr int kSeqThreads = 128;
__global__ void __launch_bounds__(kSeqThreads) canonical_kernel(const double *__restrict__ X, const int *__restrict__ gs,
                                                                const int *__restrict__ gn, int T, double vanish_tol,
                                                                const int *__restrict__ bad, double *Q, int *status) {
  __shared__ double red[kSeqThreads / 32], w[kSpeMaxTokens], dots[kSpeMaxTokens];
  const int g0 = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (gs[g0] != g0) return;
  const int r = gn[g0];
  if (r > kSeqGroup && !bad[g0]) return;
  int got = 0;
  for (int node = 0; node < T && got < r; ++node) {
    for (int c = tid; c < r; c += kSeqThreads) w[c] = X[static_cast<size_t>(g0 + c) * T + node];
    __syncthreads();
    for (int pass = 0; pass < 2 && got > 0; ++pass) {
      for (int b = warp; b < got; b += kSeqThreads / 32) {
        double s = 0.0;
        for (int c = lane; c < r; c += 32) s = fma(Q[static_cast<size_t>(g0 + b) * T + c], w[c], s);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) dots[b] = s;
      }
      __syncthreads();
      for (int c = tid; c < r; c += kSeqThreads) {
        double s = w[c];
        for (int b = 0; b < got; ++b) s = fma(-dots[b], Q[static_cast<size_t>(g0 + b) * T + c], s);
        w[c] = s;
      }
      __syncthreads();
    }
    double nv = 0.0;
    for (int c = tid; c < r; c += kSeqThreads) nv = fma(w[c], w[c], nv);
    nv = sqrt(block_sum(nv, red));
    if (nv > vanish_tol) {
      for (int c = tid; c < r; c += kSeqThreads) Q[static_cast<size_t>(g0 + got) * T + c] = w[c] / nv;
      ++got;
    }
    __syncthreads();
  }
  if (got != r && tid == 0) atomicOr(status, 1);
}

// the canonical vectors in node coordinates: U[node][i] = sum_c X[g0 + c][node] Q[i][c]
__global__ void __launch_bounds__(256) basis_kernel(const double *__restrict__ X, const double *__restrict__ Q,
                                                   const int *__restrict__ gs, const int *__restrict__ gn, int T,
                                                   double *U) {
  __shared__ double out[32][9];
  const int node = blockIdx.x * 32 + (threadIdx.x & 31), sub = threadIdx.x >> 5, i = blockIdx.y * 8 + sub;
  double s = 0.0;
  if (node < T && i < T) {
    const int g0 = gs[i], r = gn[i];
#pragma unroll 4
    for (int c = 0; c < r; ++c) s = fma(X[static_cast<size_t>(g0 + c) * T + node], Q[static_cast<size_t>(i) * T + c], s);
  }
  out[threadIdx.x & 31][sub] = s;
  __syncthreads();
  const int rn = blockIdx.x * 32 + (threadIdx.x >> 3), ri = blockIdx.y * 8 + (threadIdx.x & 7);
  if (rn < T && ri < T) U[static_cast<size_t>(rn) * T + ri] = out[threadIdx.x >> 3][threadIdx.x & 7];
}

struct MhsaCoef {
  // per head: the score form (alpha, beta, gamma, delta) / sqrt(d_e) and the value rows va, vb
  double form[kSpeMaxHeads][4];
};

// The fixed-point form of a node's attention.  Double operations are 64 times scarcer than integer ones on
// this GPU, and the T^2 exponentials of a node and head take about 27 of them each, so the softmax runs on
// 64-bit integers: scores in base 2 to 2^-52, 2^-48 in a row whose coefficients pass 2^9 (a double score of magnitude
// 8 or more is rounded to 2^-50, past 1024 to 2^-43, one near zero more finely than either), exponentials to about 2^-53
// of the row's largest one (double table entries and the series below), they and their products held with 64
// fraction bits of it (fewer significant ones the smaller they are), sums exact in 96 bits.  The table's error
// against 64 bits is that of double operations (2.5e-8 in fp32).  With l = lambda / 2^el and v = u / 2^eu in (-1, 1), a row's scores are
// A (l_k - l_min) / 2 + B (v_k + 1) / 2 up to a constant, which a softmax does not see; |A| and |B| are
// scaled by 2^(63 - er) to fill 63 bits.
// |A|, |B| < 2^9 (scores within +-1024): 52 fraction bits; < 2^13: 48, more than a double of that size holds (its
// scores near zero keep fewer than a double would); a wider row takes doubles, whose warp then takes 20 times as long as the others
constexpr int kFixNarrow = 9, kFixWide = 13;
struct FixKey {
  uint64_t l, v;  // (l - l_min) / 2 and (v + 1) / 2, 64 fraction bits
};
// the high 64 bits of x y, up to 2 short (the product of the low halves is left out): a 32 x 32-bit
// product into 64 bits runs at a quarter of the rate of other integer operations and bounds this kernel
__device__ __forceinline__ uint64_t mulhi3(uint64_t x, uint64_t y) {
  const uint32_t xl = static_cast<uint32_t>(x), xh = static_cast<uint32_t>(x >> 32);
  const uint32_t yl = static_cast<uint32_t>(y), yh = static_cast<uint32_t>(y >> 32);
  return static_cast<uint64_t>(xh) * yh + __umulhi(xh, yl) + __umulhi(xl, yh);
}
struct FixSum {  // a 96-bit unsigned sum, 64 fraction bits
  uint64_t lo;
  uint32_t hi;
  __device__ __forceinline__ void add(uint64_t x) {
    lo += x;
    hi += lo < x ? 1u : 0u;
  }
  __device__ __forceinline__ double value() const {
    return fma(static_cast<double>(hi), 18446744073709551616.0, static_cast<double>(lo));
  }
};
// 2^-y for y >= 0 with 52 fraction bits, as a fraction of 2^64: 2^-(j/4096) from the table (the top 12
// fraction bits), times 1 - C / 2^12 with C / 2^12 = 1 - 2^-r for the 40 bits r < 2^-12 that remain, by its
// Taylor series to r^3 (the next term is below 2^-54 / 24; the terms after the first need 32 bits)
constexpr int kFixTable = 4096;
__device__ __forceinline__ uint64_t fix_exp2(uint64_t y, const uint64_t *table) {
  const uint32_t n = static_cast<uint32_t>(y >> 52);
  const uint64_t t = table[static_cast<uint32_t>(y >> 40) & 4095u];
  const uint64_t r = y << 24;  // r 2^12, 64 fraction bits
  const uint32_t rh = static_cast<uint32_t>(r >> 32);
  // C = r' (ln 2 - r' ((ln 2)^2 / 2 / 2^12 - r' (ln 2)^3 / 6 / 2^24)), r' = r 2^12; the bracket's second part
  // with 44 fraction bits: (ln 2)^2 / 2 in 32 bits is 0x3D7F7BFF, (ln 2)^3 / 6 / 2^12 is 58200
  const uint32_t q = __umulhi(rh, 0x3D7F7BFFu - __umulhi(rh, 58200u));
  const uint64_t c = mulhi3(r, 0xB17217F7D1CF79ABull - (static_cast<uint64_t>(q) << 20));
  const uint64_t p = t - (mulhi3(t, c) >> 12);
  return n < 64u ? p >> n : 0ull;
}

// 2^-(j/4096) as fractions of 2^64
__global__ void exp_table_kernel(uint64_t *table) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < kFixTable)
    table[j] = j == 0 ? ~0ull : static_cast<uint64_t>(exp2(-static_cast<double>(j) / kFixTable) * 18446744073709551616.0);
}

// one CTA per node j: SPE_j[c] = sum_e sum_k (mean_i PL_i va_e[k] + mean_i PU_i vb_e[k]) Wo[e d_e + k][c]
// T = 576, 4 heads, 576 nodes: 41 ms with double operations, now 3.8 ms (6.1 while rows with scores past
// +-512, 4% of the warps, took doubles).
__global__ void __launch_bounds__(576) mhsa_kernel(const double *lam, const double *U, int T, int heads,
                                                   const MhsaCoef coef, const double *va, const double *vb,
                                                   const double *wo, const uint64_t *exp_table, int d_spe, float *spe,
                                                   double *spe64) {
  extern __shared__ __align__(16) double sh[];
  double *L = sh, *u = sh + T;
  FixKey *key = reinterpret_cast<FixKey *>(sh + 2 * T);
  uint64_t *table = reinterpret_cast<uint64_t *>(key + T);
  float2 *key32 = reinterpret_cast<float2 *>(table + kFixTable);
  __shared__ double red[32], mean[2 * kSpeMaxHeads], part[kSpeMaxHeads][18][2];  // at most 18 warps
  const int j = blockIdx.x;
  double um = 0.0;
  for (int a = threadIdx.x; a < T; a += blockDim.x) {
    L[a] = lam[a];
    u[a] = U[static_cast<int64_t>(j) * T + a];  // phi_a[j]
    um = fmax(um, fabs(u[a]));
  }
  for (int t = threadIdx.x; t < kFixTable; t += blockDim.x) table[t] = exp_table[t];
  for (int o = 16; o > 0; o >>= 1) um = fmax(um, __shfl_xor_sync(0xffffffffu, um, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = um;
  __syncthreads();
  for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) um = fmax(um, red[w]);
  // powers of two above the largest |lambda| and |u|
  const double lm = fmax(fabs(L[0]), fabs(L[T - 1]));
  const int el = lm > 0.0 ? ilogb(lm) + 1 : 0, eu = um > 0.0 ? ilogb(um) + 1 : 0;
  const double lmin = scalbn(L[0], -el);
  for (int a = threadIdx.x; a < T; a += blockDim.x) {
    const double l = scalbn(L[a], -el), v = scalbn(u[a], -eu);
    key[a] = FixKey{static_cast<uint64_t>((l - lmin) * 9223372036854775808.0),
                    static_cast<uint64_t>(static_cast<int64_t>(v * 9223372036854775808.0)) + 0x8000000000000000ull};
    key32[a] = make_float2(static_cast<float>(0.5 * (l - lmin)), static_cast<float>(fma(0.5, v, 0.5)));
  }
  __syncthreads();
  for (int e = 0; e < heads; ++e) {
    const double al = coef.form[e][0], be = coef.form[e][1], ga = coef.form[e][2], de = coef.form[e][3];
    double spl = 0.0, spu = 0.0;
    for (int i = threadIdx.x; i < T; i += blockDim.x) {
      // s_i' = (L_i al + u_i ga) L_i' + (L_i be + u_i de) u_i'
      const double A1 = L[i] * al + u[i] * ga, B1 = L[i] * be + u[i] * de;
      const double log2e = 1.4426950408889634074;
      const double A = scalbn(A1 * log2e, el + 1), B = scalbn(B1 * log2e, eu + 1), top = fmax(fabs(A), fabs(B));
      if (top < static_cast<double>(1 << kFixWide)) {
        int er = top > 0.0 ? ilogb(top) + 1 : 0;
        if (er < -40) er = -40;
        const uint64_t Ai = static_cast<uint64_t>(scalbn(fabs(A), 63 - er)), Bi = static_cast<uint64_t>(scalbn(fabs(B), 63 - er));
        // the score's negative from magnitudes: flip the bits where a coefficient is positive (-x - 1 = ~x)
        const uint64_t na = A > 0.0 ? ~0ull : 0ull, nb = B > 0.0 ? ~0ull : 0ull;
        const float Af = static_cast<float>(A), Bf = static_cast<float>(B);
        float m32 = -INFINITY;
        for (int k = 0; k < T; ++k) m32 = fmaxf(m32, __fmaf_rn(Af, key32[k].x, __fmul_rn(Bf, key32[k].y)));
        FixSum l = {0, 0}, pl = {0, 0}, pu = {0, 0};
        auto row = [&](auto wide_tag) {
          constexpr int F = decltype(wide_tag)::value ? 48 : 52;  // fraction bits of a score
          const int shift = 63 - F - er;                          // the products have 63 - er
          // any shift near the maximum serves: the single-precision one, raised above its own error (2^-11, 2^-7)
          const uint64_t m = static_cast<uint64_t>(static_cast<int64_t>((static_cast<double>(m32) + 0.015625) * static_cast<double>(1ll << F)));
#pragma unroll 2
          for (int k = 0; k < T; ++k) {
            const FixKey f = key[k];
            uint64_t y = m + ((mulhi3(Ai, f.l) >> shift) ^ na) + ((mulhi3(Bi, f.v) >> shift) ^ nb);
            if (F == 48) y = (y < (64ull << F) ? y : 64ull << F) << 4;
            const uint64_t p = fix_exp2(y, table);
            l.add(p);
            pl.add(mulhi3(p, f.l));
            pu.add(mulhi3(p, f.v));
          }
        };
        if (er <= kFixNarrow) row(std::false_type{});
        else row(std::true_type{});
        // sum p v = 2 sum p (v + 1) / 2 - sum p, formed before it is rounded
        const uint64_t tl = pu.lo << 1;
        const uint32_t th = (pu.hi << 1) | static_cast<uint32_t>(pu.lo >> 63);
        const int64_t dh = static_cast<int64_t>(th) - static_cast<int64_t>(l.hi) - (tl < l.lo ? 1 : 0);
        const double sv = fma(static_cast<double>(dh), 18446744073709551616.0, static_cast<double>(tl - l.lo));
        const double sum = l.value();
        spl += L[0] + scalbn(2.0 * (pl.value() / sum), el);
        spu += scalbn(sv / sum, eu);
      } else {
        double m = -INFINITY;
        for (int k = 0; k < T; ++k) m = fmax(m, A1 * L[k] + B1 * u[k]);
        double l = 0.0, pl = 0.0, pu = 0.0;
        for (int k = 0; k < T; ++k) {
          const double p = exp(A1 * L[k] + B1 * u[k] - m);
          l += p;
          pl += p * L[k];
          pu += p * u[k];
        }
        spl += pl / l;
        spu += pu / l;
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      spl += __shfl_xor_sync(0xffffffffu, spl, o);
      spu += __shfl_xor_sync(0xffffffffu, spu, o);
    }
    if ((threadIdx.x & 31) == 0) part[e][threadIdx.x >> 5][0] = spl, part[e][threadIdx.x >> 5][1] = spu;
  }
  __syncthreads();
  if (threadIdx.x < 2 * heads) {
    double s = 0.0;
    for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) s += part[threadIdx.x >> 1][w][threadIdx.x & 1];
    mean[threadIdx.x] = s / T;
  }
  __syncthreads();
  const int d_e = d_spe / heads;
  for (int c = threadIdx.x; c < d_spe; c += blockDim.x) {
    double s = 0.0;
    for (int e = 0; e < heads; ++e)
      for (int k = 0; k < d_e; ++k)
        s += (mean[2 * e] * va[e * d_e + k] + mean[2 * e + 1] * vb[e * d_e + k]) * wo[(e * d_e + k) * d_spe + c];
    spe[static_cast<int64_t>(j) * d_spe + c] = static_cast<float>(s);
    if (spe64) spe64[static_cast<int64_t>(j) * d_spe + c] = s;
  }
}

// Lets launches of `kernel` ask for all the shared memory that the device has.  The attribute belongs to the process: set
// to one graph's need it would stop the launches of a call with a larger graph on another thread.
template <typename... Args>
cudaError_t allow_shared(void (*kernel)(Args...)) {
  cudaFuncAttributes a;
  const cudaError_t e = cudaFuncGetAttributes(&a, kernel);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(kMaxDynSmem - a.sharedSizeBytes));
}

// one Cholesky QR of the clusters larger than rmin
void chol_qr(double *V, double *Gm, const int *gs, const int *gn, int T, int rmin, int coords, double thr, int *bad) {
  const int nt = (T + 31) / 32;
  gram_kernel<<<dim3(nt, nt), 256>>>(V, gs, gn, T, rmin, coords, Gm);
  chol_kernel<<<T, kCholThreads, kCholSmem>>>(Gm, gs, gn, T, rmin, thr, bad);
  trsm_kernel<<<dim3((T + 15) / 16, T), 256>>>(Gm, V, gs, gn, T, rmin, coords);
}

}  // namespace

cudaError_t run_spe_table(const uint8_t *H, int n, int m, int d_spe, int heads, const double *w_pe, const double *wq,
                          const double *wk, const double *wv, const double *wo, double cluster_tol, double vanish_tol,
                          float *spe_host, double *lam_host, double *U_host, double *spe64_host, int *status_host) {
  const int T = n + m, d_e = d_spe / heads;
  // the projections of the two rows of W_pe and the score forms per head
  MhsaCoef coef = {};
  std::vector<double> vah(static_cast<size_t>(d_spe)), vbh(static_cast<size_t>(d_spe));
  for (int e = 0; e < heads; ++e) {
    std::vector<double> qa(d_e), qb(d_e), ka(d_e), kb(d_e);
    for (int k = 0; k < d_e; ++k) {
      double s[6] = {0, 0, 0, 0, 0, 0};
      for (int a = 0; a < d_spe; ++a) {
        const size_t idx = (static_cast<size_t>(e) * d_spe + a) * d_e + k;
        s[0] += w_pe[a] * wq[idx], s[1] += w_pe[d_spe + a] * wq[idx];
        s[2] += w_pe[a] * wk[idx], s[3] += w_pe[d_spe + a] * wk[idx];
        s[4] += w_pe[a] * wv[idx], s[5] += w_pe[d_spe + a] * wv[idx];
      }
      qa[k] = s[0], qb[k] = s[1], ka[k] = s[2], kb[k] = s[3], vah[e * d_e + k] = s[4], vbh[e * d_e + k] = s[5];
    }
    double f[4] = {0, 0, 0, 0};
    for (int k = 0; k < d_e; ++k) f[0] += qa[k] * ka[k], f[1] += qa[k] * kb[k], f[2] += qb[k] * ka[k], f[3] += qb[k] * kb[k];
    const double sc = 1.0 / std::sqrt(static_cast<double>(d_e));
    for (int t = 0; t < 4; ++t) coef.form[e][t] = f[t] * sc;
  }
  // one allocation for everything
  size_t bytes = 0;
  auto part = [&](size_t size) {
    const size_t off = bytes;
    bytes += (size + 255) & ~static_cast<size_t>(255);
    return off;
  };
  const size_t TT = static_cast<size_t>(T) * T * sizeof(double), T1 = static_cast<size_t>(T) * sizeof(double);
  const size_t o_X = part(TT), o_V = part(TT), o_G = part(TT), o_U = part(TT), o_d = part(T1), o_e = part(T1),
               o_tau = part(T1), o_lam = part(T1), o_row = part(2 * T1), o_p = part(2 * T1),
               o_va = part(sizeof(double) * d_spe), o_vb = part(sizeof(double) * d_spe),
               o_wo = part(sizeof(double) * d_spe * d_spe), o_spe64 = part(sizeof(double) * T * d_spe),
               o_spe = part(sizeof(float) * T * d_spe), o_H = part(static_cast<size_t>(m) * n),
               o_gs = part(sizeof(int) * T), o_gn = part(sizeof(int) * T), o_bad = part(sizeof(int) * 2 * T),
               o_node = part(sizeof(int) * T), o_busy = part(sizeof(int) * (32 * 32 + 1)), o_exp = part(kFixTable * sizeof(uint64_t)), o_status = part(2 * sizeof(int));
  uint8_t *base = nullptr;
  cudaError_t e = cudaSuccess;
  auto ok = [&](cudaError_t x) { return (e = x) == cudaSuccess; };
  int dev = 0, sms = 0, per_sm = 0, R = 1, G = 1;
  std::vector<int> bad(static_cast<size_t>(T));
  if (!ok(cudaMalloc(&base, bytes))) return e;
  auto dp = [&](size_t off) { return reinterpret_cast<double *>(base + off); };
  double *X = dp(o_X), *V = dp(o_V), *Gm = dp(o_G), *U = dp(o_U), *d = dp(o_d), *ed = dp(o_e), *tau = dp(o_tau),
         *lam = dp(o_lam), *rowbuf = dp(o_row), *pbuf = dp(o_p);
  float *spe = reinterpret_cast<float *>(base + o_spe);
  uint8_t *Hd = base + o_H;
  int *gs = reinterpret_cast<int *>(base + o_gs), *gn = reinterpret_cast<int *>(base + o_gn),
      *badd = reinterpret_cast<int *>(base + o_bad), *node = reinterpret_cast<int *>(base + o_node),
      *busy = reinterpret_cast<int *>(base + o_busy), *again = busy + 32 * 32,
      *dstatus = reinterpret_cast<int *>(base + o_status);
  unsigned *count = reinterpret_cast<unsigned *>(dstatus + 1);
  const int nt = (T + 31) / 32;
  if (!ok(cudaMemcpy(Hd, H, static_cast<size_t>(m) * n, cudaMemcpyHostToDevice)) ||
      !ok(cudaMemset(dstatus, 0, 2 * sizeof(int))) ||
      !ok(cudaMemcpy(dp(o_va), vah.data(), sizeof(double) * d_spe, cudaMemcpyHostToDevice)) ||
      !ok(cudaMemcpy(dp(o_vb), vbh.data(), sizeof(double) * d_spe, cudaMemcpyHostToDevice)) ||
      !ok(cudaMemcpy(dp(o_wo), wo, sizeof(double) * d_spe * d_spe, cudaMemcpyHostToDevice)))
    goto done;
  // the tridiagonal form: one CTA per SM (fewer for a small matrix), each with R rows in shared memory
  if (!ok(cudaGetDevice(&dev)) || !ok(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) goto done;
  G = T < 2 * sms ? (T + 1) / 2 : sms;
  R = (T + G - 1) / G;
  {
    const size_t smem = sizeof(double) * T * (3 + static_cast<size_t>(R));
    if (!ok(allow_shared(tridiag_kernel)) ||
        !ok(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, tridiag_kernel, kTriThreads, smem)))
      goto done;
    if (per_sm < 1) {
      e = cudaErrorInvalidConfiguration;
      goto done;
    }
    int narg = n, marg = m;
    void *args[] = {&Hd, &narg, &marg, &V, &tau, &d, &ed, &rowbuf, &pbuf, &count, &dstatus};
    if (!ok(cudaLaunchCooperativeKernel(reinterpret_cast<void *>(tridiag_kernel), dim3(G), dim3(kTriThreads), args, smem,
                                        nullptr)))
      goto done;
  }
  bisect_kernel<<<T, 32, sizeof(double2) * T>>>(d, ed, T, lam);
  group_kernel<<<1, kSpeMaxTokens>>>(lam, T, cluster_tol, gs, gn);
  if (!ok(allow_shared(chol_kernel)) || !ok(allow_shared(select_kernel))) goto done;
  {
    // inverse iteration, vectors of a CTA bounded by the shared memory of their factors; another seed where
    // a cluster's random vectors came out dependent
    const size_t per_vec = static_cast<size_t>(T) * (5 * sizeof(double) + 1);
    int nv = static_cast<int>(220000 / per_vec);
    nv = nv < 1 ? 1 : (nv > 32 ? 32 : nv);
    const int want = (T + sms - 1) / sms;  // no more to a CTA than fills the SMs
    nv = nv > want ? want : nv;
    const size_t smem = per_vec * nv;
    if (!ok(allow_shared(invit_kernel))) goto done;
    for (uint32_t attempt = 0;; ++attempt) {
      if (!ok(cudaMemset(badd, 0, sizeof(int) * 2 * T))) goto done;
      invit_kernel<<<(T + nv - 1) / nv, 32, smem>>>(d, ed, lam, gn, T, nv, 12345u + 977u * attempt, X);
      chol_qr(X, Gm, gs, gn, T, 1, 0, 1e-14, badd);
      chol_qr(X, Gm, gs, gn, T, 1, 0, 1e-14, badd);
      if (!ok(cudaGetLastError()) ||
          !ok(cudaMemcpy(bad.data(), badd, sizeof(int) * T, cudaMemcpyDeviceToHost)))
        goto done;
      bool again = false;
      for (int b : bad) again = again || b != 0;
      if (!again) break;
      if (attempt == 4) {
        e = cudaErrorUnknown;
        goto done;
      }
    }
  }
  // orthogonal vectors to rounding: one round, and a second where that left more (U is free until the end)
  static_assert(kSpeMaxTokens <= 32 * 32, "a mark for every tile");
  if (!ok(cudaMemset(again, 0, sizeof(int)))) goto done;
  overlap_kernel<<<dim3(nt, nt), 256>>>(X, T, nullptr, Gm, busy, again);
  polish_kernel<<<dim3(nt, nt), 256>>>(X, Gm, busy, T, nullptr, U);
  overlap_kernel<<<dim3(nt, nt), 256>>>(U, T, again, Gm, busy, again);
  polish_kernel<<<dim3(nt, nt), 256>>>(U, Gm, busy, T, again, X);
  if (T > 3) pair_kernel<<<T - 3, 32>>>(V, T, pbuf);  // (pbuf: the reduction is done with it)
  // (32 elements a lane spill 812 bytes a thread; they serve every T past 576)
  if (T <= 128) back_kernel<4><<<(T + 1) / 2, 64>>>(V, tau, pbuf, T, X);
  else if (T <= 320) back_kernel<10><<<(T + 1) / 2, 64>>>(V, tau, pbuf, T, X);
  else if (T <= 576) back_kernel<18><<<(T + 1) / 2, 64>>>(V, tau, pbuf, T, X);
  else back_kernel<32><<<(T + 1) / 2, 64>>>(V, tau, pbuf, T, X);
  // the canonical basis in coordinates (V is free now), then in node coordinates
  {
    const int st = (std::min(T, kCholShared) + 31) / 32;
    proj_kernel<<<dim3(st, st, T), 256>>>(X, gs, gn, T, kSeqGroup, Gm);
  }
  select_kernel<<<T, kCholThreads, kCholSmem>>>(X, Gm, gs, gn, T, kSeqGroup, node, badd + T);
  coords_kernel<<<T, 128>>>(X, gs, gn, node, badd + T, T, kSeqGroup, V);
  chol_qr(V, Gm, gs, gn, T, kSeqGroup, 1, 1e-8, badd + T);
  chol_qr(V, Gm, gs, gn, T, kSeqGroup, 1, 1e-8, badd + T);
  canonical_kernel<<<T, kSeqThreads>>>(X, gs, gn, T, vanish_tol, badd + T, V, dstatus);
  basis_kernel<<<dim3(nt, (T + 7) / 8), 256>>>(X, V, gs, gn, T, U);
  {
    const size_t smem = static_cast<size_t>(T) * (2 * sizeof(double) + sizeof(FixKey) + sizeof(float2)) + kFixTable * sizeof(uint64_t);
    const int passes = (T + 575) / 576, threads = ((T + passes - 1) / passes + 31) / 32 * 32;  // rows per pass
    if (!ok(allow_shared(mhsa_kernel))) goto done;
    uint64_t *exp_table = reinterpret_cast<uint64_t *>(base + o_exp);
    exp_table_kernel<<<kFixTable / 256, 256>>>(exp_table);
    mhsa_kernel<<<T, threads, smem>>>(lam, U, T, heads, coef, dp(o_va), dp(o_vb), dp(o_wo), exp_table, d_spe, spe,
                                      dp(o_spe64));
  }
  if (!ok(cudaGetLastError()) || !ok(cudaDeviceSynchronize())) goto done;
  if (!ok(cudaMemcpy(spe_host, spe, sizeof(float) * T * d_spe, cudaMemcpyDeviceToHost)) ||
      !ok(cudaMemcpy(status_host, dstatus, sizeof(int), cudaMemcpyDeviceToHost)))
    goto done;
  if (*status_host & 2) {
    e = cudaErrorLaunchTimeout;
    goto done;
  }
  if (lam_host && !ok(cudaMemcpy(lam_host, lam, T1, cudaMemcpyDeviceToHost))) goto done;
  if (U_host && !ok(cudaMemcpy(U_host, U, TT, cudaMemcpyDeviceToHost))) goto done;
  if (spe64_host && !ok(cudaMemcpy(spe64_host, dp(o_spe64), sizeof(double) * T * d_spe, cudaMemcpyDeviceToHost)))
    goto done;
done:
  cudaFree(base);
  return e;
}

}  // namespace aecct
