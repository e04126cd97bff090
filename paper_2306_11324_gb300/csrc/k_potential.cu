// Potential evaluation at many points (Sec. 4.4, last part; Sec. 5.3): the scattered field
//   sound-soft  u_s(x) = -SL(t)(x) = -int G(x, y) t(y) dsigma_y
//   sound-hard  u_s(x) =  DL(u)(x) =  int dG/dn_y(x, y) u(y) dsigma_y
// summed over the Gauss points of every element, applied matrix-free by an interpolation fast
// multipole method in physical space: an octree over the bounding cube of the sources (Gauss points)
// and targets (evaluation points), tensor Chebyshev interpolation with q^3 nodes per box (rank O(q^3),
// against O(q^2) for the surface operators of the reference-domain FMM), kernel samples between box
// nodes generated on the fly once per box offset, the near field summed directly.
//
// Interpolated kernel on an admissible box pair (t, s): G~(x, y) = sum_{a, b} L^t_a(x) G(x_a, y_b)
// L^s_b(y); the double layer differentiates L^s_b(y) along n_y.  Sources carry the weighted density
// rho = w h^2 (density at the Gauss point): monopoles -a rho (soft), dipoles rho n~ (hard).
// Admissibility as on the surface: box radius rho_l = side sqrt(3)/2, admissible iff
// 2 rho_l <= eta_adm (|c_t - c_s| - 2 rho_l) and kappa 2 rho_l <= kappa_cap (when a cap is set).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <unordered_map>
#include <vector>

#include "internal.h"
#include "k_common.cuh"
#include "k_m2l.cuh"
#include "kernels.h"

namespace igabem {

namespace {

constexpr int POT_MAXQ = 10;

struct PotLevel {
  int n;                    // occupied boxes
  const double *center;     // [n][3]
  double half;              // half side
  const int *child;         // [n][8] child box on level l + 1 with sources, or -1
  double2 *W, *Z;           // multipole / local expansions [n][q^3][R]
  double2 *M;               // FP32: sum of a box's expansion [n][R], and the power of two that scales its entries to
  double *scale;            // at most 1
};

struct PotArgs {
  int q, Q, R, hard;
  double kappa;
  const double *cheb;       // q points on [-1, 1], then 1 / (c_a - c_k) [q][q] (0 for k = a)
  const double *T1;         // [2][q][q]: parent Lagrange a at child node b (child c per direction)
  const double2 *cis;       // exp(2 pi i k / CIS_N)
  // sources (Gauss points) sorted by leaf box
  const double *sy;         // [ns][3]
  const double *sn;         // [ns][3] n~ (hard)
  const double *sa;         // [ns] a
  const int *sidx;          // [ns] original Gauss point index
  const int *src_ptr;       // [nleaf + 1]
  const double2 *rho;       // weighted density [G][R]
  // targets sorted by leaf box
  const double *tx;         // [nt][3]
  const int *tidx;          // [nt] original point index
  const int *tbox;          // [nt] leaf box
  const int *near_ptr, *near_src;  // leaf box pairs summed directly
  double2 *u;               // output [n_points][R] (original order)
};

// admissible pairs of one level with the same box offset c_t - c_s = (dx, dy, dz) sides
struct PotChunk {
  int first, count, dx, dy, dz;
};

// value (and derivative) of the Lagrange polynomial a at x; inv: 1 / (c_a - c_k)
__device__ inline double lagrange_a(const double *cheb, const double *inv, int q, int a, double x, double *d) {
  double v = 1.0, dv = 0.0;
  for (int k = 0; k < q; ++k) {
    if (k == a) continue;
    const double i = inv[a * q + k], f = (x - cheb[k]) * i;
    if (d) dv = fma(dv, f, v * i);
    v *= f;
  }
  if (d) *d = dv;
  return v;
}

// source strength seen by interpolation node a of leaf box b: monopole -a rho L_a(y), dipole
// rho n~ . grad L_a(y).  One block per leaf box, the 1-D Lagrange values of its sources (in groups of
// 64) computed once in shared memory.
__global__ void __launch_bounds__(128) k_pot_p2m(PotArgs P, PotLevel L) {
  __shared__ double lag[2][3][64][POT_MAXQ];
  const int Q = P.Q, q = P.q, R = P.R, b = blockIdx.x;
  const int j0 = P.src_ptr[b], j1 = P.src_ptr[b + 1];
  if (j0 == j1) return;  // never read as a source
  const double *c = L.center + 3 * b, *inv = P.cheb + q;
  const double ih = 1.0 / L.half;
  for (int g0 = j0; g0 < j1; g0 += 64) {
    const int n = min(64, j1 - g0);
    __syncthreads();
    for (int o = threadIdx.x; o < 3 * n * q; o += blockDim.x) {
      const int d = o / (n * q), j = (o / q) % n, a = o % q;
      double dv;
      lag[0][d][j][a] = lagrange_a(P.cheb, inv, q, a, (P.sy[3 * (long)(g0 + j) + d] - c[d]) * ih, P.hard ? &dv : nullptr);
      if (P.hard) lag[1][d][j][a] = dv;
    }
    __syncthreads();
    for (int o = threadIdx.x; o < Q * R; o += blockDim.x) {
      const int a = o / R, r = o % R, a1 = a / (q * q), a2 = (a / q) % q, a3 = a % q;
      double2 acc = g0 == j0 ? cmk(0, 0) : L.W[(long)b * Q * R + o];
      for (int j = 0; j < n; ++j) {
        const double2 rho = P.rho[(long)P.sidx[g0 + j] * R + r];
        const double l1 = lag[0][0][j][a1], l2 = lag[0][1][j][a2], l3 = lag[0][2][j][a3];
        double w;
        if (!P.hard) {
          w = -P.sa[g0 + j] * l1 * l2 * l3;
        } else {
          const double *nn = P.sn + 3 * (long)(g0 + j);
          w = (nn[0] * lag[1][0][j][a1] * l2 * l3 + nn[1] * l1 * lag[1][1][j][a2] * l3 +
               nn[2] * l1 * l2 * lag[1][2][j][a3]) * ih;
        }
        acc = cadd(acc, cscale(rho, w));
      }
      L.W[(long)b * Q * R + o] = acc;
    }
  }
}

// One-dimensional transfers of one column in shared memory (Z and X: q^3 values), direction by direction:
// Z[.. o ..] = sum_i M(o, i) X[.. i ..] with M(o, i) = T(o, i) (up: parent from child) or T(i, o) (down).
// After the three passes the result is in X's place of the last call; the caller alternates the buffers.
__device__ inline void pot_pass(const double *T, int q, int Q, int stride, bool up, const double2 *X, double2 *Z) {
  for (int o = threadIdx.x; o < Q; o += blockDim.x) {
    const int k = (o / stride) % q, base = o - k * stride;
    double2 acc = cmk(0, 0);
    for (int i = 0; i < q; ++i) acc = cadd(acc, cscale(X[base + i * stride], up ? T[k * q + i] : T[i * q + k]));
    Z[o] = acc;
  }
  __syncthreads();
}

// M2M from level l + 1 into level l: W_p[a] = sum_children sum_b T_c(a, b) W_c[b], the tensor transfer one
// direction after the other (3 q^4 products a child instead of q^6); one block per (parent, column)
__global__ void __launch_bounds__(128) k_pot_m2m(PotArgs P, PotLevel Lp, PotLevel Lc) {
  extern __shared__ double2 smu[];
  const int Q = P.Q, q = P.q, R = P.R, t = blockIdx.x, r = blockIdx.y;
  double2 *X = smu, *Z = X + Q, *S = Z + Q;
  bool any = false;
  for (int o = threadIdx.x; o < Q; o += blockDim.x) S[o] = cmk(0, 0);
  for (int c = 0; c < 8; ++c) {
    const int ch = Lp.child[8 * t + c];
    if (ch < 0) continue;
    any = true;
    for (int o = threadIdx.x; o < Q; o += blockDim.x) X[o] = Lc.W[((long)ch * Q + o) * R + r];
    __syncthreads();
    pot_pass(P.T1 + (c >> 2) * q * q, q, Q, q * q, true, X, Z);
    pot_pass(P.T1 + ((c >> 1) & 1) * q * q, q, Q, q, true, Z, X);
    pot_pass(P.T1 + (c & 1) * q * q, q, Q, 1, true, X, Z);
    for (int o = threadIdx.x; o < Q; o += blockDim.x) S[o] = cadd(S[o], Z[o]);
    __syncthreads();
  }
  if (any)
    for (int o = threadIdx.x; o < Q; o += blockDim.x) Lp.W[((long)t * Q + o) * R + r] = S[o];
}

// M and scale of one level's boxes, one warp per (box, column); a box without sources gets M = 0 (never read)
__global__ void __launch_bounds__(128) k_pot_sums(PotLevel L, int Q, int R, const double2 *__restrict__ W) {
  const long o = blockIdx.x * 4L + (threadIdx.x >> 5);
  if (o >= (long)L.n * R) return;
  const long b = o / R, r = o - b * R;
  double2 sum = cmk(0, 0);
  double most = 0;
  for (int a = threadIdx.x & 31; a < Q; a += 32) {
    const double2 w = W[(b * Q + a) * R + r];
    sum = cadd(sum, w);
    most = fmax(most, fmax(fabs(w.x), fabs(w.y)));
  }
  for (int k = 16; k > 0; k >>= 1) {
    sum.x += __shfl_xor_sync(0xffffffffu, sum.x, k);
    sum.y += __shfl_xor_sync(0xffffffffu, sum.y, k);
    most = fmax(most, __shfl_xor_sync(0xffffffffu, most, k));
  }
  if ((threadIdx.x & 31) == 0) {
    int e = 0;
    if (most > 0 && isfinite(most)) frexp(most, &e);
    L.M[o] = sum;
    L.scale[o] = scalbn(1.0, -max(-1000, min(1000, e)));
  }
}

// M2L on one level.  G(x_a, y_b) depends on the box offset c_t - c_s alone, so the pairs of a level are
// grouped by it: one block takes up to POT_COLS columns (pairs of one offset times densities) and 128 target
// nodes, and generates each sample once for all of them instead of once per pair; a thread owns one target
// node with its columns' sums in registers.  The pairs' results go through a buffer of POT_BUFFER bytes, some pairs at a
// time, and are added per target in the order of the pairs (k_pot_add), so that a call repeats bit for bit.  In FP32,
// in units of the half side and about the source box's centre (distance r0 from the target node), a sample is
//   G = exp(i kappa r0) / (4 pi half) (1 / r0 + h),  h = (exp(i kappa (r - r0)) - 1) / r + (1 / r - 1 / r0),
// whose first part times the sum of the expansion is formed in FP64 and whose second, small unless the phase turns within
// the box, from r^2 - r0^2 = |y|^2 - 2 X.y without cancellation: what FP32 rounds off samples, expansions (scaled by a
// power of two per box) and products is a part of h, not of G.  The products take two columns per instruction, the
// sums of 16 source nodes are added up with their rounding errors.  Difference to the FP64 form (rms, random densities,
// sound-soft kappa = 0.3, 3, 12, 20): 0.25, 1.4, 8.0, 11e-8; sound-hard 0.5: 20e-8.  (A sample at a time with FP64
// differences, expansions and sums 4.3, 7.9, 50, 90, 128e-8; FP32 products of G, split about the box centres, 4.5, 4.4,
// 10, 14, 185e-8.)
// Measured on 4001 points around 6144 Gauss points, q = 7, 372,000 pairs, host tree included: FP32 1516 -> 29.9 ms a
// call (before: a sample per pair with FP64 differences and sums, and per-node Lagrange values in P2M), FP64 451 ms.
// Groups of 4, 8, 16, 32 nodes: 35.4, 32.6, 29.9, 28.8 ms at 1.03, 1.13, 1.38, 1.87e-8 (kappa = 3).
constexpr int POT_COLS = 16, POT_ROWS = 128, POT_STEP = 64, POT_GROUP = 16;
// Results of the pairs at a time.  Each part ends with a wave of blocks that does not fill the device: 4001 points, q = 7,
// 2 GB in all, FP32: 32 MiB 36.1, 128 MiB 35.5, 512 MiB 33.1, 2 GiB 33.2 ms (32.6 with atomics in no fixed order);
// 20000 points, 8 densities: 860, 738, 699, 689 ms (674).
constexpr size_t POT_BUFFER = size_t(512) << 20;

template <class T>
__global__ void __launch_bounds__(POT_ROWS) k_pot_m2l(PotArgs P, PotLevel L, const PotChunk *__restrict__ chunks,
                                                      const int2 *__restrict__ pairs, int p0, double2 *__restrict__ out) {
  constexpr bool F32 = sizeof(T) == 4;
  __shared__ __align__(16) T wre[POT_STEP][POT_COLS];
  __shared__ __align__(16) T wim[POT_STEP][POT_COLS];
  __shared__ __align__(16) T ys[POT_STEP][4];
  __shared__ double2 tab[F32 ? 1 : CIS_N];
  __shared__ long wcol[POT_COLS];           // a column's first entry in W
  __shared__ double scale[F32 ? POT_COLS : 1];
  const int Q = P.Q, q = P.q, R = P.R, tid = threadIdx.x;
  const PotChunk ck = chunks[blockIdx.x];
  const int ncol = ck.count * R, a = blockIdx.y * POT_ROWS + tid;
  if (tid < ncol) {
    const long s = pairs[ck.first + tid / R].y;
    wcol[tid] = s * Q * R + tid % R;
    if constexpr (F32) scale[tid] = L.scale[s * R + tid % R];
  }
  // FP32: positions in units of the half side about the source centre; FP64: lengths
  const double unit = F32 ? 1.0 : L.half;
  double X[3] = {2.0 * unit * ck.dx, 2.0 * unit * ck.dy, 2.0 * unit * ck.dz};
  if (a < Q) {
    X[0] += P.cheb[a / (q * q)] * unit;
    X[1] += P.cheb[(a / q) % q] * unit;
    X[2] += P.cheb[a % q] * unit;
  }
  double c0, c1;
  phase64_scale(F32 ? P.kappa * L.half : P.kappa, c0, c1);
  T tr[POT_COLS], ti[POT_COLS];
  float lr[F32 ? POT_COLS : 1], li[F32 ? POT_COLS : 1];  // FP32: what the sums over the groups round off
#pragma unroll
  for (int c = 0; c < POT_COLS; ++c) {
    tr[c] = ti[c] = 0;
    if constexpr (F32) lr[c] = li[c] = 0;
  }
  T x2[3] = {0, 0, 0}, r02 = 1, r0 = 1, ir0 = 1;  // FP32: -2 X, |X|^2, |X|, 1 / |X|
  const T kappa = (T)(P.kappa * L.half);
  if constexpr (F32) {
    const double d2 = X[0] * X[0] + X[1] * X[1] + X[2] * X[2], id = rsqrt64(d2);
#pragma unroll
    for (int c = 0; c < 3; ++c) x2[c] = (T)(-2.0 * X[c]);
    r02 = (T)d2;
    r0 = (T)(d2 * id);
    ir0 = (T)id;
  } else {
    for (int i = tid; i < CIS_N; i += POT_ROWS) tab[i] = P.cis[i];
  }
  for (int b0 = 0; b0 < Q; b0 += POT_STEP) {
    const int nb = min(POT_STEP, Q - b0);
    __syncthreads();
    for (int o = tid; o < nb * POT_COLS; o += POT_ROWS) {
      const int b = o / POT_COLS, c = o % POT_COLS;
      double2 v = cmk(0, 0);
      if (c < ncol) {
        v = L.W[wcol[c] + (long)(b0 + b) * R];
        if constexpr (F32) v = cscale(v, scale[c]);
      }
      wre[b][c] = (T)v.x;
      wim[b][c] = (T)v.y;
    }
    for (int b = tid; b < nb; b += POT_ROWS) {
      const int bb = b0 + b;
      const double y[3] = {P.cheb[bb / (q * q)] * unit, P.cheb[(bb / q) % q] * unit, P.cheb[bb % q] * unit};
      for (int c = 0; c < 3; ++c) ys[b][c] = (T)y[c];
      ys[b][3] = (T)(y[0] * y[0] + y[1] * y[1] + y[2] * y[2]);
    }
    __syncthreads();
    if (a >= Q) continue;
    if constexpr (F32) for (int g0 = 0; g0 < nb; g0 += POT_GROUP) {
      float2 pr[POT_COLS / 2], pi[POT_COLS / 2];
#pragma unroll
      for (int c = 0; c < POT_COLS / 2; ++c) pr[c] = pi[c] = make_float2(0.f, 0.f);
      for (int b = g0; b < min(nb, g0 + POT_GROUP); ++b) {
        const float4 y = *reinterpret_cast<const float4 *>(ys[b]);
        const float num = fmaf(x2[0], y.x, fmaf(x2[1], y.y, fmaf(x2[2], y.z, y.w)));  // r^2 - r0^2
        const float r2 = r02 + num, i0 = rsqrtf(r2), ir = fmaf(0.5f * i0, fmaf(-r2 * i0, i0, 1.f), i0);
        const float del = __fdividef(num, fmaf(r2, ir, r0));                            // r - r0
        float sn, cm;
        sin_cosm1(kappa * del, sn, cm);
        const float gx = fmaf(-del, ir0, cm) * ir, gy = sn * ir;
        const float2 gxx = make_float2(gx, gx), gyy = make_float2(gy, gy), gyn = make_float2(-gy, -gy);
        const float4 *wr = reinterpret_cast<const float4 *>(wre[b]), *wi = reinterpret_cast<const float4 *>(wim[b]);
#pragma unroll
        for (int c = 0; c < POT_COLS / 4; ++c) {
          const float4 u = wr[c], v = wi[c];
          const float2 u0 = make_float2(u.x, u.y), u1 = make_float2(u.z, u.w), v0 = make_float2(v.x, v.y),
                       v1 = make_float2(v.z, v.w);
          pr[2 * c] = fma2x(gxx, u0, fma2x(gyn, v0, pr[2 * c]));
          pi[2 * c] = fma2x(gxx, v0, fma2x(gyy, u0, pi[2 * c]));
          pr[2 * c + 1] = fma2x(gxx, u1, fma2x(gyn, v1, pr[2 * c + 1]));
          pi[2 * c + 1] = fma2x(gxx, v1, fma2x(gyy, u1, pi[2 * c + 1]));
        }
      }
#pragma unroll
      for (int c = 0; c < POT_COLS / 2; ++c) {
        two_sum(tr[2 * c], lr[2 * c], pr[c].x); two_sum(tr[2 * c + 1], lr[2 * c + 1], pr[c].y);
        two_sum(ti[2 * c], li[2 * c], pi[c].x); two_sum(ti[2 * c + 1], li[2 * c + 1], pi[c].y);
      }
    } else {
      for (int b = 0; b < nb; ++b) {
        const double d0 = X[0] - ys[b][0], d1 = X[1] - ys[b][1], d2 = X[2] - ys[b][2];
        const double r2 = d0 * d0 + d1 * d1 + d2 * d2, ir = rsqrt64(r2), f = ir * (0.25 / IGA_PI);
        const Phase64 p = phase64(tab, r2 * ir, c0, c1);
        const C2<double> G = phase_mul(p.E.x * f, p.E.y * f, p);
#pragma unroll
        for (int c = 0; c < POT_COLS; ++c) {
          if (c >= ncol) break;  // the same for every thread: no padding on the FP64 pipe
          tr[c] = fma(G.x, wre[b][c], fma(-G.y, wim[b][c], tr[c]));
          ti[c] = fma(G.x, wim[b][c], fma(G.y, wre[b][c], ti[c]));
        }
      }
    }
  }
  if (a >= Q) return;
  double fx = 0, fy = 0, id = 0;  // FP32: exp(i kappa r0) / (4 pi half), 1 / r0
  if constexpr (F32) {
    const double d2 = X[0] * X[0] + X[1] * X[1] + X[2] * X[2];
    id = rsqrt64(d2);
    const Phase64 p = phase64(P.cis, d2 * id, c0, c1);
    const double f = 0.25 / IGA_PI / L.half;
    const C2<double> E = phase_mul(p.E.x * f, p.E.y * f, p);
    fx = E.x;
    fy = E.y;
  }
#pragma unroll
  for (int c = 0; c < POT_COLS; ++c) {
    if (c >= ncol) break;
    double2 *z = out + ((long)(ck.first - p0 + c / R) * Q + a) * R + c % R;
    if constexpr (F32) {
      const double is = 1.0 / scale[c];  // exact
      const double2 M = L.M[(long)pairs[ck.first + c / R].y * R + c % R];
      const double hx = fma(id, M.x, ((double)tr[c] + (double)lr[c]) * is);
      const double hy = fma(id, M.y, ((double)ti[c] + (double)li[c]) * is);
      *z = cmk(fma(fx, hx, -fy * hy), fma(fx, hy, fy * hx));
    } else {
      *z = cmk(tr[c], ti[c]);
    }
  }
}

// Z_t += the results of the pairs p0 .. p1 with target t, in the order of the pairs (list: each target's pairs, ascending)
__global__ void __launch_bounds__(128) k_pot_add(PotLevel L, int QR, const int *__restrict__ ptr, const int *__restrict__ list,
                                                 int p0, int p1, const double2 *__restrict__ out) {
  const int t = blockIdx.x;
  auto first = [&](int p) {  // first entry of target t that is not below p
    int lo = ptr[t], hi = ptr[t + 1];
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (list[mid] < p) lo = mid + 1;
      else hi = mid;
    }
    return lo;
  };
  const int k0 = first(p0), k1 = first(p1);
  if (k0 == k1) return;
  for (int o = blockIdx.y * 128 + threadIdx.x; o < QR; o += gridDim.y * 128) {
    double2 z = L.Z[(long)t * QR + o];
    for (int k = k0; k < k1; ++k) z = cadd(z, out[(long)(list[k] - p0) * QR + o]);
    L.Z[(long)t * QR + o] = z;
  }
}

// L2L from level l into level l + 1: Z_c[b] += sum_a T_c(a, b) Z_p[a], direction by direction; one block per
// (child, column)
__global__ void __launch_bounds__(128) k_pot_l2l(PotArgs P, PotLevel Lp, PotLevel Lc, const int *parent_of,
                                                 const int *child_slot) {
  extern __shared__ double2 smd_[];
  const int Q = P.Q, q = P.q, R = P.R, ch = blockIdx.x, r = blockIdx.y;
  const int t = parent_of[ch], c = child_slot[ch];
  double2 *X = smd_, *Z = X + Q;
  for (int o = threadIdx.x; o < Q; o += blockDim.x) X[o] = Lp.Z[((long)t * Q + o) * R + r];
  __syncthreads();
  pot_pass(P.T1 + (c >> 2) * q * q, q, Q, q * q, false, X, Z);
  pot_pass(P.T1 + ((c >> 1) & 1) * q * q, q, Q, q, false, Z, X);
  pot_pass(P.T1 + (c & 1) * q * q, q, Q, 1, false, X, Z);
  for (int o = threadIdx.x; o < Q; o += blockDim.x) {
    double2 *z = Lc.Z + ((long)ch * Q + o) * R + r;
    *z = cadd(*z, Z[o]);
  }
}

// L2P and the near field at every target: u = sum_a L^t_a(x) Z_t[a] + sum_{near leaf boxes} direct.  One warp
// per target: its lanes share the nodes of the box and the sources nearby.
__global__ void __launch_bounds__(128) k_pot_eval(PotArgs P, PotLevel L, int n_pts) {
  __shared__ double lag[4][3][POT_MAXQ];
  const int q = P.q, Q = P.Q, R = P.R, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long j = blockIdx.x * 4L + warp;
  if (j >= n_pts) return;
  const int t = P.tbox[j];
  const double x[3] = {P.tx[3 * j], P.tx[3 * j + 1], P.tx[3 * j + 2]};
  double2 acc[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) acc[r] = cmk(0, 0);
  if (L.Z) {
    const double *c = L.center + 3 * t;
    const double ih = 1.0 / L.half;
    if (lane < 3 * q) {
      const int d = lane / q, k = lane % q;
      lag[warp][d][k] = lagrange_a(P.cheb, P.cheb + q, q, k, (P.tx[3 * j + d] - c[d]) * ih, nullptr);
    }
    __syncwarp();
    for (int a = lane; a < Q; a += 32) {
      const double w = lag[warp][0][a / (q * q)] * lag[warp][1][(a / q) % q] * lag[warp][2][a % q];
#pragma unroll
      for (int r = 0; r < 8; ++r)
        if (r < R) acc[r] = cadd(acc[r], cscale(L.Z[((long)t * Q + a) * R + r], w));
    }
  }
  for (int k = P.near_ptr[t]; k < P.near_ptr[t + 1]; ++k) {
    const int s = P.near_src[k];
    for (int g = P.src_ptr[s] + lane; g < P.src_ptr[s + 1]; g += 32) {
      const double *y = P.sy + 3 * (long)g;
      const double v[3] = {y[0] - x[0], y[1] - x[1], y[2] - x[2]};
      const double rr = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
      double sn, cs;
      sincos(P.kappa * rr, &sn, &cs);
      const double2 G = cmk(cs / (4.0 * IGA_PI * rr), sn / (4.0 * IGA_PI * rr));
      double2 kv;
      if (!P.hard) {
        kv = cscale(G, -P.sa[g]);
      } else {
        const double *n = P.sn + 3 * (long)g;
        const double vn = (v[0] * n[0] + v[1] * n[1] + v[2] * n[2]) / (rr * rr);
        kv = cscale(cmul(G, cmk(-1.0, P.kappa * rr)), vn);   // G (i kappa r - 1)/r^2 (y - x).n~
      }
#pragma unroll
      for (int r = 0; r < 8; ++r)
        if (r < R) acc[r] = cadd(acc[r], cmul(kv, P.rho[(long)P.sidx[g] * R + r]));
    }
  }
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    if (r >= R) break;
    for (int o = 16; o > 0; o >>= 1) {
      acc[r].x += __shfl_xor_sync(0xffffffffu, acc[r].x, o);
      acc[r].y += __shfl_xor_sync(0xffffffffu, acc[r].y, o);
    }
    if (lane == 0) P.u[(long)P.tidx[j] * R + r] = acc[r];
  }
}

struct Key {
  long long v;
  bool operator==(const Key &o) const { return v == o.v; }
};
struct KeyHash {
  size_t operator()(const Key &k) const { return std::hash<long long>()(k.v); }
};
inline long long pack(int i, int j, int k) { return ((long long)i << 42) | ((long long)j << 21) | (long long)k; }

}  // namespace

}  // namespace igabem

using namespace igabem;

extern "C" int igabem_potential(igabem_problem *P, int n_rhs, const void *density, int n_pts, const double *pts,
                                void *uout) {
  return run_guarded([&] {
    if (!P || !density || !pts || !uout || n_rhs <= 0 || n_pts <= 0) fail(IGABEM_EINVAL, "invalid potential arguments");
    if (n_rhs > 8) fail(IGABEM_EINVAL, "igabem_potential takes at most 8 densities per call");
    IGA_CUDA(cudaSetDevice(P->geom->ctx->device));
    const HostSetup &S = P->S;
    const igabem_options &o = P->opt;
    cudaStream_t st = P->stream;
    const int R = n_rhs, q = std::min(o.cheb_q, POT_MAXQ), Q = q * q * q;
    const long G = (long)S.E * S.ng * S.ng;
    const bool fp32 = o.precision != IGABEM_FP64;
    // sources: the Gauss points (positions, normals, Jacobians from the device tables)
    std::vector<double> gx(3 * G), gn(3 * G), ga(G);
    for (int c = 0; c < 3; ++c) {
      IGA_CUDA(cudaMemcpy(gx.data() + c * G, P->d.gpx + c * G, G * sizeof(double), cudaMemcpyDeviceToHost));
      IGA_CUDA(cudaMemcpy(gn.data() + c * G, P->d.gpn + c * G, G * sizeof(double), cudaMemcpyDeviceToHost));
    }
    IGA_CUDA(cudaMemcpy(ga.data(), P->d.gpa, G * sizeof(double), cudaMemcpyDeviceToHost));
    std::vector<double> tp(3L * n_pts);
    cudaPointerAttributes at{};
    const bool pdev = cudaPointerGetAttributes(&at, pts) == cudaSuccess &&
                      (at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged);
    cudaGetLastError();
    IGA_CUDA(cudaMemcpy(tp.data(), pts, tp.size() * sizeof(double), pdev ? cudaMemcpyDeviceToHost : cudaMemcpyHostToHost));
    // bounding cube
    double lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (long i = 0; i < G; ++i)
      for (int c = 0; c < 3; ++c) {
        lo[c] = std::min(lo[c], gx[c * G + i]);
        hi[c] = std::max(hi[c], gx[c * G + i]);
      }
    for (long i = 0; i < n_pts; ++i)
      for (int c = 0; c < 3; ++c) {
        lo[c] = std::min(lo[c], tp[3 * i + c]);
        hi[c] = std::max(hi[c], tp[3 * i + c]);
      }
    double side = 0;
    for (int c = 0; c < 3; ++c) side = std::max(side, hi[c] - lo[c]);
    side *= 1.0 + 1e-9;
    if (!(side > 0)) side = 1.0;
    // leaf level: at most 64 sources per leaf box (depth <= 10); everything near without the FMM
    int D = 0;
    auto cell = [&](double v, int c, int l) {
      const int n = 1 << l;
      return std::min(n - 1, std::max(0, (int)((v - lo[c]) / side * n)));
    };
    if (!o.no_fmm) {
      // a point's cell on level l is its cell on level 10 shifted: Morton codes sorted once give every level's counts
      auto spread = [](unsigned v) {  // 10 bits, two zeros between neighbours
        v = (v | v << 16) & 0x030000FFu;
        v = (v | v << 8) & 0x0300F00Fu;
        v = (v | v << 4) & 0x030C30C3u;
        return (v | v << 2) & 0x09249249u;
      };
      std::vector<unsigned> code(G);
      for (long i = 0; i < G; ++i)
        code[i] = spread(cell(gx[i], 0, 10)) << 2 | spread(cell(gx[G + i], 1, 10)) << 1 | spread(cell(gx[2 * G + i], 2, 10));
      std::sort(code.begin(), code.end());
      for (D = 1; D < 10; ++D) {
        const int sh = 3 * (10 - D);
        long mx = 0;
        for (long i = 0; i < G;) {
          long e = i;
          while (e < G && code[e] >> sh == code[i] >> sh) ++e;
          mx = std::max(mx, e - i);
          i = e;
        }
        if (mx <= 64) break;
      }
    }
    // occupied boxes per level (leaf level first, then parents)
    std::vector<std::vector<long long>> keys(D + 1);
    std::vector<std::unordered_map<Key, int, KeyHash>> index(D + 1);
    auto leaf_key = [&](const double *x, int c0stride) {
      return pack(cell(x[0], 0, D), cell(x[c0stride], 1, D), cell(x[2 * c0stride], 2, D));
    };
    std::vector<long long> skey(G), tkey(n_pts);
    for (long i = 0; i < G; ++i) skey[i] = leaf_key(&gx[i], (int)G);
    for (long i = 0; i < n_pts; ++i) tkey[i] = leaf_key(&tp[3 * i], 1);
    {
      std::vector<long long> all(skey);
      all.insert(all.end(), tkey.begin(), tkey.end());
      std::sort(all.begin(), all.end());
      all.erase(std::unique(all.begin(), all.end()), all.end());
      keys[D] = all;
    }
    for (int l = D - 1; l >= 0; --l) {
      std::vector<long long> par;
      for (long long k : keys[l + 1]) {
        const int i = int(k >> 42), j = int((k >> 21) & 0x1FFFFF), kk = int(k & 0x1FFFFF);
        par.push_back(pack(i >> 1, j >> 1, kk >> 1));
      }
      std::sort(par.begin(), par.end());
      par.erase(std::unique(par.begin(), par.end()), par.end());
      keys[l] = par;
    }
    for (int l = 0; l <= D; ++l)
      for (size_t b = 0; b < keys[l].size(); ++b) index[l][Key{keys[l][b]}] = (int)b;
    const int nleaf = (int)keys[D].size();
    // sources and targets sorted by leaf box
    std::vector<int> sperm(G), tperm(n_pts);
    for (long i = 0; i < G; ++i) sperm[i] = (int)i;
    for (long i = 0; i < n_pts; ++i) tperm[i] = (int)i;
    std::vector<int> sbox(G), tbox(n_pts);
    for (long i = 0; i < G; ++i) sbox[i] = index[D][Key{skey[i]}];
    for (long i = 0; i < n_pts; ++i) tbox[i] = index[D][Key{tkey[i]}];
    std::stable_sort(sperm.begin(), sperm.end(), [&](int a, int b) { return sbox[a] < sbox[b]; });
    std::stable_sort(tperm.begin(), tperm.end(), [&](int a, int b) { return tbox[a] < tbox[b]; });
    std::vector<int> sptr(nleaf + 1, 0), tptr(nleaf + 1, 0);
    for (long i = 0; i < G; ++i) sptr[sbox[i] + 1]++;
    for (long i = 0; i < n_pts; ++i) tptr[tbox[i] + 1]++;
    for (int b = 0; b < nleaf; ++b) {
      sptr[b + 1] += sptr[b];
      tptr[b + 1] += tptr[b];
    }
    std::vector<double> sy(3 * G), sn(3 * G), sa(G), tx(3L * n_pts);
    for (long j = 0; j < G; ++j) {
      const int i = sperm[j];
      for (int c = 0; c < 3; ++c) {
        sy[3 * j + c] = gx[c * G + i];
        sn[3 * j + c] = gn[c * G + i];
      }
      sa[j] = ga[i];
    }
    for (long j = 0; j < n_pts; ++j)
      for (int c = 0; c < 3; ++c) tx[3 * j + c] = tp[3 * (long)tperm[j] + c];
    // per level: centres, source/target presence (subtree), children
    std::vector<std::vector<double>> cen(D + 1);
    std::vector<std::vector<char>> hs(D + 1), ht(D + 1);
    std::vector<std::vector<int>> child(D + 1);
    for (int l = 0; l <= D; ++l) {
      const int n = (int)keys[l].size();
      cen[l].resize(3L * n);
      hs[l].assign(n, 0);
      ht[l].assign(n, 0);
      child[l].assign(8L * n, -1);
      const double s = side / (1 << l);
      for (int b = 0; b < n; ++b) {
        const long long k = keys[l][b];
        const int idx[3] = {int(k >> 42), int((k >> 21) & 0x1FFFFF), int(k & 0x1FFFFF)};
        for (int c = 0; c < 3; ++c) cen[l][3 * b + c] = lo[c] + (idx[c] + 0.5) * s;
      }
    }
    for (int b = 0; b < nleaf; ++b) {
      hs[D][b] = sptr[b + 1] > sptr[b];
      ht[D][b] = tptr[b + 1] > tptr[b];
    }
    std::vector<std::vector<int>> parent(D + 1), slot(D + 1);
    for (int l = D; l >= 1; --l) {
      const int n = (int)keys[l].size();
      parent[l].resize(n);
      slot[l].resize(n);
      for (int b = 0; b < n; ++b) {
        const long long k = keys[l][b];
        const int i = int(k >> 42), j = int((k >> 21) & 0x1FFFFF), kk = int(k & 0x1FFFFF);
        const int p = index[l - 1][Key{pack(i >> 1, j >> 1, kk >> 1)}];
        const int c = ((i & 1) << 2) | ((j & 1) << 1) | (kk & 1);
        parent[l][b] = p;
        slot[l][b] = c;
        child[l - 1][8 * p + c] = b;
        hs[l - 1][p] |= hs[l][b];
        ht[l - 1][p] |= ht[l][b];
      }
    }
    // dual traversal: admissible pairs per level with their box offsets, near leaf pairs.  The candidates of a level go
    // over host threads in chunks, whose lists are taken in order (as one thread would form them); a level's admissible
    // pairs are sorted at once, so that the lists of one level alone are in memory with their offsets.
    struct Box {
      int i, j, k;
    };
    std::vector<std::vector<Box>> box(D + 1);
    for (int l = 0; l <= D; ++l) {
      box[l].reserve(keys[l].size());
      for (long long v : keys[l]) box[l].push_back({int(v >> 42), int((v >> 21) & 0x1FFFFF), int(v & 0x1FFFFF)});
    }
    const double cap = o.kappa_cap > 0 ? o.kappa_cap : INFINITY;
    // admissible pairs of every level sorted by box offset, in chunks of POT_COLS columns
    const int per = std::max(1, POT_COLS / R);
    std::vector<std::vector<int2>> fpair(D + 1);
    std::vector<std::vector<PotChunk>> chunk(D + 1);
    std::vector<std::vector<int>> tptr_far(D + 1), tlist(D + 1);  // each target's pairs, ascending
    std::vector<std::pair<int, int>> near, cand{{0, 0}}, nxt;
    if (!(ht[0][0] && hs[0][0])) cand.clear();
    for (int l = 0; l <= D; ++l) {
      const double rad = side / (1 << l) * std::sqrt(3.0) / 2;
      const long n = (long)cand.size(), nch = std::min<long>(64, (n + 8191) / 8192);
      struct Part {
        std::vector<std::pair<int, int>> far, near, next;
        int most = 0;  // largest box offset in far
      };
      std::vector<Part> part(nch);
      parallel_for(nch, [&](long c) {
        Part &q_ = part[c];
        for (long i = n * c / nch; i < n * (c + 1) / nch; ++i) {
          const int t = cand[i].first, s = cand[i].second;
          const double *ct = &cen[l][3 * t], *cs = &cen[l][3 * s];
          const double dist = std::sqrt((ct[0] - cs[0]) * (ct[0] - cs[0]) + (ct[1] - cs[1]) * (ct[1] - cs[1]) +
                                        (ct[2] - cs[2]) * (ct[2] - cs[2])) - 2 * rad;
          const bool adm = !o.no_fmm && dist > 0 && 2 * rad <= o.eta_adm * dist && o.kappa * 2 * rad <= cap;
          if (adm) {
            const Box &bt = box[l][t], &bs = box[l][s];
            q_.far.push_back({t, s});
            q_.most = std::max({q_.most, std::abs(bt.i - bs.i), std::abs(bt.j - bs.j), std::abs(bt.k - bs.k)});
          } else if (l == D) {
            q_.near.push_back({t, s});
          } else {
            int sb[8], ns = 0;  // the source box's children with sources
            for (int b = 0; b < 8; ++b) {
              const int ch = child[l][8 * s + b];
              if (ch >= 0 && hs[l + 1][ch]) sb[ns++] = ch;
            }
            for (int a = 0; a < 8; ++a) {
              const int ta = child[l][8 * t + a];
              if (ta < 0 || !ht[l + 1][ta]) continue;
              for (int b = 0; b < ns; ++b) q_.next.push_back({ta, sb[b]});
            }
          }
        }
      });
      size_t n_next = 0;
      for (const Part &q_ : part) n_next += q_.next.size();
      nxt.clear();
      nxt.reserve(n_next);
      for (Part &q_ : part) {
        near.insert(near.end(), q_.near.begin(), q_.near.end());
        nxt.insert(nxt.end(), q_.next.begin(), q_.next.end());
        std::vector<std::pair<int, int>>().swap(q_.near);
        std::vector<std::pair<int, int>>().swap(q_.next);
      }
      cand.swap(nxt);
      size_t nf = 0;
      int most = 0;
      for (const Part &q_ : part) {
        nf += q_.far.size();
        most = std::max(most, q_.most);
      }
      if (nf == 0) continue;
      const long w = 2L * most + 1;
      auto id = [&](const std::pair<int, int> &f) {  // of the pair's box offset
        const Box &t = box[l][f.first], &s = box[l][f.second];
        return ((t.i - s.i + most) * w + t.j - s.j + most) * w + t.k - s.k + most;
      };
      fpair[l].resize(nf);
      auto add_chunks = [&](size_t first, size_t count, long o) {
        for (size_t i = 0; i < count; i += per)
          chunk[l].push_back({(int)(first + i), (int)std::min<size_t>(per, count - i), int(o / (w * w) - most),
                              int(o / w % w - most), int(o % w - most)});
      };
      if (w * w * w <= 1 << 20) {  // counting sort over the offsets' cube
        std::vector<int> first(w * w * w + 1, 0);
        for (const Part &q_ : part)
          for (const auto &f : q_.far) first[id(f) + 1]++;
        for (long o = 0; o < w * w * w; ++o) {
          if (first[o + 1]) add_chunks(first[o], first[o + 1], o);
          first[o + 1] += first[o];
        }
        for (Part &q_ : part) {
          for (const auto &f : q_.far) fpair[l][first[id(f)]++] = make_int2(f.first, f.second);
          std::vector<std::pair<int, int>>().swap(q_.far);
        }
      } else {
        size_t i = 0;
        for (Part &q_ : part) {
          for (const auto &f : q_.far) fpair[l][i++] = make_int2(f.first, f.second);
          std::vector<std::pair<int, int>>().swap(q_.far);
        }
        auto key = [&](const int2 &f) { return id({f.x, f.y}); };
        std::stable_sort(fpair[l].begin(), fpair[l].end(), [&](const int2 &x, const int2 &y) { return key(x) < key(y); });
        for (i = 0; i < nf;) {
          size_t e = i;
          while (e < nf && key(fpair[l][e]) == key(fpair[l][i])) ++e;
          add_chunks(i, e - i, key(fpair[l][i]));
          i = e;
        }
      }
      std::vector<int> &tp_ = tptr_far[l];
      tp_.assign(keys[l].size() + 1, 0);
      for (const int2 &f : fpair[l]) tp_[f.x + 1]++;
      for (size_t t = 0; t + 1 < tp_.size(); ++t) tp_[t + 1] += tp_[t];
      tlist[l].resize(nf);
      std::vector<int> fill(tp_.begin(), tp_.end() - 1);
      for (size_t i = 0; i < nf; ++i) tlist[l][fill[fpair[l][i].x]++] = (int)i;
    }
    auto csr = [](const std::vector<std::pair<int, int>> &pairs, int n, std::vector<int> &ptr, std::vector<int> &src) {
      ptr.assign(n + 1, 0);
      for (auto &p : pairs) ptr[p.first + 1]++;
      for (int i = 0; i < n; ++i) ptr[i + 1] += ptr[i];
      src.assign(pairs.size(), 0);
      std::vector<int> fill(ptr.begin(), ptr.end() - 1);
      for (auto &p : pairs) src[fill[p.first]++] = p.second;
    };
    std::vector<int> nptr, nsrc;
    csr(near, nleaf, nptr, nsrc);
    int lmin = D + 1;
    for (int l = 0; l <= D; ++l)
      if (!fpair[l].empty()) lmin = std::min(lmin, l);
    // interpolation tables
    std::vector<double> cheb(q + (size_t)q * q, 0.0), T1(2L * q * q);
    for (int a = 0; a < q; ++a) cheb[a] = std::cos((2 * a + 1) * M_PI / (2 * q));
    for (int a = 0; a < q; ++a)
      for (int k = 0; k < q; ++k)
        if (k != a) cheb[q + a * q + k] = 1.0 / (cheb[a] - cheb[k]);
    for (int c = 0; c < 2; ++c)
      for (int a = 0; a < q; ++a)
        for (int b = 0; b < q; ++b) {
          const double x = 0.5 * cheb[b] + (c ? 0.5 : -0.5);  // child node b in parent coordinates
          double v = 1.0;
          for (int k = 0; k < q; ++k)
            if (k != a) v *= (x - cheb[k]) / (cheb[a] - cheb[k]);
          T1[(c * q + a) * q + b] = v;
        }
    // device buffers (one allocation)
    std::vector<int> tsort(n_pts);  // leaf box of each sorted target
    for (long j = 0; j < n_pts; ++j) tsort[j] = tbox[tperm[j]];
    size_t bytes = 0;
    auto add = [&](size_t n) { bytes += (n + 255) & ~size_t(255); };
    add(sizeof(double) * 3 * G); add(sizeof(double) * 3 * G); add(sizeof(double) * G); add(sizeof(int) * G);
    add(sizeof(int) * (nleaf + 1)); add(sizeof(double) * 3 * n_pts); add(sizeof(int) * n_pts);
    add(sizeof(int) * n_pts); add(sizeof(int) * (nleaf + 1)); add(sizeof(int) * std::max<size_t>(nsrc.size(), 1));
    add(sizeof(double2) * G * R); add(sizeof(double2) * (size_t)n_pts * R); add(sizeof(double) * cheb.size());
    add(sizeof(double) * T1.size());
    for (int l = 0; l <= D; ++l) {
      const size_t n = keys[l].size();
      add(sizeof(double) * 3 * n); add(sizeof(int) * 8 * n); add(sizeof(int) * n); add(sizeof(int) * n);
      add(sizeof(int2) * std::max<size_t>(fpair[l].size(), 1));
      add(sizeof(PotChunk) * std::max<size_t>(chunk[l].size(), 1));
      add(sizeof(int) * std::max<size_t>(tptr_far[l].size(), 1));
      add(sizeof(int) * std::max<size_t>(tlist[l].size(), 1));
      if (l >= lmin) {
        add(sizeof(double2) * n * Q * R);
        add(sizeof(double2) * n * Q * R);
        add(sizeof(double2) * n * R);
        add(sizeof(double) * n * R);
      }
    }
    Arena A;
    A.reserve(bytes + 4096);
    auto up = [&](const auto &v) {
      using T = typename std::decay_t<decltype(v)>::value_type;
      T *p = A.get<T>(std::max<size_t>(v.size(), 1));
      if (!v.empty()) IGA_CUDA(cudaMemcpyAsync(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, st));
      return p;
    };
    struct Buffer {
      double2 *p = nullptr;
      ~Buffer() { cudaFree(p); }
    } out;
    try {
      // the buffer of the pairs' results: smaller where the memory for it is not there (the results do not depend on it)
      const size_t QR = (size_t)Q * R;
      size_t most_pairs = 0, room = 0;  // pairs of a level; pairs that the buffer holds
      for (int l = 0; l <= D; ++l) most_pairs = std::max(most_pairs, fpair[l].size());
      if (most_pairs) {
        room = std::min(most_pairs, std::max<size_t>(per, POT_BUFFER / (QR * sizeof(double2))));
        while (cudaMalloc(&out.p, room * QR * sizeof(double2)) != cudaSuccess) {
          cudaGetLastError();
          out.p = nullptr;
          if (room <= (size_t)per) fail(IGABEM_ENOMEM, "no device memory for the potential's buffer");
          room = std::max<size_t>(per, room / 2);
        }
      }
      PotArgs PA{};
      PA.q = q;
      PA.Q = Q;
      PA.R = R;
      PA.hard = S.hard ? 1 : 0;
      PA.kappa = o.kappa;
      PA.sy = up(sy);
      PA.sn = up(sn);
      PA.sa = up(sa);
      PA.sidx = up(sperm);
      PA.src_ptr = up(sptr);
      PA.tx = up(tx);
      PA.tidx = up(tperm);
      PA.tbox = up(tsort);
      PA.cis = reinterpret_cast<const double2 *>(P->d.cis);
      PA.near_ptr = up(nptr);
      PA.near_src = up(nsrc);
      double2 *rho = A.get<double2>(G * R);
      PA.rho = rho;
      double2 *ud = A.get<double2>((size_t)n_pts * R);
      PA.u = ud;
      PA.cheb = up(cheb);
      PA.T1 = up(T1);
      std::vector<PotLevel> LV(D + 1);
      std::vector<int *> par_d(D + 1), slot_d(D + 1);
      std::vector<int2 *> pair_d(D + 1);
      std::vector<PotChunk *> chunk_d(D + 1);
      std::vector<int *> tptr_d(D + 1), tlist_d(D + 1);
      for (int l = 0; l <= D; ++l) {
        PotLevel &L = LV[l];
        L.n = (int)keys[l].size();
        L.center = up(cen[l]);
        L.half = side / (1 << l) / 2;
        std::vector<int> with_src(child[l]);
        if (l < D)
          for (int &c : with_src)
            if (c >= 0 && !hs[l + 1][c]) c = -1;
        L.child = up(with_src);
        pair_d[l] = up(fpair[l]);
        chunk_d[l] = up(chunk[l]);
        tptr_d[l] = up(tptr_far[l]);
        tlist_d[l] = up(tlist[l]);
        par_d[l] = up(parent[l].empty() ? std::vector<int>(1, 0) : parent[l]);
        slot_d[l] = up(slot[l].empty() ? std::vector<int>(1, 0) : slot[l]);
        L.W = L.Z = L.M = nullptr;
        L.scale = nullptr;
        if (l >= lmin) {
          L.W = A.get<double2>((size_t)L.n * Q * R);
          L.Z = A.get<double2>((size_t)L.n * Q * R);
          L.M = A.get<double2>((size_t)L.n * R);
          L.scale = A.get<double>((size_t)L.n * R);
          IGA_CUDA(cudaMemsetAsync(L.Z, 0, sizeof(double2) * (size_t)L.n * Q * R, st));
        }
      }
      launch_density(P->d, S, o, R, static_cast<const double *>(density), reinterpret_cast<double *>(rho), st);
      if (lmin <= D) {
        k_pot_p2m<<<nleaf, 128, 0, st>>>(PA, LV[D]);
        note_launch();
        const size_t smt = 3 * sizeof(double2) * (size_t)Q;  // q <= 10: at most 48 KB
        IGA_CUDA(set_max_dynamic_smem(k_pot_m2m, smt));
        IGA_CUDA(set_max_dynamic_smem(k_pot_l2l, smt));
        for (int l = D - 1; l >= lmin; --l) {
          k_pot_m2m<<<dim3(LV[l].n, R), 128, smt, st>>>(PA, LV[l], LV[l + 1]);
          note_launch();
        }
        for (int l = lmin; l <= D; ++l) {
          if (fp32 && !chunk[l].empty()) {
            k_pot_sums<<<(unsigned)(((long)LV[l].n * R + 3) / 4), 128, 0, st>>>(LV[l], Q, R, LV[l].W);
            note_launch();
          }
          for (size_t i = 0; i < chunk[l].size();) {
            const int p0 = chunk[l][i].first;
            size_t e = i;
            int p1 = p0;
            for (; e < chunk[l].size() && (size_t)(p1 - p0 + chunk[l][e].count) <= room; ++e) p1 += chunk[l][e].count;
            const dim3 grid((unsigned)(e - i), (Q + POT_ROWS - 1) / POT_ROWS);
            if (fp32) k_pot_m2l<float><<<grid, POT_ROWS, 0, st>>>(PA, LV[l], chunk_d[l] + i, pair_d[l], p0, out.p);
            else k_pot_m2l<double><<<grid, POT_ROWS, 0, st>>>(PA, LV[l], chunk_d[l] + i, pair_d[l], p0, out.p);
            note_launch();
            k_pot_add<<<dim3(LV[l].n, (unsigned)((QR + 511) / 512)), 128, 0, st>>>(LV[l], (int)QR, tptr_d[l], tlist_d[l], p0, p1,
                                                                                  out.p);
            note_launch();
            i = e;
          }
        }
        for (int l = lmin; l < D; ++l) {
          k_pot_l2l<<<dim3(LV[l + 1].n, R), 128, smt, st>>>(PA, LV[l], LV[l + 1], par_d[l + 1], slot_d[l + 1]);
          note_launch();
        }
      }
      k_pot_eval<<<(n_pts + 3) / 4, 128, 0, st>>>(PA, LV[D], n_pts);
      note_launch();
      IGA_CUDA(cudaGetLastError());
      cudaPointerAttributes ua{};
      const bool udev = cudaPointerGetAttributes(&ua, uout) == cudaSuccess &&
                        (ua.type == cudaMemoryTypeDevice || ua.type == cudaMemoryTypeManaged);
      cudaGetLastError();
      IGA_CUDA(cudaMemcpyAsync(uout, ud, sizeof(double2) * (size_t)n_pts * R,
                               udev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, st));
      IGA_CUDA(cudaStreamSynchronize(st));
    } catch (...) {
      cudaStreamSynchronize(st);
      A.release();
      throw;
    }
    A.release();
  });
}
