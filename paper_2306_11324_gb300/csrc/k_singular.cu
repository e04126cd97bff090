// Touching element pairs (Sec. 4.3) for ansatz degrees up to 3 and five Gauss points per transformed variable
// (others: k_near_singular): the regularising rules summed in tensor form, FP64.
//
// The points of a rule are regions x Gauss indices (a, b, c, d).  With the region and a fixed (a slab of
// 125 points, xi = the a-th Gauss point) every coordinate of a point depends on one or two of b, c, d, and no
// index is shared between the two coordinates of one element (see slab_of):
//   * an element's points of the slab form a tensor grid (1 x 5 .. 5 x 25): its net is contracted along
//     the coordinate with fewer values once, then along the other per point;
//   * the basis functions are tensor products, so the block
//       sum_{b,c,d} s(b,c,d) u_k1(x1) u_k2(x2) u_l1(y1) u_l2(y2)
//     is contracted one index (or index pair) at a time with tables of univariate values.
// Sound-hard: the curl part gc c_k . c_l is four scalar kernels, gc times the products of the tangents, with
// derivatives in place of values of u_k1 .. u_l2, and goes the same way; it is symmetric in the two elements,
// so one sum serves both blocks.
//
// Bound: FP64 arithmetic (a warp instruction holds a quarter of an SM for about 76 cycles), so the helpers of
// k_m2l.cuh take the square root, the reciprocal and the exponential, and each step is spread over all warps.
// Measured on GB300, set-up of all touching pairs (k_near_singular -> here): sound-soft, p = 2, 24576 elements
// (3.7e8 points) 337 -> 150 ms; sound-hard, p = 2, 6144 elements (9.2e7 points) 282 -> 59 ms.
#include <algorithm>

#include "internal.h"
#include "k_common.cuh"
#include "k_m2l.cuh"
#include "kernels.h"

namespace igabem {

namespace {

constexpr int NS = 5, NP = NS * NS * NS, ST = 128;  // Gauss points, points of a slab, threads

struct TensorSing {
  const int *sing;         // 7 ints per unordered touching pair
  const double *rule[3];   // per kind (identical, edge, vertex): x1, x2, y1, y2, w of n points
  int rule_n[3];
  const int *edeg;
  const long *eoff;
  const double *ebez, *ext1, *phi1, *gpa, *gw;
  const double2 *cis;
  int n1, ng, b, nL1, nL, pg1;
  double h, kappa, eta;
  double2 *blk;
};

// Index set of each canonical coordinate (x1, x2, y1, y2) in a slab, as a mask over b (1), c (2), d (4), and the
// contraction: first over index b (pattern 0, 1) with coordinate jb or over a pair of indices (pattern 2).
struct Slab {
  int mask[4];
  // pattern 0 (edge, pyramids 0 and 1): b with jb, (c, d) with the pair (pa, pb), then the constant j0
  // pattern 1 (edge, pyramid 2; vertex): b with jb, c with jc, d with the pair (pa, pb)
  // pattern 2 (identical): two indices with the pair (pa, pb), the third (stride i5) with the pair (qa, qb)
  int pattern, jb, jc, j0, pa, pb, qa, qb;
};

__device__ inline Slab slab_of(int kind, int region) {
  Slab s{};
  if (kind == 0) {  // identical: (sign, sign, triangle)
    s.pattern = 2;
    if ((region & 1) == 0) {  // x1, y1 from c; x2, y2 from (b, d)
      s.mask[0] = s.mask[2] = 2;
      s.mask[1] = s.mask[3] = 5;
      s.pa = 1; s.pb = 3; s.qa = 0; s.qb = 2;
    } else {                  // x1, y1 from (b, c); x2, y2 from d
      s.mask[0] = s.mask[2] = 3;
      s.mask[1] = s.mask[3] = 4;
      s.pa = 0; s.pb = 2; s.qa = 1; s.qb = 3;
    }
  } else if (kind == 1) {  // common edge: (sign, pyramid)
    const int pyr = region % 3;
    s.pa = 1; s.pb = 3;
    if (pyr < 2) {
      s.pattern = 0;
      s.j0 = pyr == 0 ? 0 : 2;
      s.jb = 2 - s.j0;
      s.mask[s.jb] = 1;
      s.mask[1] = s.mask[3] = 6;
    } else {
      s.pattern = 1;
      s.jb = 0; s.jc = 2;
      s.mask[0] = 1; s.mask[2] = 2;
      s.mask[1] = s.mask[3] = 4;
    }
  } else {  // common vertex: the largest coordinate is constant, the others from b, c, d in order
    s.pattern = 1;
    s.j0 = region;
    s.jb = region == 0 ? 1 : 0;
    s.jc = region <= 1 ? 2 : 1;
    s.pb = region == 3 ? 2 : 3;
    s.pa = region;
    s.mask[s.jb] = 1; s.mask[s.jc] = 2; s.mask[s.pb] = 4;
  }
  return s;
}

// number of values of a coordinate, the value's index at (b, c, d), and a point (offset in the slab) where value i
// is taken
__device__ inline int n_values(int mask) { return mask == 0 ? 1 : (mask & (mask - 1)) ? NS * NS : NS; }
__device__ inline int value_at(int mask, int b, int c, int d) {
  switch (mask) {
    case 0: return 0;
    case 1: return b;
    case 2: return c;
    case 4: return d;
    case 3: return b * NS + c;
    case 5: return b * NS + d;
    default: return c * NS + d;
  }
}
__device__ inline int point_of(int mask, int i) {
  const int hi = i / NS, lo = i % NS;
  switch (mask) {
    case 0: return 0;
    case 1: return i * NS * NS;
    case 2: return i * NS;
    case 4: return i;
    case 3: return hi * NS * NS + lo * NS;
    case 5: return hi * NS * NS + lo;
    default: return hi * NS + lo;
  }
}

// The square symmetry k takes the canonical coordinates (r1, r2) to the local ones: which canonical coordinate
// becomes the first local one, and whether a canonical coordinate r enters as 1 - r.
__device__ inline bool d4_swaps(int k) { return (k & 1) != (k >= 4); }
__device__ inline bool d4_flips(int k, int c) { return ((c == 0 ? 0x6C : 0xC6) >> k) & 1; }

// shared-memory layout, offsets in doubles
template <int P1, bool HARD> struct Lay {
  static constexpr int G = HARD ? 6 : 2;              // kernel groups: xy, yx, and the four curl terms
  static constexpr int NV = HARD ? 4 : 1;             // value / derivative variants of a product table
  static constexpr int GEO = HARD ? 13 : 7;           // x, n, |n| (d_s x, d_t x)
  static constexpr int bas = 0;                                        // [2 variants][4][25][P1]
  static constexpr int ppa = bas + (HARD ? 2 : 1) * 4 * 25 * P1;       // [NV][25][P1^2]
  static constexpr int ppb = ppa + NV * 25 * P1 * P1;                  // [NV][5][P1^2]
  static constexpr int geo = (ppb + NV * 5 * P1 * P1 + 1) & ~1;        // [2][125][GEO]; then T1, T2
  static constexpr int t1 = geo;                                       // [G][75 or 5 P1^2 .. 25 P1][2]
  static constexpr int n1 = 25 * P1 > 5 * P1 * P1 ? 25 * P1 : 5 * P1 * P1;
  static constexpr int t2 = t1 + G * n1 * 2;                           // [G][5 P1^2 or P1^3][2]
  static constexpr int n2 = 5 * P1 * P1 > P1 * P1 * P1 ? 5 * P1 * P1 : P1 * P1 * P1;
  static constexpr int geo_end = geo + 2 * NP * GEO > t2 + G * n2 * 2 ? geo + 2 * NP * GEO : t2 + G * n2 * 2;
  static constexpr int s = (geo_end + 1) & ~1;                         // [G][125][2]; before it bern and part
};
template <int P1, bool HARD> __host__ __device__ inline int sing_tensor_doubles(int pg1) {
  const int bern = 4 * 25 * 2 * pg1 + 2 * NS * pg1 * 8, smp = Lay<P1, HARD>::G * NP * 2;
  return Lay<P1, HARD>::s + (bern > smp ? bern : smp) + 2 * 4 * pg1 * pg1;
}

template <int P1, bool HARD>
__global__ void __launch_bounds__(ST) k_sing_tensor(const __grid_constant__ TensorSing A) {
  extern __shared__ __align__(16) double sm[];
  using L = Lay<P1, HARD>;
  constexpr int G = L::G, PP = P1 * P1, P3 = PP * P1, P4 = PP * PP, NE = (P4 + ST - 1) / ST;
  const int tid = threadIdx.x, pg1 = A.pg1;
  double *bas = sm + L::bas, *ppa = sm + L::ppa, *ppb = sm + L::ppb, *geo = sm + L::geo, *t1 = sm + L::t1,
         *t2 = sm + L::t2, *S = sm + L::s;
  double *bern = S, *part = bern + 4 * 25 * 2 * pg1;
  const int bern_part = 4 * 25 * 2 * pg1 + 2 * NS * pg1 * 8, smp = G * NP * 2;
  double *net = S + (bern_part > smp ? bern_part : smp);  // [2][4 pg1^2]
  const int *W = A.sing + 7 * blockIdx.x;
  const int el[2] = {W[0], W[1]}, sym[2] = {W[3], W[4]}, kind = W[2] == 0 ? 0 : W[2] == 2 ? 1 : 2;
  const int blk_ef = W[5], blk_fe = W[6];
  const int npt = A.rule_n[kind];
  const double *R = A.rule[kind];
  const int n1 = A.n1;
  const double h4 = A.h * A.h * A.h * A.h;
  int deg[2][2], col[2][2];  // geometry degrees and element columns along the local directions
#pragma unroll
  for (int z = 0; z < 2; ++z) {
    deg[z][0] = A.edeg[2 * el[z]];
    deg[z][1] = A.edeg[2 * el[z] + 1];
    col[z][0] = (el[z] / n1) % n1;
    col[z][1] = el[z] % n1;
    const int nn = 4 * (deg[z][0] + 1) * (deg[z][1] + 1);
    for (int i = tid; i < nn; i += ST) net[z * 4 * pg1 * pg1 + i] = A.ebez[A.eoff[el[z]] + i];
  }
  // local direction (0: first) of each canonical coordinate
  auto dir_of = [&](int j) { return (j & 1) ^ (d4_swaps(sym[j >> 1]) ? 1 : 0); };
  // group g > 1 takes the derivative along local direction dx on the x side and dy on the y side: (0,0), (0,1),
  // (1,0), (1,1); is coordinate j differentiated in group g?
  auto der = [&](int g, int j) {
    if (!HARD || g < 2) return 0;
    const int dd = (j >> 1) ? (g & 1) : ((g - 2) >> 1);
    return dir_of(j) == dd ? 1 : 0;
  };
  double2 axy[NE], ayx[NE], aw[HARD ? NE : 1];
#pragma unroll
  for (int i = 0; i < NE; ++i) axy[i] = ayx[i] = cmk(0, 0);
  if constexpr (HARD) {
#pragma unroll
    for (int i = 0; i < NE; ++i) aw[i] = cmk(0, 0);
  }
  double c0, c1;
  phase64_scale(A.kappa, c0, c1);
  // identical pairs: the first half of the rule, both orientations of every point into the same block
  const int nslab = (kind == 0 ? npt / 2 : npt) / NP;
  for (int sl = 0; sl < nslab; ++sl) {
    const Slab T = slab_of(kind, sl / NS);
    const int base = sl * NP;
    __syncthreads();  // the previous slab is done
    // univariate values: Bernstein polynomials of the geometry (threads 0..63) and basis functions (64..127) at the
    // values of the four coordinates (16 to 60 of them)
    {
      const bool fun = tid >= 64;
      int i = tid & 63, j = 0;
      while (j < 4 && i >= n_values(T.mask[j])) i -= n_values(T.mask[j++]);
      if (j < 4) {
        const int z = j >> 1, d = dir_of(j);
        const double r = R[j * npt + base + point_of(T.mask[j], i)];
        const double t = d4_flips(sym[z], j & 1) ? 1.0 - r : r;
        double B[8], dB[8];
        if (!fun) {
          const int q = deg[z][d];
          bernstein_all(q, t, B, dB);
          double *o = bern + (j * 25 + i) * 2 * pg1;
          for (int k = 0; k <= q; ++k) {
            o[k] = B[k];
            o[pg1 + k] = dB[k];
          }
        } else {
          bernstein_all(P1 - 1, t, B, HARD ? dB : nullptr);
          const double *ex = A.ext1 + (long)col[z][d] * PP;
#pragma unroll
          for (int f = 0; f < P1; ++f) {
            double v = 0, dv = 0;
#pragma unroll
            for (int k = 0; k < P1; ++k) {
              const double x = ex[f * P1 + k];
              v = fma(x, B[k], v);
              if (HARD) dv = fma(x, dB[k], dv);
            }
            bas[(j * 25 + i) * P1 + f] = v;
            if (HARD) bas[(100 + j * 25 + i) * P1 + f] = dv * n1;
          }
        }
      }
    }
    __syncthreads();
    // nets contracted along the coordinate with fewer values: part[side][value][row][value 4, derivative 4]
    int js[2], nl[2];  // that coordinate of each side; number of values of the other one
#pragma unroll
    for (int z = 0; z < 2; ++z) {
      js[z] = 2 * z + (n_values(T.mask[2 * z]) <= n_values(T.mask[2 * z + 1]) ? 0 : 1);
      nl[z] = n_values(T.mask[js[z] ^ 1]);
    }
    {
      const int w0 = n_values(T.mask[js[0]]) * pg1, w1 = n_values(T.mask[js[1]]) * pg1;
      for (int w = tid; w < w0 + w1; w += ST) {
        const int z = w >= w0, ww = z ? w - w0 : w, i = ww / pg1, row = ww - i * pg1;
        const int ds = dir_of(js[z]), qs = deg[z][ds], ql = deg[z][ds ^ 1];
        if (row > ql) continue;
        const int stride = ds == 0 ? (deg[z][1] + 1) * 4 : 4, rstride = ds == 0 ? 4 : (deg[z][1] + 1) * 4;
        const double *c = net + z * 4 * pg1 * pg1 + row * rstride, *B = bern + (js[z] * 25 + i) * 2 * pg1;
        double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int k = 0; k <= qs; ++k) {
          const double b0 = B[k], b1 = B[pg1 + k];
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const double y = c[k * stride + x];
            v[x] = fma(b0, y, v[x]);
            v[4 + x] = fma(b1, y, v[4 + x]);
          }
        }
        double *o = part + ((z * NS + i) * pg1 + row) * 8;
#pragma unroll
        for (int x = 0; x < 8; ++x) o[x] = v[x];
      }
      // products of the pairs' univariate values, per derivative variant (va, vb): 2 va + vb
      const int na = T.pattern == 1 ? 0 : 25 * PP, nb = T.pattern == 0 ? 0 : 5 * PP;
      for (int w = ST - 1 - tid; w < L::NV * (na + nb); w += ST) {
        const int var = w / (na + nb), ww = w - var * (na + nb), a = ww < na;
        const int o = a ? ww : ww - na, i = o / PP, f = o % PP;
        // pattern 1: (pa, pb) over d; pattern 2: (qa, qb) over the third index
        const int ja = a || T.pattern == 1 ? T.pa : T.qa, jb = a || T.pattern == 1 ? T.pb : T.qb;
        const int ia = T.mask[ja] == 0 ? 0 : i;  // the constant coordinate of a vertex pair
        const double *ba = bas + ((var >> 1) * 100 + ja * 25 + ia) * P1, *bb = bas + ((var & 1) * 100 + jb * 25 + i) * P1;
        (a ? ppa : ppb)[(var * (a ? 25 : 5) + i) * PP + f] = ba[f / P1] * bb[f % P1];
      }
    }
    __syncthreads();
    // geometry of the elements' points: x, n = d_s x ^ d_t x, |n| (and the tangents)
    {
      const int g0 = n_values(T.mask[0]) * n_values(T.mask[1]), g1 = n_values(T.mask[2]) * n_values(T.mask[3]);
      for (int w = tid; w < g0 + g1; w += ST) {
        const int z = w >= g0, ww = z ? w - g0 : w, is = ww / nl[z], il = ww - is * nl[z];
        const int jl = js[z] ^ 1, dl = dir_of(jl), ql = deg[z][dl];
        const double *c = part + (z * NS + is) * pg1 * 8, *B = bern + (jl * 25 + il) * 2 * pg1;
        double hv[4] = {0, 0, 0, 0}, hl[4] = {0, 0, 0, 0}, hs[4] = {0, 0, 0, 0};
        for (int k = 0; k <= ql; ++k) {
          const double b0 = B[k], b1 = B[pg1 + k];
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            hv[x] = fma(b0, c[8 * k + x], hv[x]);
            hl[x] = fma(b1, c[8 * k + x], hl[x]);
            hs[x] = fma(b0, c[8 * k + 4 + x], hs[x]);
          }
        }
        const double iw = rcp64(hv[3]), iwn = iw * n1;
        double *g = geo + (z * NP + (js[z] & 1 ? il * n_values(T.mask[2 * z + 1]) + is : ww)) * L::GEO;
        double fs[3], ft[3], nn[3];
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          const double F = hv[x] * iw, u = fma(-F, hl[3], hl[x]) * iwn, v = fma(-F, hs[3], hs[x]) * iwn;
          g[x] = F;
          fs[x] = dl == 0 ? u : v;
          ft[x] = dl == 0 ? v : u;
        }
        cross3(fs, ft, nn);
        const double n2 = fma(nn[0], nn[0], fma(nn[1], nn[1], nn[2] * nn[2]));
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          g[3 + x] = nn[x];
          if (HARD) {
            g[7 + x] = fs[x];
            g[10 + x] = ft[x];
          }
        }
        g[6] = n2 > 0 ? n2 * rsqrt64(n2) : 0.0;
      }
    }
    __syncthreads();
    // kernel values of the slab's points times the weight: G0 = w exp(i kappa r) / (4 pi r),
    //   soft  ks(x, y) = G0 (A + i B), A = -a_y (d.n_x) / r^2, B = kappa a_y (d.n_x) / r - eta a_x a_y, d = x - y
    //   hard  ks(x, y) = G0 (A + i B), A = -a_x (d.n_y) / r^2, B = kappa a_x (d.n_y) / r + eta kappa^2 n_x.n_y,
    //         curl terms -i eta G0 times (t.t', -t.s', -s.t', s.s') with the tangents s = d_s x, t = d_t x
    // and ks(y, x) with the roles (and the sign of d) exchanged
    if (tid < NP) {
      const int b = tid / (NS * NS), c = tid / NS % NS, d = tid % NS;
      const double *x = geo + (value_at(T.mask[0], b, c, d) * n_values(T.mask[1]) + value_at(T.mask[1], b, c, d)) * L::GEO;
      const double *y = geo + (NP + value_at(T.mask[2], b, c, d) * n_values(T.mask[3]) + value_at(T.mask[3], b, c, d)) * L::GEO;
      const double d0 = x[0] - y[0], d1 = x[1] - y[1], d2 = x[2] - y[2];
      const double r2 = fma(d0, d0, fma(d1, d1, d2 * d2)), ir = rsqrt64(r2);
      const double2 *tab = A.cis;
      const Phase64 ph = phase64(tab, r2 * ir, c0, c1);
      const double f = R[4 * npt + base + tid] * (h4 * (0.25 / IGA_PI)) * ir;
      const C2<double> g = phase_mul(ph.E.x * f, ph.E.y * f, ph);
      const double qx = fma(d0, x[3], fma(d1, x[4], d2 * x[5])) * ir, qy = fma(d0, y[3], fma(d1, y[4], d2 * y[5])) * ir;
      double A1, B1, A2, B2;
      if constexpr (!HARD) {
        const double ea = A.eta * (x[6] * y[6]), u = y[6] * qx, v = -x[6] * qy;
        A1 = -u * ir;
        B1 = fma(A.kappa, u, -ea);
        A2 = -v * ir;
        B2 = fma(A.kappa, v, -ea);
      } else {
        const double nn = A.eta * A.kappa * A.kappa * fma(x[3], y[3], fma(x[4], y[4], x[5] * y[5]));
        const double u = x[6] * qy, v = -y[6] * qx;
        A1 = -u * ir;
        B1 = fma(A.kappa, u, nn);
        A2 = -v * ir;
        B2 = fma(A.kappa, v, nn);
      }
      double2 *S2 = reinterpret_cast<double2 *>(S);
      S2[tid] = cmk(fma(g.x, A1, -(g.y * B1)), fma(g.x, B1, g.y * A1));
      S2[NP + tid] = cmk(fma(g.x, A2, -(g.y * B2)), fma(g.x, B2, g.y * A2));
      if constexpr (HARD) {
        const double gx = A.eta * g.y, gy = -A.eta * g.x;  // -i eta G0
        const double tt = fma(x[10], y[10], fma(x[11], y[11], x[12] * y[12]));
        const double ts = -fma(x[10], y[7], fma(x[11], y[8], x[12] * y[9]));
        const double st = -fma(x[7], y[10], fma(x[8], y[11], x[9] * y[12]));
        const double ss = fma(x[7], y[7], fma(x[8], y[8], x[9] * y[9]));
        S2[2 * NP + tid] = cmk(gx * tt, gy * tt);
        S2[3 * NP + tid] = cmk(gx * ts, gy * ts);
        S2[4 * NP + tid] = cmk(gx * st, gy * st);
        S2[5 * NP + tid] = cmk(gx * ss, gy * ss);
      }
    }
    __syncthreads();
    // The contractions; a task is one real number (re / im the fastest index).
    if (T.pattern == 2) {
      // t1[g][i5][f] = sum over the 25 values of the pair (pa, pb)
      const int tri = T.qa;  // 0: the third index is c; 1: it is d
      for (int w = tid; w < G * 5 * PP * 2; w += ST) {
        const int im = w & 1, f = (w >> 1) % PP, i5 = (w >> 1) / PP % 5, g = (w >> 1) / PP / 5;
        const double *s = S + (g * NP + (tri == 0 ? i5 * NS : i5)) * 2 + im;
        const double *pp = ppa + (2 * der(g, T.pa) + der(g, T.pb)) * 25 * PP + f;
        double acc = 0;
#pragma unroll
        for (int i = 0; i < 25; ++i) {
          const int o = tri == 0 ? (i / NS) * NS * NS + i % NS : (i / NS) * NS * NS + (i % NS) * NS;
          acc = fma(s[2 * o], pp[i * PP], acc);
        }
        t1[w] = acc;  // ((g 5 + i5) PP + f) 2 + im
      }
    } else {
      // t1[g][c, d][f] = sum_b s u_f(b)
      for (int w = tid; w < G * 25 * P1 * 2; w += ST) {
        const int im = w & 1, f = (w >> 1) % P1, cd = (w >> 1) / P1 % 25, g = (w >> 1) / P1 / 25;
        const double *s = S + (g * NP + cd) * 2 + im, *u = bas + (der(g, T.jb) * 100 + T.jb * 25) * P1 + f;
        double acc = 0;
#pragma unroll
        for (int b = 0; b < NS; ++b) acc = fma(s[b * 50], u[b * P1], acc);
        t1[w] = acc;  // ((g 25 + cd) P1 + f) 2 + im
      }
      __syncthreads();
      if (T.pattern == 0) {
        // t2[g][f][kk] = sum_{c, d} t1 u_pa u_pb
        for (int w = tid; w < G * P3 * 2; w += ST) {
          const int im = w & 1, kk = (w >> 1) % PP, f = (w >> 1) / PP % P1, g = (w >> 1) / P3;
          const double *s = t1 + (g * 25 * P1 + f) * 2 + im, *pp = ppa + (2 * der(g, T.pa) + der(g, T.pb)) * 25 * PP + kk;
          double acc = 0;
#pragma unroll
          for (int i = 0; i < 25; ++i) acc = fma(s[i * P1 * 2], pp[i * PP], acc);
          t2[w] = acc;  // ((g P1 + f) PP + kk) 2 + im
        }
      } else {
        // t2[g][d][fb][fc] = sum_c t1 u_fc(c)
        for (int w = tid; w < G * 5 * PP * 2; w += ST) {
          const int im = w & 1, fc = (w >> 1) % P1, fb = (w >> 1) / P1 % P1, d = (w >> 1) / PP % 5, g = (w >> 1) / PP / 5;
          const double *s = t1 + ((g * 25 + d) * P1 + fb) * 2 + im, *u = bas + (der(g, T.jc) * 100 + T.jc * 25) * P1 + fc;
          double acc = 0;
#pragma unroll
          for (int c = 0; c < NS; ++c) acc = fma(s[c * 5 * P1 * 2], u[c * P1], acc);
          t2[w] = acc;  // ((g 5 + d) PP + fb P1 + fc) 2 + im
        }
      }
    }
    __syncthreads();
    // block entries (f[0], f[1]) of x, (f[2], f[3]) of y in canonical coordinates
#pragma unroll
    for (int sl2 = 0; sl2 < NE; ++sl2) {
      const int e = tid + sl2 * ST;
      if (e >= P4) break;
      const int f[4] = {e / P3, e / PP % P1, e / P1 % P1, e % P1};
      auto pick = [&](int j) { return j == 0 ? f[0] : j == 1 ? f[1] : j == 2 ? f[2] : f[3]; };
#pragma unroll
      for (int g = 0; g < G; ++g) {
        double2 v = cmk(0, 0);
        if (T.pattern == 0) {
          const double u = bas[(der(g, T.j0) * 100 + T.j0 * 25) * P1 + pick(T.j0)];
          const double2 s = reinterpret_cast<const double2 *>(t2)[(g * P1 + pick(T.jb)) * PP + f[1] * P1 + f[3]];
          v = cmk(u * s.x, u * s.y);
        } else {
          // pattern 1: t2[g][d][fb fc] with the pair (pa, pb) over d; pattern 2: t1[g][i5][pair] with (qa, qb)
          const bool two = T.pattern == 2;
          const int ja = two ? T.qa : T.pa, jb = two ? T.qb : T.pb;
          const double2 *s = reinterpret_cast<const double2 *>(two ? t1 : t2) + g * 5 * PP +
                             (two ? pick(T.pa) * P1 + pick(T.pb) : pick(T.jb) * P1 + pick(T.jc));
          const double *pp = ppb + (2 * der(g, ja) + der(g, jb)) * 5 * PP + pick(ja) * P1 + pick(jb);
#pragma unroll
          for (int i = 0; i < 5; ++i) {
            v.x = fma(pp[i * PP], s[i * PP].x, v.x);
            v.y = fma(pp[i * PP], s[i * PP].y, v.y);
          }
        }
        if (g == 0) axy[sl2] = cadd(axy[sl2], v);
        else if (g == 1) ayx[sl2] = cadd(ayx[sl2], v);
        else if constexpr (HARD) aw[sl2] = cadd(aw[sl2], v);
      }
    }
  }
  // into the blocks of (e, f) and (f, e); for identical pairs also 1/2 M
  const int mask = (1 << A.b) - 1;
#pragma unroll
  for (int sl2 = 0; sl2 < NE; ++sl2) {
    const int e = tid + sl2 * ST;
    if (e >= P4) break;
    const int f[4] = {e / P3, e / PP % P1, e / P1 % P1, e % P1};
    const bool s0 = d4_swaps(sym[0]), s1 = d4_swaps(sym[1]);
    const int ka = s0 ? f[1] : f[0], kb = s0 ? f[0] : f[1], la = s1 ? f[3] : f[2], lb = s1 ? f[2] : f[3];
    double2 a = axy[sl2], b = ayx[sl2];
    if constexpr (HARD) {
      a = cadd(a, aw[sl2]);
      b = cadd(b, aw[sl2]);
    }
    if (kind == 0) {  // 1/2 M_kl = 1/2 sum_q w_q h^2 a_q psi_k psi_l
      double m = 0;
      for (int q1 = 0; q1 < A.ng; ++q1)
        for (int q2 = 0; q2 < A.ng; ++q2) {
          const double *u = A.phi1 + (col[0][0] * A.ng + q1) * P1, *v = A.phi1 + (col[0][1] * A.ng + q2) * P1;
          m += A.gw[q1] * A.gw[q2] * A.gpa[((long)el[0] * A.ng + q1) * A.ng + q2] * (u[ka] * v[kb]) * (u[la] * v[lb]);
        }
      a.x += 0.5 * m * A.h * A.h;
    }
    const int row = ((col[0][0] & mask) + ka) * A.nL1 + (col[0][1] & mask) + kb;
    const int cf = ((col[1][0] & mask) + la) * A.nL1 + (col[1][1] & mask) + lb;
    double2 *d = A.blk + (size_t)blk_ef * A.nL * A.nL + (size_t)cf * A.nL + row;
    atomicAdd(&d->x, a.x);
    atomicAdd(&d->y, a.y);
    d = A.blk + (size_t)blk_fe * A.nL * A.nL + (size_t)row * A.nL + cf;
    atomicAdd(&d->x, b.x);
    atomicAdd(&d->y, b.y);
  }
}

template <int P1, bool HARD> void go(const TensorSing &A, int n, cudaStream_t st) {
  const size_t smem = sizeof(double) * sing_tensor_doubles<P1, HARD>(A.pg1);
  IGA_CUDA(set_max_dynamic_smem(k_sing_tensor<P1, HARD>, smem));
  k_sing_tensor<P1, HARD><<<n, ST, smem, st>>>(A);
  note_launch();
  IGA_CUDA(cudaGetLastError());
}

}  // namespace

// five Gauss points (the default) and p <= 3: the accumulators of (p + 1)^4 entries stay in registers
bool sing_tensor_supported(const HostSetup &S) { return S.ns == NS && S.p <= 3; }

void launch_sing_tensor(const DeviceProblem &d, const HostSetup &S, const igabem_options &o, cudaStream_t st) {
  TensorSing A{};
  A.sing = d.sing;
  for (int k = 0; k < 3; ++k) {
    A.rule[k] = d.rule[k];
    A.rule_n[k] = d.rule_n[k];
  }
  A.edeg = d.edeg; A.eoff = d.eoff; A.ebez = d.ebez; A.ext1 = d.ext1; A.phi1 = d.phi1; A.gpa = d.gpa; A.gw = d.gw;
  A.cis = reinterpret_cast<const double2 *>(d.cis);
  A.n1 = S.n1; A.ng = S.ng; A.b = S.b; A.nL1 = S.nL1; A.nL = S.nL;
  A.pg1 = 1;
  for (int v : S.edeg) A.pg1 = std::max(A.pg1, v + 1);
  A.h = S.h; A.kappa = o.kappa; A.eta = o.eta_cfie;
  A.blk = reinterpret_cast<double2 *>(d.blk);
  const int n = (int)S.sing.size() / 7;
  if (n == 0) return;
  switch (S.p) {
    case 0: go<1, false>(A, n, st); break;
    case 1: S.hard ? go<2, true>(A, n, st) : go<2, false>(A, n, st); break;
    case 2: S.hard ? go<3, true>(A, n, st) : go<3, false>(A, n, st); break;
    default: S.hard ? go<4, true>(A, n, st) : go<4, false>(A, n, st);
  }
}

}  // namespace igabem
