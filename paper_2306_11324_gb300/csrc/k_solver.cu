// Right-hand sides (Sec. 4.1), far-field pattern (Sec. 1) and the vector kernels of GMRES (Sec. 5.1).
#include <cooperative_groups.h>

#include <algorithm>

#include "internal.h"
#include "k_common.cuh"
#include "k_m2l.cuh"
#include "kernels.h"

namespace igabem {

namespace {

inline int grid_for(long n, int block = 256) {
  return (int)std::max<long>(1, std::min<long>((n + block - 1) / block, 152L * 32));
}

#define GRID_STRIDE(i, n) \
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < (n); i += (long)gridDim.x * blockDim.x)

struct RhsArgs {
  const double *gpx, *gpn, *gpa, *phi1, *gw;
  const int *g2x_ptr, *g2x_idx;
  const double *dirs;     // per right-hand side: the direction d (plane wave) or the source point z
  long gst, N;
  int n1, nb, p, ng, R;
  double h, kappa, eta;
  bool hard;
  int kind;               // 0 plane waves exp(i kappa d.x); 1 point sources G(x, z)
};

// b[i][r] = sum over the elements of the supports of psi_i of sum_q w_q h^2 psi(q) f_r(q),
//   soft: f = grad u_inc . n~ - i eta a u_inc        (a (du_inc/dn - i eta u_inc))
//   hard: f = a u_inc - i eta grad u_inc . n~        (a (u_inc - i eta du_inc/dn))
// with u_inc = exp(i kappa d.x), grad u_inc = i kappa d u_inc (plane wave), or u_inc = G(x, z),
// grad u_inc = G (i kappa r - 1) / r^2 (x - z), r = |x - z| (point source at z).
__global__ void k_rhs(RhsArgs A, double2 *__restrict__ b) {
  const int p1 = A.p + 1, nq = A.ng * A.ng;
  GRID_STRIDE(o, A.N * A.R) {
    long gi = o / A.R;
    int r = int(o % A.R);
    const double *d = A.dirs + 3 * r;
    double2 acc = cmk(0, 0);
    for (int k = A.g2x_ptr[gi]; k < A.g2x_ptr[gi + 1]; ++k) {
      long X = A.g2x_idx[k];
      int j = int(X / ((long)A.nb * A.nb)), i1 = int((X / A.nb) % A.nb), i2 = int(X % A.nb);
      for (int ix = max(0, i1 - A.p); ix <= min(A.n1 - 1, i1); ++ix)
        for (int iy = max(0, i2 - A.p); iy <= min(A.n1 - 1, i2); ++iy) {
          long e = ((long)j * A.n1 + ix) * A.n1 + iy;
          int ka = i1 - ix, kb = i2 - iy;
          for (int q1 = 0; q1 < A.ng; ++q1)
            for (int q2 = 0; q2 < A.ng; ++q2) {
              long iq = e * nq + q1 * A.ng + q2;
              double x[3] = {A.gpx[iq], A.gpx[A.gst + iq], A.gpx[2 * A.gst + iq]};
              double n[3] = {A.gpn[iq], A.gpn[A.gst + iq], A.gpn[2 * A.gst + iq]};
              double2 f;
              if (A.kind == 0) {
                double dx = d[0] * x[0] + d[1] * x[1] + d[2] * x[2];
                double dn = d[0] * n[0] + d[1] * n[1] + d[2] * n[2];
                double s, c;
                sincos(A.kappa * dx, &s, &c);
                f = A.hard ? cmk(A.gpa[iq] + A.eta * A.kappa * dn, 0.0) : cmk(0.0, A.kappa * dn - A.eta * A.gpa[iq]);
                f = cmul(f, cmk(c, s));
              } else {
                const double v[3] = {x[0] - d[0], x[1] - d[1], x[2] - d[2]};
                const double r = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
                double s, c;
                sincos(A.kappa * r, &s, &c);
                const double2 u = cmk(c / (4.0 * IGA_PI * r), s / (4.0 * IGA_PI * r));
                const double vn = (v[0] * n[0] + v[1] * n[1] + v[2] * n[2]) / (r * r);
                const double2 gn = cscale(cmul(u, cmk(-1.0, A.kappa * r)), vn);   // grad u_inc . n~
                const double2 ie_gn = cmk(-A.eta * gn.y, A.eta * gn.x);         // i eta grad u . n~
                const double2 ie_u = cmk(-A.eta * u.y * A.gpa[iq], A.eta * u.x * A.gpa[iq]);  // i eta a u
                f = A.hard ? csub(cscale(u, A.gpa[iq]), ie_gn) : csub(gn, ie_u);
              }
              double w = A.gw[q1] * A.gw[q2] * A.h * A.h *
                         A.phi1[(ix * A.ng + q1) * p1 + ka] * A.phi1[(iy * A.ng + q2) * p1 + kb];
              acc = cadd(acc, cscale(f, w));
            }
        }
    }
    b[o] = acc;
  }
}

// density at the Gauss points, weighted by w_q h^2: rho[e][q][r] = w_q h^2 sum_k psi_k(q) x[.][r], in FP64, stored as
// V (the FP32 far field rounds it here once); a thread takes four columns, so that the basis products are
// shared
template <class V>
__global__ void k_density(RhsArgs A, const int *__restrict__ x2g, const double2 *__restrict__ x, long E,
                          V *__restrict__ rho) {
  const int p1 = A.p + 1, nq = A.ng * A.ng, nc4 = (A.R + 3) / 4;
  GRID_STRIDE(o, E * nq * nc4) {
    const long iq = o / nc4, e = iq / nq;
    const int r0 = int(o - iq * nc4) * 4, nr = min(4, A.R - r0), q = int(iq - e * nq), q1 = q / A.ng, q2 = q % A.ng;
    const int j = int(e / ((long)A.n1 * A.n1)), ix = int((e / A.n1) % A.n1), iy = int(e % A.n1);
    double2 acc[4] = {cmk(0, 0), cmk(0, 0), cmk(0, 0), cmk(0, 0)};
    for (int ka = 0; ka < p1; ++ka)
      for (int kb = 0; kb < p1; ++kb) {
        const long X = ((long)j * A.nb + ix + ka) * A.nb + iy + kb;
        const double w = A.phi1[(ix * A.ng + q1) * p1 + ka] * A.phi1[(iy * A.ng + q2) * p1 + kb];
        const double2 *xr = x + (long)x2g[X] * A.R + r0;
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (r < nr) acc[r] = cadd(acc[r], cscale(xr[r], w));
      }
    const double w = A.gw[q1] * A.gw[q2] * A.h * A.h;
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (r < nr) {
        V v;
        v.x = (decltype(v.x))(acc[r].x * w);
        v.y = (decltype(v.y))(acc[r].y * w);
        rho[iq * A.R + r0 + r] = v;
      }
  }
}

// u_inf[k][r] = sum_points rho * exp(-i kappa x^_k . x) * (soft: -a/(4 pi); hard: -i kappa (x^.n~)/(4 pi)) in FP64.  One
// block per direction and four columns, which share the exponential (FP64 arithmetic bounds it: 18 operations for
// the table-driven exponential instead of CUDA's sincos per column); the points are split over a cluster of
// gridDim.z blocks where there are few directions.  A single column has a form of its own: columns that are not there cost
// the wider one as much as the others.  98304 points, 3000 directions, 1 and 4 columns: 12.1 and 17.9 ms (one column in the wide form
// 19.1, CUDA's sincos per column 18.4 and 72).
constexpr int FF64_COLS = 4;

template <int NC>
__global__ void __launch_bounds__(256, NC == 1 ? 4 : 3) k_farfield(RhsArgs A, const double2 *__restrict__ rho, long npts,
                                                  const double *__restrict__ xhat, const double2 *__restrict__ cis,
                                                  double2 *__restrict__ uinf) {
  __shared__ double2 tab[CIS_N];
  __shared__ double2 red[8][NC];
  const int k = blockIdx.x, r0 = blockIdx.y * NC, nr = min(NC, A.R - r0), nz = gridDim.z;
  const double xh[3] = {xhat[3 * k], xhat[3 * k + 1], xhat[3 * k + 2]};
  double c0, c1;
  phase64_scale(A.kappa, c0, c1);
  for (int i = threadIdx.x; i < CIS_N; i += 256) tab[i] = cis[i];
  __syncthreads();
  double2 acc[NC];
#pragma unroll
  for (int r = 0; r < NC; ++r) acc[r] = cmk(0, 0);
  for (long i = blockIdx.z * 256 + threadIdx.x; i < npts; i += 256L * nz) {
    const double d = fma(xh[0], A.gpx[i], fma(xh[1], A.gpx[A.gst + i], xh[2] * A.gpx[2 * A.gst + i]));
    const Phase64 p = phase64(tab, d, c0, c1);
    // amplitude times exp(i kappa x^.x) = (c, s): soft a, the factor is -(c - i s); hard kappa x^.n~, -(s + i c)
    double2 f;
    if (A.hard) {
      const double xn = A.kappa * fma(xh[0], A.gpn[i], fma(xh[1], A.gpn[A.gst + i], xh[2] * A.gpn[2 * A.gst + i]));
      const C2<double> e = phase_mul(p.E.x * xn, p.E.y * xn, p);
      f = cmk(-e.y, -e.x);
    } else {
      const double a = A.gpa[i];
      const C2<double> e = phase_mul(p.E.x * a, p.E.y * a, p);
      f = cmk(-e.x, e.y);
    }
#pragma unroll
    for (int r = 0; r < NC; ++r)
      if (r < nr) {
        const double2 v = rho[i * A.R + r0 + r];
        acc[r].x = fma(f.x, v.x, fma(-f.y, v.y, acc[r].x));
        acc[r].y = fma(f.x, v.y, fma(f.y, v.x, acc[r].y));
      }
  }
#pragma unroll
  for (int r = 0; r < NC; ++r) {
    for (int o = 16; o > 0; o >>= 1) {
      acc[r].x += __shfl_xor_sync(0xffffffffu, acc[r].x, o);
      acc[r].y += __shfl_xor_sync(0xffffffffu, acc[r].y, o);
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][r] = acc[r];
  }
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  if (nz > 1) cl.sync();
  else __syncthreads();
  if (blockIdx.z == 0 && (int)threadIdx.x < nr) {
    double2 s = cmk(0, 0);
    for (int z = 0; z < nz; ++z) {
      const double2(*rz)[NC] = nz > 1 ? cl.map_shared_rank(red, z) : red;
      for (int w = 0; w < 8; ++w) s = cadd(s, rz[w][threadIdx.x]);
    }
    uinf[(long)k * A.R + r0 + threadIdx.x] = cscale(s, 0.25 / IGA_PI);
  }
  if (nz > 1) cl.sync();  // no block leaves while another reads its shared memory
}

// Far field in the mixed precisions, for many directions: the Gauss points are taken in groups of
// FE x FE elements with a reference point C (the group's first Gauss point, FP64); the phase
// kappa x^.y = kappa x^.C + kappa x^.(y - C) splits into a per-(direction, group) factor exp(-i kappa
// x^.C) in FP64 and per-point exponentials of the small offsets in FP32, summed in FP32 per group and
// direction, scaled by the FP64 factor and added over the groups in FP64.  Block: one group and 64 DPT
// directions, 4 point lanes per direction, up to 8 right-hand sides per pass.
// Bound: FP32 arithmetic (41 operations a point, direction and 8 columns), if shared memory does not set the pace: a
// point's 8 densities take a warp 16 cycles to load, so a thread uses them for DPT directions; the densities are
// stored by parts, so that the products take two columns per instruction.  Measured, 393216 points,
// 2048 directions, 8 columns, with the density: 1.98 -> 1.73 ms (before, one direction a thread and FP64
// conversions in every block).
constexpr int FF_LANES = 4, FF_COLS = 8, FF_CHUNK = 256, FF_TH = 64;

template <int DPT, bool HARD>
__global__ void __launch_bounds__(FF_LANES *FF_TH) k_farfield32(RhsArgs A, const float2 *__restrict__ rho, int fe, int n_dir,
                                                               const double *__restrict__ xhat, double2 *__restrict__ uinf) {
  constexpr int NT = FF_LANES * FF_TH, ND = FF_TH * DPT;
  __shared__ float4 pts[FF_CHUNK];                       // y - C (3), a
  __shared__ float4 nrm[HARD ? FF_CHUNK : 1];            // n~ (3)
  __shared__ __align__(16) float rre[FF_CHUNK][FF_COLS], rim[FF_CHUNK][FF_COLS];  // weighted density
  const int nq = A.ng * A.ng, ge = 1 << fe, ngr1 = A.n1 >> fe;
  const int g = blockIdx.x, j = g / (ngr1 * ngr1), gx = (g / ngr1) % ngr1, gy = g % ngr1;
  const int npts = ge * ge * nq;
  const int dl = threadIdx.x % FF_TH, lane = threadIdx.x / FF_TH, k0 = blockIdx.y * ND;
  // reference point: the first Gauss point of the group
  const long e0 = ((long)j * A.n1 + gx * ge) * A.n1 + gy * ge;
  const double C0 = A.gpx[e0 * nq], C1 = A.gpx[A.gst + e0 * nq], C2v = A.gpx[2 * A.gst + e0 * nq];
  float kx[DPT][3];  // direction k0 + dl + 64 d
#pragma unroll
  for (int d = 0; d < DPT; ++d) {
    const int k = min(k0 + dl + FF_TH * d, n_dir - 1);
#pragma unroll
    for (int c = 0; c < 3; ++c) kx[d][c] = (float)(-A.kappa * xhat[3 * k + c]);
  }
  const bool work = k0 + (dl & ~31) < n_dir;  // the warp has a direction
  for (int c0 = 0; c0 < A.R; c0 += FF_COLS) {
    const int nc = min(FF_COLS, A.R - c0);
    float2 ar[DPT][FF_COLS / 2], ai[DPT][FF_COLS / 2];
#pragma unroll
    for (int d = 0; d < DPT; ++d)
#pragma unroll
      for (int c = 0; c < FF_COLS / 2; ++c) ar[d][c] = ai[d][c] = make_float2(0.f, 0.f);
    for (int p0 = 0; p0 < npts; p0 += FF_CHUNK) {
      const int np = min(FF_CHUNK, npts - p0);
      __syncthreads();
      for (int i = threadIdx.x; i < np; i += NT) {
        const int pi = p0 + i, el = pi / nq, q = pi % nq;
        const long e = ((long)j * A.n1 + gx * ge + el / ge) * A.n1 + gy * ge + el % ge;
        const long iq = e * nq + q;
        pts[i] = make_float4((float)(A.gpx[iq] - C0), (float)(A.gpx[A.gst + iq] - C1),
                             (float)(A.gpx[2 * A.gst + iq] - C2v), (float)A.gpa[iq]);
        if (HARD) nrm[i] = make_float4((float)A.gpn[iq], (float)A.gpn[A.gst + iq], (float)A.gpn[2 * A.gst + iq], 0.f);
      }
      for (int i = threadIdx.x; i < np * FF_COLS; i += NT) {
        const int pi = i / FF_COLS, c = i % FF_COLS;
        const int el = (p0 + pi) / nq, q = (p0 + pi) % nq;
        const long e = ((long)j * A.n1 + gx * ge + el / ge) * A.n1 + gy * ge + el % ge;
        const float2 v = c < nc ? rho[(e * nq + q) * A.R + c0 + c] : make_float2(0.f, 0.f);
        rre[pi][c] = v.x;
        rim[pi][c] = v.y;
      }
      __syncthreads();
      if (work) {
        for (int i = lane; i < np; i += FF_LANES) {
          const float4 y = pts[i];
          const float4 n = HARD ? nrm[i] : make_float4(0.f, 0.f, 0.f, 0.f);
          float2 re[FF_COLS / 2], im[FF_COLS / 2];
#pragma unroll
          for (int c = 0; c < FF_COLS / 4; ++c) {
            const float4 u = reinterpret_cast<const float4 *>(rre[i])[c], v = reinterpret_cast<const float4 *>(rim[i])[c];
            re[2 * c] = make_float2(u.x, u.y);
            re[2 * c + 1] = make_float2(u.z, u.w);
            im[2 * c] = make_float2(v.x, v.y);
            im[2 * c + 1] = make_float2(v.z, v.w);
          }
#pragma unroll
          for (int d = 0; d < DPT; ++d) {
            float ph = fmaf(kx[d][0], y.x, fmaf(kx[d][1], y.y, kx[d][2] * y.z));
            const float kq = rintf(ph * 0.15915494309189535f);
            ph = fmaf(-kq, 6.28318548202514648f, ph);
            ph = fmaf(-kq, -1.7484556e-07f, ph);
            float s, c;
            __sincosf(ph, &s, &c);
            float ex, ey;
            if (HARD) {  // -i kappa (x^.n~) e
              const float xn = -fmaf(kx[d][0], n.x, fmaf(kx[d][1], n.y, kx[d][2] * n.z));  // kappa x^.n~
              ex = xn * s;
              ey = -xn * c;
            } else {     // -a e
              ex = -y.w * c;
              ey = -y.w * s;
            }
            const float2 exx = make_float2(ex, ex), eyy = make_float2(ey, ey), eyn = make_float2(-ey, -ey);
#pragma unroll
            for (int cc = 0; cc < FF_COLS / 2; ++cc) {
              ar[d][cc] = fma2x(exx, re[cc], fma2x(eyn, im[cc], ar[d][cc]));
              ai[d][cc] = fma2x(exx, im[cc], fma2x(eyy, re[cc], ai[d][cc]));
            }
          }
        }
      }
    }
    // the lanes' sums, 64 directions at a time, in the chunk buffers (16 KB)
    float2(*red)[FF_TH][FF_COLS] = reinterpret_cast<float2(*)[FF_TH][FF_COLS]>(&rre[0][0]);  // [2][64][8]
    static_assert(sizeof(float) * FF_CHUNK * FF_COLS >= sizeof(float2) * FF_TH * FF_COLS * 2, "reduction buffer");
    float2(*red2)[FF_TH][FF_COLS] = reinterpret_cast<float2(*)[FF_TH][FF_COLS]>(&rim[0][0]);
#pragma unroll
    for (int d = 0; d < DPT; ++d) {
      __syncthreads();
#pragma unroll
      for (int c = 0; c < FF_COLS; ++c) {
        const float2 v = c & 1 ? make_float2(ar[d][c / 2].y, ai[d][c / 2].y) : make_float2(ar[d][c / 2].x, ai[d][c / 2].x);
        (lane < 2 ? red : red2)[lane & 1][dl][c] = v;
      }
      __syncthreads();
      // a thread per direction: the group factor exp(-i kappa x^.C) once for its columns
      const int kk = k0 + FF_TH * d + (int)threadIdx.x;
      if (threadIdx.x < FF_TH && kk < n_dir) {
        double s2, c2;
        sincos(-A.kappa * (xhat[3 * kk] * C0 + xhat[3 * kk + 1] * C1 + xhat[3 * kk + 2] * C2v), &s2, &c2);
        s2 *= 0.25 / IGA_PI;
        c2 *= 0.25 / IGA_PI;
        for (int c = 0; c < nc; ++c) {
          double sx = 0.0, sy = 0.0;
          for (int l = 0; l < FF_LANES; ++l) {
            const float2 v = (l < 2 ? red : red2)[l & 1][threadIdx.x][c];
            sx += (double)v.x;
            sy += (double)v.y;
          }
          atomicAdd(&uinf[(long)kk * A.R + c0 + c].x, c2 * sx - s2 * sy);
          atomicAdd(&uinf[(long)kk * A.R + c0 + c].y, c2 * sy + s2 * sx);
        }
      }
    }
    __syncthreads();
  }
}

// ----------------------------------------------------------------------------------------------
// GMRES vector kernels; vectors are [N][R] complex, V_i = V + i N R

constexpr int RED_BLOCKS = 304;  // most chunks of a reduction over the vectors
constexpr int DOT_V = 4;         // basis vectors a block multiplies into (w is read once for them)

// threads of a reduction block in use: a multiple of R, so that a thread keeps its column
__device__ inline int red_threads(int R) { return ((int)blockDim.x / R) * R; }

// sum over the threads of a column (thread t has column t % R), for each of n values: the threads t < R get the sums.
// A tree in shared memory ([n][blockDim]); nthr = red_threads(R).
template <int n>
__device__ inline void red_columns(double2 (&v)[n], double2 *sh, int R, int nthr) {
  const int t = threadIdx.x;
#pragma unroll
  for (int k = 0; k < n; ++k) sh[k * blockDim.x + t] = v[k];
  __syncthreads();
  int rows = nthr / R;  // threads per column left
  while (rows > 1) {
    const int half = (rows + 1) / 2;
    if (t < (rows - half) * R)
#pragma unroll
      for (int k = 0; k < n; ++k) sh[k * blockDim.x + t] = cadd(sh[k * blockDim.x + t], sh[k * blockDim.x + t + half * R]);
    __syncthreads();
    rows = half;
  }
  if (t < R)
#pragma unroll
    for (int k = 0; k < n; ++k) v[k] = sh[k * blockDim.x + t];
}

// partial sums over chunk blockIdx.x: red[(i G + g) R + r] = sum_n conj(V_i[n][r]) w[n][r] for i <= j (j = *jdev; 0
// without it), DOT_V vectors per block
__global__ void __launch_bounds__(1024) k_dot_partial(const double2 *__restrict__ V, const int *__restrict__ jdev,
                                                      const double2 *__restrict__ w, long N, int R,
                                                      double2 *__restrict__ red) {
  extern __shared__ double2 shd[];
  const int j = jdev ? *jdev : 0, i0 = blockIdx.y * DOT_V, g = blockIdx.x, G = gridDim.x;
  if (i0 > j) return;
  const int nthr = red_threads(R), nv = min(DOT_V, j + 1 - i0);
  const long chunk = (N + G - 1) / G, n0 = g * chunk, n1 = min(N, n0 + chunk), NR = N * R;
  const double2 *Vi = V + (size_t)i0 * NR;
  double2 acc[DOT_V];
#pragma unroll
  for (int k = 0; k < DOT_V; ++k) acc[k] = cmk(0, 0);
  if ((int)threadIdx.x < nthr)
    for (long idx = n0 * R + threadIdx.x; idx < n1 * R; idx += nthr) {
      const double2 x = w[idx];
#pragma unroll
      for (int k = 0; k < DOT_V; ++k)
        if (k < nv) acc[k] = cadd(acc[k], cconjmul(Vi[k * NR + idx], x));
    }
  red_columns(acc, shd, R, nthr);
  if ((int)threadIdx.x < R)
    for (int k = 0; k < nv; ++k) red[((size_t)(i0 + k) * G + g) * R + threadIdx.x] = acc[k];
}

// h[i][r] for i <= j from the partial sums of G chunks, one warp each
__global__ void k_dot_final(const double2 *__restrict__ red, const int *__restrict__ jdev, int G, int R,
                            double2 *__restrict__ h) {
  const int o = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31, j = jdev ? *jdev : 0;
  if (o >= (j + 1) * R) return;
  const int i = o / R, r = o - i * R;
  double2 s = cmk(0, 0);
  for (int g = lane; g < G; g += 32) s = cadd(s, red[((size_t)i * G + g) * R + r]);
  for (int k = 16; k > 0; k >>= 1) {
    s.x += __shfl_xor_sync(0xffffffffu, s.x, k);
    s.y += __shfl_xor_sync(0xffffffffu, s.y, k);
  }
  if (lane == 0) h[o] = s;
}

__global__ void k_multiaxpy(const double2 *__restrict__ V, int nv, const double2 *__restrict__ h,
                            double2 *__restrict__ w, long N, int R) {
  GRID_STRIDE(o, N * R) {
    int r = int(o % R);
    double2 acc = w[o];
#pragma unroll 4
    for (int i = 0; i < nv; ++i) {
      acc = cadd(acc, cmul(V[(size_t)i * N * R + o], h[i * R + r]));
    }
    w[o] = acc;
  }
}

__global__ void k_scale(const double2 *__restrict__ w, const double *__restrict__ s, double2 *dst, double2 *dst2, long N,
                        int R) {
  GRID_STRIDE(o, N * R) {
    const double2 v = cscale(w[o], s[o % R]);
    dst[o] = v;
    dst2[o] = v;
  }
}

__global__ void k_sub(const double *__restrict__ b, const double *__restrict__ y, double *__restrict__ r, long n) {
  GRID_STRIDE(o, n) r[o] = b[o] - y[o];
}

__global__ void k_sqrt_re(const double2 *__restrict__ h, double *__restrict__ nrm, int R) {
  int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r < R) nrm[r] = sqrt(fmax(h[r].x, 0.0));
}

// ---- device-side GMRES iteration: the Arnoldi index j lives on the device, so one captured graph
// serves every iteration of a cycle (the kernels read j; grids are sized for the whole cycle).  On small systems the
// launches and the serial parts are what an iteration costs, so each reduction is a tree, the second
// Gram-Schmidt update also forms the partial sums of the norm, and V_{j+1} is written together with the copy
// that the next product reads.  Measured, one column, 1944 unknowns: 0.42 -> 0.12 ms an iteration beside the
// product (before, serial sums and 13 launches). ----

// w[n][r] -= sum_{i <= j} V_i[n][r] h[i][r]; with nrm2 != nullptr also the chunks' sums of |w|^2 (same layout as the
// partial sums of one vector)
__global__ void __launch_bounds__(1024) k_orth_update(const double2 *__restrict__ V, const int *__restrict__ jdev,
                                                      const double2 *__restrict__ h, double2 *__restrict__ w, long N,
                                                      int R, double2 *__restrict__ nrm2) {
  extern __shared__ double2 shd[];
  const int nv = *jdev + 1, g = blockIdx.x, G = gridDim.x, nthr = red_threads(R), r = threadIdx.x % R;
  const long chunk = (N + G - 1) / G, n0 = g * chunk, n1 = min(N, n0 + chunk), NR = N * R;
  double2 sum[1] = {cmk(0, 0)};
  if ((int)threadIdx.x < nthr)
    for (long idx = n0 * R + threadIdx.x; idx < n1 * R; idx += nthr) {
      double2 acc = w[idx];
#pragma unroll 4
      for (int i = 0; i < nv; ++i) acc = csub(acc, cmul(V[(size_t)i * NR + idx], h[i * R + r]));
      w[idx] = acc;
      sum[0].x = fma(acc.x, acc.x, fma(acc.y, acc.y, sum[0].x));
    }
  if (!nrm2) return;
  red_columns(sum, shd, R, nthr);
  if ((int)threadIdx.x < R) nrm2[(size_t)g * R + threadIdx.x] = sum[0];
}

// V_{j} = s w for the (already advanced) index j, and its copy vj
__global__ void k_scale_vj(const double2 *__restrict__ w, const double *__restrict__ s, double2 *__restrict__ V,
                           const int *__restrict__ jdev, long N, int R, double2 *__restrict__ vj) {
  double2 *dst = V + (size_t)(*jdev) * N * R;
  GRID_STRIDE(o, N * R) {
    const double2 v = cscale(w[o], s[o % R]);
    dst[o] = v;
    vj[o] = v;
  }
}

// cycle start: H, rotations and g cleared, g_0 = beta for the active columns, s = 1 / beta, j = 0
__global__ void k_gm_init(GmDev G, const double *__restrict__ beta, const int *__restrict__ active) {
  const int R = G.R, m = G.m;
  GRID_STRIDE(o, (long)(m + 1) * m * R) G.H[o] = cmk(0, 0);
  GRID_STRIDE(o, (long)m * R) {
    G.cs[o] = cmk(1, 0);
    G.sn[o] = cmk(0, 0);
  }
  GRID_STRIDE(o, (long)(m + 1) * R) G.g[o] = o < R && active[o] ? cmk(beta[o], 0) : cmk(0, 0);
  GRID_STRIDE(o, (long)R) {
    G.done[o] = active[o] ? 0 : 1;
    G.k[o] = 0;
    G.s[o] = active[o] ? 1.0 / beta[o] : 0.0;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    G.j[0] = G.j[1] = 0;
    G.flags[0] = 0;
    G.flags[1] = 0;
  }
}

// Arnoldi column j of every active right-hand side: h = hA + hB (the two Gram-Schmidt passes), the norm from its G
// partial sums nrm2, the new column of H rotated by the previous Givens rotations, the new rotation, g updated, the
// convergence test |g_{j+1}| <= tol ||b||; s = 1 / h_{j+1,j} for the next basis vector (0 for finished
// columns); then j advances.  A warp per column: its lanes load 32 entries and rotations at a time, lane 0 runs the
// recurrence over them, 16 FP64 instructions a rotation, which hold the FP64 pipe of a quarter of an SM for 0.6 us;
// so four warps a block, and as many blocks as the columns need (the last one to finish advances j).  200 iterations on
// 216 unknowns with 16, 64, 256 columns: 48, 51, 94 ms (all columns in one block of 16 warps 73, 181, 645 ms; a thread per
// column 95, 134, 174 ms).
// flags[0] = every column finished, flags[1] = non-finite met in the cycle; j[1] counts the blocks that are done.
constexpr int ARN_WARPS = 4;

__global__ void __launch_bounds__(32 * ARN_WARPS) k_gm_arnoldi(GmDev G, const double2 *__restrict__ nrm2, int chunks) {
  __shared__ double2 hs[ARN_WARPS][32], cv[ARN_WARPS][32], sv[ARN_WARPS][32];
  __shared__ int last, all_done, unfinished[ARN_WARPS];
  const int R = G.R, m = G.m, j = *G.j, wp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = blockIdx.x * ARN_WARPS + wp;
  if (lane == 0) unfinished[wp] = 0;
  if (r < R && G.done[r]) {
    if (lane == 0) G.s[r] = 0.0;
  } else if (r < R) {
    double n2 = 0.0;
    for (int g = lane; g < chunks; g += 32) n2 += nrm2[(size_t)g * R + r].x;
    for (int k = 16; k > 0; k >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, k);
    const double hn = sqrt(fmax(n2, 0.0));
    double2 *Hc = G.H + (size_t)r;  // H[i][jj][r] at ((i * m) + jj) * R + r
    double2 a = cmk(0, 0);          // lane 0: the entry that the next rotation (or the new one) starts from
    for (int i0 = 0; i0 <= j; i0 += 32) {
      const int i = i0 + lane, n = min(32, j + 1 - i0);
      __syncwarp();
      if (i <= j) hs[wp][lane] = cadd(G.hA[i * R + r], G.hB[i * R + r]);
      if (i < j) {
        cv[wp][lane] = G.cs[i * R + r];
        sv[wp][lane] = G.sn[i * R + r];
      }
      __syncwarp();
      if (lane == 0) {
        // entry i0 + k and the rotation of rows i0 + k - 1, i0 + k: the last entry of the previous 32 is in a
        if (i0 == 0) a = hs[wp][0];
        for (int k = i0 == 0 ? 1 : 0; k < n; ++k) {
          // rotation i0 + k - 1 (of the previous 32 for k = 0): [c, s; -conj(s), conj(c)] (a, b)
          const double2 c = k ? cv[wp][k - 1] : G.cs[(i0 - 1) * R + r], q = k ? sv[wp][k - 1] : G.sn[(i0 - 1) * R + r];
          const double2 b = hs[wp][k], t = cadd(cmul(c, a), cmul(q, b));
          a = cadd(cmul(cmk(-q.x, q.y), a), cmul(cmk(c.x, -c.y), b));
          if (k) hs[wp][k - 1] = t;
          else Hc[((size_t)(i0 - 1) * m + j) * R] = t;
        }
      }
      __syncwarp();
      if (lane < n - 1) Hc[((size_t)i * m + j) * R] = hs[wp][lane];
    }
    if (lane == 0) {
      const double den = sqrt(a.x * a.x + a.y * a.y + hn * hn);
      const double2 c = den > 0 ? cmk(a.x / den, -a.y / den) : cmk(1, 0);
      const double2 q = den > 0 ? cmk(hn / den, 0.0) : cmk(0, 0);
      G.cs[j * R + r] = c;
      G.sn[j * R + r] = q;
      Hc[((size_t)j * m + j) * R] = cmk(den, 0);
      Hc[((size_t)(j + 1) * m + j) * R] = cmk(0, 0);
      const double2 gj = G.g[j * R + r];
      const double2 gn = cmul(cmk(-q.x, q.y), gj);
      G.g[(j + 1) * R + r] = gn;
      G.g[j * R + r] = cmul(c, gj);
      G.k[r] = j + 1;
      const int its = ++G.its[r];
      const double res = sqrt(gn.x * gn.x + gn.y * gn.y);
      if (!isfinite(res) || !isfinite(hn)) atomicExch(&G.flags[1], 1);
      const bool done = res <= G.tol * G.bn[r] || its >= G.maxit || hn == 0.0 || j + 1 >= m;
      G.done[r] = done ? 1 : 0;
      G.s[r] = (!done && hn > 0) ? 1.0 / hn : 0.0;
      unfinished[wp] = !done;
    }
  }
  __syncthreads();
  if (gridDim.x == 1) {  // no other block to wait for
    if (threadIdx.x == 0) {
      int any = 0;
      for (int w = 0; w < ARN_WARPS; ++w) any |= unfinished[w];
      G.flags[0] = !any;
      G.j[0] = j + 1;
    }
    return;
  }
  if (threadIdx.x == 0) {
    __threadfence();  // the block's done[] and its read of j come before its count
    last = atomicAdd(&G.j[1], 1) == (int)gridDim.x - 1;
    all_done = 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int c = threadIdx.x; c < R; c += 32 * ARN_WARPS)
    if (!__ldcg(&G.done[c])) atomicExch(&all_done, 0);
  __syncthreads();
  if (threadIdx.x == 0) {
    G.flags[0] = all_done;
    G.j[0] = j + 1;
    G.j[1] = 0;
  }
}

// y = H^-1 g per column over its Krylov dimension k (zero beyond)
__global__ void k_gm_solve(GmDev G) {
  const int R = G.R, m = G.m;
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < R; r += gridDim.x * blockDim.x) {
    const int kc = G.k[r];
    for (int i = m; i >= 0; --i) G.y[i * R + r] = cmk(0, 0);
    for (int i = kc - 1; i >= 0; --i) {
      double2 acc = G.g[i * R + r];
      for (int q = i + 1; q < kc; ++q) acc = csub(acc, cmul(G.H[((size_t)i * m + q) * R + r], G.y[q * R + r]));
      const double2 d = G.H[((size_t)i * m + i) * R + r];
      const double dd = d.x * d.x + d.y * d.y;
      G.y[i * R + r] = dd > 0 ? cmk((acc.x * d.x + acc.y * d.y) / dd, (acc.y * d.x - acc.x * d.y) / dd) : cmk(0, 0);
    }
  }
}

RhsArgs rhs_args(const DeviceProblem &d, const HostSetup &S, const igabem_options &o, int R) {
  RhsArgs A;
  A.gpx = d.gpx; A.gpn = d.gpn; A.gpa = d.gpa; A.phi1 = d.phi1; A.gw = d.gw;
  A.g2x_ptr = d.g2x_ptr; A.g2x_idx = d.g2x_idx; A.dirs = nullptr;
  A.gst = (long)S.E * S.ng * S.ng; A.N = S.N;
  A.n1 = S.n1; A.nb = S.nb; A.p = S.p; A.ng = S.ng; A.R = R;
  A.h = S.h; A.kappa = o.kappa; A.eta = o.eta_cfie; A.hard = S.hard;
  A.kind = 0;
  return A;
}

}  // namespace

void launch_rhs(const DeviceProblem &d, const HostSetup &S, const igabem_options &o, int R,
                const double *dirs_dev, double *b, cudaStream_t st, int kind) {
  Phase ph(d.prof, IGABEM_PH_RHS, st);
  RhsArgs A = rhs_args(d, S, o, R);
  A.dirs = dirs_dev;
  A.kind = kind;
  k_rhs<<<grid_for(S.N * R), 256, 0, st>>>(A, reinterpret_cast<double2 *>(b));
  note_launch();
  IGA_CUDA(cudaGetLastError());
}

void launch_density(const DeviceProblem &d, const HostSetup &S, const igabem_options &o, int R, const double *dens,
                    double *rho, cudaStream_t st) {
  RhsArgs A = rhs_args(d, S, o, R);
  const long npts = (long)S.E * S.ng * S.ng;
  k_density<double2><<<grid_for(npts * ((R + 3) / 4)), 256, 0, st>>>(
      A, d.x2g, reinterpret_cast<const double2 *>(dens), S.E, reinterpret_cast<double2 *>(rho));
  note_launch();
  IGA_CUDA(cudaGetLastError());
}

void launch_farfield(const DeviceProblem &d, const HostSetup &S, const igabem_options &o, int R,
                     const double *dens, int n_dir, const double *xhat_dev, double *uinf, double *scratch,
                     cudaStream_t st) {
  if (R > 65535) fail(IGABEM_EINVAL, "the far field takes at most 65535 right-hand sides per call");
  Phase ph(d.prof, IGABEM_PH_FARFIELD, st);
  RhsArgs A = rhs_args(d, S, o, R);
  long npts = (long)S.E * S.ng * S.ng;
  double2 *rho = reinterpret_cast<double2 *>(scratch);  // E nq R complex values
  const int dgrid = grid_for(npts * ((R + 3) / 4));
  if (o.precision != IGABEM_FP64) {
    float2 *rho32 = reinterpret_cast<float2 *>(scratch);
    k_density<float2><<<dgrid, 256, 0, st>>>(A, d.x2g, reinterpret_cast<const double2 *>(dens), S.E, rho32);
    note_launch();
    const int fe = std::min(S.m, 4);
    const long ngroups = (long)S.np << (2 * (S.m - fe));
    IGA_CUDA(cudaMemsetAsync(uinf, 0, sizeof(double2) * (size_t)n_dir * R, st));
    // Directions a thread: more of them share a load, fewer make more blocks.  A launch lasts as long as the SM with the
    // most blocks; the measured milliseconds for k blocks on it (4096 points, 24 columns, sound-soft and sound-hard alike) with
    // one direction a thread are 0.54, 0.67, -, 1.15 for k = 1, 2, 3, 4, with two 0.82, 1.09, 1.53, with four 1.07, 1.8, 2.6;
    // the least of them is taken.  24 columns, one, two, four directions a thread: 6 groups, 3000 directions 0.67, 0.82, 1.07;
    // 6000: 1.15, 1.09, 1.07; 16 groups, 6000: 2.6, 2.4, 2.6; 24 groups, 3000: 2.4, 2.2, 1.9; 96 groups, 1000: 3.2, 3.2, 3.0 ms.
    struct Form {
      int dpt;
      double first, each;
    };
    int dpt = 1;
    double least = 1e300;
    for (const Form &f : {Form{1, 0.54, 0.29}, Form{2, 0.82, 0.51}, Form{4, 1.07, 0.88}}) {
      const long blocks = ngroups * ((n_dir + FF_TH * f.dpt - 1) / (FF_TH * f.dpt));
      const double t = std::max(f.first, f.each * ((blocks + 151) / 152));
      if (t < least) {
        least = t;
        dpt = f.dpt;
      }
    }
    auto go = [&](auto kfn) {
      const dim3 g32((unsigned)ngroups, (unsigned)((n_dir + FF_TH * dpt - 1) / (FF_TH * dpt)));
      kfn<<<g32, FF_LANES * FF_TH, 0, st>>>(A, rho32, fe, n_dir, xhat_dev, reinterpret_cast<double2 *>(uinf));
    };
    if (dpt == 4) S.hard ? go(k_farfield32<4, true>) : go(k_farfield32<4, false>);
    else if (dpt == 2) S.hard ? go(k_farfield32<2, true>) : go(k_farfield32<2, false>);
    else S.hard ? go(k_farfield32<1, true>) : go(k_farfield32<1, false>);
    note_launch();
    IGA_CUDA(cudaGetLastError());
    return;
  }
  k_density<double2><<<dgrid, 256, 0, st>>>(A, d.x2g, reinterpret_cast<const double2 *>(dens), S.E, rho);
  note_launch();
  const int per = R == 1 ? 1 : FF64_COLS, cols = (R + per - 1) / per;
  int nz = 1;
  while (nz < 8 && (long)n_dir * cols * nz < 4 * 152 && npts >= 1024L * nz) nz *= 2;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(n_dir, cols, nz);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = at.val.clusterDim.y = 1;
  at.val.clusterDim.z = nz;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  IGA_CUDA(cudaLaunchKernelEx(&cfg, R == 1 ? k_farfield<1> : k_farfield<FF64_COLS>, A, (const double2 *)rho, npts, xhat_dev,
                              reinterpret_cast<const double2 *>(d.cis), reinterpret_cast<double2 *>(uinf)));
  note_launch();
  IGA_CUDA(cudaGetLastError());
}

namespace {
// threads of the reduction kernels (whole columns; at least a warp's worth of columns per thread row) and chunks of the
// vectors: 8 elements a thread on small vectors, so that few partial sums are left
int dot_threads(int R) { return std::max(R, (256 / R) * R); }
int dot_chunks(long N, int R) { return (int)std::max<long>(1, std::min<long>(RED_BLOCKS, N * R / 2048)); }

void launch_dot(const double *V, const int *jdev, int most, const double *w, long N, int R, double *red, double2 *h,
                cudaStream_t st) {
  const int threads = dot_threads(R), G = dot_chunks(N, R);
  const size_t smem = sizeof(double2) * DOT_V * threads;
  IGA_CUDA(set_max_dynamic_smem(k_dot_partial, smem));
  k_dot_partial<<<dim3(G, (most + DOT_V - 1) / DOT_V), threads, smem, st>>>(
      reinterpret_cast<const double2 *>(V), jdev, reinterpret_cast<const double2 *>(w), N, R,
      reinterpret_cast<double2 *>(red));
  note_launch();
  k_dot_final<<<(most * R * 32 + 255) / 256, 256, 0, st>>>(reinterpret_cast<const double2 *>(red), jdev, G, R, h);
  note_launch();
  IGA_CUDA(cudaGetLastError());
}
}  // namespace

void launch_gm_iteration_tail(const GmDev &G, double *red, long N, double *vj, cudaStream_t st) {
  // two classical Gram-Schmidt passes against V_0..V_j, the norm, the Arnoldi update, the next basis vector
  const int R = G.R, threads = dot_threads(R), chunks = dot_chunks(N, R);
  for (int pass = 0; pass < 2; ++pass) {
    double2 *h = pass ? G.hB : G.hA;
    launch_dot(G.V, G.j, G.m + 1, G.w, N, R, red, h, st);
    // the update on finer chunks than the sums, up to the sums' scratch
    const int blocks = (int)std::max<long>(chunks, std::min<long>(RED_BLOCKS, (N * R + threads - 1) / threads));
    k_orth_update<<<blocks, threads, threads * sizeof(double2), st>>>(reinterpret_cast<const double2 *>(G.V), G.j, h,
                                                                      reinterpret_cast<double2 *>(G.w), N, R,
                                                                      pass ? reinterpret_cast<double2 *>(red) : nullptr);
    note_launch();
    if (pass) {
      k_gm_arnoldi<<<(R + ARN_WARPS - 1) / ARN_WARPS, 32 * ARN_WARPS, 0, st>>>(G, reinterpret_cast<const double2 *>(red), blocks);
      note_launch();
    }
  }
  k_scale_vj<<<grid_for(N * R), 256, 0, st>>>(reinterpret_cast<const double2 *>(G.w), G.s,
                                               reinterpret_cast<double2 *>(G.V), G.j, N, R,
                                               reinterpret_cast<double2 *>(vj));
  note_launch();
  IGA_CUDA(cudaGetLastError());
}

void launch_gm_init(const GmDev &G, const double *beta, const int *active, cudaStream_t st) {
  k_gm_init<<<grid_for((long)(G.m + 1) * G.m * G.R), 256, 0, st>>>(G, beta, active);
  note_launch();
}

void launch_gm_solve(const GmDev &G, cudaStream_t st) {
  k_gm_solve<<<(G.R + 127) / 128, 128, 0, st>>>(G);
  note_launch();
}

void launch_update(const double *V, int nv, const double *y, double *x, long N, int R, cudaStream_t st) {
  k_multiaxpy<<<grid_for(N * R), 256, 0, st>>>(reinterpret_cast<const double2 *>(V), nv,
                                                reinterpret_cast<const double2 *>(y),
                                                reinterpret_cast<double2 *>(x), N, R);
  note_launch();
}

void launch_norms(const double *w, long N, int R, double *red, double *nrm, cudaStream_t st) {
  double2 *h = reinterpret_cast<double2 *>(red) + (size_t)RED_BLOCKS * R;  // past the partial sums of one vector
  launch_dot(w, nullptr, 1, w, N, R, red, h, st);
  k_sqrt_re<<<(R + 255) / 256, 256, 0, st>>>(h, nrm, R);
  note_launch();
}

void launch_scale(const double *w, const double *s, double *dst, double *dst2, long N, int R, cudaStream_t st) {
  k_scale<<<grid_for(N * R), 256, 0, st>>>(reinterpret_cast<const double2 *>(w), s, reinterpret_cast<double2 *>(dst),
                                            reinterpret_cast<double2 *>(dst2), N, R);
  note_launch();
}

void launch_sub(const double *b, const double *y, double *r, long n, cudaStream_t st) {
  k_sub<<<grid_for(n), 256, 0, st>>>(b, y, r, n);
  note_launch();
}

}  // namespace igabem
