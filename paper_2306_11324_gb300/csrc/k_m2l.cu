// M2L: couplings of admissible cluster pairs (Sec. 4.4), FP64 and FP32: kernel samples between the
// Chebyshev nodes generated on the fly (k_m2l_fly; k_m2l_gemm for many columns); the blocks stored at
// set-up (m2l_stored) are generated here and applied in k_stream.cu.  All levels go in one launch, each with its own q (level-adaptive
// interpolation), one block (or a cluster of blocks) per target cluster.
//
// FP32 phase split: the sample phase kappa r is formed as kappa |D| (D = c_t - c_s, the distance of
// the two cluster centres, taken in FP64 once per pair and reduced mod 2 pi) plus kappa (r - |D|),
// with r - |D| = (2 D.delta + |delta|^2)/(r + |D|) computed in FP32 from the node offsets
// delta = (x_a - c_t) - (y_b - c_s).  The FP32 error of the phase is then of the order of the
// cluster size times the unit roundoff instead of kappa r times it, and the factor
// exp(i kappa |D|) multiplies the pair's partial sums once.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "k_common.cuh"
#include "kernels.h"
#include "k_m2l.cuh"

namespace igabem {

namespace {


struct M2LLevel {
  const int *far_ptr, *far_src;
  const double *nodes;   // FP64 [7][n q^2]: x, n~, a
  const float *nodes32;  // FP32 [7][n q^2]: x - c, n~, a
  const float *pc;       // FP32 pair constants [n_far][8]: D, |D|, |D|^2, cos, sin of kappa|D| (FP32 path)
  const double2 *xhat;
  const float2 *xhat32;  // FP32 copy of xhat (the FP32 kernels read it)
  double2 *yhat;
  int n;                 // clusters on the level
  int first;             // first block index of the level in the flattened grid
  int q, Q;              // interpolation points per direction / per cluster on the level
};

struct M2LArgs {
  M2LLevel lev[16];
  int nlev;
  int QS;                // source nodes per warp in shared memory (the largest Q of the launch)
  int CR, R;
  double kappa, eta;
  bool hard;
  const double2 *cis;    // exp(2 pi i k / CIS_N), k < CIS_N
  int rows_most;         // P Q of the level that uses most of a block's threads (k_m2l_fly)
};

// Per-source-node data in shared memory: position (FP32: its offset from the cluster centre), the
// Jacobian (soft; FP64: / (4 pi)) or the normal (hard), and in FP32 the products with D = c_t - c_s.
template <class T, bool HARD> struct FlyNode;
template <> struct __align__(16) FlyNode<double, false> { double y[3], a; };
template <> struct __align__(16) FlyNode<double, true> { double y[3], n[3]; };
template <> struct __align__(16) FlyNode<float, false> { float y[3], Dy, a, pad[3]; };
template <> struct __align__(16) FlyNode<float, true> { float y[3], Dy, n[3], Dn; };

// M2L with the samples generated on the fly.  A thread owns one target node of one pair: the Q nodes of P
// pairs (P = 256 / Q) lie side by side in a block's 256 threads (Q = 49: 245 of them at work; one warp
// per pair with two rows a lane used 49 of 64).  It generates its row of the pair's coupling block in
// registers, reading the source nodes from shared memory, and multiplies it into NC columns: for
// sound-hard one sample gives K and G, which serve the columns of all seven channels.  Sums: the pair's in
// registers, then over the thread's pairs (FP32: see FLY_BLOCK), then over the P threads of a node and over the blocks
// of a cluster, in that fixed order (FP64).  A target's interaction list is split over a cluster of
// gridDim.y blocks, which add their sums through distributed shared memory, where a level has too few
// targets to fill the device.  Measured on GB300, FP64 products (before: one warp per pair, 72 FP64
// instructions a sample and CUDA's sincos, or for several columns the tile of k_m2l_gemm mostly padding): 6936
// unknowns, one column, 175 M samples 32.2 -> 16.3 ms; 150 unknowns, 8 M samples 2.20 -> 0.89 ms; sound-hard,
// 1736 unknowns, 3 columns of 7 channels 41 -> 4 ms.
// FP32 sums: FLY_BLOCK source nodes at a time within a pair.  Over the pairs: the sum and its rounding errors, in registers
// for up to 4 columns, in shared memory for up to 16 (their registers would cost them a second block on the SM); wider
// forms, which run one block anyway, add FLY_PAIRS pairs at a time in registers (shared memory costs them 6 %, by the L1
// it takes).
// Far rows against FP64 (rms; one chain of q^2 products and of all pairs -> this): q = 12 1.06 -> 1.04e-7, q = 16, short
// lists 6.8 -> 5.2e-8; 6144 elements, q = 7, lists of 256 pairs 9.4 -> 8.8e-8.  Time against the single chain, 1536
// elements: 1 to 4 columns 0.41 -> 0.38 (one), 0.54 -> 0.48 ms (four), 8 and 16 within 2 %, 24 2.25 -> 2.10 ms, 21
// (sound-hard) 2.34 -> 2.39 ms; where a target has few pairs the sums in shared memory show (1024 elements of a torus,
// 8 columns 0.26 -> 0.29 ms).
constexpr int FLY_BLOCK = 16, FLY_PAIRS = 8;
template <class T, int NC> constexpr bool fly_sums = std::is_same<T, float>::value && NC > 4 && NC <= 16;

// bytes in front of the nodes: the table of phase64, or the sums of the FP32 form
template <class T, int NC> __host__ __device__ constexpr size_t fly_head() {
  return fly_sums<T, NC> ? (size_t)NC * 256 * sizeof(float4) : std::is_same<T, float>::value ? 0 : CIS_N * sizeof(double2);
}

template <class T, int NC, bool HARD>
__global__ void __launch_bounds__(256) k_m2l_fly(const __grid_constant__ M2LArgs A) {
  extern __shared__ __align__(16) unsigned char smf[];
  constexpr bool F32 = std::is_same<T, float>::value, SUMS = fly_sums<T, NC>;
  using Node = FlyNode<T, HARD>;
  const int tid = threadIdx.x, nsplit = gridDim.y, rank = blockIdx.y, cr0 = blockIdx.z * NC;
  int li = 0;
  while (li + 1 < A.nlev && (int)blockIdx.x >= A.lev[li + 1].first) ++li;
  const M2LLevel &L = A.lev[li];
  const int t = blockIdx.x - L.first, Q = L.Q, P = 256 / Q, slot = tid / Q, a = tid - slot * Q;
  const long NQ = (long)L.n * Q;
  const int ncr = min(NC, A.CR - cr0);
  double2 *tab = reinterpret_cast<double2 *>(smf);                       // FP64: the table of phase64
  float4 *sums = reinterpret_cast<float4 *>(smf);                        // SUMS: [NC][256], sum and its rounding errors
  Node *src = reinterpret_cast<Node *>(smf + fly_head<T, NC>());         // [P Q]
  C2<T> *xs = reinterpret_cast<C2<T> *>(src + A.rows_most);              // [P Q][NC]
  C2<T> *red = xs;
  if constexpr (SUMS) {
#pragma unroll
    for (int c = 0; c < NC; ++c) sums[c * 256 + tid] = make_float4(0.f, 0.f, 0.f, 0.f);
  } else if constexpr (!F32) {
    for (int i = tid; i < CIS_N; i += 256) tab[i] = A.cis[i];
  }
  double c0, c1;
  phase64_scale(A.kappa, c0, c1);
  const T kappa = (T)A.kappa, eta = (T)A.eta;
  const bool on = slot < P;
  T tx[3] = {0, 0, 0}, tn[3] = {0, 0, 0}, ta = 0;
  if (on) {
    const long ia = (long)t * Q + a;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      tx[c] = F32 ? (T)L.nodes32[c * NQ + ia] : (T)L.nodes[c * NQ + ia];
      if (!HARD) tn[c] = F32 ? (T)L.nodes32[(3 + c) * NQ + ia] : (T)L.nodes[(3 + c) * NQ + ia];
    }
    ta = F32 ? (T)L.nodes32[6 * NQ + ia] : (T)L.nodes[6 * NQ + ia];
    if (!HARD) ta *= eta;
  }
  // FP32: few has the rounding errors of tot (up to 4 columns), or the last FLY_PAIRS pairs at most (above 16)
  C2<T> tot[SUMS ? 1 : NC], few[F32 && !SUMS ? NC : 1];
  int kept = 0;
  if constexpr (!SUMS) {
#pragma unroll
    for (int c = 0; c < NC; ++c) tot[c] = c2((T)0, (T)0);
    if constexpr (F32) {
#pragma unroll
      for (int c = 0; c < NC; ++c) few[c] = c2((T)0, (T)0);
    }
  }
  const int k0 = L.far_ptr[t], np = L.far_ptr[t + 1] - k0;
  for (int p0 = rank * P; p0 < np; p0 += nsplit * P) {
    const bool work = on && p0 + slot < np;
    const int kk = k0 + p0 + slot;
    T D[3] = {0, 0, 0}, Dn = 0, D2 = 0;
    C2<T> e0 = c2((T)1, (T)0);
    __syncthreads();  // the previous pairs' nodes and columns are read
    if (work) {
      if constexpr (F32) {
        const float4 q0 = reinterpret_cast<const float4 *>(L.pc)[2 * (long)kk];
        const float4 q1 = reinterpret_cast<const float4 *>(L.pc)[2 * (long)kk + 1];
        D[0] = q0.x; D[1] = q0.y; D[2] = q0.z; Dn = q0.w;
        D2 = q1.x;
        e0 = c2(q1.y, q1.z);
      }
      // the thread stages the source node with its own index
      const long ib = (long)L.far_src[kk] * Q + a;
      Node sn;
      T nn[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        sn.y[c] = F32 ? (T)L.nodes32[c * NQ + ib] : (T)L.nodes[c * NQ + ib];
        if (HARD) nn[c] = F32 ? (T)L.nodes32[(3 + c) * NQ + ib] : (T)L.nodes[(3 + c) * NQ + ib];
      }
      if constexpr (HARD) {
#pragma unroll
        for (int c = 0; c < 3; ++c) sn.n[c] = nn[c];
        if constexpr (F32) sn.Dn = D[0] * nn[0] + D[1] * nn[1] + D[2] * nn[2];
      } else {
        sn.a = F32 ? (T)L.nodes32[6 * NQ + ib] : (T)(L.nodes[6 * NQ + ib] * (0.25 / IGA_PI));
      }
      if constexpr (F32) sn.Dy = D[0] * sn.y[0] + D[1] * sn.y[1] + D[2] * sn.y[2];
      src[tid] = sn;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        C2<T> v = c2((T)0, (T)0);
        if (c < ncr) {
          if constexpr (F32) {
            const float2 w = L.xhat32[ib * A.CR + cr0 + c];
            v = c2((T)w.x, (T)w.y);
          } else {
            const double2 w = L.xhat[ib * A.CR + cr0 + c];
            v = c2((T)w.x, (T)w.y);
          }
        }
        xs[tid * NC + c] = v;
      }
    }
    __syncthreads();
    if (!work) continue;
    C2<T> part[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) part[c] = c2((T)0, (T)0);
    const Node *sp = src + slot * Q;
    const C2<T> *xp = xs + slot * Q * NC;
    const T Ddx = D[0] * tx[0] + D[1] * tx[1] + D[2] * tx[2];
    const T Dnx = D[0] * tn[0] + D[1] * tn[1] + D[2] * tn[2];
    auto add_node = [&](int b, C2<T> (&sum)[NC]) {
      const Node y = sp[b];
      const T d0 = tx[0] - y.y[0], d1 = tx[1] - y.y[1], d2 = tx[2] - y.y[2];
      C2<T> S0, S1 = c2((T)0, (T)0);  // soft: S0; hard: S0 = K, S1 = G
      if constexpr (F32) {
        const T num = (T)2 * (Ddx - y.Dy) + (d0 * d0 + d1 * d1 + d2 * d2);
        const T r2 = D2 + num, ir = rsqrtf(r2), r = r2 * ir;
        T ph = kappa * __fdividef(num, r + Dn);
        const T kq = rintf(ph * 0.15915494309189535f);
        ph = fmaf(-kq, 6.28318548202514648f, ph);
        ph = fmaf(-kq, -1.7484556e-07f, ph);
        T sph, cph;
        __sincosf(ph, &sph, &cph);
        const T f = ir * (T)(0.25 / IGA_PI), kr = kappa * r, g2 = f * ir * ir;
        const C2<T> G = c2(cph * f, sph * f);
        const C2<T> dG = c2((-cph - sph * kr) * g2, (-sph + cph * kr) * g2);
        if constexpr (!HARD) {
          const T w1 = y.a * (Dnx + d0 * tn[0] + d1 * tn[1] + d2 * tn[2]), w2 = ta * y.a;
          S0 = c2(dG.x * w1 + G.y * w2, dG.y * w1 - G.x * w2);
        } else {
          const T w1 = -ta * (y.Dn + d0 * y.n[0] + d1 * y.n[1] + d2 * y.n[2]);
          S0 = c2(dG.x * w1, dG.y * w1);
          S1 = G;
        }
      } else {
        const double r2 = d0 * d0 + d1 * d1 + d2 * d2, ir = rsqrt64(r2);
        const Phase64 ph = phase64(tab, r2 * ir, c0, c1);
        if constexpr (!HARD) {
          // exp(i kappa r) (A + i B), with w = a_y / (4 pi r): A = -w (d.n)/r^2, B = kappa w (d.n)/r - eta a_x w
          const double w = y.a * ir, gw = (d0 * tn[0] + d1 * tn[1] + d2 * tn[2]) * ir * w;
          const double Ar = -gw * ir, Br = fma(kappa, gw, -(ta * w));
          S0 = phase_mul(ph.E.x * Ar - ph.E.y * Br, ph.E.x * Br + ph.E.y * Ar, ph);
        } else {
          // G = exp(i kappa r) / (4 pi r); K = G (A + i B), w = -a_x (d.n_y) / r: A = -w / r, B = kappa w
          const double f = ir * (0.25 / IGA_PI);
          S1 = phase_mul(ph.E.x * f, ph.E.y * f, ph);
          const double w = -ta * (d0 * y.n[0] + d1 * y.n[1] + d2 * y.n[2]) * ir, Ar = -w * ir, Br = kappa * w;
          S0 = c2(S1.x * Ar - S1.y * Br, S1.x * Br + S1.y * Ar);
        }
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const bool k = !HARD || cr0 + c < A.R;  // the first R columns are channel 0
        sum[c] = fma2(k ? S0 : S1, xp[b * NC + c], sum[c]);
      }
    };
    if constexpr (F32) {
      int b = 0;
      for (; b + FLY_BLOCK <= Q; b += FLY_BLOCK) {
        C2<T> sum[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) sum[c] = c2((T)0, (T)0);
#pragma unroll
        for (int u = 0; u < FLY_BLOCK; ++u) add_node(b + u, sum);
#pragma unroll
        for (int c = 0; c < NC; ++c) part[c] = add(part[c], sum[c]);
      }
      for (; b < Q; ++b) add_node(b, part);
      if constexpr (SUMS) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const C2<T> v = mul(e0, part[c]);
          float4 w = sums[c * 256 + tid];
          two_sum(w.x, w.z, v.x);
          two_sum(w.y, w.w, v.y);
          sums[c * 256 + tid] = w;
        }
      } else if constexpr (NC <= 4) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const C2<T> v = mul(e0, part[c]);
          two_sum(tot[c].x, few[c].x, v.x);
          two_sum(tot[c].y, few[c].y, v.y);
        }
      } else {
#pragma unroll
        for (int c = 0; c < NC; ++c) few[c] = fma2(e0, part[c], few[c]);
        if (++kept == FLY_PAIRS) {
          kept = 0;
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            tot[c] = add(tot[c], few[c]);
            few[c] = c2((T)0, (T)0);
          }
        }
      }
    } else {
      // nodes at a time: 4 columns, 175 M samples 22.3 -> 21.1 ms with four; sound-hard, one column of 7 channels, 8 M
      // samples 1.43 -> 1.37 ms with two
      if constexpr (NC == 4) {
#pragma unroll 4
        for (int b = 0; b < Q; ++b) add_node(b, part);
      } else if constexpr (NC == 7) {
#pragma unroll 2
        for (int b = 0; b < Q; ++b) add_node(b, part);
      } else {
        for (int b = 0; b < Q; ++b) add_node(b, part);
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) tot[c] = add(tot[c], part[c]);
    }
  }
  // sums over the P threads of a node and the blocks of the cluster
  if constexpr (!SUMS) {
    __syncthreads();
    if (on)
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if constexpr (F32) tot[c] = add(tot[c], few[c]);
        red[tid * NC + c] = tot[c];
      }
  }
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  if (nsplit > 1) cl.sync();
  else __syncthreads();
  const int per = (Q * ncr + nsplit - 1) / nsplit, o1 = min(Q * ncr, (rank + 1) * per);
  for (int o = rank * per + tid; o < o1; o += 256) {
    const int aa = o / ncr, c = o - aa * ncr;
    double2 sum = make_double2(0, 0);
    for (int z = 0; z < nsplit; ++z) {
      if constexpr (SUMS) {
        const float4 *sz = nsplit > 1 ? cl.map_shared_rank(sums, z) : sums;
        for (int p = 0; p < P; ++p) {
          const float4 v = sz[c * 256 + p * Q + aa];
          sum.x += (double)v.x + (double)v.z;
          sum.y += (double)v.y + (double)v.w;
        }
      } else {
        const C2<T> *rz = nsplit > 1 ? cl.map_shared_rank(red, z) : red;
        for (int p = 0; p < P; ++p) {
          const C2<T> v = rz[(p * Q + aa) * NC + c];
          sum.x += (double)v.x;
          sum.y += (double)v.y;
        }
      }
    }
    L.yhat[((long)t * Q + aa) * A.CR + cr0 + c] = sum;
  }
  if (nsplit > 1) cl.sync();  // no block leaves while another reads its shared memory
}

// ---- stored coupling blocks (m2l_stored): the same kernel samples (node_sample, the samples of the
// multi-column M2L) generated once per problem, then streamed by every product ----

// one thread block per admissible pair k of a level: every entry S_k[type][b][a] (column-major: the
// target node a runs fastest) with the pair factor exp(i kappa |D|) folded in (FP32 path)
template <class T>
__global__ void __launch_bounds__(256) k_m2l_fill(M2LLevel L, bool hard, double kappa, double eta,
                                                  C2<T> *__restrict__ out) {
  constexpr bool F32 = std::is_same<T, float>::value;
  const long kk = blockIdx.x;
  const int Q = L.Q, ntype = hard ? 2 : 1;
  const long NQ = (long)L.n * Q;
  int lo = 0, hi = L.n;  // target t with far_ptr[t] <= kk < far_ptr[t + 1]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (L.far_ptr[mid] <= kk) lo = mid;
    else hi = mid;
  }
  const int t = lo, s = L.far_src[kk];
  T D[3] = {0, 0, 0}, Dn = 0, D2 = 0;
  C2<T> e0 = c2((T)1, (T)0);
  if constexpr (F32) {
    const float *pc = L.pc + 8 * kk;
    D[0] = pc[0]; D[1] = pc[1]; D[2] = pc[2]; Dn = pc[3]; D2 = pc[4];
    e0 = c2(pc[5], pc[6]);
  }
  C2<T> *S = out + kk * (long)ntype * Q * Q;
  for (int o = threadIdx.x; o < ntype * Q * Q; o += blockDim.x) {
    const int ty = o / (Q * Q), b = (o / Q) % Q, a = o % Q;
    T X[7], Y[7];
    for (int c = 0; c < 7; ++c) {
      X[c] = F32 ? (T)L.nodes32[c * NQ + (long)t * Q + a] : (T)L.nodes[c * NQ + (long)t * Q + a];
      Y[c] = F32 ? (T)L.nodes32[c * NQ + (long)s * Q + b] : (T)L.nodes[c * NQ + (long)s * Q + b];
    }
    const int type = hard ? (ty == 0 ? 1 : 2) : 0;
    const C2<T> v = node_sample<T>(type, X, X + 3, X[6], Y, Y + 3, Y[6], D, Dn, D2, (T)kappa, (T)eta);
    S[o] = F32 ? mul(e0, v) : v;
  }
}

// Multi-column M2L: per target cluster and column chunk, every coupling block S_ts (q^2 x q^2) is
// generated once into shared memory and applied to the chunk's columns of xhat_s with a register
// tiled product (4 x 4 complex outputs per thread).  A chunk lies within one channel, so one kernel
// type per block.
constexpr int GEMM_T = 16;  // thread tile grid 16 x 16

template <class T>
__global__ void __launch_bounds__(256) k_m2l_gemm(M2LArgs A, int Wc) {
  extern __shared__ __align__(16) unsigned char smg[];
  constexpr bool F32 = std::is_same<T, float>::value;
  int li = 0;
  while (li + 1 < A.nlev && (int)blockIdx.x >= A.lev[li + 1].first) ++li;
  const M2LLevel &L = A.lev[li];
  const int t = blockIdx.x - L.first;
  const int Q = L.Q;  // <= 64 (4 x 16 thread rows)
  const long NQ = (long)L.n * Q;
  const int cr0 = blockIdx.y * Wc, ch = cr0 / A.R;
  const int type = A.hard ? (ch == 0 ? 1 : 2) : 0;
  C2<T> *S = reinterpret_cast<C2<T> *>(smg);            // [Q][Q]
  C2<T> *Xs = S + Q * Q;                                 // [Q][Wc]
  T *tn = reinterpret_cast<T *>(Xs + Q * Wc);            // target nodes [Q][8]
  T *sn = tn + Q * 8;                                    // source nodes [Q][8]
  const T kappa = (T)A.kappa, eta = (T)A.eta;
  for (int a = threadIdx.x; a < Q; a += blockDim.x) {
    long ia = (long)t * Q + a;
    for (int c = 0; c < 7; ++c) tn[a * 8 + c] = F32 ? (T)L.nodes32[c * NQ + ia] : (T)L.nodes[c * NQ + ia];
  }
  const int ty = threadIdx.x / GEMM_T, tx = threadIdx.x % GEMM_T;
  C2<T> acc[4][4];
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j) acc[i][j] = c2((T)0, (T)0);
  for (int kk = L.far_ptr[t]; kk < L.far_ptr[t + 1]; ++kk) {
    const int s = L.far_src[kk];
    T D[3] = {0, 0, 0}, Dn = 0, D2 = 0;
    C2<T> e0 = c2((T)1, (T)0);
    if constexpr (F32) {
      const float4 p0 = reinterpret_cast<const float4 *>(L.pc)[2 * kk];
      const float4 p1 = reinterpret_cast<const float4 *>(L.pc)[2 * kk + 1];
      D[0] = p0.x; D[1] = p0.y; D[2] = p0.z; Dn = p0.w;
      D2 = p1.x;
      e0 = c2(p1.y, p1.z);
    }
    __syncthreads();  // previous contraction done with S, Xs, sn
    for (int b = threadIdx.x; b < Q; b += blockDim.x) {
      long ib = (long)s * Q + b;
      for (int c = 0; c < 7; ++c) sn[b * 8 + c] = F32 ? (T)L.nodes32[c * NQ + ib] : (T)L.nodes[c * NQ + ib];
    }
    for (int i = threadIdx.x; i < Q * Wc; i += blockDim.x) {
      int b = i / Wc, c = i % Wc;
      C2<T> xv;
      if constexpr (F32) {
        const float2 v = L.xhat32[((long)s * Q + b) * A.CR + cr0 + c];
        xv = c2((T)v.x, (T)v.y);
      } else {
        const double2 v = L.xhat[((long)s * Q + b) * A.CR + cr0 + c];
        xv = c2((T)v.x, (T)v.y);
      }
      // the pair factor exp(i kappa |D|) is folded into the source coefficients
      Xs[i] = F32 ? mul(e0, xv) : xv;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < Q * Q; i += blockDim.x) {
      int a = i / Q, b = i % Q;
      const T *X = tn + a * 8, *Y = sn + b * 8;
      S[i] = node_sample<T>(type, X, X + 3, X[6], Y, Y + 3, Y[6], D, Dn, D2, kappa, eta);
    }
    __syncthreads();
    C2<T> part[4][4];  // this pair's sums (blocked accumulation)
    for (int i = 0; i < 4; ++i)
      for (int j = 0; j < 4; ++j) part[i][j] = c2((T)0, (T)0);
    for (int b = 0; b < Q; ++b) {
      C2<T> sv[4], xv[4];
      for (int i = 0; i < 4; ++i) {
        int a = ty + GEMM_T * i;
        sv[i] = a < Q ? S[a * Q + b] : c2((T)0, (T)0);
      }
      for (int j = 0; j < 4; ++j) {
        int c = tx + GEMM_T * j;
        xv[j] = c < Wc ? Xs[b * Wc + c] : c2((T)0, (T)0);
      }
      for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) part[i][j] = fma2(sv[i], xv[j], part[i][j]);
    }
    for (int i = 0; i < 4; ++i)
      for (int j = 0; j < 4; ++j) acc[i][j] = add(acc[i][j], part[i][j]);
  }
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j) {
      int a = ty + GEMM_T * i, c = tx + GEMM_T * j;
      if (a < Q && c < Wc)
        L.yhat[((long)t * Q + a) * A.CR + cr0 + c] = make_double2((double)acc[i][j].x, (double)acc[i][j].y);
    }
}

// pair constants, per admissible pair k of a level (CSR order):
// [D (3), |D|, |D|^2, cos(kappa |D|), sin(kappa |D|), sigma] with D = c_t - c_s in FP64 and sigma a power
// of two that scales the pair's coupling block to at most 2^12 in magnitude (used by the FP16 operands
// of the tensor-core M2L).  sigma comes from a bound on the kernel samples over the two clusters' nodes:
// with rho the largest node distance from the cluster centre and a_max the largest Jacobian,
// |x - y| lies in [|D| - rho_t - rho_s, |D| + rho_t + rho_s] and every kernel type is at most
// (1 + kappa r_hi)(1 + a_t)(1 + a_s)(1 + |eta|) / (4 pi r_lo).
// per cluster: rho = the largest node distance from the centre, a_max = the largest node Jacobian
__global__ void k_cluster_extent(const double *__restrict__ nodes, const double *__restrict__ center, int n, int Q,
                                 double2 *__restrict__ ext) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  const long NQ = (long)n * Q;
  double rho = 0.0, amax = 0.0;
  for (int a = 0; a < Q; ++a) {
    const long i = (long)c * Q + a;
    const double dx = nodes[i] - center[3 * c], dy = nodes[NQ + i] - center[3 * c + 1],
                 dz = nodes[2 * NQ + i] - center[3 * c + 2];
    rho = fmax(rho, sqrt(dx * dx + dy * dy + dz * dz));
    amax = fmax(amax, nodes[6 * NQ + i]);
  }
  ext[c] = make_double2(rho, amax);
}

// one thread per admissible pair k (CSR order), its target t from the row pointers
__global__ void k_pair_consts(const int *__restrict__ far_ptr, const int *__restrict__ far_src,
                              const double *__restrict__ center, const double2 *__restrict__ ext, int n, long nfar,
                              double kappa, double eta, float *__restrict__ pc) {
  const long k = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (k >= nfar) return;
  int lo = 0, hi = n;  // t with far_ptr[t] <= k < far_ptr[t + 1]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (far_ptr[mid] <= k) lo = mid;
    else hi = mid;
  }
  const int t = lo, s = far_src[k];
  double D[3] = {center[3 * t] - center[3 * s], center[3 * t + 1] - center[3 * s + 1],
                 center[3 * t + 2] - center[3 * s + 2]};
  double nD = sqrt(D[0] * D[0] + D[1] * D[1] + D[2] * D[2]);
  double sn, cs;
  sincos(fmod(kappa * nD, TWO_PI), &sn, &cs);
  const double2 et = ext[t], es = ext[s];
  const double r_lo = fmax(nD - et.x - es.x, 1e-3 * nD), r_hi = nD + et.x + es.x;
  const double bound = (1.0 + kappa * r_hi) * (1.0 + et.y) * (1.0 + es.y) * (1.0 + fabs(eta)) / (4.0 * IGA_PI * r_lo);
  float *o = pc + 8L * k;
  o[0] = (float)D[0]; o[1] = (float)D[1]; o[2] = (float)D[2]; o[3] = (float)nD;
  o[4] = (float)(nD * nD); o[5] = (float)cs; o[6] = (float)sn;
  o[7] = (float)exp2(12.0 - ceil(log2(bound)));
}

template <class T, int NC, bool HARD>
void launch_fly(const M2LArgs &A, int nblocks, int nsplit, cudaStream_t st) {
  const size_t smem = fly_head<T, NC>() + (size_t)A.rows_most * (sizeof(FlyNode<T, HARD>) + NC * sizeof(C2<T>));
  auto kfn = k_m2l_fly<T, NC, HARD>;
  IGA_CUDA(set_max_dynamic_smem(kfn, smem));
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(nblocks, nsplit, (A.CR + NC - 1) / NC);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = 1;
  at.val.clusterDim.y = nsplit;
  at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  IGA_CUDA(cudaLaunchKernelEx(&cfg, kfn, A));
  note_launch();
}

// All columns, in passes of at most 24 (the FP64 accumulators of 24 columns fill the registers; each pass
// generates the samples again), sound-hard 21 (three columns of seven channels), the passes as even as the kernel's
// column counts allow.
template <class T>
void launch_fly_all(const M2LArgs &A, int nblocks, int nsplit, cudaStream_t st) {
  const int most = A.hard ? 21 : 24, passes = (A.CR + most - 1) / most, w = (A.CR + passes - 1) / passes;
  if (A.hard) {
    if (w > 14) launch_fly<T, 21, true>(A, nblocks, nsplit, st);
    else if (w > 7) launch_fly<T, 14, true>(A, nblocks, nsplit, st);
    else launch_fly<T, 7, true>(A, nblocks, nsplit, st);
  } else if (w > 16) {
    launch_fly<T, 24, false>(A, nblocks, nsplit, st);
  } else if (w > 8) {
    launch_fly<T, 16, false>(A, nblocks, nsplit, st);
  } else if (w > 4) {
    launch_fly<T, 8, false>(A, nblocks, nsplit, st);
  } else if (w > 2) {
    launch_fly<T, 4, false>(A, nblocks, nsplit, st);
  } else if (w == 2) {
    launch_fly<T, 2, false>(A, nblocks, nsplit, st);
  } else {
    launch_fly<T, 1, false>(A, nblocks, nsplit, st);
  }
}

}  // namespace

void launch_pair_consts(const DeviceProblem &d, const HostSetup &S, double kappa, double eta, cudaStream_t st) {
  for (int l = S.lmin; l <= S.L; ++l) {
    int n = S.lev[l].n;
    const long nfar = (long)S.lev[l].far_src.size();
    k_cluster_extent<<<(n + 127) / 128, 128, 0, st>>>(d.nodes[l], d.centers[l], n, S.lev[l].q * S.lev[l].q,
                                                      reinterpret_cast<double2 *>(d.cext[l]));
    note_launch();
    if (nfar == 0) continue;
    k_pair_consts<<<(int)((nfar + 255) / 256), 256, 0, st>>>(d.far_ptr[l], d.far_src[l], d.centers[l],
                                                             reinterpret_cast<const double2 *>(d.cext[l]), n, nfar,
                                                             kappa, eta, d.pairc[l]);
    note_launch();
  }
  IGA_CUDA(cudaGetLastError());
}

size_t m2l_stored_entries(const HostSetup &S, int l) {
  const size_t Q = (size_t)S.lev[l].q * S.lev[l].q;
  return S.lev[l].far_src.size() * Q * Q * (S.hard ? 2 : 1);
}

void launch_m2l_fill(const DeviceProblem &d, const HostSetup &S, const igabem_options &o, cudaStream_t st) {
  const bool fp32 = o.precision != IGABEM_FP64;
  for (int l = S.lmin; l <= S.L; ++l) {
    const long nfar = (long)S.lev[l].far_src.size();
    if (nfar == 0) continue;
    M2LLevel L{};
    L.far_ptr = d.far_ptr[l];
    L.far_src = d.far_src[l];
    L.nodes = d.nodes[l];
    L.nodes32 = d.nodes32[l];
    L.pc = d.pairc[l];
    L.n = S.lev[l].n;
    L.q = S.lev[l].q;
    L.Q = L.q * L.q;
    if (fp32)
      k_m2l_fill<float><<<(unsigned)nfar, 256, 0, st>>>(L, S.hard, o.kappa, o.eta_cfie,
                                                        reinterpret_cast<C2<float> *>(d.m2ls[l]));
    else
      k_m2l_fill<double><<<(unsigned)nfar, 256, 0, st>>>(L, S.hard, o.kappa, o.eta_cfie,
                                                         reinterpret_cast<C2<double> *>(d.m2ls[l]));
    note_launch();
  }
  IGA_CUDA(cudaGetLastError());
}

void launch_m2l_rows(const DeviceProblem &d, const HostSetup &S, const igabem_options &o, int R,
                     bool fp32, cudaStream_t st) {
  if (!d.m2ls.empty() && d.m2ls[S.lmin]) {  // stored coupling blocks
    launch_stream_m2l(d, S, R, fp32, st);
    return;
  }
  M2LArgs A;
  A.QS = 0;
  A.R = R;
  A.CR = (S.hard ? 7 : 1) * R;
  A.kappa = o.kappa;
  A.eta = o.eta_cfie;
  A.hard = S.hard;
  A.cis = reinterpret_cast<const double2 *>(d.cis);
  A.nlev = 0;
  A.rows_most = 0;
  if (S.L - S.lmin + 1 > 16) fail(IGABEM_EINVAL, "more than 16 cluster levels with admissible pairs");
  int nblocks = 0;
  for (int l = S.lmin; l <= S.L; ++l) {
    M2LLevel &L = A.lev[A.nlev++];
    L.far_ptr = d.far_ptr[l];
    L.far_src = d.far_src[l];
    L.nodes = d.nodes[l];
    L.nodes32 = d.nodes32[l];
    L.pc = d.pairc[l];
    L.xhat = reinterpret_cast<const double2 *>(d.xhat[l]);
    L.xhat32 = d.xhat32.empty() ? nullptr : d.xhat32[l];
    L.yhat = reinterpret_cast<double2 *>(d.yhat[l]);
    L.n = S.lev[l].n;
    L.first = nblocks;
    L.q = S.lev[l].q;
    L.Q = L.q * L.q;
    A.QS = std::max(A.QS, L.Q);
    A.rows_most = std::max(A.rows_most, 256 / L.Q * L.Q);
    nblocks += S.lev[l].n;
  }
  // column chunk of the multi-column kernel: the largest divisor of R not above 64 (chunks never straddle two
  // channels)
  int Wc = 1;
  for (int w = std::min(R, 64); w >= 1; --w)
    if (R % w == 0) {
      Wc = w;
      break;
    }
  // Its tile has room for 64 columns: below 48 the padding costs more than k_m2l_fly's regenerated samples
  // (FP64 operations per sample and 7 x 5 columns: 7 (72 + 256) here, 2 x 43 + 140 there).  Sound-hard in FP32, where
  // k_m2l_fly takes three of these columns a pass, they meet earlier, its time being that of the columns and of q^2, the
  // tile's of neither: 480 clusters, here and there in ms at q = 8, 32 columns 34.2 and 36.4; q = 7, 34: 25.7 and 25.6,
  // 36: 25.8 and 25.9, 40: 26.2 and 30.6; q = 6, 40: 18.8 and 18.0, 47: 19.3 and 20.0; q = 5, 47: 13.4 and 12.6.  Lists
  // of few clusters leave its blocks few pairs each: 120 clusters, q = 5 and 7, 24 columns 0.82 and 0.72, 1.47 and 1.36;
  // 28: 0.84 and 0.84, 1.52 and 1.59; 40: 0.92 and 1.15, 1.62 and 2.21.
  const bool filled =
      Wc >= 48 || (S.hard && fp32 && (nblocks < 2 * 152 ? Wc >= 28 : Wc >= 32 && Wc * A.QS >= 1750));
  if (filled && A.QS <= 64) {
    const size_t tsz = fp32 ? sizeof(float) : sizeof(double);
    size_t smem = (size_t)A.QS * A.QS * 2 * tsz + (size_t)A.QS * Wc * 2 * tsz + (size_t)A.QS * 16 * tsz;
    dim3 grid(nblocks, A.CR / Wc);
    if (fp32) {
      IGA_CUDA(set_max_dynamic_smem(k_m2l_gemm<float>, smem));
      k_m2l_gemm<float><<<grid, 256, smem, st>>>(A, Wc);
    } else {
      IGA_CUDA(set_max_dynamic_smem(k_m2l_gemm<double>, smem));
      k_m2l_gemm<double><<<grid, 256, smem, st>>>(A, Wc);
    }
    note_launch();
  } else {
    // split the interaction lists over clusters of blocks while the device is not filled several times and
    // every block keeps pairs for all its threads
    const int P = std::max(1, 256 / S.lev[S.L].q / S.lev[S.L].q);
    const long mean = S.n_far / std::max(1, nblocks);
    int nsplit = 1;
    while (nsplit < 8 && (long)nblocks * nsplit < 8 * 152 && 2L * nsplit * P <= mean + P) nsplit *= 2;
    if (fp32) launch_fly_all<float>(A, nblocks, nsplit, st);
    else launch_fly_all<double>(A, nblocks, nsplit, st);
  }
  IGA_CUDA(cudaGetLastError());
}

}  // namespace igabem
