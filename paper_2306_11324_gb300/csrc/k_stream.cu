// Products with stored blocks, which bound a product when the operator is kept in device memory:
//   * the near field: y_leaf[t] = sum_{(t,s) near} B_ts x_s over dense leaf-pair blocks;
//   * the stored M2L (m2l_stored): y_t = sum_{s far} S_ts x_s over coupling blocks per kernel type.
// Blocks are column-major (the target row runs fastest), FP32 in the mixed precisions, FP64 otherwise.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "k_async.cuh"
#include "k_common.cuh"
#include "k_m2l.cuh"
#include "kernels.h"

namespace igabem {

namespace {

struct StreamLevel {
  const int *ptr, *src;   // pairs of each target (CSR)
  const void *blk;        // [pairs][types][NR][NR]
  const void *x;          // source coefficients
  double2 *out;           // [targets][NR][C]
  int first, NR;          // first target in the flattened grid; rows (and columns) of a block
  long pairs;             // blocks of the level
};

struct StreamArgs {
  StreamLevel lev[16];
  int nlev;
  int C;                  // columns of x and out
  int c0, cols;           // the launch's columns c0 .. c0 + cols
  int npass, w;           // in passes of w columns
  int types, type;        // blocks per pair, and the one that applies to these columns
  int rows_most;          // most block rows in use by a thread block
  int group;              // threads that multiply
  int ring, stage;        // FP32: byte offset of the buffers of block entries; bytes of one
  int *status;            // device status word
  int L, b, nb, nL1;      // near field: leaf grid and patch-wise coefficient grid of x
};

template <int BYTES>
__device__ inline void cp_async_zfill(void *dst, const void *src, int src_bytes) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(d), "l"(src), "n"(BYTES), "r"(src_bytes)
               : "memory");
}

// The sums over the pairs in FP32 carry a compensation term (Neumaier: hi, lo), as accurate as FP64 sums here
// without FP64 arithmetic.
__device__ inline void sum_add(float4 &t, float x, float y) {
  auto one = [](float &hi, float &lo, float v) {
    const float s = hi + v;
    lo += fabsf(hi) >= fabsf(v) ? (hi - s) + v : (v - s) + hi;
    hi = s;
  };
  one(t.x, t.z, x);
  one(t.y, t.w, y);
}

// first coefficient of a pair's source: near field on the patch-wise grid, M2L by clusters
template <bool NEAR> __device__ inline long source_base(const StreamArgs &A, int NR, int s) {
  if constexpr (NEAR) {
    const int js = s >> (2 * A.L), cx = (s >> A.L) & ((1 << A.L) - 1), cy = s & ((1 << A.L) - 1);
    return (((long)js * A.nb + (cx << A.b)) * A.nb + (cy << A.b)) * A.C;
  } else {
    return (long)s * NR * A.C;
  }
}

// The target's sums [c][pair slot][row] (stride values a column) of every block of the cluster, over the P slots and
// the blocks, in a fixed order; rank r adds the r-th part of the outputs.
__device__ inline void stream_reduce(const StreamArgs &A, const StreamLevel &L, double2 *red, int stride, int t, int P,
                                     int cr0, int ncr) {
  const int NR = L.NR, nthr = blockDim.x, nsplit = gridDim.y, rank = blockIdx.y;
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  if (nsplit > 1) cl.sync();
  else __syncthreads();
  const int per = (NR * ncr + nsplit - 1) / nsplit, o1 = min(NR * ncr, (rank + 1) * per);
  for (int o = rank * per + threadIdx.x; o < o1; o += nthr) {
    const int aa = o / ncr, c = o - aa * ncr;
    double2 sum = make_double2(0, 0);
    for (int z = 0; z < nsplit; ++z) {
      const double2 *rz = nsplit > 1 ? cl.map_shared_rank(red, z) : red;
      for (int p = 0; p < P; ++p) {
        const double2 v = rz[c * stride + p * NR + aa];
        sum.x += v.x;
        sum.y += v.y;
      }
    }
    L.out[((long)t * NR + aa) * A.C + cr0 + c] = sum;
  }
  if (nsplit > 1) cl.sync();  // no block leaves while another reads its shared memory
}

// FP32 blocks: HBM bounds them (8 bytes an entry, each read once), if the arithmetic does not wait for shared
// memory: a 16-byte shared load delivers two columns' coefficients to a warp in 4 cycles, so a thread owns two rows
// of a pair's block (a and a + ceil(NR / 2)) and uses each coefficient twice; products take two multiply-adds
// per instruction (for the entry s and the coefficient (x, y) the sums of s.x (x, y) and of s.y (x, y)).  The row pairs of
// P pairs lie side by side in a thread block (NR = 49: 125 of 128 threads), for up to 8 columns a pass; a second
// thread group for 8 more columns on the same entries left one block an SM and cost more than reading the blocks
// again: near field of 384 leaves, 12 columns 0.172 -> 0.067 ms without it (other loads that wait for every row: 0.147),
// M2L of 6144 elements, 12 and 32 columns 0.65 -> 0.64 and 1.68 -> 1.59 ms, of 24576, 12 columns 2.53 -> 2.62 ms.
// The entries come by bulk copies of whole column ranges of the blocks into STREAM_STAGES buffers, issued by a warp
// of its own as the multiplying warps release the buffers (a copy starts at the 16-byte boundary below its first
// entry); the pairs' source coefficients are staged by cp.async one round ahead.  Every wait is bounded (2 s): one
// that runs out sets the status word, no further copy is issued, and the block leaves once its copies in flight have
// landed (waited for with the same bound).
// Measured on GB300, 8 columns, 98304 elements (34.6 GB of coupling blocks, 4.0 GB of near field): M2L 11.4 -> 7.7 ms
// (4.5 TB/s), near field 2.2 -> 1.1 ms; 64 columns, 24576 elements: M2L 36.7 -> 21.7, near field 7.5 -> 2.3 ms;
// sound-hard, 6144 elements, 5 columns of 7 channels: M2L 4.6 -> 2.1 ms (before, each lane waited on every row's copy and every 7 or 8 columns
// read the blocks again).  What bounds it now: two blocks of four multiplying warps an SM, latency between the
// products.
constexpr int STREAM_STAGES = 3;

template <int NC, bool NEAR>
__global__ void __launch_bounds__(160, 2) k_stream32(const __grid_constant__ StreamArgs A) {
  extern __shared__ __align__(16) unsigned char sms[];
  __shared__ __align__(8) uint64_t full[STREAM_STAGES], empty[STREAM_STAGES];
  const int tid = threadIdx.x, lane = tid & 31, nsplit = gridDim.y, rank = blockIdx.y;
  const int ncons = blockDim.x - 32;  // threads that multiply; the last warp copies
  const int tg = blockIdx.x / A.npass;
  int li = 0;
  while (li + 1 < A.nlev && tg >= A.lev[li + 1].first) ++li;
  const StreamLevel &L = A.lev[li];
  const int t = tg - L.first, NR = L.NR, HR = (NR + 1) >> 1, P = A.group / HR;
  const int slot = tid / HR, a = tid - slot * HR;
  const int cr0 = A.c0 + (blockIdx.x - tg * A.npass) * A.w, ncr = min(A.w, A.c0 + A.cols - cr0);
  float2 *xs = reinterpret_cast<float2 *>(sms);                                              // [2][P NR][NC]
  unsigned char *ring = sms + A.ring;                                                        // [STAGES][stage]
  const bool on = slot < P, two = a + HR < NR;
  const int k0 = L.ptr[t], np = L.ptr[t + 1] - k0, step = nsplit * P;
  // column ranges of BC columns, so that a buffer holds them for all P pairs
  const int slot_max = A.stage / P & ~15, BC = max(1, min(NR, (slot_max - 16) / (NR * 8))), nch = (NR + BC - 1) / BC;
  const int slot_bytes = (BC * NR * 8 + 16 + 15) & ~15;
  const int rounds = np > rank * P ? (np - rank * P + step - 1) / step : 0;
  const int total = rounds * nch;
  const bool vec = NC % 2 == 0 && ((A.C | cr0) & 1) == 0;
  const unsigned char *blk = reinterpret_cast<const unsigned char *>(L.blk);
  // byte offset of column b0 of pair k's block
  auto entry = [&](int k, int b0) { return (((size_t)k * A.types + A.type) * NR + b0) * NR * 8; };
  auto issue = [&](int j) {  // the copying warp
    const int r = j / nch, b0 = (j - r * nch) * BC, nb = min(BC, NR - b0), p0 = rank * P + r * step, s = j % STREAM_STAGES;
    const uint32_t bar = smem_u32(&full[s]);
    for (int p = lane; p < P && p0 + p < np; p += 32) {
      const size_t o = entry(k0 + p0 + p, b0);
      const uint32_t bytes = (uint32_t)((o & 8) + (size_t)nb * NR * 8 + 15) & ~15u;
      mbar_expect_only(bar, bytes);
      bulk_load(smem_u32(ring + (size_t)s * A.stage + (size_t)p * slot_bytes), blk + (o & ~size_t(15)), bytes, bar);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
  };
  auto stage_x = [&](int r) {  // this thread's two rows
    const int p0 = rank * P + r * step;
    if (on && p0 + slot < np) {
      const float2 *src0 = reinterpret_cast<const float2 *>(L.x) + source_base<NEAR>(A, NR, L.src[k0 + p0 + slot]) + cr0;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = a + h * HR;
        if (i >= NR) break;
        const float2 *src = src0 + (NEAR ? ((long)(i / A.nL1) * A.nb + i % A.nL1) * A.C : (long)i * A.C);
        float2 *dst = xs + ((size_t)(r & 1) * A.rows_most + slot * NR + i) * NC;
        if (vec) {
#pragma unroll
          for (int c = 0; c < NC; c += 2) {
            const int n = min(16, max(0, 8 * (ncr - c)));
            cp_async_zfill<16>(dst + c, n ? src + c : src, n);
          }
        } else {
#pragma unroll
          for (int c = 0; c < NC; ++c) cp_async_zfill<8>(dst + c, c < ncr ? src + c : src, c < ncr ? 8 : 0);
        }
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  if (tid == 0) {
    for (int s = 0; s < STREAM_STAGES; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), ncons / 32);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  float4 tot[2][NC];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int c = 0; c < NC; ++c) tot[h][c] = make_float4(0.f, 0.f, 0.f, 0.f);
  bool ok = true;
  if (tid >= ncons) {
    // fill j of a buffer follows the release of fill j - STREAM_STAGES by every multiplying warp
    int j = 0;
    for (; j < total && ok; ++j) {
      if (j >= STREAM_STAGES) ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&empty[j % STREAM_STAGES]), (uint32_t)(j / STREAM_STAGES - 1) & 1));
      if (ok) issue(j);
    }
    if (!ok) {
      --j;
      if (lane == 0) atomicExch(A.status, 1);
    }
    for (int i = max(0, j - STREAM_STAGES); i < j; ++i)  // the copies in flight land before the block leaves
      if (!mbar_wait(smem_u32(&full[i % STREAM_STAGES]), (uint32_t)(i / STREAM_STAGES) & 1)) break;
  } else {
    stage_x(0);
    float2 a1[2][NC], a2[2][NC];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int c = 0; c < NC; ++c) a1[h][c] = a2[h][c] = make_float2(0.f, 0.f);
    const int da = two ? HR : 0;  // the second row (the first again where there is none)
    int r = 0, ch = 0, s = 0;
    uint32_t parity = 0;
    for (int j = 0; j < total; ++j) {
      if (ch == 0) {
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        asm volatile("bar.sync 1, %0;" ::"r"(ncons) : "memory");  // coefficients landed, the other buffer is read
        stage_x(r + 1);
      }
      // after a wait that ran out the warp only keeps the others going
      if (ok) {
        ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&full[s]), parity));
        if (!ok && lane == 0) atomicExch(A.status, 1);
      }
      const int p0 = rank * P + r * step, b0 = ch * BC, nb = min(BC, NR - b0);
      if (ok && on && p0 + slot < np) {
        const size_t o = entry(k0 + p0 + slot, b0);
        const float2 *Sp = reinterpret_cast<const float2 *>(ring + (size_t)s * A.stage + (size_t)slot * slot_bytes + (o & 8)) + a;
        const float2 *X = xs + ((size_t)(r & 1) * A.rows_most + slot * NR + b0) * NC;
        constexpr int NV = (NC + 1) / 2;  // 16-byte loads of a coefficient row
        auto load_x = [&](float4 (&v)[NV], int b) {
          if constexpr (NC % 2 == 0) {
#pragma unroll
            for (int c = 0; c < NV; ++c) v[c] = reinterpret_cast<const float4 *>(X + b * NC)[c];
          } else {
            const float2 w = X[b];
            v[0] = make_float4(w.x, w.y, 0.f, 0.f);
          }
        };
        // entries and coefficients one column ahead of their use
        float2 e = Sp[0], f = Sp[da];
        float4 v[NV];
        load_x(v, 0);
#pragma unroll 2
        for (int b = 0; b < nb; ++b) {
          const int bn = min(b + 1, nb - 1);
          const float2 en = Sp[bn * NR], fn = Sp[bn * NR + da];
          float4 vn[NV];
          load_x(vn, bn);
          const float2 ex = make_float2(e.x, e.x), ey = make_float2(e.y, e.y), fx = make_float2(f.x, f.x),
                       fy = make_float2(f.y, f.y);
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            const float2 w = c & 1 ? make_float2(v[c / 2].z, v[c / 2].w) : make_float2(v[c / 2].x, v[c / 2].y);
            a1[0][c] = fma2x(ex, w, a1[0][c]);
            a2[0][c] = fma2x(ey, w, a2[0][c]);
            a1[1][c] = fma2x(fx, w, a1[1][c]);
            a2[1][c] = fma2x(fy, w, a2[1][c]);
          }
          e = en;
          f = fn;
#pragma unroll
          for (int c = 0; c < NV; ++c) v[c] = vn[c];
        }
        if (ch == nch - 1)
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int c = 0; c < NC; ++c) {
              sum_add(tot[h][c], a1[h][c].x - a2[h][c].y, a1[h][c].y + a2[h][c].x);
              a1[h][c] = a2[h][c] = make_float2(0.f, 0.f);
            }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&empty[s]));  // this warp has read the buffer
      if (++s == STREAM_STAGES) {
        s = 0;
        parity ^= 1;
      }
      if (++ch == nch) {
        ch = 0;
        ++r;
      }
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  }
  __syncthreads();
  double2 *red = reinterpret_cast<double2 *>(ring);  // [NC][P NR]
  if (on && tid < ncons)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (a + h * HR < NR)
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const float4 v = tot[h][c];
          red[(size_t)c * A.rows_most + slot * NR + a + h * HR] =
              make_double2((double)v.x + (double)v.z, (double)v.y + (double)v.w);
        }
  stream_reduce(A, L, red, A.rows_most, t, P, cr0, ncr);
}

// FP64 blocks: FP64 arithmetic bounds them (four multiply-adds per entry and column).  A thread owns one row of one
// pair's block, the rows of P = blockDim / NR pairs side by side, and reads its entries straight from memory,
// 8 ahead of their use.  Measured: torus, 1600 unknowns, 2 columns, 1.4 GB of coupling blocks 1.94 -> 1.39 ms, near
// field 0.91 -> 0.15 ms.
constexpr int STREAM_AHEAD = 8;

template <int NC, bool NEAR>
__global__ void __launch_bounds__(256) k_stream64(const __grid_constant__ StreamArgs A) {
  extern __shared__ __align__(16) unsigned char sms[];
  const int tid = threadIdx.x, nthr = blockDim.x, nsplit = gridDim.y, rank = blockIdx.y;
  const int tg = blockIdx.x / A.npass, cr0 = A.c0 + (blockIdx.x - tg * A.npass) * A.w;
  int li = 0;
  while (li + 1 < A.nlev && tg >= A.lev[li + 1].first) ++li;
  const StreamLevel &L = A.lev[li];
  const int t = tg - L.first, NR = L.NR, P = nthr / NR, slot = tid / NR, a = tid - slot * NR;
  const int ncr = min(A.w, A.c0 + A.cols - cr0);
  double2 *xs = reinterpret_cast<double2 *>(sms);          // [2][rows][NC]
  double2 *tot = xs + (size_t)2 * A.rows_most * NC;        // [NC][nthr]
  const bool on = slot < P;
  const int k0 = L.ptr[t], np = L.ptr[t + 1] - k0, step = nsplit * P;
  const long row = NEAR ? ((long)(a / A.nL1) * A.nb + a % A.nL1) * A.C : (long)a * A.C;
  auto stage = [&](int p0, int buf) {
    if (on && p0 + slot < np) {
      const double2 *src = reinterpret_cast<const double2 *>(L.x) + source_base<NEAR>(A, NR, L.src[k0 + p0 + slot]) + row + cr0;
      double2 *dst = xs + ((size_t)buf * A.rows_most + tid) * NC;
#pragma unroll
      for (int c = 0; c < NC; ++c) cp_async_zfill<16>(dst + c, c < ncr ? src + c : src, c < ncr ? 16 : 0);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  if (on)
#pragma unroll
    for (int c = 0; c < NC; ++c) tot[c * nthr + tid] = make_double2(0, 0);
  stage(rank * P, 0);
  int buf = 0;
  for (int p0 = rank * P; p0 < np; p0 += step, buf ^= 1) {
    const bool work = on && p0 + slot < np;
    const double2 *B = reinterpret_cast<const double2 *>(L.blk) + ((size_t)(k0 + p0 + slot) * A.types + A.type) * NR * NR + a;
    double2 sv[STREAM_AHEAD];
    if (work)
#pragma unroll
      for (int u = 0; u < STREAM_AHEAD; ++u)
        if (u < NR) sv[u] = __ldg(B + (size_t)u * NR);
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();  // this round's coefficients have landed, the other buffer is read
    stage(p0 + step, buf ^ 1);
    if (!work) continue;
    const double2 *X = xs + ((size_t)buf * A.rows_most + slot * NR) * NC;
    double2 acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = make_double2(0, 0);
    for (int b = 0; b < NR; b += STREAM_AHEAD) {
      double2 nx[STREAM_AHEAD];
#pragma unroll
      for (int u = 0; u < STREAM_AHEAD; ++u)
        if (b + STREAM_AHEAD + u < NR) nx[u] = __ldg(B + (size_t)(b + STREAM_AHEAD + u) * NR);
#pragma unroll
      for (int u = 0; u < STREAM_AHEAD; ++u) {
        if (b + u >= NR) break;
        const double2 s = sv[u];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const double2 v = X[(b + u) * NC + c];
          acc[c].x = fma(s.x, v.x, fma(-s.y, v.y, acc[c].x));
          acc[c].y = fma(s.x, v.y, fma(s.y, v.x, acc[c].y));
        }
      }
#pragma unroll
      for (int u = 0; u < STREAM_AHEAD; ++u) sv[u] = nx[u];
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      double2 v = tot[c * nthr + tid];
      tot[c * nthr + tid] = make_double2(v.x + acc[c].x, v.y + acc[c].y);
    }
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  stream_reduce(A, L, tot, nthr, t, P, cr0, ncr);
}

template <class T, int NC, bool NEAR>
void launch_one(StreamArgs &A, int targets, int threads, int nsplit, cudaStream_t st) {
  size_t smem;
  void (*kfn)(const StreamArgs);
  if constexpr (std::is_same<T, float>::value) {
    // buffers for two thread blocks on an SM, at least one column of every pair and room for the final sums
    A.ring = (int)(((size_t)2 * A.rows_most * NC * 8 + 15) & ~size_t(15));
    const size_t avail = 112 * 1024 - A.ring;
    size_t least = 0;
    for (int i = 0; i < A.nlev; ++i) {
      const int NR = A.lev[i].NR;
      least = std::max<size_t>(least, (size_t)(A.group / ((NR + 1) / 2)) * (NR * 8 + 32));
    }
    least = std::max(least, (size_t)NC * A.rows_most * 16 / STREAM_STAGES + 16);
    A.stage = (int)(std::max(std::min<size_t>(avail / STREAM_STAGES, 48 * 1024) & ~size_t(127), (least + 127) & ~size_t(127)));
    smem = (size_t)A.ring + (size_t)STREAM_STAGES * A.stage;
    kfn = k_stream32<NC, NEAR>;
  } else {
    smem = ((size_t)2 * A.rows_most + threads) * NC * 16;
    kfn = k_stream64<NC, NEAR>;
  }
  IGA_CUDA(set_max_dynamic_smem(kfn, smem));
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(targets * A.npass, nsplit);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = 1;
  at.val.clusterDim.y = nsplit;
  at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  IGA_CUDA(cudaLaunchKernelEx(&cfg, kfn, (const StreamArgs)A));
  note_launch();
}

// Columns c0 .. c0 + cols with the blocks of one type, in passes of at most 8 columns (their sums fill the registers).
template <class T, bool NEAR>
void launch_columns(StreamArgs &A, int c0, int cols, int type, int targets, double mean_pairs, cudaStream_t st) {
  constexpr bool F32 = std::is_same<T, float>::value;
  A.c0 = c0;
  A.cols = cols;
  A.type = type;
  A.npass = (cols + 7) / 8;
  A.w = (cols + A.npass - 1) / A.npass;
  const int nc = A.w <= 2 ? A.w : (A.w + 1) & ~1;  // 1, 2, 4, 6 or 8
  if (A.npass > 1) A.w = nc;
  A.npass = (cols + A.w - 1) / A.w;
  // threads that multiply (whole warps) that the levels' rows (FP32: row pairs) fill best, weighted by the levels' entries;
  // the larger of two equally good ones
  const int lo = F32 ? 96 : 128, hi = F32 ? 128 : 256;
  int group = hi;
  double best = -1;
  for (int n = lo; n <= hi; n += 32) {
    double use = 0, all = 0;
    for (int i = 0; i < A.nlev && use >= 0; ++i) {
      const int NR = A.lev[i].NR, k = F32 ? (NR + 1) / 2 : NR;
      const double wt = (double)A.lev[i].pairs * NR * NR;
      use = k > n ? -1 : use + wt * (n / k) * k / n;
      all += wt;
    }
    if (use >= 0 && use / std::max(all, 1.0) > best - 1e-9) {
      best = use / std::max(all, 1.0);
      group = n;
    }
  }
  A.group = group;
  A.rows_most = 0;
  for (int i = 0; i < A.nlev; ++i) {
    const int NR = A.lev[i].NR, k = F32 ? (NR + 1) / 2 : NR;
    A.rows_most = std::max(A.rows_most, group / k * NR);
  }
  // targets split over clusters of blocks while the device is not filled several times and every block keeps
  // pairs for all its threads, in FP32 for four rounds of them (its copies run three buffers ahead; near field of 384 leaves
  // of 36 rows, one column, split in 1, 2, 4, 8: 0.024, 0.021, 0.031, 0.046 ms; M2L of 120 targets of 49 rows 0.022, 0.018,
  // 0.024, 0.035 ms, of 144 rows 0.154, 0.098, 0.113, 0.102 ms)
  const int NRl = A.lev[A.nlev - 1].NR, P = std::max(1, group / (F32 ? (NRl + 1) / 2 : NRl));
  int nsplit = 1;
  const int rounds = F32 ? 4 : 1;
  while (nsplit < 8 && (long)targets * A.npass * nsplit < 4 * 152 && 2.0 * nsplit * P * rounds <= mean_pairs + P) nsplit *= 2;
  const int threads = F32 ? group + 32 : group;
  auto go = [&](auto n) { launch_one<T, decltype(n)::value, NEAR>(A, targets, threads, nsplit, st); };
  if (nc == 1) go(std::integral_constant<int, 1>{});
  else if (nc == 2) go(std::integral_constant<int, 2>{});
  else if (nc == 4) go(std::integral_constant<int, 4>{});
  else if (nc == 6) go(std::integral_constant<int, 6>{});
  else go(std::integral_constant<int, 8>{});
}

}  // namespace

bool stream_near_supported(const HostSetup &S) { return S.nL <= 256; }

void launch_stream_near(const DeviceProblem &d, const HostSetup &S, int R, cudaStream_t st) {
  StreamArgs A{};
  A.status = d.status;
  A.nlev = 1;
  A.C = R;
  A.types = 1;
  A.L = S.L;
  A.b = S.b;
  A.nb = S.nb;
  A.nL1 = S.nL1;
  const bool f32 = d.blk32 != nullptr;
  const int targets = S.lev[S.L].n;
  A.lev[0] = {d.near_ptr, d.near_src, f32 ? (const void *)d.blk32 : (const void *)d.blk,
              f32 ? (const void *)d.xX32 : (const void *)d.xX, reinterpret_cast<double2 *>(d.yleaf), 0, S.nL, (long)S.near_src.size()};
  const double mean = (double)S.near_src.size() / std::max(1, targets);
  if (f32) launch_columns<float, true>(A, 0, R, 0, targets, mean, st);
  else launch_columns<double, true>(A, 0, R, 0, targets, mean, st);
  IGA_CUDA(cudaGetLastError());
}

void launch_stream_m2l(const DeviceProblem &d, const HostSetup &S, int R, bool fp32, cudaStream_t st) {
  if (S.L - S.lmin + 1 > 16) fail(IGABEM_EINVAL, "more than 16 cluster levels with admissible pairs");
  StreamArgs A{};
  A.status = d.status;
  A.C = (S.hard ? 7 : 1) * R;
  A.types = S.hard ? 2 : 1;
  int targets = 0;
  for (int l = S.lmin; l <= S.L; ++l) {
    A.lev[A.nlev++] = {d.far_ptr[l], d.far_src[l], d.m2ls[l], fp32 ? (const void *)d.xhat32[l] : (const void *)d.xhat[l],
                       reinterpret_cast<double2 *>(d.yhat[l]), targets, S.lev[l].q * S.lev[l].q,
                       (long)S.lev[l].far_src.size()};
    targets += S.lev[l].n;
  }
  const double mean = (double)S.n_far / std::max(1, targets);
  auto go = [&](int c0, int cols, int type) {
    if (fp32) launch_columns<float, false>(A, c0, cols, type, targets, mean, st);
    else launch_columns<double, false>(A, c0, cols, type, targets, mean, st);
  };
  if (S.hard) {  // channel 0 takes the double-layer blocks, channels 1..6 the single-layer ones
    go(0, R, 0);
    go(R, 6 * R, 1);
  } else {
    go(0, R, 0);
  }
  IGA_CUDA(cudaGetLastError());
}

}  // namespace igabem
