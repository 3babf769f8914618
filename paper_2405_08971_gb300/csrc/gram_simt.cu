// Plain Gram x block product on the CUDA cores, FP32 and FP64:
//   Out[i, c] = sum_j sf2 k(xr_i, xc_j) B[j, c]     (Out, B column-major; the kernel matrix is never stored)
// and the same with d k / d log l_x.  A block owns a tile of rows and up to 72 columns of Out, so a
// kernel value is evaluated once per 72 columns; the sum over j is split over the blocks of a
// thread-block cluster (and, in FP32, over two halves of a block) whose partial tiles are added in a
// fixed order through distributed shared memory, so that few rows still fill the GPU without scratch.
#include <cooperative_groups.h>
#include "common.cuh"
#include "internal.h"

namespace cakf {
namespace {

namespace cg = cooperative_groups;

constexpr int GS_KS = 16;          // kernel columns per stage
constexpr int GS_THREADS = 256;
constexpr int GS_MAX_COLS = 72;    // columns of Out per block: 9 per thread column, 65 = i + 1 fits

// Matern correlation (DER: its d/dlog l_x) of a pair of rows against one column.
template <int KER, bool DER>
__device__ __forceinline__ uint64_t kpair_fn(uint64_t rx, uint64_t ry, uint64_t rz, uint64_t cx, uint64_t cy,
                                             uint64_t cz) {
  if constexpr (!DER) return kpair<KER>(rx, ry, rz, cx, cy, cz);
  const uint64_t dx = f2_sub(rx, cx), dy = f2_sub(ry, cy), dz = f2_sub(rz, cz);
  uint64_t d2 = f2_mul(dz, dz);
  d2 = f2_fma(dy, dy, d2);
  d2 = f2_fma(dx, dx, d2);
  float a, b;
  f2_split(d2, a, b);
  return f2_make(kval_dlogl<KER>(a, 1.0f), kval_dlogl<KER>(b, 1.0f));
}

// FP32.  256 threads = 2 groups of 128, each taking every second stage of the block's share of j.  A
// group's stage: its threads evaluate a (16 RPT rows) x 16 tile of kernel values in packed pairs of
// rows, and then hold RPT rows (consecutive, as f32x2 pairs) x CPT columns of Out each; the inner loop
// reads 4 rows or 4 columns per 16-byte shared load (5 loads per 36 f32x2 FMAs at CPT = 9, RPT = 8).  The
// stage after next's column coordinates, the next stage's values and B are written while the current
// stage is multiplied: one group barrier per stage.  Bound by the FP32 pipe: 9,600 x 9,600 x 129 takes
// 634 us (709 us with one shared load per column, which kept the shared-memory pipe 71 % busy),
// against 1,590 us for 64 x 64 x 32 tiles that evaluated the values once per 64 columns.
template <int CPT, int RPT> struct F32Tile {
  static constexpr int BM = 16 * RPT, BN = 8 * CPT;
  static constexpr int LDK = BM + 4;                    // floats; rows of the value tile
  static constexpr int LDB = BN + 4;                    // floats; rows of B
  static constexpr int LDR = BM + 4;                    // floats; columns of the reduction tile
  static constexpr size_t K_BYTES = (size_t)2 * GS_KS * LDK * 4;    // two buffers, per group
  static constexpr size_t B_BYTES = (size_t)2 * GS_KS * LDB * 4;
  static constexpr size_t X_BYTES = (size_t)2 * GS_KS * 4 * 8;
  static constexpr size_t GROUP = K_BYTES + B_BYTES + X_BYTES;
  static constexpr size_t RED = (size_t)BN * LDR * 4;
  static constexpr size_t SMEM = 2 * GROUP > RED ? 2 * GROUP : RED;
  // A thread's columns: runs of 4, then of 2 and 1, so that they are read by 16-, 8- and 4-byte loads
  static constexpr int N4 = CPT / 4, N2 = CPT % 4 / 2;
  __device__ static constexpr int col(int tx, int u) {
    return u < 4 * N4 ? (u / 4) * 32 + tx * 4 + u % 4
                      : (u < 4 * N4 + 2 * N2 ? 32 * N4 + tx * 2 + (u - 4 * N4) : 32 * N4 + 16 * N2 + tx);
  }
};

// One stage's products: acc += (RPT rows at ty RPT) x (CPT columns F32Tile::col(tx, .)), 16 terms each.
template <int CPT, int RPT>
__device__ __forceinline__ void stage_fma(const float* Ks, const float* Bs, int buf, int tx, int ty,
                                          uint64_t (&acc)[CPT][RPT / 2]) {
  using F = F32Tile<CPT, RPT>;
#pragma unroll 4
  for (int kk = 0; kk < GS_KS; ++kk) {
    const float* kp = Ks + (size_t)(buf * GS_KS + kk) * F::LDK + ty * RPT;
    uint64_t kr[RPT / 2];
    if constexpr (RPT % 4 == 0) {
#pragma unroll
      for (int q = 0; q < RPT / 4; ++q) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(kp + 4 * q);
        kr[2 * q] = v.x;
        kr[2 * q + 1] = v.y;
      }
    } else {
#pragma unroll
      for (int q = 0; q < RPT / 2; ++q) kr[q] = *reinterpret_cast<const uint64_t*>(kp + 2 * q);
    }
    const float* bp = Bs + (buf * GS_KS + kk) * F::LDB;
    float b[CPT];
#pragma unroll
    for (int q = 0; q < F::N4; ++q) {
      const float4 v = *reinterpret_cast<const float4*>(bp + q * 32 + tx * 4);
      b[4 * q] = v.x; b[4 * q + 1] = v.y; b[4 * q + 2] = v.z; b[4 * q + 3] = v.w;
    }
    if constexpr (F::N2) {
      const float2 v = *reinterpret_cast<const float2*>(bp + F::N4 * 32 + tx * 2);
      b[4 * F::N4] = v.x; b[4 * F::N4 + 1] = v.y;
    }
    if constexpr (CPT % 2) b[CPT - 1] = bp[F::N4 * 32 + F::N2 * 16 + tx];
#pragma unroll
    for (int u = 0; u < CPT; ++u) {
      const uint64_t bb = f2_make(b[u], b[u]);
#pragma unroll
      for (int p = 0; p < RPT / 2; ++p) acc[u][p] = f2_fma(kr[p], bb, acc[u][p]);
    }
  }
}
// The block's tile into Rs (column-major, LDR apart): group 1's part, then group 0's on top of it.
template <int CPT, int RPT>
__device__ __forceinline__ void reduce_groups(float* Rs, int g, int tx, int ty, const uint64_t (&acc)[CPT][RPT / 2]) {
  using F = F32Tile<CPT, RPT>;
  __syncthreads();
  for (int half = 1; half >= 0; --half) {
    if (g == half) {
#pragma unroll
      for (int u = 0; u < CPT; ++u)
#pragma unroll
        for (int p = 0; p < RPT / 2; ++p) {
          float lo, hi;
          f2_split(acc[u][p], lo, hi);
          float* o = Rs + (size_t)F::col(tx, u) * F::LDR + ty * RPT + 2 * p;
          if (half == 0) { lo += o[0]; hi += o[1]; }
          o[0] = lo;
          o[1] = hi;
        }
    }
    __syncthreads();
  }
}

template <int CPT, int RPT>
__global__ void __launch_bounds__(GS_THREADS, 2)
k_gram_block_f32(int fn, const C4<float>* __restrict__ Xr, int nr, const C4<float>* __restrict__ Xc, int nc,
                 const float* __restrict__ B, int ldb, int width, int cw, float sf2, float* __restrict__ Out, int ldo) {
  using F = F32Tile<CPT, RPT>;
  constexpr int BM = F::BM, HB = BM / 2;
  extern __shared__ __align__(16) unsigned char gsm[];
  cg::cluster_group cl = cg::this_cluster();
  const int Z = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int g = threadIdx.x >> 7, t = threadIdx.x & 127, tx = t & 7, ty = t >> 3;
  float* Ks = reinterpret_cast<float*>(gsm + (size_t)g * F::GROUP);
  float* Bs = reinterpret_cast<float*>(gsm + (size_t)g * F::GROUP + F::K_BYTES);
  uint64_t* Xs = reinterpret_cast<uint64_t*>(gsm + (size_t)g * F::GROUP + F::K_BYTES + F::B_BYTES);
  const int row0 = (int)(blockIdx.x / Z) * BM, col0 = blockIdx.y * cw, ncol = min(cw, width - col0);
  const int nst = (nc + GS_KS - 1) / GS_KS;             // stages in all; this group takes first, first + step, ...
  const int first = rank * 2 + g, step = 2 * Z;
  // rows this thread evaluates (r, r + HB) for the columns er * RPT .. of a stage
  const int er = t % HB, eg = t / HB;
  uint64_t rx, ry, rz;
  {
    C4<float> a, b;
    a.x = a.y = a.z = b.x = b.y = b.z = 0.f;
    if (row0 + er < nr) a = Xr[row0 + er];
    if (row0 + er + HB < nr) b = Xr[row0 + er + HB];
    rx = f2_make(a.x, b.x); ry = f2_make(a.y, b.y); rz = f2_make(a.z, b.z);
  }
  auto bar = [&]() { asm volatile("bar.sync %0, 128;" ::"r"(g + 1) : "memory"); };
  // 16 threads: the stage's column coordinates and sf2, duplicated (sf2 belongs to the kernel value: a sum without it
  // can overflow where the product does not; from a register it made <9, 8> spill: 744 us against 665 us a call)
  auto stage_x = [&](int st, int buf) {
    if (t < GS_KS) {
      const int j = st * GS_KS + t;
      C4<float> c;
      c.x = c.y = c.z = 0.f;
      if (j < nc) c = Xc[j];
      uint64_t* o = Xs + (buf * GS_KS + t) * 4;
      o[0] = f2_make(c.x, c.x); o[1] = f2_make(c.y, c.y); o[2] = f2_make(c.z, c.z);
      o[3] = f2_make(sf2, sf2);
    }
  };
  float br[CPT];
  auto load_b = [&](int st) {
#pragma unroll
    for (int i = 0; i < CPT; ++i) {
      const int e = t + 128 * i, kk = e & (GS_KS - 1), c = e / GS_KS, j = st * GS_KS + kk;
      br[i] = (j < nc && c < ncol) ? B[(size_t)(col0 + c) * ldb + j] : 0.f;
    }
  };
  auto store_b = [&](int buf) {
#pragma unroll
    for (int i = 0; i < CPT; ++i) {
      const int e = t + 128 * i, kk = e & (GS_KS - 1), c = e / GS_KS;
      Bs[(buf * GS_KS + kk) * F::LDB + c] = br[i];
    }
  };
  auto eval_with = [&](auto f, int buf) {
#pragma unroll
    for (int u = 0; u < RPT; ++u) {
      const int kk = eg * RPT + u;
      const ulonglong2 xy = *reinterpret_cast<const ulonglong2*>(Xs + (buf * GS_KS + kk) * 4);
      const ulonglong2 zs = *reinterpret_cast<const ulonglong2*>(Xs + (buf * GS_KS + kk) * 4 + 2);
      float lo, hi;
      f2_split(f2_mul(f(xy.x, xy.y, zs.x), zs.y), lo, hi);
      float* o = Ks + (size_t)(buf * GS_KS + kk) * F::LDK + er;
      o[0] = lo;
      o[HB] = hi;
    }
  };
  auto eval = [&](int buf) {                            // uniform choice of the function, once per stage
    switch (fn) {
      case 0: eval_with([&](uint64_t x, uint64_t y, uint64_t z) { return kpair_fn<0, false>(rx, ry, rz, x, y, z); }, buf); break;
      case 1: eval_with([&](uint64_t x, uint64_t y, uint64_t z) { return kpair_fn<1, false>(rx, ry, rz, x, y, z); }, buf); break;
      case 2: eval_with([&](uint64_t x, uint64_t y, uint64_t z) { return kpair_fn<2, false>(rx, ry, rz, x, y, z); }, buf); break;
      case 3: eval_with([&](uint64_t x, uint64_t y, uint64_t z) { return kpair_fn<0, true>(rx, ry, rz, x, y, z); }, buf); break;
      case 4: eval_with([&](uint64_t x, uint64_t y, uint64_t z) { return kpair_fn<1, true>(rx, ry, rz, x, y, z); }, buf); break;
      default: eval_with([&](uint64_t x, uint64_t y, uint64_t z) { return kpair_fn<2, true>(rx, ry, rz, x, y, z); }, buf); break;
    }
  };
  uint64_t acc[CPT][RPT / 2];
#pragma unroll
  for (int u = 0; u < CPT; ++u)
#pragma unroll
    for (int p = 0; p < RPT / 2; ++p) acc[u][p] = 0ull;
  if (first < nst) {
    stage_x(first, 0);
    load_b(first);
    bar();
    eval(0);
    store_b(0);
    if (first + step < nst) { stage_x(first + step, 1); load_b(first + step); }
    bar();
    int buf = 0;
    for (int st = first; st < nst; st += step, buf ^= 1) {
      stage_fma<CPT, RPT>(Ks, Bs, buf, tx, ty, acc);
      if (st + step < nst) {
        eval(buf ^ 1);
        store_b(buf ^ 1);
        // the coordinates of stage st were last read before the barrier that opened this stage
        if (st + 2 * step < nst) { stage_x(st + 2 * step, buf); load_b(st + 2 * step); }
      }
      bar();
    }
  }
  // ---- partial tiles: the groups' in shared memory, then the cluster's blocks
  float* Rs = reinterpret_cast<float*>(gsm);
  reduce_groups<CPT, RPT>(Rs, g, tx, ty, acc);
  cl.sync();
  const int share = (ncol + Z - 1) / Z, c0 = rank * share, c1 = min(ncol, c0 + share);
  for (int e = threadIdx.x; e < (c1 - c0) * BM; e += GS_THREADS) {
    const int c = c0 + e / BM, r = e % BM;
    if (row0 + r >= nr) continue;
    float v = 0.f;
    for (int q = 0; q < Z; ++q) v += cl.map_shared_rank(Rs, q)[(size_t)c * F::LDR + r];
    Out[(size_t)(col0 + c) * ldo + row0 + r] = v;
  }
  cl.sync();                                            // no block leaves while its tile is being read
}

// The plain FP32 factor product C (M x N) = alpha A (M x K) B (K x N) + beta C on the same tiles: a stage's
// 16 columns of A take the place of the kernel values (the next stage's A and B are in registers while the
// current one is multiplied), and the K range is split over the cluster in the same way.  B may be FP64
// (small coefficient blocks), converted when staged.
// 5,000 x 33 x 257 takes 17.9 us; a cakf_factor_gemm call of that size 49 us, against 84 us with 64 x 64 tiles (79
// blocks, 64 columns computed).
template <int CPT, int RPT, class TB>
__global__ void __launch_bounds__(GS_THREADS, 2)
k_gemm_nn_f32(int M, int N, int K, float alpha, const float* __restrict__ A, int lda, const TB* __restrict__ B, int ldb,
              int cw, float beta, float* __restrict__ C, int ldc) {
  using F = F32Tile<CPT, RPT>;
  constexpr int BM = F::BM, NA = BM * GS_KS / 128;
  extern __shared__ __align__(16) unsigned char gsm[];
  cg::cluster_group cl = cg::this_cluster();
  const int Z = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int g = threadIdx.x >> 7, t = threadIdx.x & 127, tx = t & 7, ty = t >> 3;
  float* Ks = reinterpret_cast<float*>(gsm + (size_t)g * F::GROUP);
  float* Bs = reinterpret_cast<float*>(gsm + (size_t)g * F::GROUP + F::K_BYTES);
  const int row0 = (int)(blockIdx.x / Z) * BM, col0 = blockIdx.y * cw, ncol = min(cw, N - col0);
  const int nst = (K + GS_KS - 1) / GS_KS;
  const int first = rank * 2 + g, step = 2 * Z;
  auto bar = [&]() { asm volatile("bar.sync %0, 128;" ::"r"(g + 1) : "memory"); };
  float ar[NA], br[CPT];
  auto load = [&](int st) {
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int e = t + 128 * i, r = e % BM, k = st * GS_KS + e / BM;
      ar[i] = (row0 + r < M && k < K) ? A[(size_t)k * lda + row0 + r] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < CPT; ++i) {
      const int e = t + 128 * i, k = st * GS_KS + (e & (GS_KS - 1)), c = e / GS_KS;
      br[i] = (k < K && c < ncol) ? float(B[(size_t)(col0 + c) * ldb + k]) : 0.f;
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int e = t + 128 * i;
      Ks[(size_t)(buf * GS_KS + e / BM) * F::LDK + e % BM] = ar[i];
    }
#pragma unroll
    for (int i = 0; i < CPT; ++i) {
      const int e = t + 128 * i;
      Bs[(buf * GS_KS + (e & (GS_KS - 1))) * F::LDB + e / GS_KS] = br[i];
    }
  };
  uint64_t acc[CPT][RPT / 2];
#pragma unroll
  for (int u = 0; u < CPT; ++u)
#pragma unroll
    for (int p = 0; p < RPT / 2; ++p) acc[u][p] = 0ull;
  if (first < nst) {
    load(first);
    store(0);
    if (first + step < nst) load(first + step);
    bar();
    int buf = 0;
    for (int st = first; st < nst; st += step, buf ^= 1) {
      stage_fma<CPT, RPT>(Ks, Bs, buf, tx, ty, acc);
      if (st + step < nst) {
        store(buf ^ 1);
        if (st + 2 * step < nst) load(st + 2 * step);
      }
      bar();
    }
  }
  float* Rs = reinterpret_cast<float*>(gsm);
  reduce_groups<CPT, RPT>(Rs, g, tx, ty, acc);
  cl.sync();
  const int share = (ncol + Z - 1) / Z, c0 = rank * share, c1 = min(ncol, c0 + share);
  for (int e = threadIdx.x; e < (c1 - c0) * BM; e += GS_THREADS) {
    const int c = c0 + e / BM, r = e % BM;
    if (row0 + r >= M) continue;
    float v = 0.f;
    for (int q = 0; q < Z; ++q) v += cl.map_shared_rank(Rs, q)[(size_t)c * F::LDR + r];
    float* o = C + (size_t)(col0 + c) * ldc + row0 + r;
    *o = beta == 0.f ? alpha * v : fmaf(alpha, v, beta * *o);
  }
  cl.sync();
}

// FP64.  A block owns 32 rows (one per lane) and up to 72 columns, column w + 8 u with warp w.  What
// counts is the number of FP64 instructions (a warp-wide one takes 19 cycles of its SM): a kernel
// value costs about 41 of them (Matern-5/2: 74 per value at 33 columns, by the instruction counters), so it is evaluated once per 72 columns, columns are not padded (a
// warp skips the ones beyond the width), and the cluster split keeps every SM busy.
// 4,097 x 2,000 x 33 takes 1,340 us, against 3,350 us for 64 x 64 tiles (65 blocks, 64 columns computed).
template <int KER, bool DER> __device__ __forceinline__ double kfn(const C4<double>& a, const C4<double>& b, double sf2) {
  const double d2 = dist2(a, b);
  return DER ? kval_dlogl<KER>(d2, sf2) : kval<KER>(d2, sf2);
}
template <int CPW>
__global__ void __launch_bounds__(GS_THREADS)
k_gram_block_f64(int fn, const C4<double>* __restrict__ Xr, int nr, const C4<double>* __restrict__ Xc, int nc,
                 const double* __restrict__ B, int ldb, int width, int cw, double sf2, double* __restrict__ Out,
                 int ldo) {
  constexpr int BN = 8 * CPW, NLD = (GS_KS * BN + GS_THREADS - 1) / GS_THREADS;
  constexpr int TILE = 2 * GS_KS * 33 > BN * 33 ? 2 * GS_KS * 33 : BN * 33;
  __shared__ double Ks[TILE];                           // two stages of values; later the partial tile
  __shared__ double Bs[2][GS_KS][BN + 1];
  cg::cluster_group cl = cg::this_cluster();
  const int Z = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row0 = (int)(blockIdx.x / Z) * 32, col0 = blockIdx.y * cw, ncol = min(cw, width - col0);
  const int nst = (nc + GS_KS - 1) / GS_KS;
  const C4<double> xi = Xr[min(row0 + lane, nr - 1)];
  double br[NLD];
  auto load_b = [&](int st) {
#pragma unroll
    for (int i = 0; i < NLD; ++i) {
      const int e = threadIdx.x + GS_THREADS * i, kk = e & (GS_KS - 1), c = e / GS_KS, j = st * GS_KS + kk;
      br[i] = (j < nc && c < ncol) ? B[(size_t)(col0 + c) * ldb + j] : 0.0;
    }
  };
  auto stage = [&](int st, int buf) {                   // 2 values per thread and the stage's B
#pragma unroll
    for (int u = 0; u < GS_KS / 8; ++u) {
      const int kk = warp + 8 * u, j = st * GS_KS + kk;
      double v = 0.0;
      if (j < nc) {
        const C4<double> xj = Xc[j];
        switch (fn) {
          case 0: v = kfn<0, false>(xi, xj, sf2); break;
          case 1: v = kfn<1, false>(xi, xj, sf2); break;
          case 2: v = kfn<2, false>(xi, xj, sf2); break;
          case 3: v = kfn<0, true>(xi, xj, sf2); break;
          case 4: v = kfn<1, true>(xi, xj, sf2); break;
          default: v = kfn<2, true>(xi, xj, sf2); break;
        }
      }
      Ks[(buf * GS_KS + kk) * 33 + lane] = v;
    }
#pragma unroll
    for (int i = 0; i < NLD; ++i) {
      const int e = threadIdx.x + GS_THREADS * i, kk = e & (GS_KS - 1), c = e / GS_KS;
      if (c < BN) Bs[buf][kk][c] = br[i];
    }
  };
  double acc[CPW];
#pragma unroll
  for (int u = 0; u < CPW; ++u) acc[u] = 0.0;
  if (rank < nst) {
    load_b(rank);
    stage(rank, 0);
    if (rank + Z < nst) load_b(rank + Z);
    __syncthreads();
    int buf = 0;
    for (int st = rank; st < nst; st += Z, buf ^= 1) {
      if (st + Z < nst) {
        stage(st + Z, buf ^ 1);
        if (st + 2 * Z < nst) load_b(st + 2 * Z);
      }
#pragma unroll 4
      for (int kk = 0; kk < GS_KS; ++kk) {
        const double k = Ks[(buf * GS_KS + kk) * 33 + lane];
#pragma unroll
        for (int u = 0; u < CPW; ++u)
          if (warp + 8 * u < ncol) acc[u] = fma(k, Bs[buf][kk][warp + 8 * u], acc[u]);
      }
      __syncthreads();
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < CPW; ++u) Ks[(warp + 8 * u) * 33 + lane] = acc[u];
  cl.sync();
  for (int c = rank * 8 + warp; c < ncol; c += 8 * Z) {
    double v = 0.0;
    for (int q = 0; q < Z; ++q) v += cl.map_shared_rank(Ks, q)[c * 33 + lane];
    if (row0 + lane < nr) Out[(size_t)(col0 + c) * ldo + row0 + lane] = v;
  }
  cl.sync();
}

template <class... KA, class... A>
void launch_clustered(void (*kernel)(KA...), dim3 grid, int Z, size_t smem, cudaStream_t st, A&&... args) {
  if (smem > 48 * 1024) cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid.x * Z, grid.y, 1);
  cfg.blockDim = dim3(GS_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = Z;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<KA>(args)...);
  note_launch();
}

// Blocks per cluster (1, 2, 4, 8) for `tiles` output tiles and `units` units of work along j per tile:
// the fewest rounds of resident blocks times the units each block then works through, plus the fixed
// cost of a block (`fixed` units: its prologue and the reduction).
int pick_cluster(long long tiles, int units, int slots, double fixed, double* cost) {
  int best = 1;
  double bc = 1e300;
  for (int Z = 1; Z <= 8; Z *= 2) {
    if (Z > 1 && units < Z) break;
    const double c = (double)((tiles * Z + slots - 1) / slots) * ((units + Z - 1) / Z + fixed);
    if (c < 0.97 * bc) { bc = c; best = Z; }
  }
  *cost = bc;
  return best;
}

template <int CPT, class TB>
void launch_nn(int M, int N, int K, float alpha, const float* A, int lda, const TB* B, int ldb, int cw, int nchunk,
               float beta, float* C, int ldc, cudaStream_t st) {
  const int units = ((K + GS_KS - 1) / GS_KS + 1) / 2, slots = 2 * 152;
  double c8, c2;
  const int t8 = (M + 127) / 128, t2 = (M + 31) / 32;
  const int z8 = pick_cluster((long long)t8 * nchunk, units, slots, 4.0, &c8);
  const int z2 = pick_cluster((long long)t2 * nchunk, units, slots, 4.0, &c2);
  if (2.5 * c8 <= c2)
    launch_clustered(k_gemm_nn_f32<CPT, 8, TB>, dim3(t8, nchunk), z8, F32Tile<CPT, 8>::SMEM, st, M, N, K, alpha, A, lda,
                     B, ldb, cw, beta, C, ldc);
  else
    launch_clustered(k_gemm_nn_f32<CPT, 2, TB>, dim3(t2, nchunk), z2, F32Tile<CPT, 2>::SMEM, st, M, N, K, alpha, A, lda,
                     B, ldb, cw, beta, C, ldc);
}

template <int CPT>
void launch_f32(int fn, const C4<float>* Xr, int nr, const C4<float>* Xc, int nc, const float* B, int ldb, int width,
                int cw, int nchunk, float sf2, float* Out, int ldo, cudaStream_t st) {
  // 128-row tiles use the FP32 pipe best (a stage costs about 2.5 times that of a 32-row tile for 4 times the
  // rows); 32-row tiles win where the 128-row ones, even clustered, leave SMs idle
  const int units = ((nc + GS_KS - 1) / GS_KS + 1) / 2, slots = 2 * 152;
  double c8, c2;
  const int t8 = (nr + 127) / 128, t2 = (nr + 31) / 32;
  const int z8 = pick_cluster((long long)t8 * nchunk, units, slots, 4.0, &c8);
  const int z2 = pick_cluster((long long)t2 * nchunk, units, slots, 4.0, &c2);
  if (2.5 * c8 <= c2)
    launch_clustered(k_gram_block_f32<CPT, 8>, dim3(t8, nchunk), z8, F32Tile<CPT, 8>::SMEM, st, fn, Xr, nr, Xc, nc, B,
                     ldb, width, cw, sf2, Out, ldo);
  else
    launch_clustered(k_gram_block_f32<CPT, 2>, dim3(t2, nchunk), z2, F32Tile<CPT, 2>::SMEM, st, fn, Xr, nr, Xc, nc, B,
                     ldb, width, cw, sf2, Out, ldo);
}

template <int CPW>
void launch_f64(int fn, const C4<double>* Xr, int nr, const C4<double>* Xc, int nc, const double* B, int ldb, int width,
                int cw, int nchunk, double sf2, double* Out, int ldo, cudaStream_t st) {
  const int tiles = (nr + 31) / 32;
  double c;
  const int Z = pick_cluster((long long)tiles * nchunk, (nc + GS_KS - 1) / GS_KS, 152, 2.0, &c);
  launch_clustered(k_gram_block_f64<CPW>, dim3(tiles, nchunk), Z, 0, st, fn, Xr, nr, Xc, nc, B, ldb, width, cw, sf2,
                   Out, ldo);
}

// fn: 0..2 the Matern orders, 3..5 their derivatives
template <class T>
void gram_block_fn(int fn, const C4<T>* Xr, int nr, const C4<T>* Xc, int nc, const T* B, int ldb, int width, T sf2,
                   T* Out, int ldo, cudaStream_t st) {
  if (nr <= 0 || width <= 0) return;
  const int nchunk = (width + GS_MAX_COLS - 1) / GS_MAX_COLS, cw = (width + nchunk - 1) / nchunk;
  // columns per thread (FP32) or warp (FP64), rounded up to an odd count: the filter's and smoother's blocks are
  // i + 1 columns wide, i mostly a multiple of 16 (33 and 65 columns are 5 and 9 without padding).  Even
  // counts would spare a width of 16, 32 or 64 a third to a ninth of its FP32 products; FP64 skips them anyway
  const int per = (cw + 7) / 8;
#define CAKF_GS(NAME)                                                                                             \
  if (per <= 1) NAME<1>(fn, Xr, nr, Xc, nc, B, ldb, width, cw, nchunk, sf2, Out, ldo, st);                        \
  else if (per <= 3) NAME<3>(fn, Xr, nr, Xc, nc, B, ldb, width, cw, nchunk, sf2, Out, ldo, st);                   \
  else if (per <= 5) NAME<5>(fn, Xr, nr, Xc, nc, B, ldb, width, cw, nchunk, sf2, Out, ldo, st);                   \
  else if (per <= 7) NAME<7>(fn, Xr, nr, Xc, nc, B, ldb, width, cw, nchunk, sf2, Out, ldo, st);                   \
  else NAME<9>(fn, Xr, nr, Xc, nc, B, ldb, width, cw, nchunk, sf2, Out, ldo, st)
  if constexpr (sizeof(T) == 4) { CAKF_GS(launch_f32); }
  else { CAKF_GS(launch_f64); }
#undef CAKF_GS
}

}  // namespace

template <class TB>
void gemm_nn_f32(int M, int N, int K, float alpha, const float* A, int lda, const TB* B, int ldb, float beta, float* C,
                 int ldc, cudaStream_t st) {
  constexpr int kMaxCols = 64;                          // (72 would spill: A's stage is in registers too)
  const int nchunk = (N + kMaxCols - 1) / kMaxCols, cw = (N + nchunk - 1) / nchunk, per = (cw + 7) / 8;
  if (per <= 1) launch_nn<1, TB>(M, N, K, alpha, A, lda, B, ldb, cw, nchunk, beta, C, ldc, st);
  else if (per <= 3) launch_nn<3, TB>(M, N, K, alpha, A, lda, B, ldb, cw, nchunk, beta, C, ldc, st);
  else if (per <= 5) launch_nn<5, TB>(M, N, K, alpha, A, lda, B, ldb, cw, nchunk, beta, C, ldc, st);
  else launch_nn<8, TB>(M, N, K, alpha, A, lda, B, ldb, cw, nchunk, beta, C, ldc, st);
}
template void gemm_nn_f32<float>(int, int, int, float, const float*, int, const float*, int, float, float*, int,
                                 cudaStream_t);
template void gemm_nn_f32<double>(int, int, int, float, const float*, int, const double*, int, float, float*, int,
                                  cudaStream_t);

template <class T>
void gram_block_simt(int ker, const C4<T>* Xr, int nr, const C4<T>* Xc, int nc, const T* B, int ldb, int width,
                     T sf2, T* Out, int ldo, cudaStream_t st) {
  gram_block_fn<T>(ker == 0 ? 0 : (ker == 1 ? 1 : 2), Xr, nr, Xc, nc, B, ldb, width, sf2, Out, ldo, st);
}

// Out = dK/dlog(l_x) (Xr, Xc) B  (the derivative Gram matrix, never stored)
template <class T>
void gram_block_dlogl_simt(int ker, const C4<T>* Xr, int nr, const C4<T>* Xc, int nc, const T* B, int ldb, int width,
                           T sf2, T* Out, int ldo, cudaStream_t st) {
  gram_block_fn<T>(ker == 0 ? 3 : (ker == 1 ? 4 : 5), Xr, nr, Xc, nc, B, ldb, width, sf2, Out, ldo, st);
}

#define INST(T)                                                                                                 \
  template void gram_block_simt<T>(int, const C4<T>*, int, const C4<T>*, int, const T*, int, int, T, T*, int,   \
                                   cudaStream_t);                                                               \
  template void gram_block_dlogl_simt<T>(int, const C4<T>*, int, const C4<T>*, int, const T*, int, int, T, T*,  \
                                         int, cudaStream_t);
INST(float)
INST(double)

}  // namespace cakf
