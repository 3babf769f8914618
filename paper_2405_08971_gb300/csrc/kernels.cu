// SIMT kernels of the CAKF/CAKS hot path (FP32 and FP64 instantiations):
//   - Gram matvec of the CG loop:  part[p][i] = sum_{j in split p} k(xo_i, xo_j) s_j
//   - tall-skinny GEMMs (split-K transposed products, tiled NN products)
//   - the CG / Gram-Schmidt bookkeeping of the iterative update step
//   - gathers, scatters and row epilogues of the filter and smoother.
#include <cooperative_groups.h>
#include "common.cuh"
#include <cuda_bf16.h>
#include "internal.h"

#include <atomic>

namespace cakf {

static std::atomic<long long> g_launches{0};
static thread_local int t_gemm_mode = 0;
static thread_local int* t_gemm_err = nullptr;
void set_gemm_mode(int mode) { t_gemm_mode = mode; }
int gemm_mode() { return t_gemm_mode; }
void set_gemm_err(int* err) { t_gemm_err = err; }

// Iteration limits of the bounded device-side waits (0 = the defaults of each kernel); a
// diagnostic setting for tests of the timeout path.
static std::atomic<long long> g_wait_limit{0};
void set_wait_limit(long long it) { g_wait_limit.store(it < 0 ? 0 : it); }
long long wait_limit(long long dflt) {
  const long long v = g_wait_limit.load();
  return v > 0 ? v : dflt;
}
long long launch_count() { return g_launches.load(); }
void note_launch(long long k) { g_launches += k; }

// ------------------------------------------------------------------------------------------
// Coordinates
template <class T>
__global__ void k_prep_coords(const double* __restrict__ X, int n, int dim, double scale,
                              C4<T>* __restrict__ out) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  C4<T> c;
  c.x = T(scale * X[(size_t)i * dim + 0]);
  c.y = dim > 1 ? T(scale * X[(size_t)i * dim + 1]) : T(0);
  c.z = dim > 2 ? T(scale * X[(size_t)i * dim + 2]) : T(0);
  c.w = T(0);
  out[i] = c;
}

// The same for the rows and columns of a Gram x block product, into one array (rows first): one launch.
template <class T>
__global__ void k_prep_coords2(const double* __restrict__ Xr, int nr, const double* __restrict__ Xc, int nc, int dim,
                               double scale, C4<T>* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nr + nc) return;
  const double* x = i < nr ? Xr + (size_t)i * dim : Xc + (size_t)(i - nr) * dim;
  C4<T> c;
  c.x = T(scale * x[0]);
  c.y = dim > 1 ? T(scale * x[1]) : T(0);
  c.z = dim > 2 ? T(scale * x[2]) : T(0);
  c.w = T(0);
  out[i] = c;
}

template <class T>
__global__ void k_gather_coords(const C4<T>* __restrict__ X, const int* __restrict__ idx, int m,
                                C4<T>* __restrict__ out) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m) out[i] = X[idx[i]];
}

// ------------------------------------------------------------------------------------------
// CG Gram matvec, split over columns; part is [nsplit][m].
// K(X_o, X_o) s for the CG actions, each kernel value evaluated once: the symmetric Gram is cut into
// MVS_T x MVS_T tiles and one block evaluates tile (I, J), I <= J.  Row sums (weights s_J) give tile
// I's share from J and, for I < J, column sums (weights s_I) give tile J's share from I.  The
// shares land in distinct slots -- part[J][rows of I] and part[I][rows of J] -- so every row has
// exactly nb = ceil(m / MVS_T) slots, each written once, summed in a fixed order by k_cg_combine.
// A lane owns MVS_R rows of the tile; each warp takes 32 of its columns (staged in shared memory)
// and reduces a column's MVS_R * 32 products with one warp sum.
// The first ngv blocks instead form the partials of t = Mo^T s (one warp per column of Mo and
// chunk of GV_CHUNK rows), which k_cg_combine needs next: one launch for both.
constexpr int MVS_T = 128, MVS_R = MVS_T / 32, MVS_W = MVS_T / 32;
constexpr int GV_CHUNK = 1024;

// Partials of t = Mo^T s: block b of the first ngv blocks of a matvec launch.
template <class T>
__device__ __forceinline__ void gv_block(const T* __restrict__ Mo, int ldm, int rp, const T* __restrict__ s, int m,
                                         T* __restrict__ tpart) {
  const int per_chunk = (rp + MVS_W - 1) / MVS_W;
  const int z = blockIdx.x / per_chunk;
  const int col = (blockIdx.x - z * per_chunk) * MVS_W + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (col >= rp) return;
  const int i0 = z * GV_CHUNK, i1 = min(m, i0 + GV_CHUNK);
  const T* a = Mo + (size_t)col * ldm;
  T acc = T(0);
#pragma unroll 8
  for (int i = i0 + lane; i < i1; i += 32) acc = fma(a[i], s[i], acc);
  acc = warp_sum(acc);
  if (lane == 0) tpart[(size_t)z * rp + col] = acc;
}

// The FP64 matvec on TILE x TILE tiles, R = TILE / 32 rows per lane, TILE / MVS_W columns per warp.
template <int KER, class T, int R>
__global__ void __launch_bounds__(MVS_W * 32)
k_gram_matvec(const C4<T>* __restrict__ Xo, const T* __restrict__ s, int m, int nb, T sf2, T* __restrict__ part,
              const T* __restrict__ Mo, int ldm, int rp, int ngv, T* __restrict__ tpart,
              const int* __restrict__ active) {
  constexpr int TILE = 32 * R, CW = TILE / MVS_W;
  pdl_wait();
  pdl_trigger();
  if (active && !*active) return;
  __shared__ C4<T> xs[TILE];
  __shared__ T ss[TILE];
  __shared__ T racc[MVS_W][TILE];
  if ((int)blockIdx.x < ngv) {
    gv_block(Mo, ldm, rp, s, m, tpart);
    return;
  }
  int idx = blockIdx.x - ngv, I = 0;
  while (idx >= nb - I) { idx -= nb - I; ++I; }
  const int J = I + idx;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int t = threadIdx.x; t < TILE; t += blockDim.x) {
    const int j = J * TILE + t;
    C4<T> x;
    x.x = x.y = x.z = x.w = T(0);
    T v = T(0);
    if (j < m) { x = Xo[j]; v = s[j]; }
    xs[t] = x;
    ss[t] = v;
  }
  C4<T> xi[R];
  T si[R], acc[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = I * TILE + lane + 32 * r;
    xi[r].x = xi[r].y = xi[r].z = xi[r].w = T(0);
    si[r] = T(0);
    if (i < m) { xi[r] = Xo[i]; si[r] = s[i]; }
    acc[r] = T(0);
  }
  __syncthreads();
  T cacc = T(0);
  if (I == J) {
#pragma unroll 4
    for (int jj = 0; jj < CW; ++jj) {
      const C4<T> xj = xs[warp * CW + jj];
      const T sj = ss[warp * CW + jj];
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r] = fma(kval<KER>(dist2(xi[r], xj), sf2), sj, acc[r]);
    }
  } else {
#pragma unroll 4
    for (int jj = 0; jj < CW; ++jj) {
      const C4<T> xj = xs[warp * CW + jj];
      const T sj = ss[warp * CW + jj];
      T cp = T(0);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const T kv = kval<KER>(dist2(xi[r], xj), sf2);
        acc[r] = fma(kv, sj, acc[r]);
        cp = fma(kv, si[r], cp);
      }
      cp = warp_sum(cp);
      if (lane == jj) cacc = cp;
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) racc[warp][lane + 32 * r] = acc[r];
  __syncthreads();
  for (int t = threadIdx.x; t < TILE; t += blockDim.x) {
    const int i = I * TILE + t;
    if (i >= m) continue;
    T v = racc[0][t];
#pragma unroll
    for (int w = 1; w < MVS_W; ++w) v += racc[w][t];
    part[(size_t)J * m + i] = v;
  }
  if (I != J && lane < CW) {
    const int j = J * TILE + warp * CW + lane;
    if (j < m) part[(size_t)I * m + j] = cacc;
  }
}

// The FP64 matvec for few observations, where even 32 x 32 tiles leave most SMs idle: every entry is
// evaluated (no symmetry), a block takes 32 rows (one per lane) and MVS_W * cpw columns (cpw per
// warp), and its sum goes to the slot of its column group, so the slots per row number
// ceil(m / (MVS_W cpw)) and no column sums are needed.  An FP64 Matern-5/2 value is about 41
// FP64 instructions, most of them a dependent chain (a warp-wide one takes 19 cycles of the SM's FP64 pipe), so
// what counts is how many SMs share the values.
template <int KER, class T>
__global__ void __launch_bounds__(MVS_W * 32)
k_gram_matvec_rows(const C4<T>* __restrict__ Xo, const T* __restrict__ s, int m, int nslot, int cpw, T sf2,
                   T* __restrict__ part, const T* __restrict__ Mo, int ldm, int rp, int ngv, T* __restrict__ tpart,
                   const int* __restrict__ active) {
  pdl_wait();
  pdl_trigger();
  if (active && !*active) return;
  __shared__ T racc[MVS_W][32];
  if ((int)blockIdx.x < ngv) {
    gv_block(Mo, ldm, rp, s, m, tpart);
    return;
  }
  const int b = blockIdx.x - ngv, rt = b / nslot, slot = b - rt * nslot;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = rt * 32 + lane;
  const C4<T> xi = Xo[min(i, m - 1)];
  const int j0 = (slot * MVS_W + warp) * cpw;
  T acc = T(0);
  for (int j = j0; j < min(m, j0 + cpw); ++j) acc = fma(kval<KER>(dist2(xi, Xo[j]), sf2), s[j], acc);
  racc[warp][lane] = acc;
  __syncthreads();
  if (warp == 0 && i < m) {
    T v = racc[0][lane];
#pragma unroll
    for (int w = 1; w < MVS_W; ++w) v += racc[w][lane];
    part[(size_t)slot * m + i] = v;
  }
}

// The FP32 matvec on packed pairs of rows (f32x2 arithmetic): a lane owns MVS_R = 4 rows of tile I
// as two pairs, the column records of tile J are staged duplicated ({x,x},{y,y},{z,z},{w,w} with
// w = sf2 s_j), and a warp's 32 per-column sums over its lanes' rows are reduced by one butterfly
// reduce-scatter (31 shuffles) instead of one warp sum per column.  Same tiles, slots and Mo^T s
// blocks as k_gram_matvec.
template <int KER>
__global__ void __launch_bounds__(MVS_W * 32, 7)   // 7 blocks per SM (72 registers): 24.3 -> 23.9 us
k_gram_matvec_f2(const C4<float>* __restrict__ Xo, const float* __restrict__ s, int m, int nb, float sf2,
                 float* __restrict__ part, const float* __restrict__ Mo, int ldm, int rp, int ngv,
                 float* __restrict__ tpart, const int* __restrict__ active) {
  pdl_wait();
  pdl_trigger();
  if (active && !*active) return;
  __shared__ uint64_t xs2[MVS_T][4];
  __shared__ float racc[MVS_W][MVS_T];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if ((int)blockIdx.x < ngv) {
    gv_block(Mo, ldm, rp, s, m, tpart);
    return;
  }
  int idx = blockIdx.x - ngv, I = 0;
  while (idx >= nb - I) { idx -= nb - I; ++I; }
  const int J = I + idx;
  for (int t = threadIdx.x; t < MVS_T; t += blockDim.x) {
    const int j = J * MVS_T + t;
    float x = 0.f, y = 0.f, zc = 0.f, w = 0.f;
    if (j < m) { const C4<float> c = Xo[j]; x = c.x; y = c.y; zc = c.z; w = sf2 * s[j]; }
    xs2[t][0] = f2_make(x, x);
    xs2[t][1] = f2_make(y, y);
    xs2[t][2] = f2_make(zc, zc);
    xs2[t][3] = f2_make(w, w);
  }
  uint64_t rx[2], ry[2], rz[2], rs[2], acc[2];
#pragma unroll
  for (int pr = 0; pr < 2; ++pr) {
    float xv[2] = {0.f, 0.f}, yv[2] = {0.f, 0.f}, zv[2] = {0.f, 0.f}, sv[2] = {0.f, 0.f};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = I * MVS_T + lane + 32 * (2 * pr + h);
      if (i < m) { const C4<float> c = Xo[i]; xv[h] = c.x; yv[h] = c.y; zv[h] = c.z; sv[h] = sf2 * s[i]; }
    }
    rx[pr] = f2_make(xv[0], xv[1]);
    ry[pr] = f2_make(yv[0], yv[1]);
    rz[pr] = f2_make(zv[0], zv[1]);
    rs[pr] = f2_make(sv[0], sv[1]);
    acc[pr] = f2_make(0.f, 0.f);
  }
  __syncthreads();
  const uint64_t(*xc)[4] = xs2 + warp * 32;
  float cacc = 0.f;
  if (I == J) {
#pragma unroll 8
    for (int jj = 0; jj < 32; ++jj) {
      const uint64_t cx = xc[jj][0], cy = xc[jj][1], cz = xc[jj][2], cw = xc[jj][3];
#pragma unroll
      for (int pr = 0; pr < 2; ++pr) acc[pr] = f2_fma(kpair<KER>(rx[pr], ry[pr], rz[pr], cx, cy, cz), cw, acc[pr]);
    }
  } else {
    float v[32];
#pragma unroll
    for (int jj = 0; jj < 32; ++jj) {
      const uint64_t cx = xc[jj][0], cy = xc[jj][1], cz = xc[jj][2], cw = xc[jj][3];
      const uint64_t k0 = kpair<KER>(rx[0], ry[0], rz[0], cx, cy, cz);
      const uint64_t k1 = kpair<KER>(rx[1], ry[1], rz[1], cx, cy, cz);
      acc[0] = f2_fma(k0, cw, acc[0]);
      acc[1] = f2_fma(k1, cw, acc[1]);
      v[jj] = f2_sum(f2_fma(k1, rs[1], f2_mul(k0, rs[0])));
    }
    // butterfly reduce-scatter: after the stage with offset o a lane keeps the half of its
    // column sums selected by its bit o; at the end lane l holds the sum for column l
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int q = 0; q < o; ++q) {
        const float send = up ? v[q] : v[q + o];
        const float keep = up ? v[q + o] : v[q];
        v[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    }
    cacc = v[0];
  }
#pragma unroll
  for (int pr = 0; pr < 2; ++pr) {
    float lo, hi;
    f2_split(acc[pr], lo, hi);
    racc[warp][lane + 32 * (2 * pr)] = lo;
    racc[warp][lane + 32 * (2 * pr + 1)] = hi;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < MVS_T; t += blockDim.x) {
    const int i = I * MVS_T + t;
    if (i >= m) continue;
    float vv = racc[0][t];
#pragma unroll
    for (int w = 1; w < MVS_W; ++w) vv += racc[w][t];
    part[(size_t)J * m + i] = vv;
  }
  if (I != J) {
    const int j = J * MVS_T + warp * 32 + lane;
    if (j < m) part[(size_t)I * m + j] = cacc;
  }
}

// ---- the CG iteration's vector kernels: k_cg_combine, k_cg_upd1, k_cg_upd2.  Each moves a few MB at most, so
// a chain of L2 round trips and barriers bounds them, and in FP64 the FP64 pipe of the few SMs a small step
// occupies.  Hence:
//  - Everything a kernel reads that was written two launches earlier or before (the factor rows, the previous
//    directions, s, r, v) is loaded before pdl_wait(), while the kernel in front is still running: that kernel
//    began its own work only after its pdl_wait(), that is after the one before it had completed, and this one
//    was launched only after that.  These loads bypass L1 (ldcg): the launch in front may be writing a
//    neighbouring column whose first rows share a cache line with them.
//  - Sums over the lanes are taken several at a time (warp_sum_t: half the lanes go on with half the values),
//    which for 8 FP64 sums takes 9 additions per lane instead of 40.
//  - FP64 with up to CG64_SMALL_MAX observations takes small row blocks (8 rows by 4 columns per warp), which
//    put the products on four times as many SMs.
//  - The update kernel also writes the next action where it is known (residual, replayed or stored one).
// Every FP32 sum keeps its order whatever is loaded ahead.  One iteration with its matvec, before and after:
// 128 observations, 256 columns, 32 directions (FP64) 32.0 -> 20.0 us; 8,192 x 512 x 64 (FP32) 40.6 -> 32.2 us.
constexpr int CG64_SMALL_MAX = 2048;
__device__ __forceinline__ float ldcg_if(bool p, const float* a) {
  float x;
  asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %2, 0;\n mov.b32 %0, 0;\n @q ld.global.cg.f32 %0, [%1];\n}\n"
               : "=f"(x) : "l"(a), "r"((int)p) : "memory");
  return x;
}
__device__ __forceinline__ double ldcg_if(bool p, const double* a) {
  double x;
  asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %2, 0;\n mov.b64 %0, 0;\n @q ld.global.cg.f64 %0, [%1];\n}\n"
               : "=d"(x) : "l"(a), "r"((int)p) : "memory");
  return x;
}
__device__ __forceinline__ int ldcg_i(const int* a) {
  int x;
  asm volatile("ld.global.cg.s32 %0, [%1];" : "=r"(x) : "l"(a) : "memory");
  return x;
}

// Sums of NV values (a power of two, <= 32) over the lanes of a warp; lane l gets the total of value
// warp_sum_idx<NV>(l).  Pairs lanes in warp_sum's order, so the totals equal its bit for bit.
template <int NV> __device__ __forceinline__ int warp_sum_idx(int lane) {
  int k = 0;
#pragma unroll
  for (int h = NV / 2, o = 16; h >= 1; h >>= 1, o >>= 1) k += (lane & o) ? h : 0;
  return k;
}
template <int NV, class T> __device__ __forceinline__ T warp_sum_t(T (&v)[NV]) {
  const int lane = threadIdx.x & 31;
  int o = 16;
#pragma unroll
  for (int h = NV / 2; h >= 1; h >>= 1, o >>= 1) {
#pragma unroll
    for (int k = 0; k < h; ++k) {
      const bool up = lane & o;
      const T send = up ? v[k] : v[k + h], keep = up ? v[k + h] : v[k];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  T t = v[0];
#pragma unroll
  for (; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// g = sum_p part[p] + sn2 * s - a2 * Mo t     (Mo: m x r col-major, ld = ldm).  t is summed from
// the row-chunk partials of the matvec launch's Mo^T s blocks (tz chunks) into shared memory
// first.  A block owns ROWS rows; a warp takes CC = 32 / ROWS columns of Mo at a time, every CB_WARPS-th
// group of them (CB_UNROLL independent accumulators), and the warps' sums are added
// in shared memory.  The block then forms its rows' share of the first dot pass of CG iteration j
//   q < j: V[:, q] . g ;  j: s . g ;  j+1: s . r0 ;  j+2: g . v ;  j+3: s . s
// into dpart[q * gridDim.x + block] (summed by k_cg_upd1 in a fixed order, in the working precision:
// FP64 adds would cost more than the data they sum on this GPU).
constexpr int CB_ROWS = 32, CB_ROWS_SMALL = 8, CB_WARPS = 8, CB_UNROLL = 8;
template <class T, int ROWS>
__global__ void __launch_bounds__(CB_WARPS * 32)
k_cg_combine(const T* __restrict__ part, int nsplit, const T* __restrict__ s, T sn2,
             const T* __restrict__ Mo, int ldm, int r, const T* __restrict__ tpart, int tz, T a2,
             int m, T* __restrict__ g, const T* __restrict__ V, int ldv, int j, const T* __restrict__ r0,
             const T* __restrict__ v, T* __restrict__ dpart, const int* __restrict__ active) {
  constexpr int CC = 32 / ROWS;
  constexpr int PRE = sizeof(T) == 4 ? 64 : (CC > 1 ? 16 : 32);   // columns per thread loaded ahead
  constexpr int QB = CC > 1 ? 2 : 8;                              // dots per thread whose loads are in flight together
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rl = lane % ROWS, cl = lane / ROWS;
  const int i = blockIdx.x * ROWS + rl;
  const bool valid = i < m;
  const int rv = (r + CC - 1) / CC;                    // groups of CC columns
  T x0[PRE], xq[QB];
#pragma unroll
  for (int e = 0; e < PRE; ++e) {
    const int col = (warp + e * CB_WARPS) * CC + cl;
    x0[e] = ldcg_if(valid && col < r, Mo + (size_t)col * ldm + i);
  }
#pragma unroll
  for (int u = 0; u < QB; ++u) {
    const int q = (warp + u * CB_WARPS) * CC + cl;
    xq[u] = ldcg_if(valid && q < j, V + (size_t)q * ldv + i);
  }
  const T si = ldcg_if(valid, s + i), r0i = ldcg_if(valid, r0 + i), vi = ldcg_if(valid, v + i);
  const int act = ldcg_i(active);
  pdl_wait();
  pdl_trigger();
  if (!act) return;
  extern __shared__ unsigned char sm_raw[];
  T* t = reinterpret_cast<T*>(sm_raw);                 // r coefficients, zeros up to rv * CC
  __shared__ T red[CB_WARPS][ROWS], redk[CB_WARPS][ROWS];
  __shared__ T gsh[ROWS];
  // the Gram partials: warp w sums slots w, w + CB_WARPS, ... (with CC > 1 CC of them at a time).  Every loop
  // below loads a batch of independent values before it uses any of them, so a thread waits for one L2 round
  // trip per batch rather than one per value (the summation order is the same as one value at a time).
  T kw = T(0);
  if (valid) {
    constexpr int ST = CB_WARPS * CC;
    int p = warp * CC + cl;
    for (; p + 7 * ST < nsplit; p += 8 * ST) {
      T x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) x[u] = part[(size_t)(p + u * ST) * m + i];
#pragma unroll
      for (int u = 0; u < 8; ++u) kw += x[u];
    }
    for (; p < nsplit; p += ST) kw += part[(size_t)p * m + i];
  }
  for (int l = threadIdx.x; l < rv * CC; l += blockDim.x) {
    T acc = T(0);
    if (l < r) {
      int z = 0;
      for (; z + 8 <= tz; z += 8) {
        T x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = tpart[(size_t)(z + u) * r + l];
#pragma unroll
        for (int u = 0; u < 8; ++u) acc += x[u];
      }
      for (; z < tz; ++z) acc += tpart[(size_t)z * r + l];
    }
    t[l] = acc;
  }
  __syncthreads();
  T acc[CB_UNROLL];
#pragma unroll
  for (int u = 0; u < CB_UNROLL; ++u) acc[u] = T(0);
#pragma unroll
  for (int e0 = 0; e0 < PRE; e0 += CB_UNROLL) {
    const int l = warp + e0 * CB_WARPS;
    if (l >= rv) break;
    if (l + (CB_UNROLL - 1) * CB_WARPS < rv) {
#pragma unroll
      for (int u = 0; u < CB_UNROLL; ++u) acc[u] = fma(x0[e0 + u], t[(l + u * CB_WARPS) * CC + cl], acc[u]);
    } else {
#pragma unroll
      for (int u = 0; u < CB_UNROLL; ++u) {
        if (l + u * CB_WARPS >= rv) break;
        acc[0] = fma(x0[e0 + u], t[(l + u * CB_WARPS) * CC + cl], acc[0]);
      }
    }
  }
  if (valid) {
    int l = warp + PRE * CB_WARPS;
    for (; l + (CB_UNROLL - 1) * CB_WARPS < rv; l += CB_UNROLL * CB_WARPS) {
      T x[CB_UNROLL];
#pragma unroll
      for (int u = 0; u < CB_UNROLL; ++u) {
        const int col = (l + u * CB_WARPS) * CC + cl;
        x[u] = col < r ? Mo[(size_t)col * ldm + i] : T(0);
      }
#pragma unroll
      for (int u = 0; u < CB_UNROLL; ++u) acc[u] = fma(x[u], t[(l + u * CB_WARPS) * CC + cl], acc[u]);
    }
    for (; l < rv; l += CB_WARPS) {
      const int col = l * CC + cl;
      acc[0] = fma(col < r ? Mo[(size_t)col * ldm + i] : T(0), t[col], acc[0]);
    }
  }
  T lr = T(0);
#pragma unroll
  for (int u = 0; u < CB_UNROLL; ++u) lr += acc[u];
#pragma unroll
  for (int o = ROWS; o < 32; o <<= 1) {
    lr += __shfl_xor_sync(0xffffffffu, lr, o);
    kw += __shfl_xor_sync(0xffffffffu, kw, o);
  }
  if (cl == 0) {
    red[warp][rl] = lr;
    redk[warp][rl] = kw;
  }
  __syncthreads();
  if (threadIdx.x < ROWS) {
    T gv = T(0);
    if (valid) {
      T low = T(0), kv = T(0);
#pragma unroll
      for (int w = 0; w < CB_WARPS; ++w) { low += red[w][rl]; kv += redk[w][rl]; }
      kv = fma(sn2, si, kv);
      gv = fma(-a2, low, kv);
      g[i] = gv;
    }
    gsh[rl] = gv;
  }
  __syncthreads();
  const T gi = gsh[rl];
  for (int q0 = warp * CC; q0 < j + 4; q0 += QB * CB_WARPS * CC) {
    T pr[QB];
#pragma unroll
    for (int u = 0; u < QB; ++u) {
      const int q = q0 + u * CB_WARPS * CC + cl;
      T a = si, b = si;                                // q == j + 3
      if (q < j) {
        a = q0 == warp * CC ? xq[u] : (valid ? V[(size_t)q * ldv + i] : T(0));
        b = gi;
      } else if (q == j) {
        b = gi;
      } else if (q == j + 1) {
        b = r0i;
      } else if (q == j + 2) {
        a = gi;
        b = vi;
      }
      pr[u] = (valid && q < j + 4) ? a * b : T(0);
    }
    if constexpr (CC == 1) {
      const T tot = warp_sum_t<QB>(pr);
      const int q = q0 + warp_sum_idx<QB>(lane) * CB_WARPS;
      if (lane % (32 / QB) == 0 && q < j + 4) dpart[(size_t)q * gridDim.x + blockIdx.x] = tot;
    } else {
#pragma unroll
      for (int u = 0; u < QB; ++u) {
        const int q = q0 + u * CB_WARPS * CC + cl;
        if (q - cl >= j + 4) break;   // uniform across the warp
        T tot = pr[u];
#pragma unroll
        for (int o = ROWS / 2; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
        if (rl == 0 && q < j + 4) dpart[(size_t)q * gridDim.x + blockIdx.x] = tot;
      }
    }
  }
}

// Per-thread share of a block-wide dot product a . b over m entries (strided by blockDim.x).
// FP32 data: four FP32 FMA chains combined in FP64, so the FP64 pipe (slow on this GPU) sees a
// handful of operations per thread; FP64 data: FP64 throughout.
template <class T> __device__ __forceinline__ double dot_part(const T* __restrict__ a, const T* __restrict__ b, int m) {
  const int st = blockDim.x;
  int i = threadIdx.x;
  if constexpr (sizeof(T) == 8) {
    double acc = 0.0;
    for (; i < m; i += st) acc = fma(a[i], b[i], acc);
    return acc;
  } else {
    float p0 = 0.f, p1 = 0.f, p2 = 0.f, p3 = 0.f;
    for (; i + 3 * st < m; i += 4 * st) {
      p0 = fmaf(a[i], b[i], p0);
      p1 = fmaf(a[i + st], b[i + st], p1);
      p2 = fmaf(a[i + 2 * st], b[i + 2 * st], p2);
      p3 = fmaf(a[i + 3 * st], b[i + 3 * st], p3);
    }
    for (; i < m; i += st) p0 = fmaf(a[i], b[i], p0);
    return (double(p0) + double(p1)) + (double(p2) + double(p3));
  }
}

// Sum of the per-block partials part[q * nblk + b] over b for q in [0, nq), in a fixed order, into
// out[q] (shared memory) -- and, if dots != null, into dots[q] in FP64.  Each warp takes UP_QB values
// of q at a time, BB partials per lane, so that their loads are in flight together.
constexpr int UP_QB = 4;
template <int BB, class T>
__device__ __forceinline__ void sum_partials_bb(const T* __restrict__ part, int nblk, int nq, T* out, double* dots) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int q0 = warp * UP_QB; q0 < nq; q0 += nw * UP_QB) {
    T acc[UP_QB];
#pragma unroll
    for (int u = 0; u < UP_QB; ++u) acc[u] = T(0);
    for (int b0 = lane; b0 < nblk; b0 += 32 * BB) {
      T x[UP_QB][BB];
#pragma unroll
      for (int u = 0; u < UP_QB; ++u)
#pragma unroll
        for (int e = 0; e < BB; ++e) {
          const int b = b0 + 32 * e;
          x[u][e] = (q0 + u < nq && b < nblk) ? part[(size_t)(q0 + u) * nblk + b] : T(0);
        }
#pragma unroll
      for (int u = 0; u < UP_QB; ++u)
#pragma unroll
        for (int e = 0; e < BB; ++e)
          if (b0 + 32 * e < nblk) acc[u] += x[u][e];
    }
    const T t = warp_sum_t<UP_QB>(acc);
    const int q = q0 + warp_sum_idx<UP_QB>(lane);
    if (lane % (32 / UP_QB) == 0 && q < nq) {
      out[q] = t;
      if (dots) dots[q] = double(t);
    }
  }
}
template <class T>
__device__ __forceinline__ void sum_partials(const T* __restrict__ part, int nblk, int nq, T* out, double* dots) {
  // (FP64 additions that are switched off cost as much as ones that are not: no more of them than partials)
  if (sizeof(T) == 8 && nblk <= 64) sum_partials_bb<1>(part, nblk, nq, out, dots);
  else sum_partials_bb<8>(part, nblk, nq, out, dots);
}

// Row block of the CG update kernels: ROWS rows, UP_THREADS / ROWS threads per row, each summing every
// (UP_THREADS / ROWS)-th term of a row's sum over the previous directions (the loads of a warp stay coalesced:
// its 32 threads take 32 consecutive rows of one column).
constexpr int UP_THREADS = 256, UP_ROWS = 64, UP_ROWS_SMALL = 32;
constexpr int UP_VB = 8;   // previous directions per thread whose V, GV loads are in flight together

// This thread's values of up to UP_VB directions q0, q0 + SPLIT, ... < j of V and GV.
template <int SPLIT, class T>
__device__ __forceinline__ void load_dirs(const T* V, const T* GV, int ldv, int i, bool valid, int q0, int j,
                                          T (&xv)[UP_VB], T (&xg)[UP_VB]) {
#pragma unroll
  for (int e = 0; e < UP_VB; ++e) {
    const int q = q0 + SPLIT * e;
    xv[e] = ldcg_if(valid && q < j, V + (size_t)q * ldv + i);
    xg[e] = ldcg_if(valid && q < j, GV + (size_t)q * ldv + i);
  }
}
// d -= V c, gd -= GV c over this thread's directions sp, sp + SPLIT, ...; the first UP_VB of them are in xv, xg.
template <int SPLIT, class T>
__device__ __forceinline__ void orth_pass(const T* V, const T* GV, int ldv, int i, bool valid, int sp, int j,
                                          const T* c, const T (&xv)[UP_VB], const T (&xg)[UP_VB], T& d, T& gd) {
#pragma unroll
  for (int e = 0; e < UP_VB; ++e) {
    const int q = sp + SPLIT * e;
    if (q >= j) break;
    d = fma(-xv[e], c[q], d);
    gd = fma(-xg[e], c[q], gd);
  }
  for (int q0 = sp + SPLIT * UP_VB; q0 < j; q0 += SPLIT * UP_VB) {
    T yv[UP_VB], yg[UP_VB];
    load_dirs<SPLIT>(V, GV, ldv, i, valid, q0, j, yv, yg);
#pragma unroll
    for (int e = 0; e < UP_VB; ++e) {
      const int q = q0 + SPLIT * e;
      if (q >= j) break;
      d = fma(-yv[e], c[q], d);
      gd = fma(-yg[e], c[q], gd);
    }
  }
}

// First G-orthogonalisation pass of CG iteration j.  The first-pass dots are summed from the
// combine blocks' partials (fixed order; block 0 also stores all j + 4 of them in dots1):
// c = V^T G s, then d = s - V c, G d = g - GV c, parked unnormalised in column j of V and GV.
// The block then forms its rows' share of the second-pass dots (q < j: V[:, q] . G d; j: d . G d)
// into dpart2[q * gridDim.x + block].
template <class T, int ROWS>
__global__ void __launch_bounds__(UP_THREADS)
k_cg_upd1(int j, const T* __restrict__ dpart1, int nblk1, double* __restrict__ dots1, T* V, T* GV, int ldv,
          const T* __restrict__ s, const T* __restrict__ g, int m, T* __restrict__ dpart2,
          const int* __restrict__ active) {
  constexpr int SPLIT = UP_THREADS / ROWS, RT = ROWS / 32;   // (RT rows per lane in the dots)
  constexpr int NW = UP_THREADS / 32, PQ = 2;                // passes of the dots whose loads are made ahead
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rl = threadIdx.x % ROWS, sp = threadIdx.x / ROWS;
  const int row0 = blockIdx.x * ROWS;
  const int i = row0 + rl;
  const bool valid = i < m;
  const int nrow = min(ROWS, m - row0);
  T xv[UP_VB], xg[UP_VB], xd[PQ][UP_QB][RT];
  load_dirs<SPLIT>(V, GV, ldv, i, valid, sp, j, xv, xg);
  auto load_dots = [&](int q0, T (&x)[UP_QB][RT]) {
#pragma unroll
    for (int u = 0; u < UP_QB; ++u)
#pragma unroll
      for (int e = 0; e < RT; ++e) {
        const int t = lane + 32 * e, q = q0 + u;
        x[u][e] = ldcg_if(t < nrow && q < j, V + (size_t)q * ldv + row0 + t);
      }
  };
#pragma unroll
  for (int p = 0; p < PQ; ++p) load_dots((warp + p * NW) * UP_QB, xd[p]);
  const T si = ldcg_if(valid, s + i);
  const int act = ldcg_i(active);
  pdl_wait();
  pdl_trigger();
  if (!act) return;
  __shared__ T c[1024 + 4];
  __shared__ T sd[SPLIT][ROWS], sgd[SPLIT][ROWS];
  const T gi = sp == 0 && valid ? g[i] : T(0);
  sum_partials(dpart1, nblk1, (blockIdx.x == 0) ? j + 4 : j, c, blockIdx.x == 0 ? dots1 : nullptr);
  __syncthreads();
  T d = T(0), gd = T(0);
  orth_pass<SPLIT>(V, GV, ldv, i, valid, sp, j, c, xv, xg, d, gd);
  sd[sp][rl] = d;
  sgd[sp][rl] = gd;
  __syncthreads();
  if (sp == 0) {
    d = T(0); gd = T(0);
    if (valid) {
      d = si;
      gd = gi;
#pragma unroll
      for (int u = 0; u < SPLIT; ++u) { d += sd[u][rl]; gd += sgd[u][rl]; }
      V[(size_t)j * ldv + i] = d;
      GV[(size_t)j * ldv + i] = gd;
    }
    sd[0][rl] = d;
    sgd[0][rl] = gd;
  }
  __syncthreads();
  T dl[RT], gl[RT];
#pragma unroll
  for (int e = 0; e < RT; ++e) { dl[e] = sd[0][lane + 32 * e]; gl[e] = sgd[0][lane + 32 * e]; }
  auto dots = [&](int q0, const T (&x)[UP_QB][RT]) {
    T acc[UP_QB];
#pragma unroll
    for (int u = 0; u < UP_QB; ++u) {
      acc[u] = T(0);
#pragma unroll
      for (int e = 0; e < RT; ++e) acc[u] = fma(q0 + u == j ? dl[e] : x[u][e], gl[e], acc[u]);
    }
    const T t = warp_sum_t<UP_QB>(acc);
    const int q = q0 + warp_sum_idx<UP_QB>(lane);
    if (lane % (32 / UP_QB) == 0 && q <= j) dpart2[(size_t)q * gridDim.x + blockIdx.x] = t;
  };
#pragma unroll
  for (int p = 0; p < PQ; ++p) {
    const int q0 = (warp + p * NW) * UP_QB;
    if (q0 <= j) dots(q0, xd[p]);
  }
  for (int q0 = (warp + PQ * NW) * UP_QB; q0 <= j; q0 += NW * UP_QB) {
    T x[UP_QB][RT];
    load_dots(q0, x);
    dots(q0, x);
  }
}

// Second pass and the update of the iterative CAKF step (appendix algorithm):
//   c2 = V^T G d;  d <- d - V c2;  eta = d^T G d - |c2|^2;  alpha = s^T (r0 - G v) = s^T r0 - g^T v;
//   V[:, j] = d / sqrt(eta);  GV[:, j] = G d / sqrt(eta);  v += (alpha / eta) d;  r -= (alpha / eta) G d.
// Every block sums the second-pass dots from the k_cg_upd1 partials, recomputes the scalars and
// takes the same stop decision.  The next action, if it is known by then, is written to s here: a given one
// (snext_rep: replayed actions; snext_col: a stored column), or, with only Snext (CG policy without
// re-orthogonalisation), the updated residual; Snext also receives it as column j + 1 of S.
template <class T, int ROWS>
__global__ void __launch_bounds__(UP_THREADS)
k_cg_upd2(int j, const double* __restrict__ dots1, const T* __restrict__ dpart2, int nblk2,
          T* V, T* GV, int ldv, T* r, T* v, T* s, T* __restrict__ Q, int m,
          double bd_tol, double rtol2_r0sq, int use_rtol, int* active,
          double* __restrict__ eta_out, double* __restrict__ alpha_out, int* __restrict__ count,
          T* Snext, const double* __restrict__ snext_rep, const T* snext_col) {
  constexpr int SPLIT = UP_THREADS / ROWS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rl = threadIdx.x % ROWS, sp = threadIdx.x / ROWS;
  const int i = blockIdx.x * ROWS + rl;
  const bool valid = i < m, own = sp == 0 && valid;
  T xv[UP_VB], xg[UP_VB];
  load_dirs<SPLIT>(V, GV, ldv, i, valid, sp, j, xv, xg);
  const T ri = ldcg_if(own, r + i), vi = ldcg_if(own, v + i), si = ldcg_if(own && Q, s + i);
  T sn = T(0);
  if (snext_rep) sn = T(ldcg_if(own, snext_rep + i));
  else if (snext_col) sn = ldcg_if(own, snext_col + i);
  const int act = ldcg_i(active);
  pdl_wait();
  pdl_trigger();
  if (!act) return;
  __shared__ T c[1024 + 4];
  __shared__ double sh[2];
  __shared__ T shc[3];             // 1 / sqrt(eta), alpha / eta, 1 / |s| (formed once, in FP64)
  __shared__ int stop_sh;
  __shared__ T sd[SPLIT][ROWS], sgd[SPLIT][ROWS];
  const T dj = ldcg_if(own, V + (size_t)j * ldv + i), gdj = ldcg_if(own, GV + (size_t)j * ldv + i);
  double sg = 0.0, a1 = 0.0, a2 = 0.0, ss = 0.0;
  if (warp < 4) {
    sg = ldcg_if(true, dots1 + j);
    a1 = ldcg_if(true, dots1 + j + 1);
    a2 = ldcg_if(true, dots1 + j + 2);
    ss = ldcg_if(true, dots1 + j + 3);
  }
  sum_partials(dpart2, nblk2, j + 1, c, nullptr);
  __syncthreads();
  // The scalars, one warp (on an SM partition of its own) per FP64 division or root: 0: 1 / sqrt(eta),
  // 1: alpha / eta, 2: 1 / |s|, 3: the stop decision.
  if (warp < 4) {
    double eta = 0.0;
    if (warp != 2) {
      double ccp = 0.0;
      for (int q = lane; q < j; q += 32) ccp = fma(double(c[q]), double(c[q]), ccp);
      eta = double(c[j]) - warp_sum(ccp);
    }
    const double alpha = a1 - a2;
    if (lane == 0) {
      if (warp == 0) { sh[0] = eta; shc[0] = T(1.0 / sqrt(eta)); }
      else if (warp == 1) { sh[1] = alpha; shc[1] = T(alpha / eta); }
      else if (warp == 2) { if (Q) shc[2] = T(1.0 / sqrt(ss)); }
      else {
        int stop = !(eta > bd_tol * sg) || !isfinite(eta) || !isfinite(alpha);
        if (use_rtol && ss <= rtol2_r0sq) stop = 1;
        stop_sh = stop;
      }
    }
  }
  T d = T(0), gd = T(0);
  orth_pass<SPLIT>(V, GV, ldv, i, valid, sp, j, c, xv, xg, d, gd);
  sd[sp][rl] = d;
  sgd[sp][rl] = gd;
  __syncthreads();
  if (stop_sh) {
    // breakdown / converged: this direction is not used; clear the parked column
    if (own) { V[(size_t)j * ldv + i] = T(0); GV[(size_t)j * ldv + i] = T(0); }
    if (blockIdx.x == 0 && threadIdx.x == 0) *active = 0;
    return;
  }
  if (own) {
    d = dj;
    gd = gdj;
#pragma unroll
    for (int u = 0; u < SPLIT; ++u) { d += sd[u][rl]; gd += sgd[u][rl]; }
    const T inv = shc[0];
    const T coef = shc[1];
    V[(size_t)j * ldv + i] = d * inv;
    GV[(size_t)j * ldv + i] = gd * inv;
    v[i] = fma(coef, d, vi);
    const T rn = fma(-coef, gd, ri);
    r[i] = rn;
    if (Q) Q[(size_t)j * ldv + i] = si * shc[2];
    if (snext_rep || snext_col || Snext) {
      const T val = snext_rep || snext_col ? sn : rn;
      s[i] = val;
      if (Snext) Snext[i] = val;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) { eta_out[j] = sh[0]; alpha_out[j] = sh[1]; *count = j + 1; }
}

// Projection coefficients of the action on the orthonormal basis Q of the previous actions:
// qd[l] = Q[:, l] . s  (one block per l)
template <class T>
__global__ void k_cg_qdots(const T* __restrict__ Q, int ldq, int j, const T* __restrict__ s, int m,
                           double* __restrict__ qd, const int* __restrict__ active) {
  pdl_wait();
  pdl_trigger();
  if (!*active) return;
  const int l = blockIdx.x;
  const T* a = Q + (size_t)l * ldq;
  const double acc = block_sum(dot_part(a, s, m));
  if (threadIdx.x == 0) qd[l] = acc;
}
// s -= Q[:, :j] qd   (Gram-Schmidt against the previous actions; a no-op in exact arithmetic for CG
// residuals, which are mutually orthogonal).  On the last pass S[:, j] = s.
template <class T>
__global__ void k_cg_qorth(const T* __restrict__ Q, int ldq, int j, const double* __restrict__ qd, T* __restrict__ s,
                           int m, T* __restrict__ S, int lds, const int* __restrict__ active) {
  pdl_wait();
  pdl_trigger();
  if (!*active) return;
  __shared__ T c[1024];
  for (int q = threadIdx.x; q < j; q += blockDim.x) c[q] = T(qd[q]);
  __syncthreads();
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  T v = s[i];
  for (int q = 0; q < j; ++q) v = fma(-Q[(size_t)q * ldq + i], c[q], v);
  s[i] = v;
  if (S) S[(size_t)j * lds + i] = v;
}

// s = r (CG policy: the current residual) or s = the replayed action; S[:, j] = s.
template <class T>
__global__ void k_cg_select(int j, const T* __restrict__ r, const double* __restrict__ rep, int m,
                            T* __restrict__ s, T* __restrict__ S, int lds, const int* __restrict__ active) {
  pdl_wait();
  pdl_trigger();
  if (!*active) return;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  T val = rep ? T(rep[(size_t)j * m + i]) : r[i];
  s[i] = val;
  S[(size_t)j * lds + i] = val;
}

// r0 = y - m_pred[obs] ; r = r0 ; v = 0 ; sum of squares of r0 accumulated by the caller
template <class T>
__global__ void k_cg_init(const double* __restrict__ y, const double* __restrict__ mpred,
                          const int* __restrict__ obs, int m, T* __restrict__ r, T* __restrict__ r0,
                          T* __restrict__ v, double* __restrict__ r0sq) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  double val = 0.0;
  if (i < m) {
    val = y[i] - mpred[obs[i]];
    r[i] = T(val);
    r0[i] = T(val);
    v[i] = T(0);
  }
  double sq = block_sum(val * val);
  if (threadIdx.x == 0) atomicAdd(r0sq, sq);
}

// ------------------------------------------------------------------------------------------
// Split-K transposed product: part[z][a + b*na] = sum_{t in chunk z} A[t, a] B[t, b]
// (A: K x na, B: K x nb column-major), 64 x 64 output tiles, 4 x 4 per thread, K staged 32 at a time
// (rows of A and B are contiguous along K: each warp reads 32 consecutive K values of 8 columns).
// Accumulation in the working precision, partials in double; k_reduce_splits sums them.
constexpr int TN_T = 64, TN_K = 32;
template <class T>
__global__ void __launch_bounds__(256)
k_gemm_tn_part(const T* __restrict__ A, int lda, int na, const T* __restrict__ B, int ldb, int nb,
               int K, int chunk, double* __restrict__ part) {
  __shared__ T As[TN_K][TN_T + 1];
  __shared__ T Bs[TN_K][TN_T + 1];
  const int a0 = blockIdx.x * TN_T, b0 = blockIdx.y * TN_T;
  const int k_begin = blockIdx.z * chunk, k_end = min(K, k_begin + chunk);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  T acc[4][4];
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[p][q] = T(0);
  const int kk_ld = threadIdx.x & 31, cc_ld = threadIdx.x >> 5;   // 32 K values x 8 columns per pass
  for (int k0 = k_begin; k0 < k_end; k0 += TN_K) {
    const int t = k0 + kk_ld;
#pragma unroll
    for (int pass = 0; pass < TN_T / 8; ++pass) {
      const int cc = cc_ld + 8 * pass;
      As[kk_ld][cc] = (t < k_end && a0 + cc < na) ? A[(size_t)(a0 + cc) * lda + t] : T(0);
      Bs[kk_ld][cc] = (t < k_end && b0 + cc < nb) ? B[(size_t)(b0 + cc) * ldb + t] : T(0);
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < TN_K; ++kk) {
      T aa[4], bb[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) aa[p] = As[kk][ty + 16 * p];
#pragma unroll
      for (int q = 0; q < 4; ++q) bb[q] = Bs[kk][tx + 16 * q];
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = fma(aa[p], bb[q], acc[p][q]);
    }
    __syncthreads();
  }
  const size_t stride = (size_t)na * nb;
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int a = a0 + ty + 16 * p, b = b0 + tx + 16 * q;
      if (a < na && b < nb) part[blockIdx.z * stride + (size_t)b * na + a] = double(acc[p][q]);
    }
}

// The FP64 factor products.  GB300's FP64 pipe takes 19 cycles of its SM per warp-wide FMA, so a tile
// needs no register blocking to keep it busy (one or two shared loads per FMA are free); what the
// products of the FP64 mode need is blocks on every SM and no padding: outputs are taken 32 rows by
// single columns, and the columns per warp (1, 2, 4) shrink until the grid fills the GPU.
// Measured in the gradient pass of the 1,024-point model (M = 1,024): N = 256, K = 288 takes 133 us
// against 318 us with 64 x 64 tiles (64 blocks), N = 33 about 22 us against 150 us (16 blocks).
constexpr int G64_WARPS = 8;
// C[M x N] = alpha A[M x K] B[K x N] + beta C: lane = row, CPW columns per warp, the next 4 values of k
// loaded while the current ones are used.  Every output sums over k in ascending order.
template <int CPW>
__global__ void __launch_bounds__(G64_WARPS * 32)
k_gemm_nn_f64(int M, int N, int K, double alpha, const double* __restrict__ A, int lda, const double* __restrict__ B,
              int ldb, double beta, double* __restrict__ C, int ldc) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x * 32 + lane;
  const int n0 = (blockIdx.y * G64_WARPS + warp) * CPW;
  if (n0 >= N) return;
  const double* a = A + min(row, M - 1);
  const double* b[CPW];
#pragma unroll
  for (int c = 0; c < CPW; ++c) b[c] = B + (size_t)min(n0 + c, N - 1) * ldb;
  double acc[CPW];
#pragma unroll
  for (int c = 0; c < CPW; ++c) acc[c] = 0.0;
  constexpr int U = 4;
  double av[U], bv[CPW][U];
  const int K4 = K / U * U;
  if (K4 > 0) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      av[u] = a[(size_t)u * lda];
#pragma unroll
      for (int c = 0; c < CPW; ++c) bv[c][u] = b[c][u];
    }
  }
  for (int k = 0; k < K4; k += U) {
    double an[U], bn[CPW][U];
    const int kn = k + U < K4 ? k + U : 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      an[u] = a[(size_t)(kn + u) * lda];
#pragma unroll
      for (int c = 0; c < CPW; ++c) bn[c][u] = b[c][kn + u];
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int c = 0; c < CPW; ++c) acc[c] = fma(av[u], bv[c][u], acc[c]);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      av[u] = an[u];
#pragma unroll
      for (int c = 0; c < CPW; ++c) bv[c][u] = bn[c][u];
    }
  }
  for (int k = K4; k < K; ++k) {
    const double x = a[(size_t)k * lda];
#pragma unroll
    for (int c = 0; c < CPW; ++c) acc[c] = fma(x, b[c][k], acc[c]);
  }
  if (row >= M) return;
#pragma unroll
  for (int c = 0; c < CPW; ++c) {
    if (n0 + c >= N) break;
    double* p = C + (size_t)(n0 + c) * ldc + row;
    *p = beta == 0.0 ? alpha * acc[c] : fma(alpha, acc[c], beta * *p);
  }
}

// part[z][a + b*na] = sum_{t in chunk z} A[t, a] B[t, b] (A: K x na, B: K x nb): 32 columns of A by
// G64_WARPS * CPW columns of B per block, 32 values of t staged through shared memory at a time
// (their loads in flight while the previous ones are used).  With one chunk the output is written
// directly (C = alpha sum + beta C).
template <int CPW>
__global__ void __launch_bounds__(G64_WARPS * 32)
k_gemm_tn_f64(const double* __restrict__ A, int lda, int na, const double* __restrict__ B, int ldb, int nb, int K,
              int chunk, double* __restrict__ part, double alpha, double beta, double* __restrict__ C, int ldc) {
  constexpr int NBC = G64_WARPS * CPW;
  __shared__ double As[32][33], Bs[32][NBC + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int a0 = blockIdx.x * 32, b0 = blockIdx.y * NBC;
  const int kb = blockIdx.z * chunk, ke = min(K, kb + chunk);
  double ra[4], rb[CPW], acc[CPW];
#pragma unroll
  for (int c = 0; c < CPW; ++c) acc[c] = 0.0;
  // lane = t within the stage, warp w loads columns w, w + 8, ... of both operands
  auto load = [&](int k0) {
    const int t = k0 + lane;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int col = a0 + warp + G64_WARPS * u;
      ra[u] = (t < ke && col < na) ? A[(size_t)col * lda + t] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < CPW; ++u) {
      const int col = b0 + warp + G64_WARPS * u;
      rb[u] = (t < ke && col < nb) ? B[(size_t)col * ldb + t] : 0.0;
    }
  };
  load(kb);
  for (int k0 = kb; k0 < ke; k0 += 32) {
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) As[lane][warp + G64_WARPS * u] = ra[u];
#pragma unroll
    for (int u = 0; u < CPW; ++u) Bs[lane][warp + G64_WARPS * u] = rb[u];
    __syncthreads();
    if (k0 + 32 < ke) load(k0 + 32);
    if (b0 + warp * CPW < nb) {
#pragma unroll 8
      for (int t = 0; t < 32; ++t) {
        const double x = As[t][lane];
#pragma unroll
        for (int c = 0; c < CPW; ++c) acc[c] = fma(x, Bs[t][warp * CPW + c], acc[c]);
      }
    }
  }
  const int a = a0 + lane;
  if (a >= na) return;
#pragma unroll
  for (int c = 0; c < CPW; ++c) {
    const int b = b0 + warp * CPW + c;
    if (b >= nb) break;
    if (part) {
      part[blockIdx.z * (size_t)na * nb + (size_t)b * na + a] = acc[c];
    } else {
      double* o = C + (size_t)b * ldc + a;
      *o = alpha * acc[c] + (beta != 0.0 ? beta * *o : 0.0);
    }
  }
}

// C[a + b*ldc] = alpha * sum_z part[z][a + b*na]  (+ beta * C)
template <class OutT>
__global__ void k_reduce_splits(const double* __restrict__ part, int nsplit, int na, int nb, double alpha,
                                double beta, OutT* __restrict__ C, int ldc) {
  size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  size_t tot = (size_t)na * nb;
  if (e >= tot) return;
  double acc = 0.0;
  for (int z = 0; z < nsplit; ++z) acc += part[z * tot + e];
  int a = int(e % na), b = int(e / na);
  OutT* c = C + (size_t)b * ldc + a;
  *c = OutT(alpha * acc + (beta != 0.0 ? beta * double(*c) : 0.0));
}

// ------------------------------------------------------------------------------------------
// Small FP64 product with transposes: C = alpha op(A) op(B) + beta C  (sizes up to a few hundred).  A 16 x 16 tile
// of C per cluster of blocks, which split K and add their partial tiles in rank order through distributed shared
// memory: few tiles would leave the products to the FP64 pipes of as many SMs (32 x 32 x 256: 29 us with one
// block per tile, 9 us with 8).
constexpr int GSM_SPLIT_MAX = 8;
__global__ void __launch_bounds__(256)
k_gemm_small_f64(int ta, int tb, int M, int N, int K, double alpha, const double* __restrict__ A, int lda,
                 const double* __restrict__ B, int ldb, double beta, double* __restrict__ C, int ldc) {
  __shared__ double As[16][17], Bs[16][17];
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  const int Z = gridDim.z, rank = blockIdx.z;            // (a cluster spans the z extent)
  int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int nst = (K + 15) / 16, k1 = nst * (rank + 1) / Z * 16;
  double acc = 0.0;
  for (int k0 = nst * rank / Z * 16; k0 < k1; k0 += 16) {
    int ka = k0 + tx, kb = k0 + ty;
    int ar = blockIdx.x * 16 + ty;
    As[ty][tx] = (ar < M && ka < K) ? (ta ? A[(size_t)ar * lda + ka] : A[(size_t)ka * lda + ar]) : 0.0;
    int bc = blockIdx.y * 16 + tx;
    Bs[ty][tx] = (bc < N && kb < K) ? (tb ? B[(size_t)kb * ldb + bc] : B[(size_t)bc * ldb + kb]) : 0.0;
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) acc = fma(As[ty][kk], Bs[kk][tx], acc);
    __syncthreads();
  }
  int e = threadIdx.x;                                   // element (ty, tx) of the tile this thread writes
  if (Z > 1) {
    As[ty][tx] = acc;
    cl.sync();
    const int share = 256 / Z;
    e = rank * share + threadIdx.x;
    if ((int)threadIdx.x < share) {
      acc = 0.0;
      for (int q = 0; q < Z; ++q) acc += cl.map_shared_rank(&As[0][0], q)[(e >> 4) * 17 + (e & 15)];
    } else {
      e = -1;
    }
    cl.sync();                                           // no block leaves while its tile is being read
  }
  const int row = blockIdx.x * 16 + (e >> 4), col = blockIdx.y * 16 + (e & 15);
  if (e >= 0 && row < M && col < N) {
    double* c = C + (size_t)col * ldc + row;
    *c = alpha * acc + (beta != 0.0 ? beta * *c : 0.0);
  }
}

// ------------------------------------------------------------------------------------------
// Row kernels
// Out[i, c] = In[idx[i], c] for c < cols (column-major, gather rows)
template <class T>
__global__ void k_gather_rows(const T* __restrict__ In, int ldi, const int* __restrict__ idx, int m, int cols,
                              T* __restrict__ Out, int ldo) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int c = blockIdx.y;
  if (i < m && c < cols) Out[(size_t)c * ldo + i] = In[(size_t)c * ldi + idx[i]];
}

// Out[idx[i], c] += alpha * In[i, c]
template <class T>
__global__ void k_scatter_add_rows(const T* __restrict__ In, int ldi, const int* __restrict__ idx, int m, int cols,
                                   T alpha, T* __restrict__ Out, int ldo) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int c = blockIdx.y;
  if (i < m && c < cols) Out[(size_t)c * ldo + idx[i]] += alpha * In[(size_t)c * ldi + i];
}

// sum_c A[i, c]^2 for row i of a column-major block.  FP32 factors: four compensated (Kahan) FP32
// sums combined in FP64 -- relative error about 2^-24 whatever the column count, at FP32-pipe speed
// (an FP64 accumulation chain per row is bound by GB300's narrow FP64 pipe); FP64 factors: FP64.
template <class T>
__device__ __forceinline__ double row_sumsq(const T* __restrict__ A, int lda, int i, int cols) {
  double acc = 0.0;
  if constexpr (sizeof(T) == 4) {
    float s[4] = {0.f, 0.f, 0.f, 0.f}, e[4] = {0.f, 0.f, 0.f, 0.f};
    int c = 0;
    for (; c + 3 < cols; c += 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float v = A[(size_t)(c + u) * lda + i];
        const float y = fmaf(v, v, -e[u]);
        const float t = s[u] + y;
        e[u] = (t - s[u]) - y;
        s[u] = t;
      }
    }
    for (; c < cols; ++c) {
      const float v = A[(size_t)c * lda + i];
      const float y = fmaf(v, v, -e[0]);
      const float t = s[0] + y;
      e[0] = (t - s[0]) - y;
      s[0] = t;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) acc += double(s[u]) - double(e[u]);
  } else {
    for (int c = 0; c < cols; ++c) { const double v = double(A[(size_t)c * lda + i]); acc += v * v; }
  }
  return acc;
}

// rs[i] = sum_c A[i, c]^2 (+ beta * rs[i])
template <class T>
__global__ void k_rowsumsq(const T* __restrict__ A, int lda, int n, int cols, double beta, double* __restrict__ rs) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double acc = row_sumsq(A, lda, i, cols);
  rs[i] = acc + (beta != 0.0 ? beta * rs[i] : 0.0);
}

// m_pred = a m_prev + (mu_k - a mu_{k-1})
__global__ void k_predict_mean(const double* __restrict__ mprev, const double* __restrict__ mu_k,
                               const double* __restrict__ mu_km1, double a, int n, double* __restrict__ mpred) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double b = mu_k ? (mu_k[i] - a * mu_km1[i]) : 0.0;
  mpred[i] = a * mprev[i] + b;
}

// Two-block state (Matern-3/2 temporal factor: positions in rows [0, half), velocities in rows
// [half, 2 half)): Out = (C (x) I) In for a 2 x 2 matrix C = [[c00, c01], [c10, c11]], i.e.
//   Out[i] = c00 In[i] + c01 In[half + i],  Out[half + i] = c10 In[i] + c11 In[half + i]
// per column.  In == Out is allowed: each thread reads its pair before writing it.
template <class T>
__global__ void k_mix2(const T* In, int ldi, T* Out, int ldo, int half, int cols, T c00, T c01, T c10, T c11) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int c = blockIdx.y;
  if (i >= half || c >= cols) return;
  const T x = In[(size_t)c * ldi + i], v = In[(size_t)c * ldi + half + i];
  Out[(size_t)c * ldo + i] = fma(c00, x, c01 * v);
  Out[(size_t)c * ldo + half + i] = fma(c10, x, c11 * v);
}

// Mean prediction of the two-block state with the prior mean (mu_k, 0) of the positions:
//   m^- = A (m - (mu_{k-1}, 0)) + (mu_k, 0)   (mu may be null: zero mean)
__global__ void k_predict_mean2(const double* __restrict__ mprev, const double* __restrict__ mu_k,
                                const double* __restrict__ mu_km1, double a00, double a01, double a10, double a11,
                                int n, int half, double* __restrict__ mpred) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double x = mprev[i] - (mu_km1 ? mu_km1[i] : 0.0), v = mprev[half + i];
  mpred[i] = fma(a00, x, a01 * v) + (mu_k ? mu_k[i] : 0.0);
  mpred[half + i] = fma(a10, x, a11 * v);
}

// out[i] = a[i] + b[i] (FP64 plus working precision), i < n
template <class T>
__global__ void k_add_vec(const double* __restrict__ a, const T* __restrict__ b, int n, double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = a[i] + double(b[i]);
}

// Filter outputs of step k:  m_k = m_pred + (P^- w);  var_k = sf2 - a^2 rs_plus - rowsumsq(P^- W)
template <class T>
__global__ void k_filter_out(const double* __restrict__ mpred, const T* __restrict__ PVv, int ld, int ic,
                             double sf2, double a2, const double* __restrict__ rs_plus, int n,
                             double* __restrict__ mout, double* __restrict__ vout, double* __restrict__ rs_pw) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double acc = ic > 0 ? row_sumsq(PVv, ld, i, ic) : 0.0;
  double pw = ic >= 0 ? double(PVv[(size_t)ic * ld + i]) : 0.0;
  mout[i] = mpred[i] + pw;
  vout[i] = sf2 - a2 * rs_plus[i] - acc;
  if (rs_pw) rs_pw[i] = acc;
}

// Copy of a scaled column block: Out[:, c] = alpha * In[:, c]
template <class T>
__global__ void k_scale_copy(const T* __restrict__ In, int ldi, int n, int cols, T alpha, T* __restrict__ Out, int ldo) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int c = blockIdx.y;
  if (i < n && c < cols) Out[(size_t)c * ldo + i] = alpha * In[(size_t)c * ldi + i];
}

// Smoother outputs at k: ms = m_k + Y[:, cw];  vs = v_k - rowsumsq(Y[:, 0:cw])
template <class T>
__global__ void k_smooth_out(const double* __restrict__ mk, const double* __restrict__ vk, const T* __restrict__ Y,
                             int ld, int cw, int n, double* __restrict__ ms, double* __restrict__ vs) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double acc = row_sumsq(Y, ld, i, cw);
  ms[i] = mk[i] + double(Y[(size_t)cw * ld + i]);
  vs[i] = vk[i] - acc;
}

// Dense vector from the sparse filter message:  out = x + scatter(v_obs - u_obs) ...
// ws_new[i] = X[i, cw] ; then ws_new[obs] += v - Vz (done by k_ws_obs)
template <class T>
__global__ void k_ws_obs(const int* __restrict__ obs, int m, const T* __restrict__ vk, const T* __restrict__ Vz,
                         T* __restrict__ ws) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m) ws[obs[i]] += vk[i] - Vz[i];
}

// Y[:, c] = alpha * [Ws, ws][:, c]   (X = A^T [Ws ws] in the smoother)
template <class T>
__global__ void k_build_x(const T* __restrict__ Ws, int ldw, int cw, const T* __restrict__ ws, T alpha, int n,
                          T* __restrict__ X, int ldx) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int c = blockIdx.y;
  if (i >= n || c > cw) return;
  X[(size_t)c * ldx + i] = alpha * (c < cw ? Ws[(size_t)c * ldw + i] : ws[i]);
}

// FP64 per-step NLL from the iteration: sum_j [ 1/2 log(2 pi eta_j) + 1/2 alpha_j^2 / eta_j ] - logdet(L)
// where L L^T = S^T S (Cholesky in FP64, in place on the i x i Gram).  One block.
__global__ void k_nll_step(const double* __restrict__ eta, const double* __restrict__ alpha,
                           const int* __restrict__ count, double* __restrict__ SS, int ic, double* __restrict__ nll_k,
                           int* __restrict__ err) {
  __shared__ double s_piv;
  __shared__ int s_bad;
  const int j = *count;
  if (threadIdx.x == 0) s_bad = 0;
  __syncthreads();
  // Cholesky of the leading j x j block (column-major, ld = ic), right-looking
  for (int p = 0; p < j; ++p) {
    if (threadIdx.x == 0) {
      double d = SS[(size_t)p * ic + p];
      if (!(d > 0.0) || !isfinite(d)) { s_bad = 1; d = 1.0; }
      s_piv = sqrt(d);
      SS[(size_t)p * ic + p] = s_piv;
    }
    __syncthreads();
    for (int q = p + 1 + threadIdx.x; q < j; q += blockDim.x) SS[(size_t)p * ic + q] /= s_piv;
    __syncthreads();
    for (int e = threadIdx.x; e < (j - p - 1) * (j - p - 1); e += blockDim.x) {
      int q = p + 1 + e % (j - p - 1), c = p + 1 + e / (j - p - 1);
      if (q >= c) SS[(size_t)c * ic + q] -= SS[(size_t)p * ic + q] * SS[(size_t)p * ic + c];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    double acc = 0.0;
    const double l2pi = 1.8378770664093453;
    for (int q = 0; q < j; ++q) {
      acc += 0.5 * (l2pi + log(eta[q])) + 0.5 * alpha[q] * alpha[q] / eta[q];
      acc -= log(SS[(size_t)q * ic + q]);
    }
    *nll_k = acc;
    if (s_bad || !isfinite(acc)) atomicExch(err, kErrNllChol);
  }
}

// Per-step small FP64 algebra of the NLL tangent pass (one block).  With Gh = S^T G S = R^T R
// (R upper), beta = Gh^-1 yh and, per parameter p, W_p = R^-T dGh_p R^-1:
//   grad[p] += 1/2 tr(W_p) + beta^T dyh_p - 1/2 beta^T dGh_p beta
//   Q_p      = upper triangle of W_p with halved diagonal   (dR R^-1 of the Cholesky factor)
//   u_p      = R^-T (dyh_p - dGh_p beta)                    (R dbeta_p)
// Work arrays (global, ld = ic): L (ic x ic), Rinv (ic x ic), W (ic x ic), tmp (3 ic).
__global__ void k_grad_small(int ic, int np, const double* __restrict__ Gh, const double* __restrict__ dGh,
                             const double* __restrict__ yh, const double* __restrict__ dyh, double* __restrict__ L,
                             double* __restrict__ Rinv, double* __restrict__ W, double* __restrict__ tmp,
                             double* __restrict__ Q, double* __restrict__ u, double* __restrict__ grad,
                             int* __restrict__ err) {
  __shared__ double piv;
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  for (int e = threadIdx.x; e < ic * ic; e += blockDim.x) L[e] = Gh[e];
  __syncthreads();
  // Cholesky Gh = L L^T (lower, in place, column-major)
  for (int p = 0; p < ic; ++p) {
    if (threadIdx.x == 0) {
      double d = L[(size_t)p * ic + p];
      if (!(d > 0.0) || !isfinite(d)) { bad = 1; d = 1.0; }
      piv = sqrt(d);
      L[(size_t)p * ic + p] = piv;
    }
    __syncthreads();
    for (int q = p + 1 + threadIdx.x; q < ic; q += blockDim.x) L[(size_t)p * ic + q] /= piv;
    __syncthreads();
    const int w = ic - p - 1;
    for (int e = threadIdx.x; e < w * w; e += blockDim.x) {
      int q = p + 1 + e % w, c = p + 1 + e / w;
      if (q >= c) L[(size_t)c * ic + q] -= L[(size_t)p * ic + q] * L[(size_t)p * ic + c];
    }
    __syncthreads();
  }
  // Rinv = (L^T)^-1 = upper triangular; column j solves L^T x = e_j by back substitution
  for (int j = threadIdx.x; j < ic; j += blockDim.x) {
    for (int i = ic - 1; i >= 0; --i) {
      double acc = (i == j) ? 1.0 : 0.0;
      for (int l = i + 1; l <= j; ++l) acc -= L[(size_t)i * ic + l] * Rinv[(size_t)j * ic + l];   // R_il = L_li
      Rinv[(size_t)j * ic + i] = (i > j) ? 0.0 : acc / L[(size_t)i * ic + i];
    }
  }
  __syncthreads();
  // beta = Rinv Rinv^T yh
  double* t1 = tmp;
  double* beta = tmp + ic;
  for (int i = threadIdx.x; i < ic; i += blockDim.x) {
    double acc = 0.0;
    for (int l = 0; l < ic; ++l) acc += Rinv[(size_t)i * ic + l] * yh[l];   // (Rinv^T yh)_i = sum_l Rinv[l, i] yh_l
    t1[i] = acc;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < ic; i += blockDim.x) {
    double acc = 0.0;
    for (int l = 0; l < ic; ++l) acc += Rinv[(size_t)l * ic + i] * t1[l];
    beta[i] = acc;
  }
  __syncthreads();
  double* t2 = tmp + 2 * ic;
  for (int p = 0; p < np; ++p) {
    const double* D = dGh + (size_t)p * ic * ic;
    // W = Rinv^T D Rinv : first Y = D Rinv (into Q_p as scratch), then W = Rinv^T Y
    double* Y = Q + (size_t)p * ic * ic;
    for (int e = threadIdx.x; e < ic * ic; e += blockDim.x) {
      int i = e % ic, j = e / ic;
      double acc = 0.0;
      for (int l = 0; l <= j; ++l) acc += D[(size_t)l * ic + i] * Rinv[(size_t)j * ic + l];
      Y[e] = acc;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < ic * ic; e += blockDim.x) {
      int i = e % ic, j = e / ic;
      double acc = 0.0;
      for (int l = 0; l <= i; ++l) acc += Rinv[(size_t)i * ic + l] * Y[(size_t)j * ic + l];
      W[e] = acc;
    }
    __syncthreads();
    // scalars
    double tr = 0.0, bdy = 0.0, bdb = 0.0;
    for (int i = threadIdx.x; i < ic; i += blockDim.x) {
      tr += W[(size_t)i * ic + i];
      bdy += beta[i] * dyh[(size_t)p * ic + i];
      double db = 0.0;
      for (int l = 0; l < ic; ++l) db += D[(size_t)l * ic + i] * beta[l];
      bdb += beta[i] * db;
      t2[i] = dyh[(size_t)p * ic + i] - db;
    }
    tr = block_sum(tr);
    bdy = block_sum(bdy);
    bdb = block_sum(bdb);
    if (threadIdx.x == 0) grad[p] += 0.5 * tr + bdy - 0.5 * bdb;
    // u_p = Rinv^T t2 ; Q_p = Phi(W)
    for (int i = threadIdx.x; i < ic; i += blockDim.x) {
      double acc = 0.0;
      for (int l = 0; l <= i; ++l) acc += Rinv[(size_t)i * ic + l] * t2[l];
      u[(size_t)p * ic + i] = acc;
    }
    for (int e = threadIdx.x; e < ic * ic; e += blockDim.x) {
      int i = e % ic, j = e / ic;
      Q[(size_t)p * ic * ic + e] = (i < j) ? W[e] : ((i == j) ? 0.5 * W[e] : 0.0);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0 && bad) atomicExch(err, kErrGradChol);
}

// out[i, p] = in[idx[i] + p * ld]   (gather rows of a double block into precision T)
template <class T>
__global__ void k_gather_rows_f64(const double* __restrict__ In, int ld, const int* __restrict__ idx, int m, int cols,
                                  T* __restrict__ Out, int ldo) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int c = blockIdx.y;
  if (i < m && c < cols) Out[(size_t)c * ldo + i] = T(In[(size_t)c * ld + idx[i]]);
}

// dm_new[:, p] = dmpred[:, p] + E[:, p][col] + t[:, p]    (tangent of the filter mean)
template <class T>
__global__ void k_tangent_mean(const double* __restrict__ dmpred, const T* __restrict__ E, size_t estride, int ecol,
                               int lde, const T* __restrict__ t, int ldt, int n, int np, double* __restrict__ dm) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int p = blockIdx.y;
  if (i >= n || p >= np) return;
  double v = dmpred[(size_t)p * n + i];
  if (E) v += double(E[p * estride + (size_t)ecol * lde + i]);
  if (t) v += double(t[(size_t)p * ldt + i]);
  dm[(size_t)p * n + i] = v;
}

// dmpred[:, p] = adot_p * m_prev + a * dm_prev[:, p] - adot_p * mu_{k-1}
__global__ void k_tangent_predict(const double* __restrict__ mprev, const double* __restrict__ dmprev,
                                  const double* __restrict__ mu_km1, double a, double adot_lt, int n, int np,
                                  double* __restrict__ dmpred) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int p = blockIdx.y;
  if (i >= n || p >= np) return;
  const double ad = (p == 1) ? adot_lt : 0.0;
  double v = a * dmprev[(size_t)p * n + i] + ad * mprev[i];
  if (mu_km1) v -= ad * mu_km1[i];
  dmpred[(size_t)p * n + i] = v;
}

template <class T>
__global__ void k_axpy_block(T alpha, const T* __restrict__ X, int ldx, int rows, int cols, T* __restrict__ Y, int ldy) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int c = blockIdx.y;
  if (i < rows && c < cols) Y[(size_t)c * ldy + i] += alpha * X[(size_t)c * ldx + i];
}
template <class T>
__global__ void k_scale_cols(T* A, int ld, int rows, int cols, T s) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int c = blockIdx.y;
  if (i < rows && c < cols) A[(size_t)c * ld + i] *= s;
}

// In-place Cholesky (lower) of the leading j x j block of a symmetric matrix (column-major, ld),
// symmetrised from both triangles first.  Block-wide; returns false (on all threads) if not PD.
__device__ bool block_cholesky(double* A, int ld, int j) {
  __shared__ double piv;
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  for (int e = threadIdx.x; e < j * j; e += blockDim.x) {
    int r = e % j, c = e / j;
    if (r > c) {
      double v = 0.5 * (A[(size_t)c * ld + r] + A[(size_t)r * ld + c]);
      A[(size_t)c * ld + r] = v;
    }
  }
  __syncthreads();
  for (int p = 0; p < j; ++p) {
    if (threadIdx.x == 0) {
      double d = A[(size_t)p * ld + p];
      if (!(d > 0.0) || !isfinite(d)) { bad = 1; d = 1.0; }
      piv = sqrt(d);
      A[(size_t)p * ld + p] = piv;
    }
    __syncthreads();
    for (int q = p + 1 + threadIdx.x; q < j; q += blockDim.x) A[(size_t)p * ld + q] /= piv;
    __syncthreads();
    const int w = j - p - 1;
    for (int e = threadIdx.x; e < w * w; e += blockDim.x) {
      int q = p + 1 + e % w, c = p + 1 + e / w;
      if (q >= c) A[(size_t)c * ld + q] -= A[(size_t)p * ld + q] * A[(size_t)p * ld + c];
    }
    __syncthreads();
  }
  bool ok = bad == 0;
  __syncthreads();
  return ok;
}

// Per-step NLL from its definition (eq. proj-observation with the actions S of the step):
//   nll = 1/2 [ j log 2 pi + logdet(S^T G S) ] + 1/2 yh^T (S^T G S)^-1 yh - 1/2 logdet(S^T S),
// yh = S^T r0, with both log-determinants from FP64 Cholesky factors of the leading j x j blocks.
// z (length >= j) is scratch for the forward substitution.
__global__ void k_nll_def(const int* __restrict__ count, double* __restrict__ Gh, double* __restrict__ SS, int ld,
                          const double* __restrict__ yh, double* __restrict__ z, double* __restrict__ nll_k,
                          int* __restrict__ err) {
  const int j = *count;
  const bool ok1 = block_cholesky(Gh, ld, j);
  const bool ok2 = block_cholesky(SS, ld, j);
  if (threadIdx.x == 0) {
    double ld1 = 0.0, ld2 = 0.0, quad = 0.0;
    for (int q = 0; q < j; ++q) {
      ld1 += log(Gh[(size_t)q * ld + q]);
      ld2 += log(SS[(size_t)q * ld + q]);
    }
    for (int q = 0; q < j; ++q) {          // L z = yh, L = lower Cholesky factor of S^T G S
      double acc = yh[q];
      for (int l = 0; l < q; ++l) acc -= Gh[(size_t)l * ld + q] * z[l];
      z[q] = acc / Gh[(size_t)q * ld + q];
      quad += z[q] * z[q];
    }
    const double val = 0.5 * j * 1.8378770664093453 + ld1 + 0.5 * quad - ld2;
    *nll_k = val;
    if (!ok1 || !ok2 || !isfinite(val)) atomicExch(err, kErrNllChol);
  }
}

// The same NLL term with both j x j factorisations in shared memory, side by side (2 j^2 + 3 j
// doubles of dynamic shared memory).  GB300 issues a warp-wide FP64 instruction over 16 cycles, so
// the scalar work of a pivot (square root, reciprocal) is done once per matrix, by one lane of warp 0
// (S^T G S) and one lane of warp 1 (S^T S), and broadcast through shared memory; the column scale and
// the forward substitution multiply by the stored reciprocal, and the logarithms of the pivots are
// taken in parallel.
constexpr int NLL_THREADS = 256;
__global__ void __launch_bounds__(NLL_THREADS)
k_nll_def_smem(const int* __restrict__ count, const double* __restrict__ Gh, const double* __restrict__ SS, int ld,
               const double* __restrict__ yh, double* __restrict__ nll_k, int* __restrict__ err) {
  extern __shared__ double nsm[];
  const int j = min(*count, ld);
  double* S1 = nsm;                      // S^T G S, j x j (ld j), lower triangle used
  double* S2 = nsm + (size_t)j * j;      // S^T S
  double* inv1 = S2 + (size_t)j * j;     // reciprocal pivots of S1
  double* inv2 = inv1 + j;
  double* b = inv2 + j;                  // right-hand side of the forward substitution
  __shared__ int bad;
  __shared__ double red[NLL_THREADS / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (threadIdx.x == 0) bad = 0;
  for (int e = threadIdx.x; e < j * j; e += blockDim.x) {
    const int r = e % j, c = e / j;
    if (r >= c) {
      S1[c * j + r] = (r == c) ? Gh[(size_t)c * ld + r] : 0.5 * (Gh[(size_t)c * ld + r] + Gh[(size_t)r * ld + c]);
      S2[c * j + r] = (r == c) ? SS[(size_t)c * ld + r] : 0.5 * (SS[(size_t)c * ld + r] + SS[(size_t)r * ld + c]);
    }
  }
  for (int q = threadIdx.x; q < j; q += blockDim.x) b[q] = yh[q];
  __syncthreads();
  for (int p = 0; p < j; ++p) {
    if (lane == 0 && warp < 2) {
      double* S = warp == 0 ? S1 : S2;
      double d = S[p * j + p];
      if (!(d > 0.0) || !isfinite(d)) { bad = 1; d = 1.0; }
      const double piv = sqrt(d);
      S[p * j + p] = piv;
      (warp == 0 ? inv1 : inv2)[p] = 1.0 / piv;
    }
    __syncthreads();
    const double i1 = inv1[p], i2 = inv2[p];
    for (int q = p + 1 + threadIdx.x; q < j; q += blockDim.x) {
      S1[p * j + q] *= i1;
      S2[p * j + q] *= i2;
    }
    __syncthreads();
    // trailing updates: warps take the columns c of both matrices round robin, lanes the rows q >= c
    const int w = j - p - 1;
    for (int cc = warp; cc < 2 * w; cc += nw) {
      double* S = cc < w ? S1 : S2;
      const int c = p + 1 + (cc < w ? cc : cc - w);
      const double* lp = S + p * j;
      const double lc = lp[c];
      double* col = S + c * j;
      for (int q = c + lane; q < j; q += 32) col[q] = fma(-lp[q], lc, col[q]);
    }
    __syncthreads();
  }
  // L z = yh for the factor of S^T G S (column oriented)
  double quad = 0.0;
  for (int q = 0; q < j; ++q) {
    const double zq = b[q] * inv1[q];
    quad = fma(zq, zq, quad);
    for (int l = q + 1 + threadIdx.x; l < j; l += blockDim.x) b[l] = fma(-S1[q * j + l], zq, b[l]);
    __syncthreads();
  }
  // sum_q log L1_qq - sum_q log L2_qq, logarithms in parallel
  double lg = 0.0;
  for (int q = threadIdx.x; q < j; q += blockDim.x) lg += log(S1[q * j + q]) - log(S2[q * j + q]);
  lg = warp_sum(lg);
  if (lane == 0) red[warp] = lg;
  __syncthreads();
  if (threadIdx.x == 0) {
    double ldiff = 0.0;
    for (int w2 = 0; w2 < nw; ++w2) ldiff += red[w2];
    const double val = 0.5 * j * 1.8378770664093453 + ldiff + 0.5 * quad;
    *nll_k = val;
    if (bad || !isfinite(val)) atomicExch(err, kErrNllChol);
  }
}

__global__ void k_set_diag(double* __restrict__ G, int ld, const double* __restrict__ lam, double scale, int r) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < r) G[(size_t)i * ld + i] = scale * lam[i];
}

// Fill the upper-right / lower-left border of the truncation Gram from an r x i block B (double)
__global__ void k_put_block_sym(double* __restrict__ G, int ld, int row0, int col0, const double* __restrict__ B,
                                int ldb, int nr, int nc, double scale) {
  int a = blockIdx.x * blockDim.x + threadIdx.x;
  int b = blockIdx.y;
  if (a >= nr || b >= nc) return;
  double v = scale * B[(size_t)b * ldb + a];
  G[(size_t)(col0 + b) * ld + row0 + a] = v;
  G[(size_t)(row0 + a) * ld + col0 + b] = v;
}

__global__ void k_check_finite(const double* __restrict__ x, size_t n, int* __restrict__ err) {
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n && !isfinite(x[i])) atomicExch(err, kErrNonFinite);
}


__global__ void k_scale_f64(double* __restrict__ A, int ld, int rows, int cols, double s) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int c = blockIdx.y;
  if (i < rows && c < cols) A[(size_t)c * ld + i] *= s;
}

template <class T>
__global__ void k_convert_from_f64(const double* __restrict__ In, int ldi, int rows, int cols, T* __restrict__ Out,
                                   int ldo) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int c = blockIdx.y;
  if (i < rows && c < cols) Out[(size_t)c * ldo + i] = T(In[(size_t)c * ldi + i]);
}

// ------------------------------------------------------------------------------------------
// Host-side launchers
static inline unsigned cdiv(size_t a, size_t b) { return unsigned((a + b - 1) / b); }

template <class T>
void prep_coords(const double* X, int n, int dim, double scale, C4<T>* out, cudaStream_t st) {
  if (n <= 0) return;
  k_prep_coords<T><<<cdiv(n, 256), 256, 0, st>>>(X, n, dim, scale, out); note_launch();
}
template <class T>
void prep_coords2(const double* Xr, int nr, const double* Xc, int nc, int dim, double scale, C4<T>* out,
                  cudaStream_t st) {
  k_prep_coords2<T><<<cdiv((size_t)nr + nc, 256), 256, 0, st>>>(Xr, nr, Xc, nc, dim, scale, out); note_launch();
}
template <class T>
void gather_coords(const C4<T>* X, const int* idx, int m, C4<T>* out, cudaStream_t st) {
  if (m <= 0) return;
  k_gather_coords<T><<<cdiv(m, 256), 256, 0, st>>>(X, idx, m, out); note_launch();
}

// Tiling of the FP64 matvec by the observation count (Matern-5/2; a 128 x 128 tile costs 185 us on its
// SM whatever the others do, a 32 x 32 one about 18 us):
//   m <= 416        every entry, one row per lane: 5.7 us a launch at m = 128 against 185 us for the one
//                   128-wide tile.  Its cost grows as m^2 / 152 SMs and meets the one wave of 32 x 32
//                   tiles (m <= 544: 152 blocks) between m = 400 and 500
//   m <= 2048       32 x 32 tiles of the upper triangle: m = 2048 has 2,080 of them, the block count of
//                   m = 8,192 with 128 x 128 tiles, and the same 64 slots
//   above           128 x 128 tiles, whose slots grow as m / 128
constexpr int MV64_ROWS_MAX = 416, MV64_SMALL_TILE_MAX = 2048;
static int mv64_cpw(int m) { return std::max(1, (m + 255) / 256); }   // columns per warp: at most 64 slots
int gram_matvec_slots(int m, int elem_size) {
  if (m <= 0) return 1;
  if (elem_size == 8 && m <= MV64_ROWS_MAX) return (m + MVS_W * mv64_cpw(m) - 1) / (MVS_W * mv64_cpw(m));
  if (elem_size == 8 && m <= MV64_SMALL_TILE_MAX) return (m + 31) / 32;
  return (m + MVS_T - 1) / MVS_T;
}
size_t gram_matvec_part_elems(int mmax) {
  return (size_t)std::max(mmax, 1) * std::max(64, (mmax + MVS_T - 1) / MVS_T);
}

template <int KER, class T>
static void launch_matvec(const C4<T>* Xo, const T* s, int m, T sf2, T* part, const T* Mo, int ldm, int rp, T* tpart,
                          const int* active, cudaStream_t st) {
  const int nb = gram_matvec_slots(m, sizeof(T));
  const int ngv = rp > 0 ? (int)cdiv(m, GV_CHUNK) * (int)cdiv(rp, MVS_W) : 0;
  const int grid = ngv + nb * (nb + 1) / 2;
  if constexpr (sizeof(T) == 4) {
    launch_pdl(k_gram_matvec_f2<KER>, dim3(grid), dim3(MVS_W * 32), 0, st, Xo, s, m, nb, sf2, part, Mo, ldm, rp, ngv,
               tpart, active);
  } else if (m <= MV64_ROWS_MAX) {
    launch_pdl(k_gram_matvec_rows<KER, T>, dim3(ngv + nb * (int)cdiv(m, 32)), dim3(MVS_W * 32), 0, st, Xo, s, m, nb,
               mv64_cpw(m), sf2, part, Mo, ldm, rp, ngv, tpart, active);
  } else if (m <= MV64_SMALL_TILE_MAX) {
    launch_pdl(k_gram_matvec<KER, T, 1>, dim3(grid), dim3(MVS_W * 32), 0, st, Xo, s, m, nb, sf2, part, Mo, ldm, rp,
               ngv, tpart, active);
  } else {
    launch_pdl(k_gram_matvec<KER, T, MVS_R>, dim3(grid), dim3(MVS_W * 32), 0, st, Xo, s, m, nb, sf2, part, Mo, ldm, rp,
               ngv, tpart, active);
  }
}
template <class T>
void gram_matvec(int ker, const C4<T>* Xo, const T* s, int m, T sf2, T* part, const T* Mo, int ldm, int rp, T* tpart,
                 const int* active, cudaStream_t st) {
  if (m <= 0) return;
  switch (ker) {
    case 0: launch_matvec<0, T>(Xo, s, m, sf2, part, Mo, ldm, rp, tpart, active, st); break;
    case 1: launch_matvec<1, T>(Xo, s, m, sf2, part, Mo, ldm, rp, tpart, active, st); break;
    default: launch_matvec<2, T>(Xo, s, m, sf2, part, Mo, ldm, rp, tpart, active, st); break;
  }
}

static bool cg_small(int m, size_t es) { return es == 8 && m <= CG64_SMALL_MAX; }
static int cg_blocks1(int m, size_t es) { return (int)cdiv(m, cg_small(m, es) ? CB_ROWS_SMALL : CB_ROWS); }
static int cg_blocks2(int m, size_t es) { return (int)cdiv(m, cg_small(m, es) ? UP_ROWS_SMALL : UP_ROWS); }
template <class T>
void cg_combine(const T* part, int nsplit, const T* s, T sn2, const T* Mo, int ldm, int r, const T* t, T a2, int m,
                T* g, const T* V, int ldv, int j, const T* r0, const T* v, T* dpart1, const int* active,
                cudaStream_t st) {
  const int tz = std::max(1, (m + GV_CHUNK - 1) / GV_CHUNK);
  auto fn = k_cg_combine<T, CB_ROWS>;
  const size_t smem = std::max(cg_small(m, sizeof(T)) ? (r + 3) / 4 * 4 : r, 1) * sizeof(T);
  if constexpr (sizeof(T) == 8)
    if (cg_small(m, 8)) fn = k_cg_combine<T, CB_ROWS_SMALL>;
  launch_pdl(fn, dim3(cg_blocks1(m, sizeof(T))), dim3(CB_WARPS * 32), smem, st, part, nsplit, s, sn2, Mo, ldm,
              r, t, tz, a2, m, g, V, ldv, j, r0, v, dpart1, active);
}
size_t cg_dpart2_offset(int m, int budget, size_t elem_size) { return (size_t)(budget + 4) * cg_blocks1(m, elem_size); }
size_t cg_dpart_elems(int mmax, int budget) {
  // (the small FP64 blocks of a step with fewer observations can outnumber the blocks of the largest step)
  const int mb = std::max(mmax, 1), ms = std::min(mb, CG64_SMALL_MAX);
  return (size_t)(budget + 4) * std::max(cg_blocks1(mb, 4), cg_blocks1(ms, 8)) +
         (size_t)(budget + 1) * std::max(cg_blocks2(mb, 4), cg_blocks2(ms, 8));
}
template <class T>
void cg_upd1(int j, const T* dpart1, double* dots1, T* V, T* GV, int ldv, const T* s, const T* g, int m,
             T* dpart2, const int* active, cudaStream_t st) {
  auto fn = k_cg_upd1<T, UP_ROWS>;
  if constexpr (sizeof(T) == 8)
    if (cg_small(m, 8)) fn = k_cg_upd1<T, UP_ROWS_SMALL>;
  launch_pdl(fn, dim3(cg_blocks2(m, sizeof(T))), dim3(UP_THREADS), 0, st, j, dpart1, cg_blocks1(m, sizeof(T)), dots1, V, GV,
             ldv, s, g, m, dpart2, active);
}
template <class T>
void cg_upd2(int j, const double* dots1, const T* dpart2, T* V, T* GV, int ldv, T* r, T* v, T* s, T* Q,
             int m, double bd_tol, double rtol2_r0sq, int use_rtol, int* active, double* eta, double* alpha,
             int* count, T* Snext, const double* snext_rep, const T* snext_col, cudaStream_t st) {
  auto fn = k_cg_upd2<T, UP_ROWS>;
  if constexpr (sizeof(T) == 8)
    if (cg_small(m, 8)) fn = k_cg_upd2<T, UP_ROWS_SMALL>;
  launch_pdl(fn, dim3(cg_blocks2(m, sizeof(T))), dim3(UP_THREADS), 0, st, j, dots1, dpart2, cg_blocks2(m, sizeof(T)), V, GV,
             ldv, r, v, s, Q, m, bd_tol, rtol2_r0sq, use_rtol, active, eta, alpha, count, Snext, snext_rep, snext_col);
}
template <class T>
void cg_reorth(const T* Q, int ldq, int j, T* s, int m, double* qd, T* S, int lds, const int* active, cudaStream_t st) {
  // two classical Gram-Schmidt passes against the previous (orthonormal) action basis
  for (int pass = 0; pass < 2; ++pass) {
    if (j > 0) {
      launch_pdl(k_cg_qdots<T>, dim3(j), dim3(256), 0, st, Q, ldq, j, s, m, qd, active);
    }
    launch_pdl(k_cg_qorth<T>, dim3(cdiv(m, 256)), dim3(256), 0, st, Q, ldq, j, qd, s, m, pass == 1 ? S : nullptr, lds, active);
  }
}
template <class T>
void cg_select(int j, const T* r, const double* rep, int m, T* s, T* S, int lds, const int* active, cudaStream_t st) {
  launch_pdl(k_cg_select<T>, dim3(cdiv(m, 256)), dim3(256), 0, st, j, r, rep, m, s, S, lds, active);
}
template <class T>
void cg_init(const double* y, const double* mpred, const int* obs, int m, T* r, T* r0, T* v, double* r0sq,
             cudaStream_t st) {
  k_cg_init<T><<<cdiv(m, 256), 256, 0, st>>>(y, mpred, obs, m, r, r0, v, r0sq); note_launch();
}

__global__ void k_axpby_f32_f64(const float* __restrict__ X, int ldx, int rows, int cols, double alpha, double beta,
                                double* __restrict__ C, int ldc) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int c = blockIdx.y;
  if (i >= rows || c >= cols) return;
  double* p = C + (size_t)c * ldc + i;
  *p = alpha * double(X[(size_t)c * ldx + i]) + (beta != 0.0 ? beta * *p : 0.0);
}

// FP32 <-> BF16 (round to nearest even) copies of column-major blocks, for the BF16 factor store
__global__ void k_to_bf16(const float* __restrict__ In, int ldi, int rows, int cols, uint16_t* __restrict__ Out,
                          int ldo) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int c = blockIdx.y;
  if (i >= rows || c >= cols) return;
  const __nv_bfloat16 b = __float2bfloat16_rn(In[(size_t)c * ldi + i]);
  Out[(size_t)c * ldo + i] = *reinterpret_cast<const uint16_t*>(&b);
}
__global__ void k_from_bf16(const uint16_t* __restrict__ In, int ldi, int rows, int cols, float* __restrict__ Out,
                            int ldo) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int c = blockIdx.y;
  if (i >= rows || c >= cols) return;
  Out[(size_t)c * ldo + i] = __uint_as_float((uint32_t)In[(size_t)c * ldi + i] << 16);
}
void to_bf16(const float* In, int ldi, int rows, int cols, uint16_t* Out, int ldo, cudaStream_t st) {
  if (rows <= 0 || cols <= 0) return;
  k_to_bf16<<<dim3(cdiv(rows, 256), cols), 256, 0, st>>>(In, ldi, rows, cols, Out, ldo); note_launch();
}
void from_bf16(const uint16_t* In, int ldi, int rows, int cols, float* Out, int ldo, cudaStream_t st) {
  if (rows <= 0 || cols <= 0) return;
  k_from_bf16<<<dim3(cdiv(rows, 256), cols), 256, 0, st>>>(In, ldi, rows, cols, Out, ldo); note_launch();
}

void convert_to_f64(const float* In, int ldi, int rows, int cols, double* Out, int ldo, cudaStream_t st) {
  if (rows <= 0 || cols <= 0) return;
  k_axpby_f32_f64<<<dim3(cdiv(rows, 256), cols), 256, 0, st>>>(In, ldi, rows, cols, 1.0, 0.0, Out, ldo); note_launch();
}

template <class T>
void gemm_tn(const T* A, int lda, int na, const T* B, int ldb, int nb, int K, double alpha, double beta, double* C,
             int ldc, double* part, size_t part_elems, cudaStream_t st) {
  if (na <= 0 || nb <= 0) return;
  if (sizeof(T) == 4 && t_gemm_mode == 2 && (double)na * nb * K > 2e7 && K >= 64) {
    // FP32 operands on the tensor cores (split TF32), FP32 partial tiles summed by k_gemm_reduce
    if (gemm_tc_tn((const float*)A, lda, na, (const float*)B, ldb, nb, K, alpha, beta, C, ldc, part,
                   part_elems * sizeof(double), t_gemm_err, st) == 0)
      return;
    cudaGetLastError();
  }
  const size_t tile_elems = (size_t)na * nb;
  if constexpr (sizeof(T) == 8) {
    // about two blocks per SM: single columns per warp while that alone does not fill the GPU, then
    // splits of K (at least 64 values each)
    const int gx = cdiv(na, 32);
    int cpw = 4;
    while (cpw > 1 && gx * (int)cdiv(nb, G64_WARPS * cpw) < 2 * 152) cpw /= 2;
    const int gy = cdiv(nb, G64_WARPS * cpw);
    int nsplit = std::max(1, std::min({2 * 152 / (gx * gy), K / 64, (int)std::min<size_t>(part_elems / tile_elems, 1 << 20)}));
    const int chunk = std::max(32, (int)cdiv(cdiv(std::max(K, 1), nsplit), 32) * 32);
    nsplit = std::max(1, (int)cdiv(std::max(K, 1), chunk));
    double* out = nsplit > 1 ? part : nullptr;
    const dim3 grid(gx, gy, nsplit);
    const double *Ad = (const double*)A, *Bd = (const double*)B;
    const int Kp = std::max(K, 0);
    switch (cpw) {
      case 1: k_gemm_tn_f64<1><<<grid, G64_WARPS * 32, 0, st>>>(Ad, lda, na, Bd, ldb, nb, Kp, chunk, out, alpha, beta, C, ldc); break;
      case 2: k_gemm_tn_f64<2><<<grid, G64_WARPS * 32, 0, st>>>(Ad, lda, na, Bd, ldb, nb, Kp, chunk, out, alpha, beta, C, ldc); break;
      default: k_gemm_tn_f64<4><<<grid, G64_WARPS * 32, 0, st>>>(Ad, lda, na, Bd, ldb, nb, Kp, chunk, out, alpha, beta, C, ldc); break;
    }
    note_launch();
    if (out) {
      k_reduce_splits<double><<<cdiv(tile_elems, 256), 256, 0, st>>>(part, nsplit, na, nb, alpha, beta, C, ldc);
      note_launch();
    }
    return;
  }
  int gx = cdiv(na, TN_T), gy = cdiv(nb, TN_T);
  int want = std::max(1, (int)(4 * 152 / std::max(1, gx * gy)));
  int chunk_min = 256;
  int nsplit = std::max(1, std::min(want, (K + chunk_min - 1) / chunk_min));
  nsplit = std::max(1, std::min<int>(nsplit, (int)(part_elems / tile_elems)));
  int chunk = (K + nsplit - 1) / nsplit;
  chunk = ((chunk + TN_K - 1) / TN_K) * TN_K;
  nsplit = std::max(1, (K + chunk - 1) / chunk);
  if (K <= 0) { nsplit = 1; chunk = TN_K; }
  k_gemm_tn_part<T><<<dim3(gx, gy, nsplit), 256, 0, st>>>(A, lda, na, B, ldb, nb, std::max(K, 0), chunk, part); note_launch();
  k_reduce_splits<double><<<cdiv(tile_elems, 256), 256, 0, st>>>(part, nsplit, na, nb, alpha, beta, C, ldc); note_launch();
}

// FP32 copy of a small double coefficient block for the tensor-core path (device scratch per host
// thread and current device)
static thread_local float* t_bscratch = nullptr;
static thread_local size_t t_bscratch_elems = 0;
static thread_local int t_bscratch_dev = -1;
static float* bscratch(size_t elems) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return nullptr; }
  if (dev != t_bscratch_dev) {        // a buffer of another device is not reachable from this one
    if (t_bscratch) cudaFree(t_bscratch);
    t_bscratch = nullptr;
    t_bscratch_elems = 0;
    t_bscratch_dev = dev;
  }
  if (elems > t_bscratch_elems) {
    if (t_bscratch) cudaFree(t_bscratch);
    t_bscratch = nullptr;
    t_bscratch_elems = 0;
    if (cudaMalloc(&t_bscratch, elems * sizeof(float)) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    t_bscratch_elems = elems;
  }
  return t_bscratch;
}

template <class T, class TB>
void gemm_nn(int M, int N, int K, T alpha, const T* A, int lda, const TB* B, int ldb, T beta, T* C, int ldc,
             cudaStream_t st) {
  if (M <= 0 || N <= 0) return;
  if (K <= 0) {
    if (beta == T(1)) return;
  }
  if (sizeof(T) == 4 && t_gemm_mode == 2 && K >= 16 && M >= 4096 && (double)M * N * K > 2e7) {
    // tall factor times a small coefficient block on the tensor cores (split TF32)
    const float* Bf = reinterpret_cast<const float*>(B);
    int ldbf = ldb;
    if (sizeof(TB) == 8) {
      float* sb = bscratch((size_t)K * N);
      if (sb) {
        convert_from_f64<float>(reinterpret_cast<const double*>(B), ldb, K, N, sb, K, st);
        Bf = sb;
        ldbf = K;
      } else {
        Bf = nullptr;
      }
    }
    if (Bf && gemm_tc_nn(M, N, K, (float)alpha, (const float*)A, lda, Bf, ldbf, (float)beta, (float*)C, ldc,
                         t_gemm_err, st) == 0)
      return;
    cudaGetLastError();
  }
  if constexpr (sizeof(T) == 8 && sizeof(TB) == 8) {
    const int gx = cdiv(M, 32);
    int cpw = 4;
    while (cpw > 1 && gx * (int)cdiv(N, G64_WARPS * cpw) < 2 * 152) cpw /= 2;
    const dim3 grid(gx, cdiv(N, G64_WARPS * cpw));
    switch (cpw) {
      case 1: k_gemm_nn_f64<1><<<grid, G64_WARPS * 32, 0, st>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc); break;
      case 2: k_gemm_nn_f64<2><<<grid, G64_WARPS * 32, 0, st>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc); break;
      default: k_gemm_nn_f64<4><<<grid, G64_WARPS * 32, 0, st>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc); break;
    }
    note_launch();
  } else {
    gemm_nn_f32<TB>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, st);
  }
}

void gemm_small_f64(int ta, int tb, int M, int N, int K, double alpha, const double* A, int lda, const double* B,
                    int ldb, double beta, double* C, int ldc, cudaStream_t st) {
  if (M <= 0 || N <= 0) return;
  // K is split while the tiles leave SMs free (152) and every block keeps two stages of 16
  const int tiles = (int)(cdiv(M, 16) * cdiv(N, 16));
  int Z = 1;
  while (Z < GSM_SPLIT_MAX && tiles * Z * 2 <= 152 && K >= 64 * Z) Z *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cdiv(M, 16), cdiv(N, 16), Z);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = Z;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  note_launch();
  cudaLaunchKernelEx(&cfg, k_gemm_small_f64, ta, tb, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc);
}

template <class T>
void gather_rows(const T* In, int ldi, const int* idx, int m, int cols, T* Out, int ldo, cudaStream_t st) {
  if (m <= 0 || cols <= 0) return;
  k_gather_rows<T><<<dim3(cdiv(m, 256), cols), 256, 0, st>>>(In, ldi, idx, m, cols, Out, ldo); note_launch();
}
template <class T>
void scatter_add_rows(const T* In, int ldi, const int* idx, int m, int cols, T alpha, T* Out, int ldo, cudaStream_t st) {
  if (m <= 0 || cols <= 0) return;
  k_scatter_add_rows<T><<<dim3(cdiv(m, 256), cols), 256, 0, st>>>(In, ldi, idx, m, cols, alpha, Out, ldo); note_launch();
}
template <class T>
void rowsumsq(const T* A, int lda, int n, int cols, double beta, double* rs, cudaStream_t st) {
  k_rowsumsq<T><<<cdiv(n, 256), 256, 0, st>>>(A, lda, n, cols, beta, rs); note_launch();
}
void predict_mean(const double* mprev, const double* mu_k, const double* mu_km1, double a, int n, double* mpred,
                  cudaStream_t st) {
  k_predict_mean<<<cdiv(n, 256), 256, 0, st>>>(mprev, mu_k, mu_km1, a, n, mpred); note_launch();
}
template <class T>
void mix2(const T* In, int ldi, T* Out, int ldo, int half, int cols, const double C[4], cudaStream_t st) {
  if (half <= 0 || cols <= 0) return;
  k_mix2<T><<<dim3(cdiv(half, 256), cols), 256, 0, st>>>(In, ldi, Out, ldo, half, cols, T(C[0]), T(C[1]), T(C[2]),
                                                         T(C[3])); note_launch();
}
void predict_mean2(const double* mprev, const double* mu_k, const double* mu_km1, const double A[4], int n, int half,
                   double* mpred, cudaStream_t st) {
  k_predict_mean2<<<cdiv(n, 256), 256, 0, st>>>(mprev, mu_k, mu_km1, A[0], A[1], A[2], A[3], n, half, mpred);
  note_launch();
}
template <class T>
void add_vec(const double* a, const T* b, int n, double* out, cudaStream_t st) {
  if (n <= 0) return;
  k_add_vec<T><<<cdiv(n, 256), 256, 0, st>>>(a, b, n, out); note_launch();
}
template <class T>
void filter_out(const double* mpred, const T* PVv, int ld, int ic, double sf2, double a2, const double* rs_plus, int n,
                double* mout, double* vout, double* rs_pw, cudaStream_t st) {
  k_filter_out<T><<<cdiv(n, 256), 256, 0, st>>>(mpred, PVv, ld, ic, sf2, a2, rs_plus, n, mout, vout, rs_pw); note_launch();
}
template <class T>
void scale_copy(const T* In, int ldi, int n, int cols, T alpha, T* Out, int ldo, cudaStream_t st) {
  if (n <= 0 || cols <= 0) return;
  k_scale_copy<T><<<dim3(cdiv(n, 256), cols), 256, 0, st>>>(In, ldi, n, cols, alpha, Out, ldo); note_launch();
}
template <class T>
void smooth_out(const double* mk, const double* vk, const T* Y, int ld, int cw, int n, double* ms, double* vs,
                cudaStream_t st) {
  k_smooth_out<T><<<cdiv(n, 256), 256, 0, st>>>(mk, vk, Y, ld, cw, n, ms, vs); note_launch();
}
template <class T>
void ws_obs(const int* obs, int m, const T* vk, const T* Vz, T* ws, cudaStream_t st) {
  if (m <= 0) return;
  k_ws_obs<T><<<cdiv(m, 256), 256, 0, st>>>(obs, m, vk, Vz, ws); note_launch();
}
template <class T>
void build_x(const T* Ws, int ldw, int cw, const T* ws, T alpha, int n, T* X, int ldx, cudaStream_t st) {
  k_build_x<T><<<dim3(cdiv(n, 256), cw + 1), 256, 0, st>>>(Ws, ldw, cw, ws, alpha, n, X, ldx); note_launch();
}
void nll_step(const double* eta, const double* alpha, const int* count, double* SS, int ic, double* nll_k, int* err,
              cudaStream_t st) {
  k_nll_step<<<1, 256, 0, st>>>(eta, alpha, count, SS, ic, nll_k, err); note_launch();
}
void grad_small(int ic, int np, const double* Gh, const double* dGh, const double* yh, const double* dyh, double* L,
                double* Rinv, double* W, double* tmp, double* Q, double* u, double* grad, int* err, cudaStream_t st) {
  k_grad_small<<<1, 256, 0, st>>>(ic, np, Gh, dGh, yh, dyh, L, Rinv, W, tmp, Q, u, grad, err); note_launch();
}
template <class T>
void gather_rows_f64(const double* In, int ld, const int* idx, int m, int cols, T* Out, int ldo, cudaStream_t st) {
  if (m <= 0 || cols <= 0) return;
  k_gather_rows_f64<T><<<dim3(cdiv(m, 256), cols), 256, 0, st>>>(In, ld, idx, m, cols, Out, ldo); note_launch();
}
template <class T>
void tangent_mean(const double* dmpred, const T* E, size_t estride, int ecol, int lde, const T* t, int ldt, int n,
                  int np, double* dm, cudaStream_t st) {
  k_tangent_mean<T><<<dim3(cdiv(n, 256), np), 256, 0, st>>>(dmpred, E, estride, ecol, lde, t, ldt, n, np, dm);
  note_launch();
}
void tangent_predict(const double* mprev, const double* dmprev, const double* mu_km1, double a, double adot_lt, int n,
                     int np, double* dmpred, cudaStream_t st) {
  k_tangent_predict<<<dim3(cdiv(n, 256), np), 256, 0, st>>>(mprev, dmprev, mu_km1, a, adot_lt, n, np, dmpred);
  note_launch();
}
template <class T>
void axpy_block(T alpha, const T* X, int ldx, int rows, int cols, T* Y, int ldy, cudaStream_t st) {
  if (rows <= 0 || cols <= 0) return;
  k_axpy_block<T><<<dim3(cdiv(rows, 256), cols), 256, 0, st>>>(alpha, X, ldx, rows, cols, Y, ldy); note_launch();
}
template <class T>
void scale_cols(T* A, int ld, int rows, int cols, T s, cudaStream_t st) {
  if (rows <= 0 || cols <= 0) return;
  k_scale_cols<T><<<dim3(cdiv(rows, 256), cols), 256, 0, st>>>(A, ld, rows, cols, s); note_launch();
}
template void axpy_block<float>(float, const float*, int, int, int, float*, int, cudaStream_t);
template void axpy_block<double>(double, const double*, int, int, int, double*, int, cudaStream_t);
template void scale_cols<float>(float*, int, int, int, float, cudaStream_t);
template void scale_cols<double>(double*, int, int, int, double, cudaStream_t);
template void gather_rows_f64<float>(const double*, int, const int*, int, int, float*, int, cudaStream_t);
template void gather_rows_f64<double>(const double*, int, const int*, int, int, double*, int, cudaStream_t);
template void tangent_mean<float>(const double*, const float*, size_t, int, int, const float*, int, int, int, double*,
                                  cudaStream_t);
template void tangent_mean<double>(const double*, const double*, size_t, int, int, const double*, int, int, int,
                                   double*, cudaStream_t);

void nll_def(const int* count, double* Gh, double* SS, int ld, const double* yh, double* z, double* nll_k, int* err,
             cudaStream_t st) {
  const size_t smem = (2 * (size_t)ld * ld + 3 * (size_t)ld) * sizeof(double);
  if (smem <= 200 * 1024) {
    if (smem > 40 * 1024) cudaFuncSetAttribute(k_nll_def_smem, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_nll_def_smem<<<1, NLL_THREADS, smem, st>>>(count, Gh, SS, ld, yh, nll_k, err); note_launch();
    return;
  }
  k_nll_def<<<1, 256, 0, st>>>(count, Gh, SS, ld, yh, z, nll_k, err); note_launch();
}

// ------------------------------------------------------------------------------------------
// Batch update (Alg. 2) helpers: the actions S are fixed up front, Ghat = S^T G S = L L^T,
// W = H^T S L^-T, w = H^T S Ghat^-1 S^T r0.

// Coordinate actions (reading R18 of the oracle): S = 0 except S[floor((q + 1/2) m / i), q] = 1.
template <class T>
__global__ void k_coord_actions(int m, int i, T* __restrict__ S) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= i) return;
  const int row = (int)(((double)q + 0.5) * (double)m / (double)i);
  S[(size_t)q * m + min(row, m - 1)] = T(1);
}

// Cholesky Ghat = L L^T (FP64, i x i, lower triangle of Ghat read symmetrised; L in shared memory,
// written to Lout with ld i) and z = L^-1 yh.  One block.  A non-positive or non-finite pivot
// raises the numeric error flag (the step's projected Gram must be positive definite).
constexpr int BCH_THREADS = 256;
__global__ void __launch_bounds__(BCH_THREADS)
k_batch_chol(const double* __restrict__ Gh, int i, const double* __restrict__ yh, double* __restrict__ Lout,
             double* __restrict__ z, double* __restrict__ eta, int* __restrict__ err) {
  extern __shared__ double bsm[];
  double* L = bsm;                  // i x i, column-major
  double* zz = bsm + (size_t)i * i;
  __shared__ double piv;
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  for (int e = threadIdx.x; e < i * i; e += blockDim.x) {
    const int r = e % i, c = e / i;
    L[e] = r >= c ? 0.5 * (Gh[(size_t)c * i + r] + Gh[(size_t)r * i + c]) : 0.0;
  }
  for (int q = threadIdx.x; q < i; q += blockDim.x) zz[q] = yh[q];
  __syncthreads();
  for (int p = 0; p < i; ++p) {
    if (threadIdx.x == 0) {
      double d = L[(size_t)p * i + p];
      if (eta) eta[p] = d;            // the pivot: eta_j of the iterative form (S^T G S = U^-T diag(eta) U^-1)
      if (!(d > 0.0) || !isfinite(d)) { bad = 1; d = 1.0; }
      piv = sqrt(d);
      L[(size_t)p * i + p] = piv;
      zz[p] /= piv;
    }
    __syncthreads();
    const double ip = 1.0 / piv, zp = zz[p];
    for (int q = p + 1 + threadIdx.x; q < i; q += blockDim.x) {
      const double lq = L[(size_t)p * i + q] * ip;
      L[(size_t)p * i + q] = lq;
      zz[q] -= lq * zp;
    }
    __syncthreads();
    // trailing update of the lower triangle: column c, rows q >= c
    const int w = i - p - 1;
    for (int e = threadIdx.x; e < w * w; e += blockDim.x) {
      const int c = p + 1 + e / w, q = p + 1 + e % w;
      if (q >= c) L[(size_t)c * i + q] -= L[(size_t)p * i + q] * L[(size_t)p * i + c];
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < i * i; e += blockDim.x) Lout[e] = L[e];
  for (int q = threadIdx.x; q < i; q += blockDim.x) z[q] = zz[q];
  if (threadIdx.x == 0 && bad) atomicExch(err, kErrBatchChol);
}

// V = S L^-T (row by row: x L^T = s, forward substitution in FP64) into columns 0..i-1 of Vv, and
// v = V z into column i.  One thread per row of S.
template <class T>
__global__ void k_batch_v(const T* __restrict__ S, int m, int i, const double* __restrict__ L,
                          const double* __restrict__ z, T* __restrict__ Vv) {
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= m) return;
  double x[160];
  double v = 0.0;
  for (int j = 0; j < i; ++j) {
    double acc = (double)S[(size_t)j * m + row];
    for (int l = 0; l < j; ++l) acc = fma(-x[l], L[(size_t)l * i + j], acc);
    x[j] = acc / L[(size_t)j * i + j];
    Vv[(size_t)j * m + row] = T(x[j]);
    v = fma(x[j], z[j], v);
  }
  Vv[(size_t)i * m + row] = T(v);
}

template <class T>
void coord_actions(int m, int i, T* S, cudaStream_t st) {
  if (m <= 0 || i <= 0) return;
  cudaMemsetAsync(S, 0, (size_t)m * i * sizeof(T), st);
  k_coord_actions<T><<<cdiv(i, 128), 128, 0, st>>>(m, i, S); note_launch();
}
int batch_chol(const double* Gh, int i, const double* yh, double* L, double* z, double* eta, int* err,
               cudaStream_t st) {
  if (i <= 0) return 0;
  if (i > kBatchMaxActions) return 1;
  const size_t smem = ((size_t)i * i + i) * sizeof(double);
  if (smem > 48 * 1024) cudaFuncSetAttribute(k_batch_chol, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k_batch_chol<<<1, BCH_THREADS, smem, st>>>(Gh, i, yh, L, z, eta, err); note_launch();
  return 0;
}
template <class T>
void batch_v(const T* S, int m, int i, const double* L, const double* z, T* Vv, cudaStream_t st) {
  if (m <= 0 || i <= 0) return;
  k_batch_v<T><<<cdiv(m, 128), 128, 0, st>>>(S, m, i, L, z, Vv); note_launch();
}
template void coord_actions<float>(int, int, float*, cudaStream_t);
template void coord_actions<double>(int, int, double*, cudaStream_t);
template void batch_v<float>(const float*, int, int, const double*, const double*, float*, cudaStream_t);
template void batch_v<double>(const double*, int, int, const double*, const double*, double*, cudaStream_t);

// ------------------------------------------------------------------------------------------
// Per-step diagnostics: the squared norm of a vector (the final residual of a step's update), the
// trace of the truncation Gram before the eigensolver and the discarded mass after it.
template <class T>
__global__ void k_sqnorm(const T* __restrict__ x, int m, double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const double v = i < m ? (double)x[i] : 0.0;
  const double s = block_sum(v * v);
  if (threadIdx.x == 0) atomicAdd(out, s);
}
__global__ void k_trace(const double* __restrict__ G, int N, int ld, double* __restrict__ out) {
  double acc = 0.0;
  for (int i = threadIdx.x; i < N; i += blockDim.x) acc += G[(size_t)i * ld + i];
  acc = block_sum(acc);
  if (threadIdx.x == 0) *out = acc;
}
__global__ void k_sub_sum(const double* __restrict__ w, int keep, double* __restrict__ out) {
  double acc = 0.0;
  for (int i = threadIdx.x; i < keep; i += blockDim.x) acc += w[i];
  acc = block_sum(acc);
  if (threadIdx.x == 0) *out -= acc;
}
// r_final = r0 - (G S) L^-T z for the batch update: squared norm accumulated into out
template <class T>
__global__ void k_batch_resid(const T* __restrict__ GS, int m, int i, const double* __restrict__ L,
                              const double* __restrict__ z, const T* __restrict__ r0, double* __restrict__ out) {
  extern __shared__ double yc[];   // L^-T z, by back substitution (thread 0), shared by the block
  if (threadIdx.x == 0) {
    for (int j = i - 1; j >= 0; --j) {
      double acc = z[j];
      for (int l = j + 1; l < i; ++l) acc = fma(-L[(size_t)j * i + l], yc[l], acc);
      yc[j] = acc / L[(size_t)j * i + j];
    }
  }
  __syncthreads();
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  double r = 0.0;
  if (row < m) {
    r = (double)r0[row];
    for (int j = 0; j < i; ++j) r = fma(-(double)GS[(size_t)j * m + row], yc[j], r);
  }
  const double s = block_sum(r * r);
  if (threadIdx.x == 0) atomicAdd(out, s);
}
template <class T> void sqnorm_acc(const T* x, int m, double* out, cudaStream_t st) {
  if (m <= 0) return;
  k_sqnorm<T><<<cdiv(m, 256), 256, 0, st>>>(x, m, out); note_launch();
}
void trace_into(const double* G, int N, int ld, double* out, cudaStream_t st) {
  k_trace<<<1, 256, 0, st>>>(G, N, ld, out); note_launch();
}
void sub_sum(const double* w, int keep, double* out, cudaStream_t st) {
  k_sub_sum<<<1, 256, 0, st>>>(w, keep, out); note_launch();
}
template <class T>
void batch_resid(const T* GS, int m, int i, const double* L, const double* z, const T* r0, double* out, cudaStream_t st) {
  if (m <= 0 || i <= 0) return;
  k_batch_resid<T><<<cdiv(m, 256), 256, i * sizeof(double), st>>>(GS, m, i, L, z, r0, out); note_launch();
}
template void sqnorm_acc<float>(const float*, int, double*, cudaStream_t);
template void sqnorm_acc<double>(const double*, int, double*, cudaStream_t);
template void batch_resid<float>(const float*, int, int, const double*, const double*, const float*, double*, cudaStream_t);
template void batch_resid<double>(const double*, int, int, const double*, const double*, const double*, double*,
                                  cudaStream_t);

// ------------------------------------------------------------------------------------------
// Posterior sampler (the CAKF/CAKS sampler algorithm): S draws as the columns of n x S blocks.
// xp = a xprev + (mu_k - a mu_{k-1}) + q   (FP64; mu pointers may be null)
__global__ void k_samp_predict(const double* __restrict__ xprev, const double* __restrict__ q,
                               const double* __restrict__ mu_k, const double* __restrict__ mu_km1, double a, int n,
                               int S, double* __restrict__ xp) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int s = blockIdx.y;
  if (j >= n || s >= S) return;
  const double b = mu_k ? mu_k[j] - a * mu_km1[j] : 0.0;
  xp[(size_t)s * n + j] = fma(a, xprev[(size_t)s * n + j], b + q[(size_t)s * n + j]);
}
// d = y - xp[obs] - eps  (m x S, precision T)
template <class T>
__global__ void k_samp_resid(const double* __restrict__ y, const double* __restrict__ xp, const int* __restrict__ obs,
                             const double* __restrict__ eps, int m, int n, int S, T* __restrict__ d) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int s = blockIdx.y;
  if (i >= m || s >= S) return;
  d[(size_t)s * m + i] = T(y[i] - xp[(size_t)s * n + obs[i]] - eps[(size_t)s * m + i]);
}
// x = xa + alpha * t  (x, xa FP64 n x S with ld n; t precision T with ld ldt)
template <class T>
__global__ void k_samp_add(const double* __restrict__ xa, const T* __restrict__ t, int ldt, double alpha, int n, int S,
                           double* __restrict__ x) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int s = blockIdx.y;
  if (j >= n || s >= S) return;
  x[(size_t)s * n + j] = fma(alpha, (double)t[(size_t)s * ldt + j], xa[(size_t)s * n + j]);
}
void samp_predict(const double* xprev, const double* q, const double* mu_k, const double* mu_km1, double a, int n,
                  int S, double* xp, cudaStream_t st) {
  k_samp_predict<<<dim3(cdiv(n, 256), S), 256, 0, st>>>(xprev, q, mu_k, mu_km1, a, n, S, xp); note_launch();
}
template <class T>
void samp_resid(const double* y, const double* xp, const int* obs, const double* eps, int m, int n, int S, T* d,
                cudaStream_t st) {
  if (m <= 0) return;
  k_samp_resid<T><<<dim3(cdiv(m, 256), S), 256, 0, st>>>(y, xp, obs, eps, m, n, S, d); note_launch();
}
template <class T>
void samp_add(const double* xa, const T* t, int ldt, double alpha, int n, int S, double* x, cudaStream_t st) {
  k_samp_add<T><<<dim3(cdiv(n, 256), S), 256, 0, st>>>(xa, t, ldt, alpha, n, S, x); note_launch();
}
template void samp_resid<float>(const double*, const double*, const int*, const double*, int, int, int, float*, cudaStream_t);
template void samp_resid<double>(const double*, const double*, const int*, const double*, int, int, int, double*,
                                 cudaStream_t);
template void samp_add<float>(const double*, const float*, int, double, int, int, double*, cudaStream_t);
template void samp_add<double>(const double*, const double*, int, double, int, int, double*, cudaStream_t);

// Filter marginal at a query time t_k + tau (the interpolation corollary, OU prior): m(t) = at m_k +
// mu(t) - at mu_k, var(t) = sf2 - at^2 (sf2 - var_k).
__global__ void k_interp_filter(const double* __restrict__ mk, const double* __restrict__ vk,
                                const double* __restrict__ mu_t, const double* __restrict__ mu_k, double at,
                                double sf2, int n, double* __restrict__ m, double* __restrict__ v) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const double b = mu_t ? mu_t[j] - (mu_k ? at * mu_k[j] : 0.0) : 0.0;
  m[j] = fma(at, mk[j], b);
  v[j] = sf2 - at * at * (sf2 - vk[j]);
}
void interp_filter(const double* mk, const double* vk, const double* mu_t, const double* mu_k, double at, double sf2,
                   int n, double* m, double* v, cudaStream_t st) {
  k_interp_filter<<<cdiv(n, 256), 256, 0, st>>>(mk, vk, mu_t, mu_k, at, sf2, n, m, v); note_launch();
}

void set_diag(double* G, int ld, const double* lam, double scale, int r, cudaStream_t st) {
  if (r <= 0) return;
  k_set_diag<<<cdiv(r, 256), 256, 0, st>>>(G, ld, lam, scale, r); note_launch();
}
void put_block_sym(double* G, int ld, int row0, int col0, const double* B, int ldb, int nr, int nc, double scale,
                   cudaStream_t st) {
  if (nr <= 0 || nc <= 0) return;
  k_put_block_sym<<<dim3(cdiv(nr, 256), nc), 256, 0, st>>>(G, ld, row0, col0, B, ldb, nr, nc, scale); note_launch();
}
void scale_f64(double* A, int ld, int rows, int cols, double s, cudaStream_t st) {
  if (rows <= 0 || cols <= 0) return;
  k_scale_f64<<<dim3(cdiv(rows, 256), cols), 256, 0, st>>>(A, ld, rows, cols, s); note_launch();
}
template <class T>
void convert_from_f64(const double* In, int ldi, int rows, int cols, T* Out, int ldo, cudaStream_t st) {
  if (rows <= 0 || cols <= 0) return;
  k_convert_from_f64<T><<<dim3(cdiv(rows, 256), cols), 256, 0, st>>>(In, ldi, rows, cols, Out, ldo); note_launch();
}
template void convert_from_f64<float>(const double*, int, int, int, float*, int, cudaStream_t);
template void convert_from_f64<double>(const double*, int, int, int, double*, int, cudaStream_t);

void check_finite(const double* x, size_t n, int* err, cudaStream_t st) {
  if (n == 0) return;
  k_check_finite<<<cdiv(n, 256), 256, 0, st>>>(x, n, err); note_launch();
}

#define INST(T)                                                                                                  \
  template void prep_coords<T>(const double*, int, int, double, C4<T>*, cudaStream_t);                           \
  template void prep_coords2<T>(const double*, int, const double*, int, int, double, C4<T>*, cudaStream_t);      \
  template void gather_coords<T>(const C4<T>*, const int*, int, C4<T>*, cudaStream_t);                          \
  template void gram_matvec<T>(int, const C4<T>*, const T*, int, T, T*, const T*, int, int, T*, const int*,     \
                               cudaStream_t);                                                                   \
  template void cg_combine<T>(const T*, int, const T*, T, const T*, int, int, const T*, T, int, T*, const T*,     \
                              int, int, const T*, const T*, T*, const int*, cudaStream_t);                       \
  template void cg_upd1<T>(int, const T*, double*, T*, T*, int, const T*, const T*, int, T*,                    \
                           const int*, cudaStream_t);                                                            \
  template void cg_upd2<T>(int, const double*, const T*, T*, T*, int, T*, T*, T*, T*, int, double, double,       \
                           int, int*, double*, double*, int*, T*, const double*, const T*, cudaStream_t);                                 \
  template void cg_reorth<T>(const T*, int, int, T*, int, double*, T*, int, const int*, cudaStream_t);          \
  template void cg_select<T>(int, const T*, const double*, int, T*, T*, int, const int*, cudaStream_t);          \
  template void cg_init<T>(const double*, const double*, const int*, int, T*, T*, T*, double*, cudaStream_t);    \
  template void gemm_tn<T>(const T*, int, int, const T*, int, int, int, double, double, double*, int, double*,   \
                           size_t, cudaStream_t);                                                                \
  template void gemm_nn<T, T>(int, int, int, T, const T*, int, const T*, int, T, T*, int, cudaStream_t);         \
  template void gather_rows<T>(const T*, int, const int*, int, int, T*, int, cudaStream_t);                      \
  template void scatter_add_rows<T>(const T*, int, const int*, int, int, T, T*, int, cudaStream_t);              \
  template void rowsumsq<T>(const T*, int, int, int, double, double*, cudaStream_t);                             \
  template void filter_out<T>(const double*, const T*, int, int, double, double, const double*, int, double*,   \
                              double*, double*, cudaStream_t);                                                   \
  template void scale_copy<T>(const T*, int, int, int, T, T*, int, cudaStream_t);                                \
  template void smooth_out<T>(const double*, const double*, const T*, int, int, int, double*, double*,           \
                              cudaStream_t);                                                                     \
  template void ws_obs<T>(const int*, int, const T*, const T*, T*, cudaStream_t);                                \
  template void build_x<T>(const T*, int, int, const T*, T, int, T*, int, cudaStream_t);                        \
  template void mix2<T>(const T*, int, T*, int, int, int, const double*, cudaStream_t);                          \
  template void add_vec<T>(const double*, const T*, int, double*, cudaStream_t);

INST(float)
INST(double)
template void gemm_nn<float, double>(int, int, int, float, const float*, int, const double*, int, float, float*, int,
                                     cudaStream_t);

}  // namespace cakf
