// FP64 symmetric eigensolver for the truncation step (Truncate, Sec. 3.2: the top-r eigen-directions
// of the (r+i) x (r+i) Gram of the downdate factor).
//
//   1. Householder tridiagonalisation, one cooperative kernel; the blocks exchange each column's
//      matvec and pivot column through write-once words (no grid barrier), with bounded polling.
//   2. Divide and conquer on the tridiagonal (Cuppen's tearing; deflation of small z components and
//      close poles by Givens rotations; secular roots by a two-pole rational model guarded by
//      bisection; eigenvectors from the Loewner-corrected z (Gu-Eisenstat), which keeps them
//      orthogonal without re-orthogonalisation).
//   3. Back-transformation of the wanted columns through the Householder reflectors.
// All arithmetic is FP64; only the final eigenvector block is stored in the caller's precision.
#include <type_traits>
#include <vector>
#include <map>
#include <mutex>
#include "internal.h"
#include "fp64_ops.cuh"

namespace cakf {

namespace {

constexpr double kEps = 2.220446049250313e-16;

// Exchange between the blocks of the tridiagonalisation without barriers or flags: every step has its own
// slots, filled with the sentinel (all bits set: a NaN that arithmetic only passes on from an operand, and
// td_load() replaces it in the input) before the kernel starts; an owner writes each 8-byte word once, and a consumer polls the words it needs
// until none is the sentinel.  Each word is written and read as one access.
constexpr unsigned long long kSlotEmpty = ~0ULL;
__device__ __forceinline__ void publish(double* p, double x) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(__double_as_longlong(x)) : "memory");
}
__device__ __forceinline__ double td_load(const double* p) {
  const double x = *p;
  return __isnan(x) ? __longlong_as_double(0x7FF8000000000000LL) : x;
}
__device__ __forceinline__ void ld_slot(const double* p, unsigned long long& s, unsigned long long& c) {
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(s), "=l"(c) : "l"(p) : "memory");
}
__device__ __forceinline__ int ld_relaxed_int(const int* p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
constexpr long long kPollLimit = 4000000LL;

// Power of two that brings a largest magnitude amax (its bit pattern; as far as the exponent range goes, a zero or
// denormal one too) to about 2^target, and its inverse; 1 for a non-finite one.
__device__ __forceinline__ void pow2_scale(unsigned long long amax, int target, double& sc, double& inv) {
  const int ex = (int)(amax >> 52) & 0x7FF;
  if (ex == 2047) { sc = inv = 1.0; return; }
  const long long E = max(1, min(2045, 2046 + target - ex));
  sc = __longlong_as_double(E << 52);
  inv = __longlong_as_double((2046 - E) << 52);
}

// *amax = largest magnitude of the N x N matrix, as a bit pattern (zero before the launch)
__global__ void __launch_bounds__(256)
k_absmax(const double* __restrict__ A, int lda, int N, unsigned long long* __restrict__ amax) {
  unsigned long long m = 0;
  for (int j = blockIdx.x; j < N; j += gridDim.x)
    for (int t = threadIdx.x; t < N; t += blockDim.x) {
      const unsigned long long b = (unsigned long long)__double_as_longlong(A[(size_t)j * lda + t]) & 0x7FFFFFFFFFFFFFFFULL;
      m = b > m ? b : m;
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long x = __shfl_xor_sync(0xffffffffu, m, o);
    m = x > m ? x : m;
  }
  if ((threadIdx.x & 31) == 0) atomicMax(amax, m);
}

// ---------------------------------------------------------------------------------- tridiagonal
// Householder tridiagonalisation (lower).  Columns of the trailing block are owned by blocks round-robin
// (column j: block j % G, slot j / G) and stay in shared memory; vectors along the trailing rows are held
// by every block.  With c the first column of the trailing block B_k (rows k..), x = c1^2 + sigma, sigma =
// sum_{t>=2} c_t^2, s = sqrt(x) and gamma = c1 + sign(c1) s, the reflector is I - tau v v^T on rows k + 1..
// with v = (gamma, c_2, c_3, ...), tau = 1 / (s |gamma|) -- unscaled, so that
//   p = B v = S + gamma C,   S_j = sum_{t>=1} B_{tj} v_t,  C = column k + 1 of B (rows k + 1..),
// where S depends on c but not on sigma.  Since C is also row k + 1, p_0 = C . v, so q = p . v =
// sum_{t>=1} S_t v_t + gamma (S_0 + p_0) needs no p.  Step k:
//   warps 0-3  poll S and C, with the partial sums of S_t v_t on the way                    -- barrier
//   warp 4     their sum; warps 0-3 form p and C - gamma tau p                                -- barrier
//   warps 0-3  next c = C - gamma tau p - e3 v, e3 = tau (p_0 - gamma tau q)                   -- barrier
//   warps 0-3  owned columns: B_tj -= v_t a_j + p_t b_j  (a_j = tau (p_j - tau q v_j), b_j = tau v_j) and, in
//              the same pass, the next S_j; publish S_j, and the next pivot column as it is formed
//   warp 4     sigma and the scalars of the next reflector, which nobody waits for before the next
//              exchange has arrived
// What bounds it: an FP64 instruction holds its quarter of the SM (one warp here) for 64 cycles, 77 when all
// four are busy, whatever its lanes or their predicates, and a shuffle level of an FP64 sum 126.  So warps
// take whole columns, sums go through integers (warp_sum_int: 460 cycles instead of 690), loops have no padded
// turns, and warp 4 takes what is not on the chain.  Per column at N = 576, about: column pass 2,700 cycles
// (three FP64 instructions per 32 entries), its sum 460, exchange 1,800 (store to L2, load) plus the wait for
// the slowest block, block sum 600, the next c 400.  The words go to REP replicas (a block polls one of
// them): 152 blocks polling the same lines queue at their L2 slices (N = 576: 2.73 ms with one replica, 2.52
// with 4, 2.66 with 16).  N = 576 takes 2.52 ms, N = 288 0.94 ms; 2.79 and 1.15 ms with scaled reflectors,
// whose scalars stood between the column pass and the exchange, shuffle sums and pairs of 16 bytes a value.
// The matrix is scaled by a power of two to about 2^TD_SCALE, which keeps the unscaled reflectors' products in
// range: they go up to N^1.5 c^3 (2^936 at N = 2,048) and, for a decoupled block far below the rest, down to c^3 and
// its reciprocal.  A column whose square is below TD_TINY (2^-620 of the matrix) is left alone (tau = 0).  v and tau are kept for the back-transformation, v
// below the subdiagonal of column k.
constexpr int TD_SCALE = 300;                // exponents: the scaled matrix,
constexpr double TD_TINY = 0x1p-640;         // and the squared norm of a column that is left alone
constexpr int TD_VEC = 128;                  // threads of the vector work: 4 warps, the owner warps
constexpr int TD_THREADS = TD_VEC + 32;      // warp 4: block reductions and scalars
constexpr int TD_MAX_SLOTS = 64;             // owned columns per block
// Replicas of the exchange slots (template parameter REP; N (N + 1) words each): 4 up to order 1,024, one above,
// where the fill of 32 N^2 bytes would begin to count.
inline int td_replicas(int N) { return N <= 1024 ? 4 : 1; }
constexpr int TD_BATCH = 5;                  // exchange entries a thread polls with their loads in flight together

__host__ __device__ inline size_t td_slot_offset(int N, int k) {   // slots (S, C) of step k: N - 1 - k of them
  return (size_t)k * (size_t)(N - 1) - (size_t)k * (size_t)(k - 1) / 2;
}

// Sum of red[0 .. TD_VEC) by one warp; the result is in every lane.
__device__ __forceinline__ double td_sum(const double* red) {
  const double2* r = reinterpret_cast<const double2*>(red) + 2 * (threadIdx.x & 31);
  const double2 a = r[0], b = r[1];
  const double x[4] = {a.x, a.y, b.x, b.y};
  return warp_sum_int<4>(x);
}
__device__ __forceinline__ double td_warp_sum(double v) {
  const double x[1] = {v};
  return warp_sum_int<1>(x);
}

struct TdScalars { double gamma, gt, tau, beta; };   // gt = gamma tau; beta: the new subdiagonal entry
__device__ __forceinline__ TdScalars td_scalars(double c1, double sigma) {
  TdScalars r;
  const double x = fma(c1, c1, sigma);
  // (comparisons on the bit patterns: they stay off the FP64 pipe)
  if (__double_as_longlong(sigma) == 0 || __double_as_longlong(x) < __double_as_longlong(TD_TINY)) {
    r.gamma = 1.0; r.gt = r.tau = 0.0; r.beta = c1;
    return r;
  }
  double sq, rs;
  fast_sqrt(x, sq, rs);
  const double ss = copysign(sq, c1);
  r.gamma = c1 + ss;
  r.beta = -ss;
  r.gt = copysign(rs, c1);
  r.tau = rs * fast_rcp(fabs(r.gamma));
  return r;
}

// With q' = sum_{t>=1} S_t v_t, q = q' + gamma (2 S_0 + gamma C_0) and p_0 = S_0 + gamma C_0:
//   e3 = tau (p_0 - gamma tau q) = (bc[3] S_0 + bc[4] C_0) - bc[5] q',   tau q = (2 bc[1] S_0 + bc[6] C_0) + tau q'
__device__ __forceinline__ void td_coefficients(const TdScalars& h, double* bc) {
  const double e2 = h.tau * h.gt, tg = h.gamma * h.gt;
  bc[0] = h.gamma; bc[1] = h.gt; bc[2] = h.tau;
  bc[3] = fma(-2.0 * e2, h.gamma, h.tau);
  bc[4] = fma(-h.gt, tg, h.gt);
  bc[5] = e2;
  bc[6] = tg;
}

// Column pass of one owned column (col, v, p, cn from local row 0 = row k + 1): rows t >= 1 get the rank-2
// update, and the sum over t >= 2 of the updated entries times cn is returned (the lane's part; cn[1] counts
// as zero).  The next entry's operands are read while the current one's three dependent operations run (64
// to 77 cycles each).  With out, entry t also goes to the next step's slots t - 1 (as its C).
template <int REP>
__device__ __forceinline__ double td_column(double* col, const double* v, const double* p, const double* cn, double aj,
                                            double bj, int L, int lane, double* out, size_t rep) {
  double s = 0.0;
  int t = 1 + lane, i = min(t, L - 1);
  double xc = col[i], xv = v[i], xp = p[i], xn = i >= 2 && t < L ? cn[i] : 0.0;
#pragma unroll 1
  for (int b = 1; b < L; b += 32) {
    double x = fma(-xp, bj, xc);
    const int tn = t + 32;
    i = min(tn, L - 1);
    xc = col[i];
    xp = p[i];
    x = fma(-xv, aj, x);
    const double cv = xn;
    xv = v[i];
    xn = tn < L ? cn[i] : 0.0;
    if (t < L) {
      col[t] = x;
      if (out) {
#pragma unroll
        for (int r = 0; r < REP; ++r) publish(out + r * rep + 2 * (t - 1) + 1, x);
      }
    }
    s = fma(x, cv, s);
    t = tn;
  }
  return s;
}

template <int REP>
__global__ void __launch_bounds__(TD_THREADS)
k_tridiag(double* __restrict__ A, int lda, int N, double* __restrict__ d, double* __restrict__ e,
          double* __restrict__ tau, double* __restrict__ slots, const unsigned long long* __restrict__ amax, int* err,
          long long poll_limit) {
  extern __shared__ __align__(16) double sm[];
  // c of three steps (a step's, the next one's, and the one that the words of the next exchange go to while
  // slower warps still read this step's) and p of two; v of a step is its c from entry 1 on
  double* cbuf = sm;
  double* pbuf = sm + 3 * N;
  double* cols = sm + 5 * N;        // owned columns (full length N)
  __shared__ __align__(16) double red[TD_VEC];
  // broadcast scalars: gamma, gamma tau, tau and the coefficients of (6) below, written by warp 4; q' (warp 4);
  // S_0, C_0 (thread 0); e1, h1 (warp 3)
  __shared__ double bc[12];
  __shared__ double cS[TD_MAX_SLOTS], cB[TD_MAX_SLOTS], cT[TD_MAX_SLOTS];   // owned columns: S_j, tau v_j, tau p_j
  const int G = gridDim.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nslot = (N + G - 1) / G;
  const int ob = (N - 1) % G;       // the block that owns the last column writes the outputs
  const int maxcol = (int)blockIdx.x + G * ((N - 1 - (int)blockIdx.x) / G);
  const size_t rep = (size_t)N * (N + 1);     // words of a replica of the slots
  double msc, minv;
  pow2_scale(*amax, TD_SCALE, msc, minv);
  if (N <= 2) {
    if (blockIdx.x == 0 && tid == 0) {
      d[0] = A[0];
      if (N == 2) { e[0] = A[1]; d[1] = A[(size_t)lda + 1]; tau[0] = 0.0; }
    }
    return;
  }
  for (int q = 0; q < nslot; ++q) {
    const int j = q * G + blockIdx.x;
    if (j >= N) break;
    for (int t = tid; t < N; t += TD_THREADS) cols[(size_t)q * N + t] = msc * td_load(A + (size_t)j * lda + t);
  }
  // ---- c_0 = column 0, its scalars; S and C of step 0
  TdScalars h = {};                 // warp 4: the current reflector's scalars
  {
    for (int t = tid; t < N; t += TD_THREADS) cbuf[t] = msc * td_load(A + t);
    __syncthreads();
    if (warp == 4) {
      double part = 0.0;
      for (int t = 2 + lane; t < N; t += 32) part = fma(cbuf[t], cbuf[t], part);
      const double sigma = td_warp_sum(part);
      h = td_scalars(cbuf[1], sigma);
      __syncwarp();
      if (lane == 0) {
        if (blockIdx.x == ob) d[0] = minv * cbuf[0];
        td_coefficients(h, bc);
        cbuf[1] = h.gamma;
      }
    } else {
      for (int q = warp; q < nslot; q += 4) {
        const int j = q * G + blockIdx.x;
        if (j < 1 || j >= N) continue;
        const double* col = cols + (size_t)q * N;
        double acc = 0.0;
        for (int t = 2 + lane; t < N; t += 32) acc = fma(col[t], cbuf[t], acc);
        acc = td_warp_sum(acc);
        if (lane == 0) cS[q] = acc;
        if (lane < REP) publish(slots + lane * rep + 2 * (j - 1), acc);
        if (j == 1)
          for (int t = 1 + lane; t < N; t += 32)
            for (int r = 0; r < REP; ++r) publish(slots + r * rep + 2 * (t - 1) + 1, col[t]);
      }
    }
  }
  for (int k = 0; k + 2 < N; ++k) {
    // a block with no column to publish for step k + 1 has nothing left to do
    if ((int)blockIdx.x != ob && maxcol < k + 2) return;
    const int L = N - k - 1;
    const double* in = slots + (blockIdx.x % REP) * rep + 2 * td_slot_offset(N, k);
    double* out = slots + 2 * td_slot_offset(N, k + 1);
    double* c = cbuf + (size_t)(k % 3) * N;          // c_k, with gamma in entry 1
    double* cn = cbuf + (size_t)((k + 1) % 3) * N;   // c_{k+1}
    double* pv = pbuf + (size_t)(k & 1) * N;
    const double* v = c + 1;
    const bool next = (k + 3 < N);            // a reflector for column k + 1 exists
    // (1) poll this step's S and C (into pv and cn), and the partial sums of S_t v_t, t >= 1
    bool ok = true;
    if (warp < 4) {
      for (int t0 = tid; t0 < L && ok; t0 += TD_VEC * TD_BATCH) {
        unsigned long long bs[TD_BATCH], bcl[TD_BATCH];
        unsigned pend = 0;
#pragma unroll
        for (int u = 0; u < TD_BATCH; ++u)
          if (t0 + u * TD_VEC < L) pend |= 1u << u;
        long long spins = 0;
        while (pend) {
#pragma unroll
          for (int u = 0; u < TD_BATCH; ++u)
            if ((pend >> u) & 1u) ld_slot(in + 2 * (t0 + u * TD_VEC), bs[u], bcl[u]);
#pragma unroll
          for (int u = 0; u < TD_BATCH; ++u)
            if (((pend >> u) & 1u) && bs[u] != kSlotEmpty && bcl[u] != kSlotEmpty) {
              pend &= ~(1u << u);
              pv[t0 + u * TD_VEC] = __longlong_as_double((long long)bs[u]);
              cn[t0 + u * TD_VEC] = __longlong_as_double((long long)bcl[u]);
            }
          if (!pend) break;
          if (++spins > poll_limit) { atomicExch(err, kErrTimeout); ok = false; break; }
          if ((spins & 255) == 0 && ld_relaxed_int(err)) { ok = false; break; }
        }
      }
      double q0 = 0.0;
      if (ok) {
        if (tid == 0) { bc[8] = pv[0]; bc[9] = cn[0]; }
#pragma unroll 1
        for (int t = tid ? tid : TD_VEC; t < L; t += TD_VEC) q0 = fma(pv[t], v[t], q0);
      }
      red[tid] = q0;
    }
    if (!__syncthreads_and(ok)) return;       // also: gamma, gamma tau, tau of this step are written
    // (2) warp 4: q; the others: p and C - gamma tau p
    const double gamma = bc[0], gt = bc[1], ta = bc[2];
    if (warp == 4) {
      const double q = td_sum(red);
      if (lane == 0) bc[7] = q;
    } else {
      {
        int t = tid;
        double ct = cn[min(t, L - 1)], st = pv[min(t, L - 1)];
#pragma unroll 1
        for (; t < L; t += TD_VEC) {
          const double c0 = ct, pt = fma(gamma, ct, st);
          ct = cn[min(t + TD_VEC, L - 1)];
          st = pv[min(t + TD_VEC, L - 1)];
          pv[t] = pt;
          cn[t] = fma(-gt, pt, c0);
        }
      }
      if (warp == 3) {
        const double S0 = bc[8], C0 = bc[9];
        const double e1 = fma(bc[4], C0, bc[3] * S0), h1 = fma(bc[6], C0, 2.0 * gt * S0);
        if (lane == 0) { bc[10] = e1; bc[11] = h1; }
      }
      // the owned columns' scalars that do not wait for q (p_j from the warp's own S_j and row k + 1)
#pragma unroll 1
      for (int q = warp; q < nslot; q += 4) {
        const int j = q * G + blockIdx.x;
        if (j < k + 2 || j >= N) continue;
        const double bj = ta * v[j - (k + 1)];
        const double tp = ta * fma(gamma, cols[(size_t)q * N + k + 1], cS[q]);
        if (lane == 0) { cB[q] = bj; cT[q] = tp; }
      }
    }
    __syncthreads();
    // (3) c_{k+1}
    if (warp < 4) {
      const double e3 = fma(-bc[5], bc[7], bc[10]);
      int t = tid;
      double gr = cn[min(t, L - 1)], vt = v[min(t, L - 1)];
#pragma unroll 1
      for (; t < L; t += TD_VEC) {
        const double x = fma(-e3, vt, gr);
        gr = cn[min(t + TD_VEC, L - 1)];
        vt = v[min(t + TD_VEC, L - 1)];
        cn[t] = x;
      }
    }
    __syncthreads();
    if (warp == 4) {
      // (4) sigma and the scalars of column k + 1, beside the column passes
      const double c0 = cn[0], c1 = cn[1], beta = h.beta;
      if (next) {
        double part = 0.0;
        int t = 2 + lane;
        double x = t < L ? cn[t] : 0.0;
#pragma unroll 1
        for (int b = 2; b < L; b += 32) {
          const double y = x;
          t += 32;
          x = t < L ? cn[t] : 0.0;
          part = fma(y, y, part);
        }
        h = td_scalars(c1, td_warp_sum(part));
        __syncwarp();
        if (lane == 0) {
          td_coefficients(h, bc);
          cn[1] = h.gamma;
        }
      }
      if (blockIdx.x == ob && lane == 0) {
        d[k + 1] = minv * c0;
        e[k] = minv * beta;
        tau[k] = ta;
        if (!next) { e[k + 1] = minv * c1; tau[k + 1] = 0.0; }
      }
    } else {
      const double hq = fma(ta, bc[7], bc[11]);
#pragma unroll 1
      for (int q = warp; q < nslot; q += 4) {
        const int j = q * G + blockIdx.x;
        if (j < k + 2 || j >= N) continue;
        const int tj = j - (k + 1);
        double* col = cols + (size_t)q * N + k + 1;
        const double bj = cB[q], aj = fma(-bj, hq, cT[q]);
        double S = td_column<REP>(col, v, pv, cn, aj, bj, L, lane, next && tj == 1 ? out : nullptr, rep);   // tj = 1: the next C
        if (next) {
          S = td_warp_sum(S);
          if (lane == 0) cS[q] = S;
          if (lane < REP) publish(out + lane * rep + 2 * (tj - 1), S);
        } else if (lane == 0) {
          d[N - 1] = minv * col[1];           // L = 2: the last diagonal entry
        }
      }
    }
    // (5) warp 4 stores the reflector below the subdiagonal of column k
    if (blockIdx.x == ob && warp == 4)
      for (int t = lane; t < L; t += 32) A[(size_t)k * lda + k + 1 + t] = v[t];
  }
}

// ------------------------------------------------------------------------------ divide & conquer
struct MergeDesc { int lo, mid, hi; };

struct DcWork {
  double *lam, *lamk, *Zw, *Dk, *Zk, *Dd, *Q, *Qtmp, *Delta, *rho, *rot, *z2, *Tm;
  float2* Df;      // kept poles / rho as FP32 pairs, and the squared z components in FP32: for the secular guess
  float* zf;
  int *colk, *cold, *rank, *Kp, *nrot, *mergeof, *gperm, *gcnt;
};

// Eigenvalues of the leaves, and Q = Qtmp = I: a merge's row tiles that straddle its children
// read zeros outside them, and a leaf without a merge at the deepest level is valid in both.  (Both lie under
// the exchange slots, so they are filled here, after the tridiagonalisation; as a memset of its own the fill took
// 7 us of a call at N = 576 and 12 at 288.)
__global__ void __launch_bounds__(256)
k_dc_init(const double* __restrict__ d, const double* __restrict__ e, int N, double* lam, double* Q, double* Qtmp) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
  if (t >= N) return;
  const double one = t == j ? 1.0 : 0.0;
  Q[(size_t)j * N + t] = one;
  Qtmp[(size_t)j * N + t] = one;
  if (t != j) return;
  double v = d[j];
  if (j > 0) v -= fabs(e[j - 1]);
  if (j + 1 < N) v -= fabs(e[j]);
  lam[j] = v;
}

// Order-preserving integer key of a double (IEEE bit pattern; negative values mirrored), so the
// sorting below compares on the integer units instead of the FP64 pipe.
__device__ __forceinline__ long long order_key(double x) {
  const long long b = __double_as_longlong(x);
  return b >= 0 ? b : (b ^ 0x7FFFFFFFFFFFFFFFLL);
}

// Block-wide exclusive prefix sum of one int per thread (thread order); *total gets the sum.
__device__ int block_excl_scan(int v, int* total) {
  __shared__ int ws[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  __syncthreads();
  if (lane == 31) ws[wid] = x;
  __syncthreads();
  if (wid == 0) {
    int t = (lane < nw) ? ws[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    ws[lane] = t;
  }
  __syncthreads();
  const int before = (wid > 0 ? ws[wid - 1] : 0) + x - v;
  *total = ws[nw - 1];
  __syncthreads();
  return before;
}

constexpr int DC_THREADS = 256;

// Shared memory of k_dc_prep for a merge of order K: four FP64 arrays, one int64 key array, six int arrays.
__host__ __device__ inline size_t prep_smem_bytes(int K) { return (size_t)K * (4 * sizeof(double) + sizeof(long long) + 6 * sizeof(int)); }

// Phase 1 of a merge: z vector, sorted poles, deflation.  One block per merge.
//   1. The two ascending child spectra are merged by rank (each entry's position is its index
//      plus the number of entries of the other list before it, found by binary search).
//   2. Small z components are deflated (all entries in parallel).
//   3. Close poles are deflated by a Givens rotation: a scan in pole order, since a rotation changes
//      the entries the next test reads; one thread, operands carried in registers.  The rotations
//      are written to W.rot and applied to the eigenvector rows by k_dc_rot.
//   4. Kept and deflated entries are compacted (block prefix sums); the kept poles are re-sorted
//      by rank when a rotation moved one.
//   5. The kept columns are grouped by their row support (child 1 only, both, child 2 only) for the
//      eigenvector product of phase 5.
// Poles, rho and with them the distances of phases 2 to 4 are in units of a power of two near the merge's
// largest magnitude (W.rho[lo + 1] takes them back): the secular function divides by distances of rho z^2, 1e-30
// of that magnitude, and squares them, which leaves FP64's range for a matrix (or a decoupled block of one) below
// 2^-430 or above 2^506 in its own units.  Eigenvalues go in and out unscaled.
// (device function: every thread of the block calls it; psm holds prep_smem_bytes(K))
__device__ void dc_prep(const MergeDesc mg, const double* __restrict__ e, int N, DcWork W, double* psm) {
  const int lo = mg.lo, mid = mg.mid, K = mg.hi - mg.lo, n1 = mg.mid - mg.lo;
  double* sLam = psm;
  double* sZr = psm + K;
  double* sD = psm + 2 * K;
  double* sZ = psm + 3 * K;
  long long* sKey = reinterpret_cast<long long*>(psm + 4 * K);
  int* sPerm = reinterpret_cast<int*>(psm + 5 * K);
  int* sStat = sPerm + K;       // 0 kept, 1 deflated (small z), 2 deflated (rotated away)
  int* sType = sStat + K;       // row support: 1 child 1, 3 child 2, 2 both
  int* sKeep = sType + K;
  int* sDefl = sKeep + K;
  int* sSort = sDefl + K;
  __shared__ int s_nrot;
  const double rho0 = e[mid - 1];
  const double sgn = rho0 >= 0.0 ? 1.0 : -1.0;
  double zz = 0.0;
  for (int t = threadIdx.x; t < K; t += blockDim.x) {
    const double z = (t < n1) ? W.Q[(size_t)(lo + t) * N + (mid - 1)] : sgn * W.Q[(size_t)(lo + t) * N + mid];
    sZr[t] = z;
    const double l = W.lam[lo + t];
    sLam[t] = l;
    sKey[t] = order_key(l);
    sPerm[t] = t;
    zz += z * z;
  }
  zz = block_sum(zz);
  double zn, rzn;
  fast_sqrt(fmax(zz, 1e-280), zn, rzn);
  // the children's spectra ascend: their ends have the largest magnitudes
  const double lmax = fmax(fmax(fabs(sLam[0]), fabs(sLam[n1 - 1])), fmax(fabs(sLam[n1]), fabs(sLam[K - 1])));
  double sc, isc;
  pow2_scale((unsigned long long)__double_as_longlong(fmax(lmax, fabs(rho0) * zz)), 0, sc, isc);
  const double rho = fabs(rho0) * sc * zz;
  // 1. merge by rank (ties: child 1 first)
  for (int t = threadIdx.x; t < K; t += blockDim.x) {
    const long long kt = sKey[t];
    int pos;
    if (t < n1) {
      int a = n1, b = K;
      while (a < b) { const int m = (a + b) >> 1; if (sKey[m] < kt) a = m + 1; else b = m; }
      pos = t + (a - n1);
    } else {
      int a = 0, b = n1;
      while (a < b) { const int m = (a + b) >> 1; if (sKey[m] <= kt) a = m + 1; else b = m; }
      pos = (t - n1) + a;
    }
    sPerm[pos] = t;
    sD[pos] = sc * sLam[t];
    sZ[pos] = sZr[t] * rzn;
    sType[pos] = (t < n1) ? 1 : 3;
  }
  __syncthreads();
  // 2. tolerance and small-z deflation
  const double dm = fmax(fabs(sD[0]), fabs(sD[K - 1]));   // sD ascends
  const double tol = 8.0 * kEps * fmax(dm, rho);
  for (int t = threadIdx.x; t < K; t += blockDim.x) sStat[t] = (rho * fabs(sZ[t]) <= tol) ? 1 : 0;
  __syncthreads();
  // 3. close poles.  The test |(D_j - D_l) c s| <= tol with c s = -z_l z_j / t^2 is evaluated
  // without the division, as |D_j - D_l| |z_l z_j| <= tol t^2; c and s are formed only for a
  // rotation.  The pairs of consecutive candidates (entries not deflated by small z) are first tested
  // in parallel on the merged values; a pair's test can only change after a rotation, so the
  // sequential scan starts at the first pair that fires (in the common case none does).
  const int ch0 = (K + (int)blockDim.x - 1) / (int)blockDim.x;
  const int a0 = min(K, (int)threadIdx.x * ch0), a1 = min(K, a0 + ch0);
  int ncl = 0;
  for (int t = a0; t < a1; ++t) ncl += (sStat[t] == 0);
  int nc = 0;
  int oc = block_excl_scan(ncl, &nc);
  int* sCand = sSort;                 // free until the kept poles are re-sorted below
  for (int t = a0; t < a1; ++t)
    if (sStat[t] == 0) sCand[oc++] = t;
  __shared__ int s_first;
  if (threadIdx.x == 0) s_first = nc;
  __syncthreads();
  for (int u = 1 + threadIdx.x; u < nc; u += blockDim.x) {
    const int l = sCand[u - 1], jj = sCand[u];
    const double zl = sZ[l], zj = sZ[jj];
    const double t2 = fma(zl, zl, zj * zj);
    if (fabs(sD[jj] - sD[l]) * fabs(zl * zj) <= tol * t2) atomicMin(&s_first, u);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int nrot = 0;
    const int first = s_first;
    if (first < nc) {
      int last = sCand[first - 1];
      double zl = sZ[last], dl = sD[last];
      for (int u = first; u < nc; ++u) {
        const int j = sCand[u];
        double zj = sZ[j], dj = sD[j];
        const double t2 = fma(zl, zl, zj * zj);
        if (fabs(dj - dl) * fabs(zl * zj) <= tol * t2) {
          const double t = sqrt(t2);
          const double c = zj / t, sn = -zl / t;
          double* rr = W.rot + (size_t)4 * (lo + nrot);
          rr[0] = (double)(lo + sPerm[last]);
          rr[1] = (double)(lo + sPerm[j]);
          rr[2] = c;
          rr[3] = sn;
          ++nrot;
          sD[last] = c * c * dl + sn * sn * dj;
          dj = sn * sn * dl + c * c * dj;
          sD[j] = dj;
          sZ[last] = 0.0;
          sZ[j] = t;
          zj = t;
          sStat[last] = 2;
          if (sType[last] != sType[j]) sType[j] = 2;
        }
        last = j;
        zl = zj;
        dl = dj;
      }
    }
    s_nrot = nrot;
    W.nrot[lo] = nrot;
  }
  __syncthreads();
  const int nrot = s_nrot;
  // 4. compaction: kept and deflated entries in pole order
  const int ch = (K + (int)blockDim.x - 1) / (int)blockDim.x;
  const int c0 = min(K, (int)threadIdx.x * ch), c1 = min(K, c0 + ch);
  int nk = 0;
  for (int t = c0; t < c1; ++t) nk += (sStat[t] == 0);
  int kp = 0;
  int ok = block_excl_scan(nk, &kp);
  int od = c0 - ok;
  for (int t = c0; t < c1; ++t) {
    if (sStat[t] == 0) sKeep[ok++] = t;
    else sDefl[od++] = t;
  }
  __syncthreads();
  const int* keep = sKeep;
  if (nrot > 0) {
    // a rotation can move a kept pole past its neighbours: rank sort by (value, position)
    for (int q = threadIdx.x; q < kp; q += blockDim.x) sKey[q] = order_key(sD[sKeep[q]]);
    __syncthreads();
    for (int q = threadIdx.x; q < kp; q += blockDim.x) {
      const long long kq = sKey[q];
      int rank = 0;
      for (int u = 0; u < kp; ++u) {
        const long long ku = sKey[u];
        rank += (ku < kq) || (ku == kq && u < q);
      }
      sSort[rank] = sKeep[q];
    }
    __syncthreads();
    keep = sSort;
  }
  const double irho = rho > 0.0 ? 1.0 / rho : 0.0;
  for (int q = threadIdx.x; q < kp; q += blockDim.x) {
    const int j = keep[q];
    const double zj2 = sZ[j] * sZ[j], ds = sD[j] * irho;
    const float dh = __double2float_rn(ds);
    W.Dk[lo + q] = sD[j];
    W.Zk[lo + q] = sZ[j];
    W.z2[lo + q] = rho * zj2;
    W.Df[lo + q] = make_float2(dh, __double2float_rn(ds - (double)dh));
    W.zf[lo + q] = __double2float_rn(zj2);
    W.colk[lo + q] = lo + sPerm[j];
  }
  for (int q = threadIdx.x; q < K - kp; q += blockDim.x) {
    const int j = sDefl[q];
    W.Dd[lo + q] = isc * sD[j];
    W.cold[lo + q] = lo + sPerm[j];
  }
  // 5. kept columns grouped by row support: child 1 only, both children, child 2 only
  {
    const int kc = (kp + (int)blockDim.x - 1) / (int)blockDim.x;
    const int q0 = min(kp, (int)threadIdx.x * kc), q1 = min(kp, q0 + kc);
    int cnt[3] = {0, 0, 0};
    for (int q = q0; q < q1; ++q) ++cnt[sType[keep[q]] - 1];
    int tot[3];
    int off[3];
    for (int g = 0; g < 3; ++g) off[g] = block_excl_scan(cnt[g], &tot[g]);
    off[1] += tot[0];
    off[2] += tot[0] + tot[1];
    for (int q = q0; q < q1; ++q) W.gperm[lo + off[sType[keep[q]] - 1]++] = q;
    if (threadIdx.x == 0) {
      W.gcnt[2 * lo] = tot[0];
      W.gcnt[2 * lo + 1] = tot[1];
      W.rho[lo] = rho;
      W.rho[lo + 1] = isc;
      W.Kp[lo] = kp;
    }
  }
}
__global__ void __launch_bounds__(DC_THREADS)
k_dc_prep(const MergeDesc* __restrict__ merges, const double* __restrict__ e, int N, DcWork W) {
  extern __shared__ double psm[];
  dc_prep(merges[blockIdx.x], e, N, W, psm);
}

// Phase 1b: the deflation rotations applied to the child eigenvector columns, one thread per row of
// the merge.  Rotation q acts on (a_q, b_q) with b_q a column no earlier rotation touched, and a_q
// either untouched as well or equal to b_{q-1}; so each group of RG rotations loads its operands up
// front (independent loads), and the a_q = b_{q-1} chain is carried in a register.
__device__ void dc_rot_row(const MergeDesc mg, int N, DcWork W, int row) {
  const int lo = mg.lo, K = mg.hi - mg.lo;
  if (row >= K) return;
  const int nrot = W.nrot[lo];
  if (nrot == 0) return;
  const double* rot = W.rot + (size_t)4 * lo;
  double* qrow = W.Q + lo + row;
  constexpr int RG = 8;
  double carry = 0.0;
  int carry_col = -1;
  for (int q0 = 0; q0 < nrot; q0 += RG) {
    const int nq = min(RG, nrot - q0);
    int ca[RG], cb[RG];
    double xa[RG], xb[RG];
#pragma unroll
    for (int u = 0; u < RG; ++u) {
      if (u >= nq) break;
      const double* rr = rot + 4 * (q0 + u);
      ca[u] = (int)rr[0];
      cb[u] = (int)rr[1];
      const int prev = (u == 0) ? carry_col : cb[u - 1];
      xb[u] = qrow[(size_t)cb[u] * N];
      xa[u] = (ca[u] == prev) ? 0.0 : qrow[(size_t)ca[u] * N];
    }
#pragma unroll
    for (int u = 0; u < RG; ++u) {
      if (u >= nq) break;
      const double* rr = rot + 4 * (q0 + u);
      const double c = rr[2], sn = rr[3];
      const int prev = (u == 0) ? carry_col : cb[u - 1];
      const double a = (ca[u] == prev) ? carry : xa[u];
      const double na = c * a + sn * xb[u];
      const double nb = -sn * a + c * xb[u];
      qrow[(size_t)ca[u] * N] = na;
      qrow[(size_t)cb[u] * N] = nb;
      carry = nb;
      carry_col = cb[u];
    }
  }
}
__global__ void __launch_bounds__(128)
k_dc_rot(const MergeDesc* __restrict__ merges, int N, DcWork W) {
  dc_rot_row(merges[blockIdx.y], N, W, blockIdx.x * blockDim.x + threadIdx.x);
}

// Sum over the LANES lanes that share one root (LANES = 32: a warp; otherwise an aligned group of lanes of a
// warp named by mask, which lets the groups of one warp run different iteration counts).
template <int LANES> __device__ __forceinline__ double group_sum(double v, unsigned mask = 0xffffffffu) {
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
  return v;
}
// The same for four values at once, by a transposing butterfly: log2(LANES) + 1 additions per lane instead of
// 4 log2(LANES) (each holds the FP64 pipe for 64 cycles); every lane gets all four sums.
template <int LANES>
__device__ __forceinline__ void group_sum4(double& a, double& b, double& c, double& d, int lane, unsigned mask) {
  constexpr int H = LANES / 2, Q = LANES / 4;
  const bool up = lane & H, up2 = lane & Q;
  double x = up ? c : a, y = up ? d : b;
  x += __shfl_xor_sync(mask, up ? a : c, H);
  y += __shfl_xor_sync(mask, up ? b : d, H);
  double v = up2 ? y : x;
  v += __shfl_xor_sync(mask, up2 ? x : y, Q);
#pragma unroll
  for (int o = Q / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
  a = __shfl_sync(mask, v, 0, LANES);
  b = __shfl_sync(mask, v, Q, LANES);
  c = __shfl_sync(mask, v, H, LANES);
  d = __shfl_sync(mask, v, H + Q, LANES);
}
template <int LANES> __device__ __forceinline__ float group_sumf(float v, unsigned mask) {
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
  return v;
}

__device__ __forceinline__ float rcp_r(float x) { return __fdividef(1.0f, x); }
__device__ __forceinline__ double rcp_r(double x) { return fast_rcp(x); }
__device__ __forceinline__ float sqrt_r(float x) { return approx_sqrt(x); }
__device__ __forceinline__ double sqrt_r(double x) {
  if (!(x > 1e-280)) return 0.0;
  double sq, rs;
  fast_sqrt(x, sq, rs);
  return sq;
}
// One step of the two-pole rational model of the secular function at tau (poles at distances Dl < 0 < Dr, in
// the real type R): f ~ c + sl / (Dl - x) + sr / (Dr - x) with the parts' values and slopes matched.  Returns
// the root inside (lo, hi), or NaN.
template <class R>
__device__ __forceinline__ R secular_step(R f, R dpsi, R dphi, R Dl, R Dr, bool inner, R tau, R lo, R hi) {
  const R sl = Dl * Dl * dpsi;
  R c1, c2;
  if (inner) {
    const R sr = Dr * Dr * dphi;
    const R c = f - Dl * dpsi - Dr * dphi;
    const R B2 = -(c * (Dl + Dr) + sl + sr), C2 = c * Dl * Dr + sl * Dr + sr * Dl;
    R disc = B2 * B2 - R(4) * c * C2;
    disc = disc > R(0) ? disc : R(0);
    const R q = R(-0.5) * (B2 + copysign(sqrt_r(disc), B2));
    c1 = q * rcp_r(c);
    c2 = C2 * rcp_r(q);
  } else {
    const R c = f - Dl * dpsi;
    c1 = c2 = Dl + sl * rcp_r(c);
  }
  const R t1 = tau + c1, t2 = tau + c2;
  if (t1 > lo && t1 < hi) return t1;     // (false for NaN)
  if (t2 > lo && t2 < hi) return t2;
  return R(NAN);
}

// Phase 2: secular roots, LANES lanes per (merge, root); the sums over poles are split across the lanes.
// delta column i: Delta[(lo+i)*N + lo + j] = Dk_j - lam_i, computed from the origin pole.
// A guess is found in FP32 first (poles as FP32 pairs, so that their differences keep their leading digits;
// about 30 times cheaper per evaluation than FP64); the FP64 iteration starts there, on the whole interval
// between the poles as its bracket, and decides convergence alone: about 3 evaluations instead of 7.
template <int LANES>
__device__ void dc_secular_root(int lo, int i, int N, DcWork W, int* err, int lane, unsigned gmask) {
  const int Kp = W.Kp[lo];
  if (i >= Kp) return;
  const double* Dk = W.Dk + lo;
  const double* z2 = W.z2 + lo;
  const double rho = W.rho[lo];
  double* delta = W.Delta + (size_t)(lo + i) * N + lo;
  const bool inner = i < Kp - 1;
  // ---- FP32 guess, in units of rho
  int org = i;
  float tg;
  {
    const float2* Df = W.Df + lo;
    const float* zf = W.zf + lo;
    float2 o = Df[i];
    const float gap = inner ? (Df[i + 1].x - o.x) + (Df[i + 1].y - o.y) : 1.0f;
    float tl = 0.f, th = gap;
    tg = 0.5f * gap;
    for (int it = 0; it < 40; ++it) {
      float psi = 0.f, dpsi = 0.f, phi = 0.f, dphi = 0.f;
      for (int j = lane; j < Kp; j += LANES) {
        const float2 dj = Df[j];
        const float r = __fdividef(1.0f, ((dj.x - o.x) + (dj.y - o.y)) - tg);
        const float tv = zf[j] * r;
        if (j <= i) { psi += tv; dpsi = fmaf(tv, r, dpsi); }
        else { phi += tv; dphi = fmaf(tv, r, dphi); }
      }
      psi = group_sumf<LANES>(psi, gmask); dpsi = group_sumf<LANES>(dpsi, gmask);
      phi = group_sumf<LANES>(phi, gmask); dphi = group_sumf<LANES>(dphi, gmask);
      const float f = 1.0f + psi + phi;
      if (it == 0 && inner && f < 0.f) {     // the root is nearer to the right pole
        org = i + 1;
        o = Df[org];
        tl = -gap; th = 0.f;
        tg = -0.5f * gap;
      }
      if (!(fabsf(f) > 1e-6f * (1.0f - psi + phi))) break;
      if (f > 0.f) th = tg; else tl = tg;
      const float2 dl = Df[i], dr = inner ? Df[i + 1] : o;
      const float Dl = ((dl.x - o.x) + (dl.y - o.y)) - tg, Dr = ((dr.x - o.x) + (dr.y - o.y)) - tg;
      float nt = secular_step(f, dpsi, dphi, Dl, Dr, inner, tg, tl, th);
      if (!(nt > tl && nt < th)) nt = 0.5f * (tl + th);
      const bool done = fabsf(nt - tg) <= 1e-6f * fabsf(nt);
      tg = nt;
      if (done) break;
    }
  }
  // ---- FP64
  const double Dorg = Dk[org];
  double tlo, thi;
  if (!inner) { tlo = 0.0; thi = rho * (1.0 + 1e-12); }      // |z| = 1
  else if (org == i) { tlo = 0.0; thi = Dk[i + 1] - Dorg; }
  else { tlo = Dk[i] - Dorg; thi = 0.0; }
  double tau = (double)tg * rho;
  if (!(tau > tlo && tau < thi)) tau = 0.5 * (tlo + thi);
  bool conv = false;
  for (int it = 0; it < 200 && !conv; ++it) {
    double psi = 0.0, dpsi = 0.0, phi = 0.0, dphi = 0.0;
    int j = lane;
#pragma unroll 2
    for (; j <= i; j += LANES) {
      const double rinv = fast_rcp((Dk[j] - Dorg) - tau);
      const double tv = z2[j] * rinv;
      psi += tv;
      dpsi = fma(tv, rinv, dpsi);
    }
#pragma unroll 2
    for (; j < Kp; j += LANES) {
      const double rinv = fast_rcp((Dk[j] - Dorg) - tau);
      const double tv = z2[j] * rinv;
      phi += tv;
      dphi = fma(tv, rinv, dphi);
    }
    __syncwarp(gmask);
    group_sum4<LANES>(psi, dpsi, phi, dphi, lane, gmask);
    const double f = 1.0 + psi + phi;
    if (f == 0.0) break;
    // residual test: f is as small as rounding of its terms allows (psi < 0 < phi term-wise)
    if (fabs(f) <= 8.0 * kEps * (1.0 - psi + phi)) break;
    if (f > 0.0) thi = tau; else tlo = tau;
    // the model step is a guess: the bracket and the residual test decide convergence
    const double Dl = (Dk[i] - Dorg) - tau, Dr = inner ? (Dk[i + 1] - Dorg) - tau : 0.0;
    double nt = secular_step(f, dpsi, dphi, Dl, Dr, inner, tau, tlo, thi);
    if (!isfinite(nt)) nt = 0.5 * (tlo + thi);
    conv = fabs(nt - tau) <= 2.0 * kEps * fmax(fabs(nt), fabs(tau)) ||
           (thi - tlo) <= 4.0 * kEps * fmax(fabs(tlo), fabs(thi));
    tau = nt;
    if (it == 199 && !conv && lane == 0) atomicExch(err, kErrSecular);
  }
  for (int j = lane; j < Kp; j += LANES) delta[j] = (Dk[j] - Dorg) - tau;
  if (lane == 0) W.lamk[lo + i] = W.rho[lo + 1] * (Dorg + tau);
}
template <int LANES>
__global__ void k_dc_secular(const MergeDesc* __restrict__ merges, const int* __restrict__ mergeof, int N, DcWork W,
                             int* err) {
  const int p = (blockIdx.x * blockDim.x + threadIdx.x) / LANES;
  const int lane = threadIdx.x % LANES;
  if (p >= N) return;
  const int mi = mergeof[p];
  if (mi < 0) return;
  const int lo = merges[mi].lo;
  dc_secular_root<LANES>(lo, p - lo, N, W, err, lane, 0xffffffffu);
}

// Phase 3: Loewner-corrected z:
//   zhat_j^2 = (lam_last - D_j)/rho * prod_{i<j} (lam_i - D_j)/(D_i - D_j) * prod_{i>j} (lam_{i-1} - D_j)/(D_i - D_j)
// Numerators and denominators are multiplied as mantissas in [1, 2) with their exponents summed in integers
// (no division, logarithm or overflow per factor), rescaled every 512 factors of a lane.
template <int LANES>
__device__ void dc_zhat_one(int lo, int j, int N, DcWork W, int lane, unsigned gmask) {
  const int Kp = W.Kp[lo];
  if (j >= Kp) return;
  const double* Dk = W.Dk + lo;
  const double rho = W.rho[lo];
  const double Dj = Dk[j];
  double pn = 1.0, pd = 1.0;
  int ex = 0;
  const long long kOne = 0x3FFLL << 52, kExp = 0x7FFLL << 52;
  auto split = [&](double x, int sign) {      // mantissa of |x| in [1, 2); its exponent into ex
    const long long b = __double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFLL;
    ex += sign * ((int)(b >> 52) - 1023);
    return __longlong_as_double((b & ~kExp) | kOne);
  };
  int cnt = 0;
  for (int i = lane; i < Kp; i += LANES) {
    if (i == j) continue;
    const int ii = (i < j) ? i : i - 1;                       // lam_i for i < j, lam_{i-1} for i > j
    pn *= split(W.Delta[(size_t)(lo + ii) * N + lo + j], 1);
    pd *= split(Dk[i] - Dj, -1);
    if (++cnt == 512) { pn = split(pn, 1); pd = split(pd, -1); cnt = 0; }
  }
  pn = split(pn, 1);
  pd = split(pd, -1);
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) {
    pn *= __shfl_xor_sync(gmask, pn, o);
    pd *= __shfl_xor_sync(gmask, pd, o);
    ex += __shfl_xor_sync(gmask, ex, o);
  }
  if (lane == 0) {
    // sqrt(last prod) with the exponent halved: an odd one leaves a factor 2 under the root
    const double last = split(W.Delta[(size_t)(lo + Kp - 1) * N + lo + j], 1);
    const double r = split(rho, -1);
    double m = last * pn / (r * pd);
    if (ex & 1) m *= 2.0;
    W.Zw[lo + j] = copysign(ldexp(sqrt(m), ex >> 1), W.Zk[lo + j]);
  }
}
// Position of item t (roots, then deflated poles) in the merged spectrum: its rank on (value key, item).
template <int LANES>
__device__ void dc_rank_one(const MergeDesc mg, int t, DcWork W, int lane, unsigned gmask) {
  const int lo = mg.lo, K = mg.hi - mg.lo, Kp = W.Kp[lo];
  const double v = (t < Kp) ? W.lamk[lo + t] : W.Dd[lo + t - Kp];
  const long long kt = order_key(v);
  int r = 0;
  for (int u = lane; u < K; u += LANES) {
    const long long ku = order_key((u < Kp) ? W.lamk[lo + u] : W.Dd[lo + u - Kp]);
    r += (ku < kt) || (ku == kt && u < t);
  }
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) r += __shfl_xor_sync(gmask, r, o);
  if (lane == 0) {
    W.lam[lo + r] = v;
    W.rank[lo + t] = r;
  }
}
template <int LANES>
__global__ void k_dc_zhat(const MergeDesc* __restrict__ merges, const int* __restrict__ mergeof, int N, DcWork W) {
  const int p = (blockIdx.x * blockDim.x + threadIdx.x) / LANES;
  const int lane = threadIdx.x % LANES;
  if (p >= N) return;
  const int mi = mergeof[p];
  if (mi < 0) return;
  const int lo = merges[mi].lo;
  dc_zhat_one<LANES>(lo, p - lo, N, W, lane, 0xffffffffu);
  dc_rank_one<LANES>(merges[mi], p - lo, W, lane, 0xffffffffu);
}

// Phase 4: eigenvector columns u_i = zhat / delta_i, normalised, written over Delta (one warp per i).
template <int LANES>
__device__ void dc_vecs_one(int lo, int i, int N, DcWork W, int lane, unsigned gmask) {
  const int Kp = W.Kp[lo];
  if (i >= Kp) return;
  double* col = W.Delta + (size_t)(lo + i) * N + lo;
  double nrm = 0.0;
  for (int j = lane; j < Kp; j += LANES) { double u = W.Zw[lo + j] * fast_rcp(col[j]); col[j] = u; nrm = fma(u, u, nrm); }
  nrm = group_sum<LANES>(nrm, gmask);
  double nv, inv;
  fast_sqrt(nrm, nv, inv);
  for (int j = lane; j < Kp; j += LANES) col[j] *= inv;
}
template <int LANES>
__global__ void k_dc_vecs(const MergeDesc* __restrict__ merges, const int* __restrict__ mergeof, int N, DcWork W) {
  const int p = (blockIdx.x * blockDim.x + threadIdx.x) / LANES;
  const int lane = threadIdx.x % LANES;
  if (p >= N) return;
  const int mi = mergeof[p];
  if (mi < 0) return;
  const int lo = merges[mi].lo;
  dc_vecs_one<LANES>(lo, p - lo, N, W, lane, 0xffffffffu);
}

// Phase 5: Qtmp[lo:hi, lo + rank] = Q[lo:hi, colk] U[:, i] (i < Kp), and the deflated columns copied; the columns
// land in ascending order of the merged spectrum, and Q and Qtmp change places for the next level.  Columns
// of rank below cmin (the final merge's, where the caller keeps only the top) are left out.  The sum over kept
// poles runs in the support order of phase 1 (gperm): a row tile inside child 1 skips the columns supported
// on child 2 only and vice versa, about half of the products.  FP64-bound, so nothing is computed for
// padding: the last stage has its own length and halves of a tile beyond the merge are skipped.
constexpr int DG_T = 32;
__global__ void __launch_bounds__(256)
k_dc_gemm(const MergeDesc* __restrict__ merges, int N, DcWork W, int cmin) {
  const MergeDesc mg = merges[blockIdx.z];
  const int r0 = blockIdx.x * DG_T, c0 = blockIdx.y * DG_T;
  const int lo = mg.lo, K = mg.hi - mg.lo, n1 = mg.mid - mg.lo;
  const int Kp = W.Kp[lo];
  if (r0 >= K || c0 >= K) return;
  __shared__ double As[DG_T][DG_T + 1], Bs[DG_T][DG_T + 1];
  __shared__ int srank[DG_T];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  int want = 0;
  if (threadIdx.x < DG_T) {
    const int c = c0 + threadIdx.x;
    const int r = c < K ? W.rank[lo + c] : -1;
    srank[threadIdx.x] = r >= cmin ? r : -1;
    want = r >= cmin;
  }
  if (!__syncthreads_or(want)) return;
  const int g1 = W.gcnt[2 * lo], g2 = W.gcnt[2 * lo + 1];
  int kb = 0, ke = Kp;
  if (r0 + DG_T <= n1) ke = g1 + g2;        // rows of child 1 only
  else if (r0 >= n1) kb = g1;               // rows of child 2 only
  const int* gp = W.gperm + lo;
  const bool a2 = r0 + 16 < K, b2 = c0 + 16 < Kp;
  double acc[2][2] = {{0, 0}, {0, 0}};
  if (c0 < Kp) {
    for (int k0 = kb; k0 < ke; k0 += DG_T) {
      for (int e2 = threadIdx.x; e2 < DG_T * DG_T; e2 += 256) {
        const int i32 = e2 % DG_T, o32 = e2 / DG_T;
        // A tile: consecutive threads take consecutive rows of one column
        {
          const int row = r0 + i32, kidx = k0 + o32;
          As[o32][i32] = (row < K && kidx < ke) ? W.Q[(size_t)W.colk[lo + gp[kidx]] * N + lo + row] : 0.0;
        }
        // B tile: consecutive threads take consecutive poles of one eigenvector column
        {
          const int kidx = k0 + i32, ci = c0 + o32;
          Bs[i32][o32] = (ci < Kp && kidx < ke) ? W.Delta[(size_t)(lo + ci) * N + lo + gp[kidx]] : 0.0;
        }
      }
      __syncthreads();
      const int kn = min(DG_T, ke - k0);
      if (a2 && b2) {
#pragma unroll 4
        for (int kk = 0; kk < kn; ++kk)
#pragma unroll
          for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) acc[a][b] = fma(As[kk][ty + 16 * a], Bs[kk][tx + 16 * b], acc[a][b]);
      } else if (a2) {
#pragma unroll 4
        for (int kk = 0; kk < kn; ++kk)
#pragma unroll
          for (int a = 0; a < 2; ++a) acc[a][0] = fma(As[kk][ty + 16 * a], Bs[kk][tx], acc[a][0]);
      } else if (b2) {
#pragma unroll 4
        for (int kk = 0; kk < kn; ++kk)
#pragma unroll
          for (int b = 0; b < 2; ++b) acc[0][b] = fma(As[kk][ty], Bs[kk][tx + 16 * b], acc[0][b]);
      } else {
#pragma unroll 4
        for (int kk = 0; kk < kn; ++kk) acc[0][0] = fma(As[kk][ty], Bs[kk][tx], acc[0][0]);
      }
      __syncthreads();
    }
  }
  // through shared memory, so that consecutive threads store consecutive rows
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) As[tx + 16 * b][ty + 16 * a] = acc[a][b];
  __syncthreads();
  for (int e2 = threadIdx.x; e2 < DG_T * DG_T; e2 += 256) {
    const int rr = e2 % DG_T, cc = e2 / DG_T, row = r0 + rr, c = c0 + cc, r = srank[cc];
    if (row >= K || r < 0) continue;
    W.Qtmp[(size_t)(lo + r) * N + lo + row] =
        c < Kp ? As[cc][rr] : W.Q[(size_t)W.cold[lo + (c - Kp)] * N + lo + row];
  }
}

// All phases of a merge of order at most DC_SMALL_K in one block (one block per merge of the level):
// the levels near the leaves have many small merges, where six launches per level cost more than the
// work.  The phases run in the order of the per-phase kernels, separated by block barriers; every phase
// touches only the merge's own rows and columns.  Roots, z entries and eigenvector columns are taken by
// groups of L lanes; the child eigenvectors and U are multiplied out of shared memory.  Blocks beyond the
// merges (the first level's launch has them) run the back-transformation's bt_tmat, which depends on the
// tridiagonalisation alone.
constexpr int DC_SMALL_K = 40;
inline size_t small_smem_bytes(int K) { return prep_smem_bytes(K) + (size_t)2 * K * (K + 1) * sizeof(double); }
__device__ void bt_tmat(const double* A, int lda, const double* tau, int N, int g, double* Tm, float2* Vff, float2* Tff);
struct TmatArgs { const double* A; int lda; const double* tau; double* Tm; float2 *Vff, *Tff; };

template <int L>
__device__ __forceinline__ void dc_small_roots(int lo, int K, int N, DcWork W, const MergeDesc mg, int* err) {
  const int grp = threadIdx.x / L, lane = threadIdx.x % L, ngrp = blockDim.x / L;
  const unsigned gmask = (L == 32 ? 0xffffffffu : ((1u << L) - 1u)) << ((threadIdx.x & 31) & ~(L - 1));
  const int Kp = W.Kp[lo];
  for (int i = grp; i < Kp; i += ngrp) dc_secular_root<L>(lo, i, N, W, err, lane, gmask);
  __syncthreads();
  for (int j = grp; j < K; j += ngrp) {
    dc_zhat_one<L>(lo, j, N, W, lane, gmask);
    dc_rank_one<L>(mg, j, W, lane, gmask);
  }
  __syncthreads();
  for (int i = grp; i < Kp; i += ngrp) dc_vecs_one<L>(lo, i, N, W, lane, gmask);
  __syncthreads();
}
__global__ void __launch_bounds__(DC_THREADS)
k_dc_small(const MergeDesc* __restrict__ merges, int nm, const double* __restrict__ e, int N, DcWork W, int* err,
           TmatArgs ta) {
  extern __shared__ double ssm[];
  if ((int)blockIdx.x >= nm) {
    bt_tmat(ta.A, ta.lda, ta.tau, N, blockIdx.x - nm, ta.Tm, ta.Vff, ta.Tff);
    return;
  }
  const MergeDesc mg = merges[blockIdx.x];
  const int lo = mg.lo, K = mg.hi - mg.lo, n1 = mg.mid - mg.lo;
  dc_prep(mg, e, N, W, ssm);
  __syncthreads();
  for (int row = threadIdx.x; row < K; row += blockDim.x) dc_rot_row(mg, N, W, row);
  __syncthreads();
  if (K <= DC_THREADS / 8) dc_small_roots<8>(lo, K, N, W, mg, err);
  else dc_small_roots<4>(lo, K, N, W, mg, err);
  const int Kp = W.Kp[lo], g1 = W.gcnt[2 * lo], g2 = W.gcnt[2 * lo + 1], ld = K + 1;
  double* Qs = ssm + prep_smem_bytes(K) / sizeof(double);
  double* Us = Qs + (size_t)K * ld;
  const int* gp = W.gperm + lo;
  for (int x = threadIdx.x; x < Kp * K; x += blockDim.x) {     // kept columns and U in support order
    const int row = x % K, q = x / K, g = gp[q];
    Qs[q * ld + row] = W.Q[(size_t)W.colk[lo + g] * N + lo + row];
    if (row < Kp) Us[row * ld + q] = W.Delta[(size_t)(lo + row) * N + lo + g];
  }
  __syncthreads();
  for (int x = threadIdx.x; x < K * K; x += blockDim.x) {
    const int row = x % K, c = x / K;
    double v;
    if (c < Kp) {
      const int kb = row < n1 ? 0 : g1, ke = row < n1 ? g1 + g2 : Kp;
      v = 0.0;
      for (int q = kb; q < ke; ++q) v = fma(Qs[q * ld + row], Us[c * ld + q], v);
    } else {
      v = W.Q[(size_t)W.cold[lo + (c - Kp)] * N + lo + row];
    }
    W.Qtmp[(size_t)(lo + W.rank[lo + c]) * N + lo + row] = v;
  }
}

// ---- double-FP32 arithmetic (pairs hi + lo of FP32 numbers).  The _rn intrinsics keep the compiler
// from contracting the error-free transformations into FMAs.
__device__ __forceinline__ float2 ff_from_double(double x) {
  const float h = __double2float_rn(x);
  return make_float2(h, __double2float_rn(x - (double)h));
}
// (s, c) <- (s, c) + (s2, c2): two_sum of the leading terms (Knuth), errors into the compensation
__device__ __forceinline__ void ff_acc_add(float& s, float& c, float s2, float c2) {
  const float t = __fadd_rn(s, s2);
  const float bb = __fsub_rn(t, s);
  const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(s2, bb));
  s = t;
  c = __fadd_rn(__fadd_rn(c, c2), e);
}
// (s, c) <- (s, c) + a b: the product of the leading parts exactly (its error by FMA), the cross
// terms into its error, the lo * lo term (2^-48 relative) dropped
__device__ __forceinline__ void ff_fma_acc(float& s, float& c, float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  float pe = __fmaf_rn(a.x, b.x, -p);
  pe = __fmaf_rn(a.x, b.y, pe);
  pe = __fmaf_rn(a.y, b.x, pe);
  ff_acc_add(s, c, p, pe);
}
// normalised pair of s + c (two_sum, valid for any magnitudes)
__device__ __forceinline__ float2 ff_norm(float s, float c) {
  const float h = __fadd_rn(s, c);
  const float bb = __fsub_rn(h, s);
  const float l = __fadd_rn(__fsub_rn(s, __fsub_rn(h, bb)), __fsub_rn(c, bb));
  return make_float2(h, l);
}
// z - (s + c)
__device__ __forceinline__ float2 ff_sub(float2 z, float s, float c) {
  float hs = z.x, cs = z.y;
  ff_acc_add(hs, cs, -s, -c);
  return ff_norm(hs, cs);
}

// Back-transformation of the top columns through the reflectors, RB reflectors at a time in the
// compact WY form: H_k0 H_k0+1 ... H_k0+RB-1 = I - V T V^T (V the RB reflectors, T upper
// triangular).  A block owns CB output columns; per group it stages V in shared memory once for
// all its columns, forms Y = V^T Z (RB x CB dots), Y <- T Y, and Z -= V Y.
constexpr int RB = 16;
constexpr int CB = 4;

// T of every group (one block per group): T_ii = tau_i, T[0:i, i] = -tau_i T[0:i, 0:i] V[:, 0:i]^T v_i.
// The RB (RB - 1) / 2 reflector dots are spread over the warps.
__device__ void bt_tmat(const double* __restrict__ A, int lda, const double* __restrict__ tau, int N, int g,
                        double* __restrict__ Tm, float2* __restrict__ Vff, float2* __restrict__ Tff) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int nref = N - 2;
  const int k0 = g * RB, nb = min(RB, nref - k0);
  __shared__ double vv[RB][RB];
  for (int pr = warp; pr < RB * RB; pr += nw) {
    const int a = pr / RB, b = pr - a * RB;
    if (!(a < b && b < nb)) continue;
    const double* va = A + (size_t)(k0 + a) * lda;
    const double* vb = A + (size_t)(k0 + b) * lda;
    double acc = 0.0;
    for (int row = k0 + b + 1 + lane; row < N; row += 32) acc = fma(va[row], vb[row], acc);
    acc = warp_sum(acc);
    if (lane == 0) vv[a][b] = acc;
  }
  __syncthreads();
  // T column by column: thread r < i forms T[r][i] from the finished columns 0 .. i-1
  __shared__ double Ts[RB][RB];
  for (int e = threadIdx.x; e < RB * RB; e += blockDim.x) Ts[e / RB][e % RB] = 0.0;
  __syncthreads();
  for (int i = 0; i < nb; ++i) {
    const double ti = tau[k0 + i];
    const int r = threadIdx.x;
    if (r < i) {
      double acc = 0.0;
      for (int c = r; c < i; ++c) acc = fma(Ts[r][c], vv[c][i], acc);
      Ts[r][i] = -ti * acc;
    } else if (r == i) {
      Ts[i][i] = ti;
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < RB * RB; e += blockDim.x) Tm[(size_t)g * RB * RB + e] = Ts[e / RB][e % RB];
  if (Vff) {
    // the group's reflectors (zero outside their support) and T as double-FP32 pairs, for
    // k_backtransform_ff: converted once here instead of in every block of the back-transform, and scaled to
    // v_0 = 1 (T by v_0 on both sides), which keeps the pairs in FP32's range
    __shared__ double v0[RB], r0[RB];
    if (threadIdx.x < RB) {
      const double x = threadIdx.x < nb ? A[(size_t)(k0 + threadIdx.x) * lda + k0 + threadIdx.x + 1] : 1.0;
      v0[threadIdx.x] = x;
      r0[threadIdx.x] = 1.0 / x;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < RB * RB; e += blockDim.x)
      Tff[(size_t)g * RB * RB + e] = ff_from_double(Ts[e / RB][e % RB] * v0[e / RB] * v0[e % RB]);
    for (int e = threadIdx.x; e < RB * N; e += blockDim.x) {
      const int a = e / N, row = e - a * N;
      const double x = (a < nb && row >= k0 + a + 1) ? A[(size_t)(k0 + a) * lda + row] * r0[a] : 0.0;
      Vff[((size_t)g * RB + a) * N + row] = ff_from_double(x);
    }
  }
}

// One block per CB output columns (descending eigenvalue order: column c holds Q[:, N-1-c]); 4, or 2 where 4
// leave SMs without a block: the columns' FP64 work is what a group costs (N = 288, 256 columns: 64 blocks of
// 4 took 245 us, 128 blocks of 2 take 200 us).
template <class T, int CB>
__global__ void __launch_bounds__(256)
k_backtransform(const double* __restrict__ A, int lda, const double* __restrict__ Tm, int N,
                const double* __restrict__ Q, const double* __restrict__ lam, int nkeep,
                double* __restrict__ w, T* __restrict__ U, int ldu) {
  extern __shared__ double bsm[];
  double* Vs = bsm;                      // RB x N, the group's reflectors (zero outside support)
  double* Z = bsm + (size_t)RB * N;      // CB x N, the columns being transformed
  __shared__ double Y[RB][CB], Yt[RB][CB];
  const int c0 = blockIdx.x * CB;
  const int ncol = min(CB, nkeep - c0);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int e = threadIdx.x; e < CB * N; e += blockDim.x) {
    const int c = e / N, t = e - c * N;
    Z[e] = (c < ncol) ? Q[(size_t)(N - 1 - (c0 + c)) * N + t] : 0.0;
  }
  const int nref = N - 2, ng = (nref + RB - 1) / RB;
  for (int g = ng - 1; g >= 0; --g) {
    const int k0 = g * RB, nb = min(RB, nref - k0), r0 = k0 + 1, L = N - r0;
    __syncthreads();
    for (int e = threadIdx.x; e < RB * L; e += blockDim.x) {
      const int a = e / L, row = r0 + (e - a * L);
      Vs[(size_t)a * N + row] = (a < nb && row >= k0 + a + 1) ? A[(size_t)(k0 + a) * lda + row] : 0.0;
    }
    __syncthreads();
    // Y = V^T Z: warp w takes reflectors 2w, 2w + 1 for all CB columns, 2 * CB = 8 partial dots
    // per lane, summed over the warp by a transposing butterfly (each exchange halves the values a
    // lane holds; 9 adds per lane instead of 5 per dot)
    {
      static_assert(RB == 16 && (CB == 4 || CB == 2), "the butterfly assumes 16 reflectors over 8 warps");
      const int a0 = 2 * warp;
      double acc[2 * CB];
#pragma unroll
      for (int u = 0; u < 2 * CB; ++u) acc[u] = 0.0;
      const double* va0 = Vs + (size_t)a0 * N;
      const double* va1 = va0 + N;
      for (int row = r0 + lane; row < N; row += 32) {
        const double x0 = va0[row], x1 = va1[row];
#pragma unroll
        for (int c = 0; c < CB; ++c) {
          const double z = Z[(size_t)c * N + row];
          acc[c] = fma(x0, z, acc[c]);
          acc[CB + c] = fma(x1, z, acc[CB + c]);
        }
      }
      int idx = 0, o = 16;
#pragma unroll
      for (int nv = 2 * CB; nv > 1; nv >>= 1, o >>= 1) {
        const bool up = lane & o;
        idx = 2 * idx + up;
#pragma unroll
        for (int u = 0; u < nv / 2; ++u) {
          const double send = up ? acc[u] : acc[u + nv / 2];
          const double keep = up ? acc[u + nv / 2] : acc[u];
          acc[u] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      }
      const int last = o;                     // lanes that differ below here hold parts of the same dot
#pragma unroll
      for (; o > 0; o >>= 1) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
      if ((lane & (2 * last - 1)) == 0) Y[a0 + idx / CB][idx % CB] = acc[0];   // idx = CB (a - a0) + c
    }
    __syncthreads();
    // Yt = T Y (T upper triangular), then Z -= V Yt
    if (threadIdx.x < RB * CB) {
      const int i = threadIdx.x / CB, c = threadIdx.x - i * CB;
      const double* Tg = Tm + (size_t)g * RB * RB + i * RB;
      double acc = 0.0;
      for (int j = i; j < RB; ++j) acc = fma(Tg[j], Y[j][c], acc);
      Yt[i][c] = acc;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < CB * L; e += blockDim.x) {
      const int c = e / L, row = r0 + (e - c * L);
      double upd = 0.0;
#pragma unroll
      for (int a = 0; a < RB; ++a) upd = fma(Vs[(size_t)a * N + row], Yt[a][c], upd);
      Z[(size_t)c * N + row] -= upd;
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < ncol * N; e += blockDim.x) {
    const int c = e / N, t = e - c * N;
    U[(size_t)(c0 + c) * ldu + t] = T(Z[e]);
  }
  if (threadIdx.x < ncol) w[c0 + threadIdx.x] = lam[N - 1 - (c0 + threadIdx.x)];
}

// The same back-transformation in double-FP32 arithmetic, for callers that round U to FP32: every
// value is an unevaluated pair hi + lo of FP32 numbers (about 48 significant bits), products are
// formed exactly by FMA and sums carry their rounding errors in a compensation term (the Dot2 scheme
// of Ogita, Rump and Oishi), so each dot product is as accurate as if computed in twice FP32's
// precision.  It runs on the FP32 pipe (128 lanes per SM per clock against FP64's 1.67 FMA), so it
// is several times faster than the FP64 kernel; its error in U (about 1e-14 relative) stays far
// below the FP32 rounding that the FP32-based modes apply to U next.  Same grouping as
// k_backtransform (RB reflectors in compact WY form per group, CB output columns per block); the
// next group's reflectors are copied into the other half of a double buffer (cp.async) while the
// current group is applied, and in Z -= V Yt each thread owns rows and updates all CB columns of a
// row together (CB independent accumulations sharing the V loads).
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void cp_async8(void* sdst, const void* gsrc) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(sdst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING> __device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}

__global__ void __launch_bounds__(256)
k_backtransform_ff(const float2* __restrict__ Vff, const float2* __restrict__ Tff, int N,
                   const double* __restrict__ Q, const double* __restrict__ lam, int nkeep,
                   double* __restrict__ w, double* __restrict__ U, int ldu) {
  extern __shared__ float2 bsf[];
  // bsf: two buffers of RB x N (the reflectors of a group), then Z
  float2* Z = bsf + (size_t)2 * RB * N;            // CB x N, the columns being transformed
  __shared__ float2 Y[RB][CB], Yt[RB][CB];
  const int c0 = blockIdx.x * CB;
  const int ncol = min(CB, nkeep - c0);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nref = N - 2, ng = (nref + RB - 1) / RB;
  // rows [g RB + 1, N) of the RB reflectors of group g into buffer b (the rest of the group's
  // column range is zero and never read)
  auto stage = [&](int g, int b) {
    const int r0 = g * RB + 1, L = N - r0;
    float2* dst = bsf + (size_t)b * RB * N;
    for (int e = threadIdx.x; e < RB * L; e += blockDim.x) {
      const int a = e / L, row = r0 + (e - a * L);
      cp_async8(dst + (size_t)a * N + row, Vff + ((size_t)g * RB + a) * N + row);
    }
    cp_async_commit();
  };
  stage(ng - 1, (ng - 1) & 1);
  for (int e = threadIdx.x; e < CB * N; e += blockDim.x) {
    const int c = e / N, t = e - c * N;
    Z[e] = (c < ncol) ? ff_from_double(Q[(size_t)(N - 1 - (c0 + c)) * N + t]) : make_float2(0.f, 0.f);
  }
  for (int g = ng - 1; g >= 0; --g) {
    const int k0 = g * RB, r0 = k0 + 1;
    const float2* Vs = bsf + (size_t)(g & 1) * RB * N;
    if (g > 0) {
      stage(g - 1, (g - 1) & 1);   // its buffer was last read in the previous iteration (synced below)
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    // Y = V^T Z: warp w takes reflectors 2w, 2w + 1 for all CB columns; the 8 (sum, compensation)
    // pairs of a lane are combined over the warp by a transposing butterfly
    {
      static_assert(RB == 16 && CB == 4, "the butterfly assumes 16 reflectors over 8 warps and 4 columns");
      const int a0 = 2 * warp;
      float sa[8], ca[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) { sa[u] = 0.f; ca[u] = 0.f; }
      const float2* va0 = Vs + (size_t)a0 * N;
      const float2* va1 = va0 + N;
      for (int row = r0 + lane; row < N; row += 32) {
        const float2 x0 = va0[row], x1 = va1[row];
#pragma unroll
        for (int c = 0; c < CB; ++c) {
          const float2 z = Z[(size_t)c * N + row];
          ff_fma_acc(sa[c], ca[c], x0, z);
          ff_fma_acc(sa[CB + c], ca[CB + c], x1, z);
        }
      }
      const bool b16 = lane & 16, b8 = lane & 8, b4 = lane & 4;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float ss = b16 ? sa[u] : sa[u + 4], cs = b16 ? ca[u] : ca[u + 4];
        const float sk = b16 ? sa[u + 4] : sa[u], ck = b16 ? ca[u + 4] : ca[u];
        sa[u] = sk; ca[u] = ck;
        ff_acc_add(sa[u], ca[u], __shfl_xor_sync(0xffffffffu, ss, 16), __shfl_xor_sync(0xffffffffu, cs, 16));
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float ss = b8 ? sa[u] : sa[u + 2], cs = b8 ? ca[u] : ca[u + 2];
        const float sk = b8 ? sa[u + 2] : sa[u], ck = b8 ? ca[u + 2] : ca[u];
        sa[u] = sk; ca[u] = ck;
        ff_acc_add(sa[u], ca[u], __shfl_xor_sync(0xffffffffu, ss, 8), __shfl_xor_sync(0xffffffffu, cs, 8));
      }
      {
        const float ss = b4 ? sa[0] : sa[1], cs = b4 ? ca[0] : ca[1];
        const float sk = b4 ? sa[1] : sa[0], ck = b4 ? ca[1] : ca[0];
        sa[0] = sk; ca[0] = ck;
        ff_acc_add(sa[0], ca[0], __shfl_xor_sync(0xffffffffu, ss, 4), __shfl_xor_sync(0xffffffffu, cs, 4));
      }
      ff_acc_add(sa[0], ca[0], __shfl_xor_sync(0xffffffffu, sa[0], 2), __shfl_xor_sync(0xffffffffu, ca[0], 2));
      ff_acc_add(sa[0], ca[0], __shfl_xor_sync(0xffffffffu, sa[0], 1), __shfl_xor_sync(0xffffffffu, ca[0], 1));
      if ((lane & 3) == 0) {
        const int idx = (b16 ? 4 : 0) + (b8 ? 2 : 0) + (b4 ? 1 : 0);   // = 4 * (a - a0) + c
        Y[a0 + (idx >> 2)][idx & 3] = ff_norm(sa[0], ca[0]);
      }
    }
    __syncthreads();
    // Yt = T Y (T upper triangular): output (i, c) by the 4 threads of a quad, each summing every
    // fourth term, combined by two shuffles
    {
      const int o = threadIdx.x >> 2, part = threadIdx.x & 3;   // 64 outputs x 4 parts = 256 threads
      const int i = o / CB, c = o - i * CB;
      const float2* Tg = Tff + (size_t)g * RB * RB + i * RB;
      float sacc = 0.f, cacc = 0.f;
      for (int j = i + part; j < RB; j += 4) ff_fma_acc(sacc, cacc, Tg[j], Y[j][c]);
      ff_acc_add(sacc, cacc, __shfl_xor_sync(0xffffffffu, sacc, 1), __shfl_xor_sync(0xffffffffu, cacc, 1));
      ff_acc_add(sacc, cacc, __shfl_xor_sync(0xffffffffu, sacc, 2), __shfl_xor_sync(0xffffffffu, cacc, 2));
      if (part == 0) Yt[i][c] = ff_norm(sacc, cacc);
    }
    __syncthreads();
    // Z -= V Yt: two rows per thread at a time, CB columns each (2 CB independent accumulations)
    for (int row = r0 + threadIdx.x; row < N; row += 2 * blockDim.x) {
      const int row2 = row + blockDim.x;
      const bool two = row2 < N;
      float sacc[2][CB], cacc[2][CB];
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int c = 0; c < CB; ++c) { sacc[h][c] = 0.f; cacc[h][c] = 0.f; }
#pragma unroll
      for (int a = 0; a < RB; ++a) {
        const float2 v0 = Vs[(size_t)a * N + row];
        const float2 v1 = two ? Vs[(size_t)a * N + row2] : make_float2(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < CB; ++c) {
          const float2 y = Yt[a][c];
          ff_fma_acc(sacc[0][c], cacc[0][c], v0, y);
          ff_fma_acc(sacc[1][c], cacc[1][c], v1, y);
        }
      }
#pragma unroll
      for (int c = 0; c < CB; ++c) {
        float2& z = Z[(size_t)c * N + row];
        z = ff_sub(z, sacc[0][c], cacc[0][c]);
        if (two) {
          float2& z2 = Z[(size_t)c * N + row2];
          z2 = ff_sub(z2, sacc[1][c], cacc[1][c]);
        }
      }
    }
    __syncthreads();   // every thread is done with Vs before it is refilled two groups later
  }
  for (int e = threadIdx.x; e < ncol * N; e += blockDim.x) {
    const int c = e / N, t = e - c * N;
    const float2 z = Z[e];
    U[(size_t)(c0 + c) * ldu + t] = (double)z.x + (double)z.y;   // exact: 48 bits fit in FP64
  }
  if (threadIdx.x < ncol) w[c0 + threadIdx.x] = lam[N - 1 - (c0 + threadIdx.x)];
}

// ------------------------------------------------------------------------------------ host side
struct Plan {
  std::vector<MergeDesc> merges;      // all levels, deepest first
  std::vector<int> level_off;         // offsets into merges per level (+ end)
  std::vector<int> mergeof;           // per level: N entries
};

void build_plan(int N, Plan& pl) {
  std::vector<std::vector<MergeDesc>> by_depth;
  struct Node { int lo, hi, depth; };
  std::vector<Node> stack{{0, N, 0}};
  while (!stack.empty()) {
    Node nd = stack.back();
    stack.pop_back();
    if (nd.hi - nd.lo <= 1) continue;
    int mid = (nd.lo + nd.hi) / 2;
    if ((int)by_depth.size() <= nd.depth) by_depth.resize(nd.depth + 1);
    by_depth[nd.depth].push_back({nd.lo, mid, nd.hi});
    stack.push_back({nd.lo, mid, nd.depth + 1});
    stack.push_back({mid, nd.hi, nd.depth + 1});
  }
  pl.merges.clear();
  pl.level_off.clear();
  pl.mergeof.clear();
  for (int dpt = (int)by_depth.size() - 1; dpt >= 0; --dpt) {
    pl.level_off.push_back((int)pl.merges.size());
    std::vector<int> mo(N, -1);
    int base = (int)pl.merges.size();
    for (size_t q = 0; q < by_depth[dpt].size(); ++q) {
      const MergeDesc& m = by_depth[dpt][q];
      for (int t = m.lo; t < m.hi; ++t) mo[t] = (int)q;
      pl.merges.push_back(m);
    }
    (void)base;
    pl.mergeof.insert(pl.mergeof.end(), mo.begin(), mo.end());
  }
  pl.level_off.push_back((int)pl.merges.size());
}

struct PlanCacheEntry {
  MergeDesc* d_merges = nullptr;
  int* d_mergeof = nullptr;
  Plan plan;
};

std::mutex g_plan_mu;
std::map<std::pair<int, int>, PlanCacheEntry> g_plans;   // (device, N)

const PlanCacheEntry* get_plan(int N) {
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lk(g_plan_mu);
  auto key = std::make_pair(dev, N);
  auto it = g_plans.find(key);
  if (it != g_plans.end()) return &it->second;
  PlanCacheEntry ent;
  build_plan(N, ent.plan);
  size_t nm = std::max<size_t>(1, ent.plan.merges.size());
  size_t nmo = std::max<size_t>(1, ent.plan.mergeof.size());
  if (cudaMalloc(&ent.d_merges, nm * sizeof(MergeDesc)) != cudaSuccess) return nullptr;
  if (cudaMalloc(&ent.d_mergeof, nmo * sizeof(int)) != cudaSuccess) return nullptr;
  if (!ent.plan.merges.empty())
    cudaMemcpy(ent.d_merges, ent.plan.merges.data(), ent.plan.merges.size() * sizeof(MergeDesc), cudaMemcpyHostToDevice);
  if (!ent.plan.mergeof.empty())
    cudaMemcpy(ent.d_mergeof, ent.plan.mergeof.data(), ent.plan.mergeof.size() * sizeof(int), cudaMemcpyHostToDevice);
  auto res = g_plans.emplace(key, std::move(ent));
  return &res.first->second;
}

inline size_t align_up(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

// Workspace of every order up to nmax: each part grows with the order.  (The exchange slots of the
// tridiagonalisation, whose replicas drop from 4 to 1 above order 1,024, have no part of their own: they lie over
// Q, Qtmp, Delta and the reflector groups, at least 4 N^2 + 17 N words that are first written after it.)
size_t eig_workspace_bytes(int nmax) {
  size_t N = std::max(nmax, 1);
  size_t b = 0;
  b += align_up((3 * N + 1) * sizeof(double));    // d, e, tau, largest magnitude
  b += 3 * align_up(N * N * sizeof(double));      // Q, Qtmp, Delta
  b += align_up((N / RB + 2) * RB * N * sizeof(float2));    // reflector groups as double-FP32 pairs
  b += 10 * align_up(N * sizeof(double));         // lam, lamk, Df, zf, Zw, Dk, Zk, Dd, rho, z2
  b += align_up(4 * N * sizeof(double));          // rot
  b += align_up((N / RB + 2) * RB * RB * sizeof(double));   // back-transform T blocks
  b += align_up((N / RB + 2) * RB * RB * sizeof(float2));   // T blocks as double-FP32 pairs
  b += 7 * align_up(N * sizeof(int));             // colk, cold, rank, Kp, nrot, gperm, spare
  b += align_up(2 * N * sizeof(int));             // gcnt
  return b + 4096;
}

template <class T>
int eig_sym_topk(double* A, int lda, int N, int nkeep, double* w, T* U, int ldu, void* work, size_t work_bytes,
                 int* err, cudaStream_t st, cudaEvent_t* marks, int assembly) {
  if (N <= 0 || nkeep <= 0) return 0;
  if (nkeep > N) nkeep = N;
  if (work_bytes < eig_workspace_bytes(N)) return 1;
  const PlanCacheEntry* pe = get_plan(N);
  if (!pe) return 2;
  char* p = (char*)work;
  auto take = [&](size_t bytes) { void* q = p; p += align_up(bytes); return q; };
  double* d = (double*)take((3 * (size_t)N + 1) * sizeof(double));
  double* e = d + N;
  double* tau = e + N;
  unsigned long long* amax = (unsigned long long*)(tau + N);
  DcWork W;
  W.Q = (double*)take((size_t)N * N * sizeof(double));
  W.Qtmp = (double*)take((size_t)N * N * sizeof(double));
  W.Delta = (double*)take((size_t)N * N * sizeof(double));
  float2* Vff = (float2*)take(((size_t)N / RB + 2) * RB * (size_t)N * sizeof(float2));
  double* slots = W.Q;
  const size_t slot_bytes = td_replicas(N) * (size_t)N * (N + 1) * sizeof(double);
  W.lam = (double*)take(N * sizeof(double));
  W.lamk = (double*)take(N * sizeof(double));
  W.Df = (float2*)take(N * sizeof(float2));
  W.zf = (float*)take(N * sizeof(double));
  W.Zw = (double*)take(N * sizeof(double));
  W.Dk = (double*)take(N * sizeof(double));
  W.Zk = (double*)take(N * sizeof(double));
  W.Dd = (double*)take(N * sizeof(double));
  W.rho = (double*)take(N * sizeof(double));
  W.z2 = (double*)take(N * sizeof(double));
  W.rot = (double*)take(4 * N * sizeof(double));
  W.Tm = (double*)take(((size_t)N / RB + 2) * RB * RB * sizeof(double));
  float2* Tff = (float2*)take(((size_t)N / RB + 2) * RB * RB * sizeof(float2));
  W.colk = (int*)take(N * sizeof(int));
  W.cold = (int*)take(N * sizeof(int));
  W.rank = (int*)take(N * sizeof(int));
  W.Kp = (int*)take(N * sizeof(int));
  W.nrot = (int*)take(N * sizeof(int));
  W.gperm = (int*)take(N * sizeof(int));
  W.gcnt = (int*)take(2 * N * sizeof(int));
  W.mergeof = nullptr;

  cudaMemsetAsync(slots, 0xFF, slot_bytes, st);      // every slot empty
  cudaMemsetAsync(d, 0, (3 * (size_t)N + 1) * sizeof(double), st);
  k_absmax<<<std::min(N, 304), 256, 0, st>>>(A, lda, N, amax); note_launch();

  // 1. tridiagonalisation (cooperative: all blocks co-resident)
  {
    const void* fn = td_replicas(N) == 4 ? (const void*)k_tridiag<4> : (const void*)k_tridiag<1>;
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    int G = N >= 3 ? std::max(1, std::min(nsm, (N + 1) / 2)) : 1;
    cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    size_t smem = 0;
    for (int attempt = 0; attempt < 8; ++attempt) {
      const int nslot = (N + G - 1) / G;
      smem = (5 + (size_t)nslot) * N * sizeof(double);
      cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)std::max<size_t>(smem, 48 * 1024));
      int occ = 0;
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, TD_THREADS, smem);
      if ((long long)occ * nsm >= G) break;
      G = std::max(1, occ * nsm);     // fewer blocks own more columns each
      if (occ == 0) { cudaGetLastError(); return 1000 + (int)cudaErrorCooperativeLaunchTooLarge; }
    }
    if ((N + G - 1) / G > TD_MAX_SLOTS) return 1000 + (int)cudaErrorInvalidValue;
    long long poll_limit = wait_limit(kPollLimit);
    void* args[] = {&A, &lda, &N, &d, &e, &tau, &slots, &amax, &err, &poll_limit};
    cudaError_t ce = cudaLaunchCooperativeKernel(fn, dim3(G), dim3(TD_THREADS), args, smem, st);
    note_launch();
    if (ce != cudaSuccess) return 1000 + (int)ce;
  }
  if (marks) cudaEventRecord(marks[0], st);
  // 2. divide and conquer; the T matrices of the back-transformation ride on the first launch of small merges
  const bool ff = sizeof(T) == sizeof(double) && assembly == kAssemblyFF && N >= 3 &&
                  (size_t)(2 * RB + CB) * N * sizeof(float2) <= 227 * 1024;   // (the double-buffered staging fits)
  const TmatArgs ta{A, lda, tau, W.Tm, ff ? Vff : nullptr, ff ? Tff : nullptr};
  int tmat_blocks = N >= 3 ? (N - 2 + RB - 1) / RB : 0;
  k_dc_init<<<dim3((N + 255) / 256, N), 256, 0, st>>>(d, e, N, W.lam, W.Q, W.Qtmp); note_launch();
  const Plan& pl = pe->plan;
  const int nlev = (int)pl.level_off.size() - 1;
  for (int lv = 0; lv < nlev; ++lv) {
    const int m0 = pl.level_off[lv], m1 = pl.level_off[lv + 1];
    const int nm = m1 - m0;
    if (nm <= 0) continue;
    const MergeDesc* dm = pe->d_merges + m0;
    const int* dmo = pe->d_mergeof + (size_t)lv * N;
    int kmax = 0;
    for (int q = m0; q < m1; ++q) kmax = std::max(kmax, pl.merges[q].hi - pl.merges[q].lo);
    if (kmax <= DC_SMALL_K) {
      k_dc_small<<<nm + tmat_blocks, DC_THREADS, small_smem_bytes(kmax), st>>>(dm, nm, e, N, W, err, ta); note_launch();
      tmat_blocks = 0;
      std::swap(W.Q, W.Qtmp);
      continue;
    }
    const size_t psmem = prep_smem_bytes(kmax);
    if (psmem > 40 * 1024) cudaFuncSetAttribute(k_dc_prep, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psmem);
    k_dc_prep<<<nm, DC_THREADS, psmem, st>>>(dm, e, N, W); note_launch();
    k_dc_rot<<<dim3((kmax + 127) / 128, nm), 128, 0, st>>>(dm, N, W); note_launch();
    // The per-root work is FP64-bound, so the grids use two-warp blocks (one warp per root) to spread the
    // roots over all SMs.  (One thread per root for the small merges measured 3x slower: one warp per SM
    // leaves its FP64 dependency chains uncovered.)
    k_dc_secular<32><<<(N + 1) / 2, 64, 0, st>>>(dm, dmo, N, W, err); note_launch();
    k_dc_zhat<32><<<(N + 1) / 2, 64, 0, st>>>(dm, dmo, N, W); note_launch();
    k_dc_vecs<32><<<(N + 1) / 2, 64, 0, st>>>(dm, dmo, N, W); note_launch();
    dim3 gg((kmax + DG_T - 1) / DG_T, (kmax + DG_T - 1) / DG_T, nm);
    k_dc_gemm<<<gg, 256, 0, st>>>(dm, N, W, lv == nlev - 1 ? N - nkeep : 0); note_launch();
    std::swap(W.Q, W.Qtmp);
  }
  if (marks) cudaEventRecord(marks[1], st);
  // 3. back-transformation of the top nkeep columns (descending eigenvalues)
  if (ff) {
    const size_t smem = (size_t)(2 * RB + CB) * N * sizeof(float2);
    if (smem > 40 * 1024) cudaFuncSetAttribute(k_backtransform_ff, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_backtransform_ff<<<(nkeep + CB - 1) / CB, 256, smem, st>>>(Vff, Tff, N, W.Q, W.lam, nkeep, w, (double*)U, ldu); note_launch();
  } else {
    const int cb = (nkeep + 3) / 4 < 128 ? 2 : 4;
    auto fn = cb == 2 ? k_backtransform<T, 2> : k_backtransform<T, 4>;
    const size_t smem = (size_t)(RB + cb) * N * sizeof(double);
    if (smem > 40 * 1024) cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    fn<<<(nkeep + cb - 1) / cb, 256, smem, st>>>(A, lda, W.Tm, N, W.Q, W.lam, nkeep, w, U, ldu); note_launch();
  }
  return cudaGetLastError() == cudaSuccess ? 0 : 4;
}

template int eig_sym_topk<float>(double*, int, int, int, double*, float*, int, void*, size_t, int*, cudaStream_t,
                                  cudaEvent_t*, int);
template int eig_sym_topk<double>(double*, int, int, int, double*, double*, int, void*, size_t, int*, cudaStream_t,
                                   cudaEvent_t*, int);

}  // namespace cakf
