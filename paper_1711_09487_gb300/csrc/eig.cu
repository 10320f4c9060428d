// Dense symmetric eigensolver used by the Rayleigh-Ritz steps (Alg. 3 step 7 and the
// completion passes).  Textbook algorithms: Householder reduction to tridiagonal form,
// bisection on Sturm counts for the eigenvalues of the tridiagonal matrix, inverse iteration
// with Gram-Schmidt inside clusters of close eigenvalues, back-transformation.
#include "eig.cuh"
#include "dense.cuh"
#include "grid_barrier.cuh"
#include "tc_gemm.cuh"

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>

namespace rfdd {

constexpr int EIG_MAXB = 64;

struct SymBatchP {
  SymItem it[EIG_MAXB];
};

// 1/q by the hardware's approximate reciprocal refined with one Newton-Raphson step
// (r <- r + r (1 - q r)), which doubles the number of correct bits: relative error about 2^-44,
// far below what a Sturm count needs (it is a tiny backward perturbation of e_k^2).  |q| >= pivmin
// keeps q a normal number.
__device__ inline double recip_nr(double q) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(q));
  return fma(r, fma(-q, r, 1.0), r);
}

// Block-wide sum, the same value in every thread.  One thread adds the warp partials (FP64
// arithmetic is scarce on this GPU: every thread adding them would cost nw FP64 adds each).
__device__ double block_sum(double v, double *red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int q = 0; q < nw; ++q) s += red[q];
    red[32] = s;
  }
  __syncthreads();
  return red[32];
}

// Householder tridiagonalisation, one pass over the trailing block per step.  Step i reflects row
// i (columns i+1..n-1) with H_i = I - tau v v^T, v[0] = 1, H_i x = beta e_1 (LAPACK convention;
// v is kept in row i for the back-transformation); the trailing block then takes the rank-2
// update -v q^T - q v^T with p = tau H_t v, q = p - (tau/2)(p^T v) v.  The update of step i-1 is
// applied lazily: house_kernel(i) forms q_{i-1} and applies it to row i only (O(n) work: on this
// GPU one SM's FP64 rate is far too low for more), and update_symv_kernel(i) applies it to rows
// and columns i+1..n-1 while forming p_i from the updated entries, so each step reads and writes
// the trailing block once.

// Step i, part 1 (one CTA per item): q_{i-1} into qbuf, row i updated by step i-1, then the
// Householder vector of row i.
__global__ void __launch_bounds__(512) house_kernel(SymBatchP b, int i, double *qbuf, int64_t qstride) {
  SymItem it = b.it[blockIdx.x];
  const int n = it.n;
  if (i >= n) return;
  double *q = qbuf + (int64_t)blockIdx.x * qstride;
  double *row = it.H + (int64_t)i * it.ld;
  __shared__ double red[33];
  const int ip = i - 1;
  if (ip >= 0 && ip < n - 2) {
    // p_{i-1} covers rows i..n-1 (work[0..len)); v_{i-1} is row i-1 from column i on
    const int len = n - i;
    const double *v = it.H + (int64_t)ip * it.ld + i;
    double ss = 0.0;
    for (int k = threadIdx.x; k < len; k += blockDim.x) ss = fma(it.work[k], v[k], ss);
    const double K = 0.5 * it.tau[ip] * block_sum(ss, red);
    for (int k = threadIdx.x; k < len; k += blockDim.x) q[i + k] = it.work[k] - K * v[k];
    __syncthreads();
    const double vi = v[0], qi = q[i];
    for (int k = threadIdx.x; k < len; k += blockDim.x) row[i + k] = fma(-qi, v[k], fma(-vi, q[i + k], row[i + k]));
    __syncthreads();
  }
  if (i >= n - 1) {
    if (threadIdx.x == 0) { it.d[i] = row[i]; it.tau[i] = 0.0; }
    return;
  }
  const int len = n - i - 1;
  double *x = row + i + 1;
  double ss = 0.0;
  for (int k = 1 + threadIdx.x; k < len; k += blockDim.x) ss = fma(x[k], x[k], ss);
  const double sig = block_sum(ss, red);
  const double alpha = x[0];
  __shared__ double scale_s, beta_s, tau_s;
  if (threadIdx.x == 0) {
    it.d[i] = row[i];
    if (sig == 0.0) {
      tau_s = 0.0;
      beta_s = alpha;
      scale_s = 0.0;
    } else {
      const double nrm = sqrt(alpha * alpha + sig);
      const double beta = alpha <= 0.0 ? nrm : -nrm;
      tau_s = (beta - alpha) / beta;
      scale_s = 1.0 / (alpha - beta);
      beta_s = beta;
    }
    it.e[i] = beta_s;
    it.tau[i] = tau_s;
  }
  __syncthreads();
  const double sc = scale_s;
  for (int k = 1 + threadIdx.x; k < len; k += blockDim.x) x[k] *= sc;
  if (threadIdx.x == 0) x[0] = 1.0;
}

// Step i, part 2 (TRD_WPR warps per row r of the trailing block i+1..n-1): apply step i-1's rank-2
// update as two FMAs (the FP64 pipes bound this kernel; the block stays symmetric to rounding, a
// backward perturbation of the order of the update's rounding), then p_i[r] = tau_i (H_t v_i)[r]
// into work.  Runs for i <= n-2 (at i = n-2 only the pending update is left).
constexpr int TRD_WPR = 2;
__global__ void __launch_bounds__(256) update_symv_kernel(SymBatchP b, int i, const double *qbuf, int64_t qstride) {
  SymItem it = b.it[blockIdx.y];
  const int n = it.n;
  if (i > n - 2) return;
  const int len = n - i - 1;
  constexpr int TPR = 32 * TRD_WPR;                 // threads per row
  const int rloc = threadIdx.x / TPR, tr = threadIdx.x % TPR;
  const int r = blockIdx.x * (256 / TPR) + rloc;
  __shared__ double part[256 / 32];
  const int c0 = i + 1;
  const bool upd = i >= 1 && i - 1 < n - 2;
  const bool sym = i < n - 2;
  double s = 0.0;
  if (r < len) {
    double *h = it.H + (int64_t)(c0 + r) * it.ld + c0;
    const double *v = it.H + (int64_t)i * it.ld + c0;         // v_i (row i)
    const double *vp = it.H + (int64_t)(i - 1) * it.ld + c0;  // v_{i-1} from column i+1 on
    const double *q = qbuf + (int64_t)blockIdx.y * qstride + c0;
    const double vr = upd ? vp[r] : 0.0, qr = upd ? q[r] : 0.0;
    for (int c = tr; c < len; c += TPR) {
      double h0 = h[c];
      if (upd) {
        h0 = fma(-qr, vp[c], fma(-vr, q[c], h0));
        h[c] = h0;
      }
      s = fma(h0, v[c], s);
    }
  }
  if (!sym) return;  // uniform over the block
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
  __syncthreads();
  if (tr == 0 && r < len) {
    double t = 0.0;
    for (int w = 0; w < TRD_WPR; ++w) t += part[rloc * TRD_WPR + w];
    it.work[r] = it.tau[i] * t;
  }
}

// --------------------------------------------------------------------------------------
// Eigenvalues of the tridiagonal matrix by multisection on Sturm counts.  The Sturm count of x is
// the number of negative pivots of the LDL^T factorisation of T - x I (Sylvester's law).
// --------------------------------------------------------------------------------------
__device__ inline int sturm_count(const double *d, const double *e, int n, double x, double pivmin) {
  int cnt = 0;
  double q = d[0] - x;
  if (fabs(q) < pivmin) q = -pivmin;
  cnt += q < 0.0;
  for (int k = 1; k < n; ++k) {
    q = d[k] - x - e[k - 1] * e[k - 1] / q;
    if (fabs(q) < pivmin) q = -pivmin;
    cnt += q < 0.0;
  }
  return cnt;
}

// Number of eigenvalues below x.  e2[k] = e[k]^2 (tri_prep_kernel).  The FP64 pipe issues one warp
// instruction in 16 cycles, so a step has four FP64 instructions: the shift, the Newton pair and the
// recurrence; the guard |q| < pivmin and the sign are read off the high word with integer
// instructions.
__device__ __forceinline__ int sturm_count_nr(const double *__restrict__ d, const double *__restrict__ e2, int n,
                                              double x, double pivmin) {
  const int pv_hi = __double2hiint(pivmin);
  int cnt = 0;
  double q = d[0] - x;
  if ((__double2hiint(q) & 0x7fffffff) < pv_hi) q = -pivmin;
  cnt += (int)((unsigned)__double2hiint(q) >> 31);
#pragma unroll 4
  for (int k = 1; k < n; ++k) {
    q = fma(-e2[k - 1], recip_nr(q), d[k] - x);
    if ((__double2hiint(q) & 0x7fffffff) < pv_hi) q = -pivmin;
    cnt += (int)((unsigned)__double2hiint(q) >> 31);
  }
  return cnt;
}

// Per item: e2 = e^2 into work, and into info the Gershgorin bounds of the spectrum, the smallest
// pivot of the counts and the largest absolute row sum.
constexpr int TRI_INFO = 4;
__global__ void __launch_bounds__(256) tri_prep_kernel(SymBatchP b, double *info) {
  const SymItem it = b.it[blockIdx.x];
  const int n = it.n;
  double gl = INFINITY, gu = -INFINITY, em = 0.0, tn = 0.0;
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const double dk = it.d[k], el = k > 0 ? fabs(it.e[k - 1]) : 0.0, er = k < n - 1 ? fabs(it.e[k]) : 0.0;
    gl = fmin(gl, dk - (el + er));
    gu = fmax(gu, dk + (el + er));
    tn = fmax(tn, fabs(dk) + el + er);
    em = fmax(em, er * er);
    it.work[k] = er * er;
  }
  for (int o = 16; o > 0; o >>= 1) {
    gl = fmin(gl, __shfl_xor_sync(0xffffffffu, gl, o));
    gu = fmax(gu, __shfl_xor_sync(0xffffffffu, gu, o));
    em = fmax(em, __shfl_xor_sync(0xffffffffu, em, o));
    tn = fmax(tn, __shfl_xor_sync(0xffffffffu, tn, o));
  }
  __shared__ double red[4][8];
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    red[0][w] = gl;
    red[1][w] = gu;
    red[2][w] = em;
    red[3][w] = tn;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < 8; ++q) {
      gl = fmin(gl, red[0][q]);
      gu = fmax(gu, red[1][q]);
      em = fmax(em, red[2][q]);
      tn = fmax(tn, red[3][q]);
    }
    double *o = info + (int64_t)blockIdx.x * TRI_INFO;
    o[0] = gl;
    o[1] = gu;
    o[2] = 2.2250738585072014e-308 * fmax(1.0, em);
    o[3] = tn;
  }
}

// G lanes per eigenvalue: each round the lanes take the Sturm counts at G points that cut [lo, hi]
// into G + 1 equal parts, and the part holding eigenvalue i becomes the new interval (log2(G + 1)
// bits per round instead of one, at G times the counting work).  One warp per CTA: the FP64 pipe of
// an SM serves one warp as fast as it does eight, so the warps are spread over all SMs (with eight
// warps a CTA the order-120 problem ran on 4 SMs: 1.23 ms, now 0.23; order 1885 on 59: 19.8 ms, now
// 8.1).
template <int G>
__global__ void __launch_bounds__(32) bisect_kernel(SymBatchP b, const double *__restrict__ info) {
  const SymItem it = b.it[blockIdx.y];
  const int n = it.n;
  const int lane = threadIdx.x, base = lane & ~(G - 1), g = lane - base;
  const int i = blockIdx.x * (32 / G) + lane / G;  // eigenvalue index
  const unsigned gmask = (G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u)) << base;
  if (i >= n) return;  // the lanes of a group share i, so a group leaves together
  const double *f = info + (int64_t)blockIdx.y * TRI_INFO;
  const double gl = f[0], gu = f[1], pivmin = f[2];
  const double eps = 2.220446049250313e-16;
  const double span = fmax(fabs(gl), fabs(gu));
  double lo = gl - 2.0 * eps * span * n - pivmin, hi = gu + 2.0 * eps * span * n + pivmin;
  for (int round = 0; round < 100; ++round) {
    if (hi - lo <= 2.0 * eps * fmax(fabs(lo), fabs(hi)) + 4.0 * pivmin) break;
    const double step = (hi - lo) / (G + 1);
    const double x = lo + step * (g + 1);
    const bool above = (x > lo && x < hi) ? sturm_count_nr(it.d, it.work, n, x, pivmin) > i : (x >= hi);
    // the first cut point whose count exceeds i bounds the eigenvalue from above
    const unsigned m = __ballot_sync(gmask, above) & gmask;
    const int first = m ? (__ffs(m) - 1 - base) : G;
    const double nlo = first > 0 ? lo + step * first : lo;
    const double nhi = first < G ? lo + step * (first + 1) : hi;
    if (!(nlo > lo || nhi < hi)) break;  // no progress in floating point
    lo = nlo;
    hi = nhi;
  }
  if (g == 0) it.lam[i] = 0.5 * (lo + hi);
}

// Eigenvalues of the tridiagonal matrices (d, e) of the batch.  G is the lanes per eigenvalue with
// the least estimated time: rounds (52 bits at log2(G + 1) a round) times a step, which takes the
// chain of dependent instructions (about 150 cycles) or, with w warps on an SM, 64 cycles of FP64
// issue for each.
static void tridiagonal_values(cudaStream_t st, const SymBatchP &b, int cnt, int nmax) {
  double *info = nullptr;
  RFDD_CUDA(cudaMallocAsync((void **)&info, (size_t)cnt * TRI_INFO * sizeof(double), st));
  tri_prep_kernel<<<cnt, 256, 0, st>>>(b, info);
  RFDD_CHECK_LAUNCH();
  int64_t total = 0;
  for (int i = 0; i < cnt; ++i) total += b.it[i].n;
  int G = 4;
  double best = 0.0;
  for (int c = 4; c <= 32; c *= 2) {
    const double w = std::ceil((double)total * c / 32.0 / sm_count());
    const double t = std::ceil(52.0 / std::log2(c + 1.0)) * std::max(150.0, 64.0 * w);
    if (c == 4 || t < best) {
      best = t;
      G = c;
    }
  }
  const dim3 grid(ceil_div((int64_t)nmax * G, 32), cnt);
  if (G == 4) bisect_kernel<4><<<grid, 32, 0, st>>>(b, info);
  else if (G == 8) bisect_kernel<8><<<grid, 32, 0, st>>>(b, info);
  else if (G == 16) bisect_kernel<16><<<grid, 32, 0, st>>>(b, info);
  else bisect_kernel<32><<<grid, 32, 0, st>>>(b, info);
  RFDD_CHECK_LAUNCH();
  RFDD_CUDA(cudaFreeAsync(info, st));
}

// Householder reduction of every item of the batch to tridiagonal form (d, e)
//
// Up to order TRD_NMAX one cooperative launch does every step: G CTAs per item, row r of the
// trailing block held by CTA r % G (its own rows stay in that SM's L1 / L2), one barrier among the
// item's CTAs per step.  After the barrier every CTA forms q_{i-1}, the updated row i and the
// Householder vector from it for itself (O(n) work, cheaper than a second barrier), then updates its
// rows and their entries of p_i.  p alternates between two buffers, and row i takes v_i one step
// late, so that no CTA overwrites what a slower one still reads.  Bound: below order 400 the chain of
// one step (barrier, two block reductions, the reflector's scalars: about 5 us), above it the three
// FP64 operations per trailing entry (n^3 FMAs are 11 ms of the chip's FP64 rate at order 1885).
// Measured: order 120 0.63 ms (1.04 ms in 240 launches, 1.7 ms with their gaps), order 1885 27.8 ms
// (37.2 in 3769 launches, 44 with gaps).
constexpr int TRD_THREADS = 512;  // at most; 256 below order 512
constexpr int TRD_NMAX = 8192;  // three vectors of the order in shared memory
// Block-wide sum over the first nact warps, given to f by one thread of warp 0; what f leaves in
// shared memory is visible to all on return.  A warp's FP64 instruction takes 16 cycles of an SM's
// FP64 pipe, whatever its lanes do: warps without data add nothing, and the scalars that follow from
// the sum are formed by one warp (formed by all sixteen they took longer than the sum).
template <typename F>
__device__ __forceinline__ void trd_sum(double v, double *red, int nact, F &&f) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w < nact) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) red[w] = v;
  }
  __syncthreads();
  if (w == 0) {
    v = lane < nact ? red[lane] : 0.0;
    for (int o = nact > 8 ? 8 : nact > 4 ? 4 : nact > 2 ? 2 : 1; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) f(v);
  }
  __syncthreads();
}

// The Householder reflector I - tau u u^T of a vector x with first entry alpha and the sum of squares sig of
// the others: beta = -sign(alpha) ||x||, u = x - beta e_1 (first entry u0, the others those of x, which so need no
// scaling), tau = 2 / ||u||^2 = 1 / (||x|| (||x|| + |alpha|)).  1 / ||x|| and the reciprocals come from the hardware's
// approximations refined by Newton's iteration, about half the dependent FP64 operations of a square root and a
// division.  Far from 1, where products with u and tau could leave the range of a double, the plain operations on the
// reflector scaled to u0 = 1: sc is the factor of the other entries (else 1).
__device__ __forceinline__ void householder(double alpha, double sig, double &beta, double &tau, double &u0,
                                            double &sc) {
  beta = alpha;
  tau = 0.0;
  u0 = sc = 1.0;
  if (sig == 0.0) return;
  const double S = fma(alpha, alpha, sig), a = fabs(alpha);
  double nrm;
  if (S > 1e-90 && S < 1e60) {
    double r;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(S));
    r = fma(0.5 * r, fma(-S * r, r, 1.0), r);
    r = fma(0.5 * r, fma(-S * r, r, 1.0), r);
    nrm = S * r;
    const double D = fma(nrm, a, S);
    double t = recip_nr(D);
    tau = fma(t, fma(-D, t, 1.0), t);
    beta = alpha <= 0.0 ? nrm : -nrm;
    u0 = alpha - beta;
  } else {
    nrm = sqrt(S);
    beta = alpha <= 0.0 ? nrm : -nrm;
    tau = (beta - alpha) / beta;
    sc = 1.0 / (alpha - beta);
  }
}

// CTAs off[j] .. off[j+1]-1 of the grid work on item j.
struct TridSplit {
  int off[EIG_MAXB + 1];
};

__global__ void __launch_bounds__(TRD_THREADS) tridiag_kernel(SymBatchP b, TridSplit sp, int nmax, double *pbuf,
                                                              unsigned *bars, int *status) {
  int item = 0;
  while (sp.off[item + 1] <= (int)blockIdx.x) ++item;
  const int me = (int)blockIdx.x - sp.off[item], G = sp.off[item + 1] - sp.off[item];
  const SymItem it = b.it[item];
  const int n = it.n, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nthr = blockDim.x, NW = nthr >> 5;
  extern __shared__ double sm[];
  double *vp = sm, *q = sm + nmax, *v = sm + 2 * nmax;  // v_{i-1}, q_{i-1}, v_i, indexed by row
  __shared__ double red[32];
  __shared__ double K_s, qi_s, tau_s, sc_s;  // tau_s: of the last reflector formed
  __shared__ double st_s[2];                 // 2^-exponent of u0, by the parity of the step
  double *p0 = pbuf + (int64_t)item * 2 * nmax;
  unsigned *bar = bars + item;
  for (int i = 0; i < n; ++i) {
    // q_{i-1} and row i
    double *row = it.H + (int64_t)i * it.ld;
    const bool upd = i >= 1 && i - 1 < n - 2;
    const int nact = min(NW, (n - i + 31) >> 5);
    double ss = 0.0;
    if (upd) {
      const double *p = p0 + (int64_t)((i - 1) & 1) * nmax;
      for (int k = i + tid; k < n; k += nthr) {
        const double pk = __ldcg(p + k);
        q[k] = pk;
        ss = fma(pk, vp[k], ss);
        v[k] = __ldcg(row + k);
      }
      trd_sum(ss, red, nact, [&](double t) {
        K_s = 0.5 * tau_s * t;
        qi_s = q[i] - K_s * vp[i];
      });
      const double K = K_s, vi = vp[i], qi = qi_s;
      ss = 0.0;
      for (int k = i + tid; k < n; k += nthr) {
        const double qk = q[k] - K * vp[k];
        const double x = fma(-qi, vp[k], fma(-vi, qk, v[k]));
        if (k > i) q[k] = qk;  // q[i] stays as it is: other threads may still read it
        v[k] = x;
        if (k > i + 1) ss = fma(x, x, ss);
      }
    } else {  // the first row, and the last one (complete after the pass of step n - 2)
      for (int k = i + tid; k < n; k += nthr) {
        const double x = __ldcg(row + k);
        v[k] = x;
        if (k > i + 1) ss = fma(x, x, ss);
      }
    }
    trd_sum(ss, red, nact, [&](double sig) {
      double beta = 0.0, tau = 0.0, u0 = 1.0, sc = 1.0;
      if (i < n - 1) {
        householder(v[i + 1], sig, beta, tau, u0, sc);
        v[i + 1] = u0;
      }
      if (me == 0) {
        // the stored reflector has its first entry in [1, 2) and tau to match (exact, powers of two): the
        // back-transformation adds many reflectors up and wants them of one size
        const int ex = (__double2hiint(u0) >> 20) & 0x7ff;
        const double p2 = __hiloint2double(ex << 20, 0);
        it.d[i] = v[i];
        it.tau[i] = tau * p2 * p2;
        st_s[i & 1] = __hiloint2double((2046 - ex) << 20, 0);
        if (i < n - 1) it.e[i] = beta;
      }
      tau_s = tau;
      sc_s = sc;
    });
    if (sc_s != 1.0) {
      for (int k = i + 2 + tid; k < n; k += nthr) v[k] *= sc_s;
      __syncthreads();
    }
    // v_{i-1} into row i-1, for the back-transformation (every CTA has read that row)
    if (me == 0 && i >= 1) {
      const double st = st_s[(i - 1) & 1];
      for (int k = i + tid; k < n; k += nthr) it.H[(int64_t)(i - 1) * it.ld + k] = st * vp[k];
    }
    if (i > n - 2) break;
    // this CTA's rows of the trailing block: pending rank-2 update, then p_i
    const bool sym = i < n - 2;
    double *pn = p0 + (int64_t)(i & 1) * nmax;
    const int first = i + 1 + ((me - (i + 1)) % G + G) % G;
    for (int r = first + warp * G; r < n; r += NW * G) {
      double *h = it.H + (int64_t)r * it.ld;
      const double vr = upd ? vp[r] : 0.0, qr = upd ? q[r] : 0.0;
      double s0 = 0.0, s1 = 0.0;
      int c = i + 1 + lane;
      if (upd) {
        double h4[4];
        if (c + 96 < n) {
#pragma unroll
          for (int u = 0; u < 4; ++u) h4[u] = h[c + 32 * u];
        }
        for (; c + 96 < n; c += 128) {
          const bool more = c + 224 < n;  // the next four entries are loaded ahead of this four's chain
          double g4[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) g4[u] = more ? h[c + 128 + 32 * u] : 0.0;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            h4[u] = fma(-qr, vp[c + 32 * u], fma(-vr, q[c + 32 * u], h4[u]));
            h[c + 32 * u] = h4[u];
          }
          s0 = fma(h4[0], v[c], s0);
          s1 = fma(h4[1], v[c + 32], s1);
          s0 = fma(h4[2], v[c + 64], s0);
          s1 = fma(h4[3], v[c + 96], s1);
#pragma unroll
          for (int u = 0; u < 4; ++u) h4[u] = g4[u];
        }
        for (; c < n; c += 32) {
          const double x = fma(-qr, vp[c], fma(-vr, q[c], h[c]));
          h[c] = x;
          s0 = fma(x, v[c], s0);
        }
      } else {
        for (; c < n; c += 32) s0 = fma(h[c], v[c], s0);
      }
      if (sym) {
        double t = s0 + s1;
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if (lane == 0) pn[r] = tau_s * t;
      }
    }
    if (!grid_barrier(bar, (unsigned)(G * (i + 1)))) {
      if (tid == 0) atomicOr(status, DS_GRID_TIMEOUT);
      return;
    }
    double *t = vp;  // v_i is the next step's v_{i-1}
    vp = v;
    v = t;
  }
}

// ctas CTAs over all items, shared in proportion to n^2 (the work of a step), at least four rows to a CTA at the start
// and one CTA to an item
static TridSplit trid_split(const SymBatchP &b, int cnt, int ctas) {
  TridSplit sp;
  double sq = 0.0;
  for (int j = 0; j < cnt; ++j) sq += (double)b.it[j].n * b.it[j].n;
  sp.off[0] = 0;
  for (int j = 0; j < cnt; ++j) {
    const double nj = b.it[j].n;
    const int g = 1 + (int)(std::max(0, ctas - cnt) * nj * nj / sq);
    sp.off[j + 1] = sp.off[j] + std::max(1, std::min(g, b.it[j].n / 4));
  }
  for (int j = cnt; j < EIG_MAXB; ++j) sp.off[j + 1] = sp.off[cnt];
  return sp;
}

static void tridiagonalize(cudaStream_t st, const SymBatchP &b, int cnt, int nmax, int *status) {
  if (nmax > 2 && nmax <= TRD_NMAX && status) {
    const int nv = (nmax + 1) & ~1;
    const size_t smem = (size_t)3 * nv * sizeof(double);
    // always the same limit: several host threads launch this kernel at once
    RFDD_CUDA(cudaFuncSetAttribute(tridiag_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   3 * TRD_NMAX * (int)sizeof(double)));
    double *pbuf = nullptr;
    const size_t pb = (size_t)cnt * 2 * nv * sizeof(double);
    RFDD_CUDA(cudaMallocAsync((void **)&pbuf, pb + (size_t)cnt * sizeof(unsigned), st));
    unsigned *bars = reinterpret_cast<unsigned *>(reinterpret_cast<char *>(pbuf) + pb);
    RFDD_CUDA(cudaMemsetAsync(bars, 0, (size_t)cnt * sizeof(unsigned), st));
    // one CTA per SM
    const int got = cooperative_launch(std::max(cnt, sm_count()), cnt, [&](int ctas) {
      SymBatchP bb = b;
      TridSplit sp = trid_split(b, cnt, ctas);
      int nvv = nv;
      void *args[] = {&bb, &sp, &nvv, &pbuf, &bars, &status};
      return cudaLaunchCooperativeKernel((const void *)tridiag_kernel, dim3(sp.off[cnt]),
                                         dim3(nmax <= 512 ? 256 : TRD_THREADS), args, smem, st);
    });
    RFDD_CUDA(cudaFreeAsync(pbuf, st));
    if (got > 0) return;
  }
  double *qbuf = nullptr;
  RFDD_CUDA(cudaMallocAsync((void **)&qbuf, (size_t)cnt * std::max(nmax, 1) * sizeof(double), st));
  for (int i = 0; i < nmax; ++i) {
    house_kernel<<<cnt, 512, 0, st>>>(b, i, qbuf, nmax);
    RFDD_CHECK_LAUNCH();
    if (i <= nmax - 2) {
      const int len = nmax - i - 1;
      update_symv_kernel<<<dim3(ceil_div((int64_t)len * 32 * TRD_WPR, 256), cnt), 256, 0, st>>>(b, i, qbuf, nmax);
      RFDD_CHECK_LAUNCH();
    }
  }
  RFDD_CUDA(cudaFreeAsync(qbuf, st));
}

// counts[i] = number of eigenvalues of item i's tridiagonal matrix below shift (Sturm count)
__global__ void sturm_count_kernel(SymBatchP b, int cnt, double shift, long long *counts) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= cnt) return;
  const SymItem it = b.it[q];
  const int n = it.n;
  if (n <= 0) {
    counts[q] = 0;
    return;
  }
  double emax2 = 0.0;
  for (int k = 0; k + 1 < n; ++k) emax2 = fmax(emax2, it.e[k] * it.e[k]);
  const double pivmin = 2.2250738585072014e-308 * fmax(1.0, emax2);
  counts[q] = sturm_count(it.d, it.e, n, shift, pivmin);
}

void sym_negative_counts(cudaStream_t st, const std::vector<SymItem> &items, double shift, long long *counts_dev,
                         int *status) {
  for (size_t s0 = 0; s0 < items.size(); s0 += EIG_MAXB) {
    SymBatchP b;
    memset(&b, 0, sizeof(b));
    const int cnt = (int)std::min<size_t>(EIG_MAXB, items.size() - s0);
    int nmax = 0;
    for (int i = 0; i < cnt; ++i) { b.it[i] = items[s0 + i]; nmax = std::max(nmax, b.it[i].n); }
    if (nmax > 0) tridiagonalize(st, b, cnt, nmax, status);
    sturm_count_kernel<<<1, 64, 0, st>>>(b, cnt, shift, counts_dev + s0);
    RFDD_CHECK_LAUNCH();
  }
}

void sym_eig_values(cudaStream_t st, const std::vector<SymItem> &items, int *status) {
  for (size_t s0 = 0; s0 < items.size(); s0 += EIG_MAXB) {
    SymBatchP b;
    memset(&b, 0, sizeof(b));
    const int cnt = (int)std::min<size_t>(EIG_MAXB, items.size() - s0);
    int nmax = 0;
    for (int i = 0; i < cnt; ++i) { b.it[i] = items[s0 + i]; nmax = std::max(nmax, b.it[i].n); }
    if (nmax == 0) continue;
    tridiagonalize(st, b, cnt, nmax, status);
    tridiagonal_values(st, b, cnt, nmax);
  }
}

// --------------------------------------------------------------------------------------
// Eigenvectors of the tridiagonal matrix by inverse iteration, one CTA per cluster.  Thread 0
// factors T - lambda I with partial pivoting (rows k, k+1 swapped when |sub| > |diagonal|) and
// runs the triangular solves; all threads share the Gram-Schmidt against the cluster's earlier
// vectors and the normalisation.
// --------------------------------------------------------------------------------------
struct Cluster {
  int item;   // index into the batch
  int first;  // position in the item's selection list
  int size;
};
struct InvIterP {
  SymItem it[EIG_MAXB];
  const int *sel[EIG_MAXB];   // device copies of the selections
};

__global__ void __launch_bounds__(256) inviter_kernel(InvIterP p, const Cluster *__restrict__ cl, double *scratch,
                                                      int64_t scratch_per_cta, double ctol) {
  const Cluster c = cl[blockIdx.x];
  const SymItem it = p.it[c.item];
  const int *sel = p.sel[c.item];
  const int n = it.n;
  const double *d = it.d, *e = it.e;
  double *u1 = scratch + (int64_t)blockIdx.x * scratch_per_cta;
  double *u2 = u1 + n, *u3 = u2 + n, *ml = u3 + n, *pv = ml + n, *x = pv + n, *ru = x + n;
  __shared__ double red[33];
  __shared__ double tnorm_s;
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int k = 0; k < n; ++k) t = fmax(t, fabs(d[k]) + (k > 0 ? fabs(e[k - 1]) : 0.0) + (k < n - 1 ? fabs(e[k]) : 0.0));
    tnorm_s = t;
  }
  __syncthreads();
  const double eps = 2.220446049250313e-16;
  const double delta = eps * fmax(tnorm_s, 1e-300);
  for (int q = 0; q < c.size; ++q) {
    const int row = c.first + q;  // output row in Zt
    const double lam = it.lam[sel[row]];
    // start vector: counter-based hash of (eigen index, component)
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      uint64_t z = (uint64_t)(sel[row] + 1) * 0x9E3779B97F4A7C15ull + (uint64_t)(k + 1) * 0xBF58476D1CE4E5B9ull;
      z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
      z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
      z ^= z >> 31;
      x[k] = (double)(z >> 11) * 0x1p-53 + 0.5;
    }
    if (threadIdx.x == 0) {
      double cd = d[0] - lam, ce1 = n > 1 ? e[0] : 0.0, ce2 = 0.0;
      for (int k = 0; k < n - 1; ++k) {
        const double sub = e[k];
        const double an = d[k + 1] - lam;
        const double bn = (k + 1 < n - 1) ? e[k + 1] : 0.0;
        if (fabs(cd) >= fabs(sub)) {
          if (cd == 0.0) cd = delta;
          const double l = sub / cd;
          u1[k] = cd;
          u2[k] = ce1;
          u3[k] = ce2;
          pv[k] = 0.0;
          ml[k] = l;
          cd = an - l * ce1;
          ce1 = bn - l * ce2;
          ce2 = 0.0;
        } else {
          const double l = cd / sub;
          u1[k] = sub;
          u2[k] = an;
          u3[k] = bn;
          pv[k] = 1.0;
          ml[k] = l;
          const double nd = ce1 - l * an;
          const double ne1 = ce2 - l * bn;
          cd = nd;
          ce1 = ne1;
          ce2 = 0.0;
        }
      }
      u1[n - 1] = (fabs(cd) < delta) ? (cd < 0 ? -delta : delta) : cd;
    }
    __syncthreads();
    // reciprocals of the pivots, once, by all threads: the solves below then multiply
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      const double u = (k < n - 1 && fabs(u1[k]) < delta) ? (u1[k] < 0 ? -delta : delta) : u1[k];
      ru[k] = 1.0 / u;
    }
    __syncthreads();
    for (int iter = 0; iter < 3; ++iter) {
      if (threadIdx.x == 0) {
        for (int k = 0; k < n - 1; ++k) {
          if (pv[k] != 0.0) {
            const double t = x[k];
            x[k] = x[k + 1];
            x[k + 1] = t;
          }
          x[k + 1] -= ml[k] * x[k];
        }
        x[n - 1] *= ru[n - 1];
        if (n > 1) x[n - 2] = (x[n - 2] - u2[n - 2] * x[n - 1]) * ru[n - 2];
        for (int k = n - 3; k >= 0; --k) x[k] = (x[k] - u2[k] * x[k + 1] - u3[k] * x[k + 2]) * ru[k];
      }
      __syncthreads();
      // scale to unit max-norm first so that the dot products below cannot overflow
      double mx = 0.0;
      for (int k = threadIdx.x; k < n; k += blockDim.x) mx = fmax(mx, fabs(x[k]));
      for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, o));
      __syncthreads();
      if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
      __syncthreads();
      double m2 = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m2 = fmax(m2, red[w]);
      const double inv = m2 > 0.0 ? 1.0 / m2 : 1.0;
      for (int k = threadIdx.x; k < n; k += blockDim.x) x[k] *= inv;
      __syncthreads();
      // Gram-Schmidt against the earlier vectors of the cluster (twice)
      for (int pass = 0; pass < 2; ++pass)
        for (int pq = 0; pq < q; ++pq) {
          const double *v = it.Zt + (int64_t)(c.first + pq) * n;
          double s = 0.0;
          for (int k = threadIdx.x; k < n; k += blockDim.x) s = fma(x[k], v[k], s);
          const double dot = block_sum(s, red);
          for (int k = threadIdx.x; k < n; k += blockDim.x) x[k] -= dot * v[k];
          __syncthreads();
        }
      double s = 0.0;
      for (int k = threadIdx.x; k < n; k += blockDim.x) s = fma(x[k], x[k], s);
      const double nrm = sqrt(block_sum(s, red));
      const double sc = nrm > 0.0 ? 1.0 / nrm : 0.0;
      for (int k = threadIdx.x; k < n; k += blockDim.x) x[k] *= sc;
      __syncthreads();
    }
    double *out = it.Zt + (int64_t)row * n;
    for (int k = threadIdx.x; k < n; k += blockDim.x) out[k] = x[k];
    __syncthreads();
  }
  (void)ctol;
}

// Inverse iteration for eigenvalues that stand alone (clusters of one), one lane per eigenvalue:
// the factorisation and the triangular solves are serial chains, so a warp runs 32 of them at the
// cost of one (all vectors of order 1885: 4.4 ms, 14.2 with one thread of a CTA per eigenvalue).
// Scratch is lane-interleaved (entry k of lane l at k * 32 + l), so every access is coalesced, and
// IV_U steps are loaded ahead of the chain.  Same start vectors, factorisation and number of
// iterations as inviter_kernel.
struct SingleWarp {
  int item, first, count;  // rows[first .. first + count): positions in the item's selection list
};
constexpr int IV_ARRAYS = 5;
constexpr int IV_U = 8;
// 1 / u to about 2^-52: two Newton steps on the hardware's approximation; the division for tiny and huge u
__device__ __forceinline__ double recip_any(double u) {
  const double a = fabs(u);
  if (!(a > 1e-290 && a < 1e290)) return 1.0 / u;
  const double r = recip_nr(u);
  return fma(r, fma(-u, r, 1.0), r);
}
__global__ void __launch_bounds__(32) inviter_single_kernel(InvIterP p, const SingleWarp *__restrict__ sw,
                                                            const int *__restrict__ rows, double *scratch,
                                                            int64_t per_warp, unsigned *flags, int64_t flags_per_warp) {
  const SingleWarp c = sw[blockIdx.x];
  const SymItem it = p.it[c.item];
  const int n = it.n, lane = threadIdx.x;
  const int row = rows[c.first + min(lane, c.count - 1)];
  const int ei = p.sel[c.item][row];
  const double lam = it.lam[ei];
  const double *__restrict__ d = it.d, *__restrict__ e = it.e;
  const int64_t len = (int64_t)n * 32;
  double *__restrict__ ru = scratch + (int64_t)blockIdx.x * per_warp + lane;
  double *__restrict__ u2 = ru + len, *__restrict__ u3 = u2 + len, *__restrict__ ml = u3 + len,
         *__restrict__ x = ml + len;
  unsigned *__restrict__ fl = flags + (int64_t)blockIdx.x * flags_per_warp;
  double tn = 0.0;
  for (int k = lane; k < n; k += 32)
    tn = fmax(tn, fabs(d[k]) + (k > 0 ? fabs(e[k - 1]) : 0.0) + (k < n - 1 ? fabs(e[k]) : 0.0));
  for (int o = 16; o > 0; o >>= 1) tn = fmax(tn, __shfl_xor_sync(0xffffffffu, tn, o));
  const double delta = 2.220446049250313e-16 * fmax(tn, 1e-300);
  auto hash = [&](int k) {
    uint64_t z = (uint64_t)(ei + 1) * 0x9E3779B97F4A7C15ull + (uint64_t)(k + 1) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (double)(z >> 11) * 0x1p-53 + 0.5;
  };
  // T - lam I = P L U with row interchanges of neighbours; ru = 1 / U_kk
  double cd = d[0] - lam, ce1 = n > 1 ? e[0] : 0.0, ce2 = 0.0;
  for (int k = 0; k < n - 1; ++k) {
    const double sub = e[k], an = d[k + 1] - lam, bn = (k + 1 < n - 1) ? e[k + 1] : 0.0;
    const bool piv = fabs(cd) < fabs(sub);
    if (!piv && cd == 0.0) cd = delta;
    double u = piv ? sub : cd;
    const double l = (piv ? cd : sub) * recip_any(u);
    if (fabs(u) < delta) u = u < 0 ? -delta : delta;
    ru[(int64_t)k * 32] = recip_any(u);
    u2[(int64_t)k * 32] = piv ? an : ce1;
    u3[(int64_t)k * 32] = piv ? bn : ce2;
    ml[(int64_t)k * 32] = l;
    x[(int64_t)k * 32] = hash(k);
    const unsigned f = __ballot_sync(0xffffffffu, piv);
    if (lane == 0) fl[k] = f;
    const double nd = piv ? ce1 - l * an : an - l * ce1;
    ce1 = piv ? ce2 - l * bn : bn - l * ce2;
    ce2 = 0.0;
    cd = nd;
  }
  {
    const double u = (fabs(cd) < delta) ? (cd < 0 ? -delta : delta) : cd;
    ru[(int64_t)(n - 1) * 32] = recip_any(u);
    u2[(int64_t)(n - 1) * 32] = u3[(int64_t)(n - 1) * 32] = 0.0;
    x[(int64_t)(n - 1) * 32] = hash(n - 1);
  }
  __syncwarp();
  double scale = 1.0, ss = 0.0;
  for (int iter = 0; iter < 3; ++iter) {
    // forward: the largest entry of the last solve is scaled to [1, 2) on the way in
    double cur = x[0] * scale;
    for (int k0 = 0; k0 < n - 1; k0 += IV_U) {
      double xn[IV_U], mk[IV_U];
      unsigned fk[IV_U];
#pragma unroll
      for (int q = 0; q < IV_U; ++q)
        if (k0 + q < n - 1) {
          xn[q] = x[(int64_t)(k0 + q + 1) * 32];
          mk[q] = ml[(int64_t)(k0 + q) * 32];
          fk[q] = fl[k0 + q];
        }
#pragma unroll
      for (int q = 0; q < IV_U; ++q)
        if (k0 + q < n - 1) {
          const double nx = xn[q] * scale;
          const bool piv = (fk[q] >> lane) & 1u;
          const double top = piv ? nx : cur, bot = piv ? cur : nx;
          x[(int64_t)(k0 + q) * 32] = top;
          cur = bot - mk[q] * top;
        }
    }
    // backward
    // (x_k - u2 x_{k+1} - u3 x_{k+2}) / U_kk with the factors multiplied by 1 / U_kk ahead: the chain from one step to
    // the next is one FMA.  The largest entry is tracked by its high word (integer instructions).
    double x1 = cur * ru[(int64_t)(n - 1) * 32], x2 = 0.0;
    int mx = __double2hiint(x1) & 0x7fffffff;
    x[(int64_t)(n - 1) * 32] = x1;
    for (int k0 = n - 2; k0 >= 0; k0 -= IV_U) {
      double xk[IV_U], a2[IV_U], a3[IV_U], rk[IV_U];
#pragma unroll
      for (int q = 0; q < IV_U; ++q)
        if (k0 - q >= 0) {
          const int64_t o = (int64_t)(k0 - q) * 32;
          xk[q] = x[o];
          a2[q] = u2[o];
          a3[q] = u3[o];
          rk[q] = ru[o];
        }
#pragma unroll
      for (int q = 0; q < IV_U; ++q)
        if (k0 - q >= 0) {
          const double v = fma(-a2[q] * rk[q], x1, fma(-a3[q] * rk[q], x2, xk[q] * rk[q]));
          x[(int64_t)(k0 - q) * 32] = v;
          x2 = x1;
          x1 = v;
          mx = max(mx, __double2hiint(v) & 0x7fffffff);
        }
    }
    // a power of two that brings the largest entry to [1, 2); 1 for zero, subnormal and not finite ones
    const int ex = mx >> 20;
    scale = ex >= 1 && ex <= 2045 ? __hiloint2double((2046 - ex) << 20, 0) : 1.0;
  }
  for (int k = 0; k < n; ++k) {
    const double v = x[(int64_t)k * 32] * scale;
    ss = fma(v, v, ss);
  }
  const double sc = ss > 0.0 ? scale / sqrt(ss) : 0.0;
  // rows of Zt through shared memory, so that the stores run along them
  __shared__ double tile[32][33];
  double *Zt = it.Zt;
  for (int k0 = 0; k0 < n; k0 += 32) {
    const int w = min(32, n - k0);
    for (int q = 0; q < w; ++q) tile[lane][q] = x[(int64_t)(k0 + q) * 32] * sc;
    __syncwarp();
    for (int r = 0; r < c.count; ++r) {
      const int rr = __shfl_sync(0xffffffffu, row, r);
      if (lane < w) Zt[(int64_t)rr * n + k0 + lane] = tile[r][lane];
    }
    __syncwarp();
  }
}

// x = H_0 H_1 ... H_{n-3} z for each tridiagonal eigenvector z (row of Zt); one CTA per vector,
// the vector in shared memory.
struct BackBatchP {
  SymItem s[EIG_MAXB];
  double *out[EIG_MAXB];
  int nsel[EIG_MAXB];
  int ld_out[EIG_MAXB];
};

__global__ void back_kernel(BackBatchP b) {
  const int bi = blockIdx.y;
  const int r = blockIdx.x;
  if (r >= b.nsel[bi]) return;
  const SymItem it = b.s[bi];
  const int n = it.n;
  extern __shared__ double x[];
  __shared__ double red[33];
  for (int k = threadIdx.x; k < n; k += blockDim.x) x[k] = it.Zt[(int64_t)r * n + k];
  __syncthreads();
  for (int i = n - 3; i >= 0; --i) {
    const double tau = it.tau[i];
    if (tau == 0.0) continue;
    const double *v = it.H + (int64_t)i * it.ld + i + 1;
    const int len = n - i - 1;
    double s = 0.0;
    for (int k = threadIdx.x; k < len; k += blockDim.x) s = fma(v[k], x[i + 1 + k], s);
    const double t = tau * block_sum(s, red);
    for (int k = threadIdx.x; k < len; k += blockDim.x) x[i + 1 + k] -= t * v[k];
    __syncthreads();
  }
  double *o = b.out[bi] + (int64_t)r * b.ld_out[bi];
  for (int k = threadIdx.x; k < n; k += blockDim.x) o[k] = x[k];
}

// --------------------------------------------------------------------------------------
// Back-transformation in blocks (compact WY form: Schreiber and Van Loan 1989).  Reflectors i = s .. s + WY_NB - 1
// make I - V T V^T with T upper triangular; on the vectors as rows, X <- X - (X V) (T^T V^T).  The blocks' clean
// copies of V^T, T and U = T^T V^T are formed for all blocks at once, then two products per block, last block
// first.  The products are FP64 by digit products on the tensor cores where they are large; one CTA per vector
// with two passes of FP64 instructions over every reflector (back_kernel) is at the chip's FP64 rate: 26.9 ms
// for the 1885 vectors of order 1885, about 5 ms in blocks.
// --------------------------------------------------------------------------------------
constexpr int WY_NB = 128;

// V^T of block b (rows i = s + j, columns c0 = s + 1 .. n - 1): zeros left of the reflector
__global__ void wy_copy_kernel(SymItem it, const int64_t *__restrict__ off, double *Vc) {
  const int b = blockIdx.y, s = b * WY_NB, n = it.n, len = n - s - 1;
  double *V = Vc + off[b];
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < (int64_t)WY_NB * len;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int i = s + (int)(e / len), c = s + 1 + (int)(e % len);
    V[e] = i <= n - 3 && c > i ? it.H[(int64_t)i * it.ld + c] : 0.0;
  }
}

// T of every block from S = V^T V (in WY_NB x WY_NB blocks): T_ii = tau_i, T_ji = -tau_i sum_l T_jl S_li (j <= l < i); one
// thread per row
__global__ void __launch_bounds__(WY_NB) wy_t_kernel(SymItem it, const double *__restrict__ S_all, double *T_all) {
  extern __shared__ double Ts[];  // WY_NB x (WY_NB + 1)
  const int b = blockIdx.x, s = b * WY_NB, j = threadIdx.x;
  const double *S = S_all + (int64_t)b * WY_NB * WY_NB;
  double *row = Ts + j * (WY_NB + 1);
  for (int i = 0; i < WY_NB; ++i) {
    const double tau = s + i <= it.n - 3 ? it.tau[s + i] : 0.0;
    double v = 0.0;
    if (j == i) v = tau;
    else if (j < i && tau != 0.0) {
      double a0 = 0.0, a1 = 0.0;
      int l = j;
      for (; l + 1 < i; l += 2) {
        a0 = fma(row[l], S[l * WY_NB + i], a0);
        a1 = fma(row[l + 1], S[(l + 1) * WY_NB + i], a1);
      }
      if (l < i) a0 = fma(row[l], S[l * WY_NB + i], a0);
      v = -tau * (a0 + a1);
    }
    row[i] = v;
  }
  double *T = T_all + (int64_t)b * WY_NB * WY_NB;
  for (int i = 0; i < WY_NB; ++i) T[j * WY_NB + i] = row[i];
}

// whether an item's back-transformation runs in blocks: the products are large enough and there is a status word
static bool wy_takes(int n, int nsel) { return tc_status_word() && n >= 512 && nsel >= 96; }

// out (nsel x n, ld) holds the tridiagonal eigenvectors as rows and receives those of H
static void wy_back(cudaStream_t st, const SymItem &it, int nsel, double *out, int ld) {
  const int n = it.n, nblk = ceil_div(n - 2, WY_NB);
  std::vector<int64_t> off(nblk);
  int64_t tot = 0;
  for (int b = 0; b < nblk; ++b) {
    off[b] = tot;
    tot += (int64_t)WY_NB * (n - b * WY_NB - 1);
  }
  const size_t sq = (size_t)nblk * WY_NB * WY_NB;
  double *ws = nullptr;
  int64_t *off_dev = nullptr;
  RFDD_CUDA(cudaMallocAsync((void **)&ws, (2 * (size_t)tot + 2 * sq + (size_t)nsel * WY_NB) * sizeof(double), st));
  RFDD_CUDA(cudaMallocAsync((void **)&off_dev, nblk * sizeof(int64_t), st));
  RFDD_CUDA(cudaMemcpyAsync(off_dev, off.data(), nblk * sizeof(int64_t), cudaMemcpyHostToDevice, st));
  double *V = ws, *U = V + tot, *S = U + tot, *T = S + sq, *P = T + sq;
  wy_copy_kernel<<<dim3(128, nblk), 256, 0, st>>>(it, off_dev, V);
  RFDD_CHECK_LAUNCH();
  std::vector<GemmItem<double>> g;
  for (int b = 0; b < nblk; ++b) {
    const int len = n - b * WY_NB - 1;
    g.push_back({V + off[b], V + off[b], S + (int64_t)b * WY_NB * WY_NB, WY_NB, WY_NB, len, len, len, WY_NB});
  }
  gemm_f64_basis_batched(st, g, false, true, 1.0, 0.0);
  const int tsm = WY_NB * (WY_NB + 1) * (int)sizeof(double);
  RFDD_CUDA(cudaFuncSetAttribute(wy_t_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, tsm));
  wy_t_kernel<<<nblk, WY_NB, tsm, st>>>(it, S, T);
  RFDD_CHECK_LAUNCH();
  g.clear();
  for (int b = 0; b < nblk; ++b) {
    const int len = n - b * WY_NB - 1;
    g.push_back({T + (int64_t)b * WY_NB * WY_NB, V + off[b], U + off[b], WY_NB, len, WY_NB, WY_NB, len, len});
  }
  gemm_f64_basis_batched(st, g, true, false, 1.0, 0.0);
  for (int b = nblk - 1; b >= 0; --b) {
    const int c0 = b * WY_NB + 1, len = n - c0;
    gemm_f64_basis_batched(st, {{out + c0, V + off[b], P, nsel, WY_NB, len, ld, len, WY_NB}}, false, true, 1.0, 0.0);
    gemm_f64_basis_batched(st, {{P, U + off[b], out + c0, nsel, len, WY_NB, WY_NB, len, ld}}, false, false, -1.0, 1.0);
  }
  RFDD_CUDA(cudaFreeAsync(ws, st));
  RFDD_CUDA(cudaFreeAsync(off_dev, st));
  RFDD_CUDA(cudaStreamSynchronize(st));  // off is read by an asynchronous copy
}

void sym_eig_vectors(cudaStream_t st, const std::vector<BackItem> &items, double ctol) {
  for (size_t s0 = 0; s0 < items.size(); s0 += EIG_MAXB) {
    const int cnt = (int)std::min<size_t>(EIG_MAXB, items.size() - s0);
    InvIterP ip;
    memset(&ip, 0, sizeof(ip));
    BackBatchP bb;
    memset(&bb, 0, sizeof(bb));
    std::vector<Cluster> clusters;
    std::vector<SingleWarp> singles;  // eigenvalues that stand alone, 32 of one item to a warp
    std::vector<int> srows;
    std::vector<int> allsel;
    std::vector<size_t> seloff(cnt);
    int nmax = 1, selmax = 0;
    for (int i = 0; i < cnt; ++i) {
      const BackItem &bi = items[s0 + i];
      const SymItem &it = *bi.s;
      ip.it[i] = it;
      bb.s[i] = it;
      bb.out[i] = bi.out;
      bb.nsel[i] = wy_takes(it.n, (int)bi.sel.size()) ? 0 : (int)bi.sel.size();
      bb.ld_out[i] = bi.ld_out;
      nmax = std::max(nmax, it.n);
      selmax = std::max(selmax, bb.nsel[i]);
      seloff[i] = allsel.size();
      allsel.insert(allsel.end(), bi.sel.begin(), bi.sel.end());
      if (bi.sel.empty()) continue;
      // clusters of close selected eigenvalues (needs the eigenvalues and the matrix scale)
      std::vector<double> lam(it.n), dd(it.n), ee(it.n);
      RFDD_CUDA(cudaMemcpyAsync(lam.data(), it.lam, it.n * sizeof(double), cudaMemcpyDeviceToHost, st));
      RFDD_CUDA(cudaMemcpyAsync(dd.data(), it.d, it.n * sizeof(double), cudaMemcpyDeviceToHost, st));
      RFDD_CUDA(cudaMemcpyAsync(ee.data(), it.e, it.n * sizeof(double), cudaMemcpyDeviceToHost, st));
      RFDD_CUDA(cudaStreamSynchronize(st));
      double tnorm = 0.0;
      for (int k = 0; k < it.n; ++k)
        tnorm = std::max(tnorm, std::fabs(dd[k]) + (k > 0 ? std::fabs(ee[k - 1]) : 0.0) +
                                    (k < it.n - 1 ? std::fabs(ee[k]) : 0.0));
      int start = 0;
      for (int q = 1; q <= (int)bi.sel.size(); ++q) {
        if (q == (int)bi.sel.size() || lam[bi.sel[q]] - lam[bi.sel[q - 1]] > ctol * tnorm) {
          if (q - start == 1) {
            if (singles.empty() || singles.back().item != i || singles.back().count == 32)
              singles.push_back({i, (int)srows.size(), 0});
            ++singles.back().count;
            srows.push_back(start);
          } else {
            clusters.push_back({i, start, q - start});
          }
          start = q;
        }
      }
    }
    if (clusters.empty() && singles.empty()) continue;
    int *sel_dev = nullptr;
    RFDD_CUDA(cudaMallocAsync((void **)&sel_dev, allsel.size() * sizeof(int), st));
    RFDD_CUDA(cudaMemcpyAsync(sel_dev, allsel.data(), allsel.size() * sizeof(int), cudaMemcpyHostToDevice, st));
    for (int i = 0; i < cnt; ++i) ip.sel[i] = sel_dev + seloff[i];
    if (!clusters.empty()) {
      Cluster *cl_dev = nullptr;
      double *scratch = nullptr;
      const int64_t per = (int64_t)7 * nmax;
      RFDD_CUDA(cudaMallocAsync((void **)&cl_dev, clusters.size() * sizeof(Cluster), st));
      RFDD_CUDA(cudaMallocAsync((void **)&scratch, (size_t)clusters.size() * per * sizeof(double), st));
      RFDD_CUDA(cudaMemcpyAsync(cl_dev, clusters.data(), clusters.size() * sizeof(Cluster), cudaMemcpyHostToDevice, st));
      inviter_kernel<<<(unsigned)clusters.size(), 256, 0, st>>>(ip, cl_dev, scratch, per, ctol);
      RFDD_CHECK_LAUNCH();
      RFDD_CUDA(cudaFreeAsync(cl_dev, st));
      RFDD_CUDA(cudaFreeAsync(scratch, st));
    }
    if (!singles.empty()) {
      SingleWarp *sw_dev = nullptr;
      int *rows_dev = nullptr;
      double *scratch = nullptr;
      const int64_t per = (int64_t)IV_ARRAYS * 32 * nmax, fper = nmax;
      RFDD_CUDA(cudaMallocAsync((void **)&sw_dev, singles.size() * sizeof(SingleWarp), st));
      RFDD_CUDA(cudaMallocAsync((void **)&rows_dev, srows.size() * sizeof(int), st));
      RFDD_CUDA(cudaMallocAsync((void **)&scratch,
                                singles.size() * ((size_t)per * sizeof(double) + (size_t)fper * sizeof(unsigned)), st));
      RFDD_CUDA(cudaMemcpyAsync(sw_dev, singles.data(), singles.size() * sizeof(SingleWarp), cudaMemcpyHostToDevice, st));
      RFDD_CUDA(cudaMemcpyAsync(rows_dev, srows.data(), srows.size() * sizeof(int), cudaMemcpyHostToDevice, st));
      inviter_single_kernel<<<(unsigned)singles.size(), 32, 0, st>>>(
          ip, sw_dev, rows_dev, scratch, per, reinterpret_cast<unsigned *>(scratch + singles.size() * per), fper);
      RFDD_CHECK_LAUNCH();
      RFDD_CUDA(cudaFreeAsync(sw_dev, st));
      RFDD_CUDA(cudaFreeAsync(rows_dev, st));
      RFDD_CUDA(cudaFreeAsync(scratch, st));
    }
    const size_t smem = (size_t)nmax * sizeof(double);
    RFDD_REQUIRE(smem <= 200 * 1024, RFDD_EINVAL, "sym_eig: order too large");
    RFDD_CUDA(cudaFuncSetAttribute(back_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    if (selmax > 0) {
      back_kernel<<<dim3(selmax, cnt), 256, smem, st>>>(bb);
      RFDD_CHECK_LAUNCH();
    }
    for (int i = 0; i < cnt; ++i) {
      const BackItem &bi = items[s0 + i];
      const SymItem &it = *bi.s;
      const int ns = (int)bi.sel.size();
      if (ns == 0 || bb.nsel[i] > 0) continue;
      RFDD_CUDA(cudaMemcpy2DAsync(bi.out, (size_t)bi.ld_out * sizeof(double), it.Zt, (size_t)it.n * sizeof(double),
                                  (size_t)it.n * sizeof(double), ns, cudaMemcpyDeviceToDevice, st));
      wy_back(st, it, ns, bi.out, bi.ld_out);
    }
    RFDD_CUDA(cudaFreeAsync(sel_dev, st));
    // host vectors referenced by async copies must outlive them
    RFDD_CUDA(cudaStreamSynchronize(st));
  }
}

}  // namespace rfdd
