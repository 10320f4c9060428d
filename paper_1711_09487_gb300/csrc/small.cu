// Small dense FP64 kernels for block orthonormalisation and Rayleigh-Ritz bookkeeping.
#include "small.cuh"
#include "dense.cuh"
#include "grid_barrier.cuh"

#include <algorithm>
#include <climits>

namespace rfdd {

constexpr int CH_MAXB = 64;
struct CholBatchP {
  CholItem it[CH_MAXB];
};

// Right-looking Cholesky G = R^T R on the upper triangle, one CTA per matrix (global memory).
// A pivot <= tol * (largest diagonal) marks its column dead: its row of R is zeroed and the
// column is skipped, so the kept columns get an orthonormal basis and dead ones a zero column.
__global__ void __launch_bounds__(512) chol_inv_kernel(CholBatchP bp, double tol) {
  const CholItem it = bp.it[blockIdx.x];
  const int b = it.b;
  double *G = it.G;
  __shared__ double dmax_s;
  __shared__ int dead_s;
  if (threadIdx.x == 0) {
    double m = 0.0;
    for (int i = 0; i < b; ++i) m = fmax(m, G[(int64_t)i * b + i]);
    dmax_s = m;
  }
  __syncthreads();
  const double thr = tol * dmax_s;
  for (int t = 0; t < b; ++t) {
    if (threadIdx.x == 0) {
      const double pv = G[(int64_t)t * b + t];
      dead_s = !(pv > thr) || !isfinite(pv);
      it.dead[t] = dead_s;
      if (!dead_s) G[(int64_t)t * b + t] = sqrt(pv);
    }
    __syncthreads();
    const double rtt = G[(int64_t)t * b + t];
    if (dead_s) {
      for (int c = t + threadIdx.x; c < b; c += blockDim.x) G[(int64_t)t * b + c] = 0.0;
    } else {
      for (int c = t + 1 + threadIdx.x; c < b; c += blockDim.x) G[(int64_t)t * b + c] /= rtt;
    }
    __syncthreads();
    if (!dead_s) {
      const int w = b - t - 1;
      for (int e = threadIdx.x; e < w * w; e += blockDim.x) {
        const int i = t + 1 + e / w, c = t + 1 + e % w;
        if (c >= i) G[(int64_t)i * b + c] -= G[(int64_t)t * b + i] * G[(int64_t)t * b + c];
      }
    }
    __syncthreads();
  }
  // zero the strict lower triangle so that G holds exactly R
  for (int e = threadIdx.x; e < b * b; e += blockDim.x)
    if (e / b > e % b) G[e] = 0.0;
  __syncthreads();
  // R^{-1} by back substitution, thread per column
  for (int c = threadIdx.x; c < b; c += blockDim.x) {
    for (int i = b - 1; i >= 0; --i) {
      double v;
      if (it.dead[i]) {
        v = 0.0;
      } else {
        v = (i == c) ? 1.0 : 0.0;
        for (int k = i + 1; k <= c; ++k) v -= G[(int64_t)i * b + k] * it.Rinv[(int64_t)k * b + c];
        v /= G[(int64_t)i * b + i];
      }
      if (i > c) v = 0.0;
      it.Rinv[(int64_t)i * b + c] = v;
    }
  }
}

// 1/sqrt(x): the hardware's approximation refined by two Newton steps; the plain operations far
// from 1
__device__ __forceinline__ double rsqrt_nr(double x) {
  if (!(x > 1e-280 && x < 1e280)) return 1.0 / sqrt(x);
  double r;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  r = fma(0.5 * r, fma(-x * r, r, 1.0), r);
  return fma(0.5 * r, fma(-x * r, r, 1.0), r);
}

// Up to order CH_SMALL (the widths of the Krylov and V_j blocks) the matrix lives in shared memory
// and the work is split in two launches: the factorisation, one CTA per matrix (b^3 / 6 FMAs at the 2
// per cycle of one SM, and a chain of about 0.5 us a step), then the inverse with CHI_COLS columns
// per CTA, so that its b^3 / 6 FMAs spread over the chip.  Order 120: 0.22 + 0.06 ms; 0.77 ms with
// chol_inv_kernel, whose inverse is one global-memory chain per column.
constexpr int CH_SMALL = 160;
constexpr int CHI_COLS = 8;
__global__ void __launch_bounds__(512) chol_small_kernel(CholBatchP bp, double tol, double *dinv_all) {
  const CholItem it = bp.it[blockIdx.x];
  const int b = it.b, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  extern __shared__ double S[];
  __shared__ double diag[CH_SMALL], dinv[CH_SMALL];
  __shared__ double thr_s;
  for (int e = tid; e < b * b; e += blockDim.x) S[e] = it.G[e];
  __syncthreads();
  if (warp == 0) {
    double m = 0.0;
    for (int i = lane; i < b; i += 32) m = fmax(m, S[i * b + i]);
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) thr_s = tol * m;
  }
  __syncthreads();
  const double thr = thr_s;
  // warp 0 turns row t (complete) into a row of R; one warp, because every warp that computes the
  // scalars takes 16 cycles of the SM's FP64 pipe per instruction
  auto finish_row = [&](int t) {
    const double pv = S[t * b + t];
    const bool dead = !(pv > thr) || !isfinite(pv);
    const double r = dead ? 0.0 : rsqrt_nr(pv);
    for (int c = t + 1 + lane; c < b; c += 32) S[t * b + c] *= r;
    if (lane == 0) {
      diag[t] = dead ? 0.0 : pv * r;
      dinv[t] = r;
      it.dead[t] = dead;
    }
  };
  if (warp == 0 && b > 0) finish_row(0);
  __syncthreads();
  for (int t = 0; t + 1 < b; ++t) {
    const bool live = dinv[t] != 0.0;
    // row t + 1 by warp 0, the others by the other warps
    for (int i = t + 1 + warp; i < b; i += warp == 0 ? b : nw - 1) {
      if (live) {
        const double g = S[t * b + i];
        for (int c = i + lane; c < b; c += 32) S[i * b + c] = fma(-g, S[t * b + c], S[i * b + c]);
      }
    }
    if (warp == 0) {
      __syncwarp();
      finish_row(t + 1);
    }
    __syncthreads();
  }
  for (int e = tid; e < b * b; e += blockDim.x) {
    const int i = e / b, c = e % b;
    it.G[e] = i < c ? (dinv[i] != 0.0 ? S[e] : 0.0) : i == c ? diag[i] : 0.0;
    if (i == c) dinv_all[(int64_t)blockIdx.x * CH_SMALL + i] = dinv[i];
  }
}

// X = R^{-1}, columns c0 .. c0 + CHI_COLS - 1: row i of X is final once every row below it has been
// eliminated, and is then subtracted from the rows above it.  Rows are scaled by 1/R_ii on the way
// out (0 for a dropped one).
__global__ void __launch_bounds__(256) chol_small_inv_kernel(CholBatchP bp, const double *__restrict__ dinv_all) {
  const CholItem it = bp.it[blockIdx.y];
  const int b = it.b, c0 = blockIdx.x * CHI_COLS, tid = threadIdx.x;
  if (c0 >= b) return;
  extern __shared__ double sm[];
  const int m = min(b, c0 + CHI_COLS);  // rows that can be nonzero
  double *R = sm, *X = sm + b * b;
  __shared__ double dinv[CH_SMALL];
  for (int e = tid; e < m * b; e += blockDim.x) R[e] = it.G[e];
  for (int e = tid; e < m; e += blockDim.x) dinv[e] = dinv_all[(int64_t)blockIdx.y * CH_SMALL + e];
  const int c = tid % CHI_COLS, rg = tid / CHI_COLS;
  constexpr int RG = 256 / CHI_COLS;
  for (int r = rg; r < m; r += RG) X[r * CHI_COLS + c] = r == c0 + c ? 1.0 : 0.0;
  __syncthreads();
  for (int i = m - 1; i > 0; --i) {
    const double xi = X[i * CHI_COLS + c] * dinv[i];
    for (int r = rg; r < i; r += RG) X[r * CHI_COLS + c] = fma(-R[r * b + i], xi, X[r * CHI_COLS + c]);
    __syncthreads();
  }
  if (c0 + c < b)
    for (int r = rg; r < b; r += RG)
      it.Rinv[(int64_t)r * b + c0 + c] = r < m ? X[r * CHI_COLS + c] * dinv[r] : 0.0;
}

void chol_inv_batched(cudaStream_t st, const std::vector<CholItem> &items, double tol) {
  for (size_t s = 0; s < items.size(); s += CH_MAXB) {
    CholBatchP b;
    memset(&b, 0, sizeof(b));
    const int cnt = (int)std::min<size_t>(CH_MAXB, items.size() - s);
    int bmax = 0;
    for (int i = 0; i < cnt; ++i) {
      b.it[i] = items[s + i];
      bmax = std::max(bmax, b.it[i].b);
    }
    if (bmax > CH_SMALL) {
      chol_inv_kernel<<<cnt, 512, 0, st>>>(b, tol);
      RFDD_CHECK_LAUNCH();
      continue;
    }
    const int sm1 = bmax * bmax * (int)sizeof(double), sm2 = sm1 + bmax * CHI_COLS * (int)sizeof(double);
    // always the same limits: several host threads launch these kernels at once
    RFDD_CUDA(cudaFuncSetAttribute(chol_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   CH_SMALL * CH_SMALL * (int)sizeof(double)));
    RFDD_CUDA(cudaFuncSetAttribute(chol_small_inv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   CH_SMALL * (CH_SMALL + CHI_COLS) * (int)sizeof(double)));
    double *dinv = nullptr;
    RFDD_CUDA(cudaMallocAsync((void **)&dinv, (size_t)cnt * CH_SMALL * sizeof(double), st));
    chol_small_kernel<<<cnt, 512, sm1, st>>>(b, tol, dinv);
    RFDD_CHECK_LAUNCH();
    chol_small_inv_kernel<<<dim3(ceil_div(bmax, CHI_COLS), cnt), 256, sm2, st>>>(b, dinv);
    RFDD_CHECK_LAUNCH();
    RFDD_CUDA(cudaFreeAsync(dinv, st));
  }
}

static int gridn(int64_t n) { return (int)std::min<int64_t>(std::max<int64_t>(1, (n + 255) / 256), 152 * 32); }

__global__ void scale_sym_kernel(double *A, int64_t k, const double *__restrict__ d) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < k * k; e += (int64_t)gridDim.x * blockDim.x)
    A[e] *= d[e / k] * d[e % k];
}
void scale_sym(cudaStream_t st, double *A, int64_t k, const double *d) {
  if (k <= 0) return;
  scale_sym_kernel<<<gridn(k * k), 256, 0, st>>>(A, k, d);
  RFDD_CHECK_LAUNCH();
}

__global__ void scale_rows_cols_kernel(const double *__restrict__ U, int64_t r, int64_t k, const double *__restrict__ d,
                                       const double *__restrict__ f, double *out) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < r * k; e += (int64_t)gridDim.x * blockDim.x)
    out[e] = U[e] * d[e % k] * f[e / k];
}
void scale_rows_cols(cudaStream_t st, const double *U, int64_t r, int64_t k, const double *d, const double *f,
                     double *out) {
  if (r * k <= 0) return;
  scale_rows_cols_kernel<<<gridn(r * k), 256, 0, st>>>(U, r, k, d, f, out);
  RFDD_CHECK_LAUNCH();
}

__global__ void inv_sqrt_diag_kernel(const double *__restrict__ G, int64_t k, double *d) {
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < k; c += (int64_t)gridDim.x * blockDim.x) {
    const double g = G[c * k + c];
    d[c] = g > 0.0 ? 1.0 / sqrt(g) : 0.0;
  }
}
void inv_sqrt_diag(cudaStream_t st, const double *G, int64_t k, double *d) {
  if (k <= 0) return;
  inv_sqrt_diag_kernel<<<gridn(k), 256, 0, st>>>(G, k, d);
  RFDD_CHECK_LAUNCH();
}

__global__ void inv_sqrt_vec_kernel(const double *__restrict__ lam, int64_t r, double *f) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < r; q += (int64_t)gridDim.x * blockDim.x)
    f[q] = 1.0 / sqrt(lam[q]);
}
void inv_sqrt_vec(cudaStream_t st, const double *lam, int64_t r, double *f) {
  if (r <= 0) return;
  inv_sqrt_vec_kernel<<<gridn(r), 256, 0, st>>>(lam, r, f);
  RFDD_CHECK_LAUNCH();
}

__global__ void ritz_residuals_kernel(const double *__restrict__ AX, const double *__restrict__ MX,
                                      const double *__restrict__ theta, int64_t n, int64_t b, double *res) {
  const int64_t c = blockIdx.x;
  const double th = theta[c];
  double sr = 0.0, sm = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
    const double mx = MX[i * b + c];
    const double r = AX[i * b + c] - th * mx;
    sr = fma(r, r, sr);
    sm = fma(mx, mx, sm);
  }
  __shared__ double r1[256], r2[256];
  r1[threadIdx.x] = sr;
  r2[threadIdx.x] = sm;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) { r1[threadIdx.x] += r1[threadIdx.x + o]; r2[threadIdx.x] += r2[threadIdx.x + o]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) res[c] = sqrt(r1[0]) / (fabs(th) * sqrt(r2[0]));
}
void ritz_residuals(cudaStream_t st, const double *AX, const double *MX, const double *theta, int64_t n, int64_t b,
                    double *res) {
  if (b <= 0) return;
  ritz_residuals_kernel<<<(unsigned)b, 256, 0, st>>>(AX, MX, theta, n, b, res);
  RFDD_CHECK_LAUNCH();
}

// out[c] = sum_i X[i][c] Y[i][c]  (n x b row-major blocks; fixed-order block reduction)
__global__ void col_dots_kernel(const double *__restrict__ X, const double *__restrict__ Y, int64_t n, int64_t b,
                                double *out) {
  const int64_t c = blockIdx.x;
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) s = fma(X[i * b + c], Y[i * b + c], s);
  __shared__ double r1[256];
  r1[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) r1[threadIdx.x] += r1[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[c] = r1[0];
}
void col_dots(cudaStream_t st, const double *X, const double *Y, int64_t n, int64_t b, double *out) {
  if (b <= 0) return;
  col_dots_kernel<<<(unsigned)b, 256, 0, st>>>(X, Y, n, b, out);
  RFDD_CHECK_LAUNCH();
}

template <typename T>
__global__ void sub_inplace_kernel(const T *__restrict__ x, T *__restrict__ y, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = y[i] - x[i];
}
template <typename T>
void sub_inplace(cudaStream_t st, const T *x, T *y, int64_t n) {
  if (n <= 0) return;
  sub_inplace_kernel<T><<<gridn(n), 256, 0, st>>>(x, y, n);
  RFDD_CHECK_LAUNCH();
}
template void sub_inplace<cx<float>>(cudaStream_t, const cx<float> *, cx<float> *, int64_t);
template void sub_inplace<cx<double>>(cudaStream_t, const cx<double> *, cx<double> *, int64_t);
template void sub_inplace<double>(cudaStream_t, const double *, double *, int64_t);

}  // namespace rfdd

namespace rfdd {

// ---------------------------------------------------------------------------------------
// Pivoted Cholesky P^T G P = R^T R in one cooperative launch, left-looking: G stays as it is (only its
// rows of chosen pivots are read), CTA c owns columns j = c mod G, and column j of R grows in row j of
// Rt.  Step t: every CTA offers the largest of its remaining diagonal entries (bit patterns compared as
// integers, smallest index on ties), one barrier, every CTA reads the offers of all, and the largest is the pivot p; the factorisation stops (rank = t) when it is <= tol
// or not finite.  Then r_t[j] = (G[p][j] - sum_s R[s][p] R[s][j]) / sqrt(d_p) and d_j -= r_t[j]^2 for the CTA's columns.
// k r^2 / 2 FP64 FMAs in all (7.7 ms of the chip's FP64 rate for k = 2720, r = 1884) and about 5 us a step: 384
// steps 2.1 ms (4.15 in two launches a step on the trailing triangle), the 2720 columns about 20 ms (50).
// *rank is 0 before the launch and written once, by a factorisation that has come to its end: where a barrier
// ran out it stays 0, and nothing indexes through perm, whose entries from the step on are not set.
// ---------------------------------------------------------------------------------------
constexpr int PCH_THREADS = 512;
constexpr int PCH_XMAX = 24 * 1024;  // entries of the pivot's column kept in shared memory

struct PchOffer {
  long long bits;  // of the largest remaining diagonal entry
  long long col;
};

__global__ void __launch_bounds__(PCH_THREADS) pchol_kernel(const double *__restrict__ Gm, int k, double *Rt, int *perm,
                                                            double tol, int *rank, PchOffer *offers, unsigned *bar,
                                                            int polls, int *status) {
  extern __shared__ double sm[];
  const int me = blockIdx.x, ng = gridDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = PCH_THREADS / 32;
  const int own = me < k ? (k - me + ng - 1) / ng : 0;
  double *d = sm, *xs = sm + (k + ng - 1) / ng;  // remaining diagonal of the own columns (-1: chosen); pivot column
  const bool x_in_smem = k <= PCH_XMAX;
  __shared__ int p_s;
  __shared__ double rinv_s, rdiag_s;
  for (int c = tid; c < own; c += PCH_THREADS) d[c] = Gm[(int64_t)(me + c * ng) * (k + 1)];
  __syncthreads();
  for (int t = 0; t < k; ++t) {
    long long bv = LLONG_MIN;
    int bi = INT_MAX;
    auto best = [&] {
      for (int o = 16; o > 0; o >>= 1) {
        const long long v2 = __shfl_xor_sync(0xffffffffu, bv, o);
        const int i2 = __shfl_xor_sync(0xffffffffu, bi, o);
        if (v2 > bv || (v2 == bv && i2 < bi)) { bv = v2; bi = i2; }
      }
    };
    PchOffer *of = offers + (size_t)(t & 1) * ng;  // two sets: a slow CTA may still read the last step's
    if (warp == 0) {
      for (int c = lane; c < own; c += 32) {
        const long long v = __double_as_longlong(d[c]);
        if (v > bv) { bv = v; bi = me + c * ng; }  // columns increase within a lane: the first maximum stays
      }
      best();
      if (lane == 0) of[me] = {bv, bi};
    }
    if (!grid_barrier(bar, (unsigned)ng * (unsigned)(t + 1), polls)) {
      if (tid == 0) atomicOr(status, DS_GRID_TIMEOUT);
      return;
    }
    if (warp == 0) {
      bv = LLONG_MIN;
      bi = INT_MAX;
      for (int c = lane; c < ng; c += 32) {
        const longlong2 w = __ldcg(reinterpret_cast<const longlong2 *>(of + c));
        if (w.x > bv || (w.x == bv && (int)w.y < bi)) { bv = w.x; bi = (int)w.y; }
      }
      best();
      if (lane == 0) {
        const double dp = bi < k ? __longlong_as_double(bv) : -1.0;
        const bool go = dp > tol && isfinite(dp);
        const double r = go ? rsqrt_nr(dp) : 0.0;
        p_s = go ? bi : -1;
        rinv_s = r;
        rdiag_s = dp * r;
      }
    }
    __syncthreads();
    const int p = p_s;
    if (p < 0) {
      if (me == 0 && tid == 0) *rank = t;
      return;
    }
    if (me == 0 && tid == 0) perm[t] = p;
    // column p of R (written by its owner, through L2)
    const double *xg = Rt + (int64_t)p * k;
    if (x_in_smem) {
      for (int s = tid; s < t; s += PCH_THREADS) xs[s] = __ldcg(xg + s);
      __syncthreads();
    }
    const double rinv = rinv_s;
    for (int c = warp; c < own; c += NW) {
      const int j = me + c * ng;
      if (d[c] < 0.0) continue;  // chosen before (the same in every lane)
      double *rj = Rt + (int64_t)j * k;
      if (j == p) {
        __syncwarp();
        if (lane == 0) {
          rj[t] = rdiag_s;
          d[c] = -1.0;
        }
        continue;
      }
      const double g = lane == 0 ? Gm[(int64_t)p * k + j] : 0.0;
      double a0 = 0.0, a1 = 0.0;
      int s = lane;
      if (x_in_smem) {
        for (; s + 96 < t; s += 128) {
          double r4[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) r4[u] = rj[s + 32 * u];
          a0 = fma(r4[0], xs[s], a0);
          a1 = fma(r4[1], xs[s + 32], a1);
          a0 = fma(r4[2], xs[s + 64], a0);
          a1 = fma(r4[3], xs[s + 96], a1);
        }
        for (; s < t; s += 32) a0 = fma(rj[s], xs[s], a0);
      } else {
        for (; s < t; s += 32) a0 = fma(rj[s], __ldcg(xg + s), a0);
      }
      a0 += a1;
      for (int o = 16; o > 0; o >>= 1) a0 += __shfl_xor_sync(0xffffffffu, a0, o);
      if (lane == 0) {
        const double v = (g - a0) * rinv;
        rj[t] = v;
        const double nd = fma(-v, v, d[c]);
        d[c] = nd <= 0.0 ? 0.0 : fabs(nd);  // a NaN stays and, being the largest pattern, ends the factorisation
      }
    }
    __syncthreads();
  }
  if (me == 0 && tid == 0) *rank = k;
}

// R into the leading r x r upper triangle of G: G[t][i] = Rt[perm[i]][t] for t <= i < r
__global__ void __launch_bounds__(256) pchol_gather_kernel(const double *__restrict__ Rt, const int *__restrict__ perm,
                                                           int k, const int *rank_p, double *G) {
  const int r = *rank_p;
  __shared__ double tile[32][33];
  const int i0 = blockIdx.x * 32, t0 = blockIdx.y * 32, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (i0 >= r || t0 >= r || i0 + 31 < t0) return;
  for (int q = w; q < 32; q += 8)
    if (i0 + q < r && t0 + lane < r) tile[q][lane] = Rt[(int64_t)perm[i0 + q] * k + t0 + lane];
  __syncthreads();
  for (int q = w; q < 32; q += 8) {
    const int t = t0 + q, i = i0 + lane;
    if (t < r && i < r && i >= t) G[(int64_t)t * k + i] = tile[lane][q];
  }
}

int pivoted_cholesky(cudaStream_t st, double *G, int k, int *perm, double tol, int *rank_dev, int *status, int polls,
                     int ctas) {
  if (polls <= 0) polls = GRID_SPIN;
  const int want = std::max(1, std::min(ctas > 0 ? ctas : sm_count(), k));
  auto smem_of = [&](int ng) { return ((size_t)ceil_div(k, ng) + (k <= PCH_XMAX ? k : 0)) * sizeof(double); };
  RFDD_REQUIRE(smem_of(want) <= 220 * 1024, RFDD_EINVAL, "pivoted Cholesky: order too large");
  RFDD_CUDA(cudaMemsetAsync(rank_dev, 0, sizeof(int), st));
  double *Rt = nullptr;
  PchOffer *offers = nullptr;
  RFDD_CUDA(cudaMallocAsync((void **)&Rt, (size_t)k * k * sizeof(double), st));
  RFDD_CUDA(cudaMallocAsync((void **)&offers, (size_t)2 * want * sizeof(PchOffer) + sizeof(unsigned), st));
  unsigned *bar = reinterpret_cast<unsigned *>(offers + 2 * want);
  RFDD_CUDA(cudaMemsetAsync(bar, 0, sizeof(unsigned), st));
  RFDD_CUDA(cudaFuncSetAttribute(pchol_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
  const int got = cooperative_launch(want, 1, [&](int ng) {
    if (smem_of(ng) > 220 * 1024) return cudaErrorCooperativeLaunchTooLarge;
    const double *Gc = G;
    void *args[] = {&Gc, &k, &Rt, &perm, &tol, &rank_dev, &offers, &bar, &polls, &status};
    return cudaLaunchCooperativeKernel((const void *)pchol_kernel, dim3(ng), dim3(PCH_THREADS), args, smem_of(ng), st);
  });
  RFDD_REQUIRE(got > 0, RFDD_ECUDA, "pivoted Cholesky: no room for its CTAs");
  const unsigned nt = (unsigned)ceil_div(k, 32);
  pchol_gather_kernel<<<dim3(nt, nt), 256, 0, st>>>(Rt, perm, k, rank_dev, G);
  RFDD_CHECK_LAUNCH();
  RFDD_CUDA(cudaFreeAsync(Rt, st));
  RFDD_CUDA(cudaFreeAsync(offers, st));
  int rank = 0;
  RFDD_CUDA(cudaMemcpyAsync(&rank, rank_dev, sizeof(int), cudaMemcpyDeviceToHost, st));
  RFDD_CUDA(cudaStreamSynchronize(st));
  return rank;
}

// out[i][j] = K[perm[i]][perm[j]] for i, j < r
__global__ void gather_sym_kernel(const double *__restrict__ K, int k, const int *__restrict__ perm, int r,
                                  double *out) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < (int64_t)r * r; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / r), j = (int)(e % r);
    out[e] = K[(int64_t)perm[i] * k + perm[j]];
  }
}
void gather_sym(cudaStream_t st, const double *K, int k, const int *perm, int r, double *out) {
  if (r <= 0) return;
  gather_sym_kernel<<<gridn((int64_t)r * r), 256, 0, st>>>(K, k, perm, r, out);
  RFDD_CHECK_LAUNCH();
}

// Lt[i][j] = R[j][i] / R[j][j] (j < i), 1 (j == i), 0 (j > i): unit lower, from upper R (ld ldr)
__global__ void unit_lower_from_upper_kernel(const double *__restrict__ R, int ldr, int r, double *Lt) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < (int64_t)r * r; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / r), j = (int)(e % r);
    Lt[e] = j < i ? R[(int64_t)j * ldr + i] / R[(int64_t)j * ldr + j] : (i == j ? 1.0 : 0.0);
  }
}
void unit_lower_from_upper(cudaStream_t st, const double *R, int ldr, int r, double *Lt) {
  if (r <= 0) return;
  unit_lower_from_upper_kernel<<<gridn((int64_t)r * r), 256, 0, st>>>(R, ldr, r, Lt);
  RFDD_CHECK_LAUNCH();
}

// out[i][j] = (A[i][j] + A[j][i]) / (2 R_ii R_jj) (r x r), into a separate buffer
__global__ void symmetrize_scaled_kernel(const double *__restrict__ A, int r, const double *__restrict__ R, int ldr,
                                         double *out) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < (int64_t)r * r; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / r), j = (int)(e % r);
    const double d = R[(int64_t)i * (ldr + 1)] * R[(int64_t)j * (ldr + 1)];
    out[e] = 0.5 * (A[e] + A[(int64_t)j * r + i]) / d;
  }
}
void symmetrize_scaled(cudaStream_t st, const double *A, int r, const double *R, int ldr, double *out) {
  if (r <= 0) return;
  symmetrize_scaled_kernel<<<gridn((int64_t)r * r), 256, 0, st>>>(A, r, R, ldr, out);
  RFDD_CHECK_LAUNCH();
}

// out (b x a) = in^T (in: a x b row-major)
__global__ void transpose_kernel(const double *__restrict__ in, int a, int b, double *out) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < (int64_t)a * b; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / b), j = (int)(e % b);
    out[(int64_t)j * a + i] = in[e];
  }
}
void transpose(cudaStream_t st, const double *in, int a, int b, double *out) {
  if ((int64_t)a * b <= 0) return;
  transpose_kernel<<<gridn((int64_t)a * b), 256, 0, st>>>(in, a, b, out);
  RFDD_CHECK_LAUNCH();
}

// Cfull[perm[i]][c] = d[perm[i]] * Cr[i][c] for i < r (other rows untouched; caller zeroes)
__global__ void scatter_rows_kernel(const double *__restrict__ Cr, int r, int ns, const int *__restrict__ perm,
                                    const double *__restrict__ d, double *Cfull) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < (int64_t)r * ns; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / ns), c = (int)(e % ns);
    const int row = perm[i];
    Cfull[(int64_t)row * ns + c] = d[row] * Cr[e];
  }
}
void scatter_rows_perm(cudaStream_t st, const double *Cr, int r, int ns, const int *perm, const double *d,
                       double *Cfull) {
  if ((int64_t)r * ns <= 0) return;
  scatter_rows_kernel<<<gridn((int64_t)r * ns), 256, 0, st>>>(Cr, r, ns, perm, d, Cfull);
  RFDD_CHECK_LAUNCH();
}


// G[c][r] = G[r][c] for r in [r0, r1), c in [c0, c1)  (k x k row-major)
__global__ void mirror_block_kernel(double *G, int64_t k, int64_t r0, int64_t r1, int64_t c0, int64_t c1) {
  const int64_t w = c1 - c0, total = (r1 - r0) * w;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = r0 + e / w, c = c0 + e % w;
    G[c * k + r] = G[r * k + c];
  }
}
void mirror_block(cudaStream_t st, double *G, int64_t k, int64_t r0, int64_t r1, int64_t c0, int64_t c1) {
  if (r1 <= r0 || c1 <= c0) return;
  mirror_block_kernel<<<gridn((r1 - r0) * (c1 - c0)), 256, 0, st>>>(G, k, r0, r1, c0, c1);
  RFDD_CHECK_LAUNCH();
}

}  // namespace rfdd
