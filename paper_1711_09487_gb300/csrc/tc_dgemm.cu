// FP64 GEMM on the tensor cores by exact digit products.
//
// Every row of op(A) and every column of op(B) is scaled by a power of two and rounded to a 63-bit
// fixed-point integer (entries down to 2^-9 of the largest are exact), which is cut into eight balanced base-256
// digits (-128 .. 127), each exact in fp16.  The products of digit planes with equal weight, i + j = g, are summed by
// tcgen05 kind::f16 MMAs into one of eight FP32 accumulators: all addends are integers and their sums stay within 2^24
// (8 pairs x 128 x 2^14), so every accumulator is exact.  After at most 128 terms of K (256 for the four of the leading
// planes, which sum fewer products) they are read back and added into two 64-bit integers per entry, which hold the sum
// exactly up to the planes that are left out (i + j > 7); one rounding to FP64 at the end.  This is the splitting of
// Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012) with integer digits.
//
// Before that, the terms of the sum are brought to one size: column k of op(A) is divided, and row k of op(B) multiplied, by the
// power of two of the column's largest entry (exponents only, exact).  Rows and columns scaled by factors of their own
// (D A D for a diagonal D, whose factors and bases are graded along the sums) then lose nothing.
//
// Error of an entry: k 2^-57 (largest |a| of its row) (largest |b| of its column) of the operands so scaled, and the
// roundings of the result.  For operands within a few powers of two of their largest entries that is below the
// error of the sum in FP64, whatever its order.  (Digits of seven bits, 512 terms to a read-back, left out planes of
// 2^-49 of the largest product: 7 ulp on operands whose digits have one sign.)
//
// What bounds it: the 36 plane products of a 128 x 64 x 32 stage read 12 KB of shared memory per 32
// cycles of MMA, by the descriptors, and a stage takes about 3500 cycles; the read-back (conversions and 64-bit
// additions of 64 k sums, about 7000 cycles for all eight accumulators) comes on top, because they fill the tensor
// memory.  Measured, without the packing: symmetric 1920 x 1920 x 64000 10.0 ms, 1885 x 1885 x 8000 1.27 ms (symmetric)
// and 1.90; with seven-bit digits, one read-back in 512 terms, 8.9, 1.12 and 1.67; with eight warps for the read-back and all
// accumulators every 128 terms 11.0, 1.39 and 2.07.
#include "dense.cuh"
#include "tc_common.cuh"
#include "tc_gemm.cuh"

#include <algorithm>

namespace rfdd {

namespace {

constexpr int DG_BM = 128, DG_BN = 64, DG_KT = 32;  // output tile, K of a stage
constexpr int DG_PLANES = 8, DG_PAIRS = DG_PLANES / 2;  // a 128-byte tile row holds 32 K-values of two planes
constexpr int DG_ATILE = DG_BM * 128, DG_BTILE = DG_BN * 128;  // bytes of one plane pair
constexpr int DG_ABYTES = DG_PAIRS * DG_ATILE, DG_BBYTES = DG_PAIRS * DG_BTILE;
constexpr int DG_STAGE = DG_ABYTES + DG_BBYTES;  // 96 KB
constexpr int DG_STAGES = 2;
constexpr int DG_BITS = 8;     // bits of a digit
constexpr int DG_CHUNK = 4;    // stages between two read-backs (128 terms)
constexpr int DG_SPLIT = 16;   // stages of the shallowest share of a split K (512 terms)
// Accumulator g sums g + 1 plane products: the four of the upper half stay exact for two chunks and are read back, and
// start anew, with every second one.
static_assert(DG_PLANES * DG_CHUNK * DG_KT << 2 * (DG_BITS - 1) <= 1 << 24, "the accumulators stay exact");
static_assert(DG_PLANES / 2 * 2 * DG_CHUNK * DG_KT << 2 * (DG_BITS - 1) <= 1 << 24, "the upper ones for two chunks");
constexpr int DG_SMEM = DG_STAGES * DG_STAGE + 1024;
constexpr int DG_EPI_WARPS = 16;  // four to each lane quarter of the accumulators
constexpr int DG_EC = DG_BN / (DG_EPI_WARPS / 4);  // columns a read-back warp takes
static_assert(DG_EC == 16, "tcgen05.ld x16");
constexpr int DG_THREADS = 64 + 32 * DG_EPI_WARPS;
constexpr int DG_MAXB = 32;

// One operand: vectors (rows of op(A), columns of op(B)) of length k
struct DigitItem {
  const double *src;
  long long ld;
  int nv, k;        // vectors, length
  int mode;         // entry (v, k): 0 at src[k * ld + v]; 1 at src[v * ld + k]; 2: vector 2j + t, entry 2p + u of
                    // the realified complex column j, [[re, im], [-im, re]] (rows u, columns t) of src[p * ld + j]
  int vb;           // vectors per tile (128 or 64)
  int nkt;
  uint8_t *dst;
  int *emax;        // per vector: largest scaled exponent (term_exp)
  int *kexp;        // per K-value: exponent of the largest entry of the column of op(A)
  int ksign;        // -1: op(A), which is divided by these powers of two; 1: op(B)
};
struct DigitBatch {
  DigitItem it[2 * DG_MAXB];
  int count;
};

constexpr int DG_INF = 1 << 20;          // "exponent" of infinities and NaN
constexpr int DG_NONE_BYTE = 0x80;       // exponents start as words of this byte, below that of any entry (zeros)
constexpr int DG_NONE = (int)0x80808080u;

// Biased exponent of x (1 for subnormal numbers), DG_NONE for zero, DG_INF for infinities and NaN; integer instructions
__device__ __forceinline__ int term_exp(double x) {
  const int hi = __double2hiint(x) & 0x7fffffff;
  if ((hi | __double2loint(x)) == 0) return DG_NONE;
  const int ex = hi >> 20;
  return ex == 0x7ff ? DG_INF : max(ex, 1);
}
// the same with off added to the exponent of a finite nonzero x
__device__ __forceinline__ int term_exp(double x, int off) {
  const int ex = term_exp(x);
  return ex == DG_NONE || ex == DG_INF ? ex : ex + off;
}

// Largest exponent of every column of op(A), into kexp (DG_NONE before); entries that are not finite do not count.
__global__ void __launch_bounds__(256) digit_kexp_kernel(const __grid_constant__ DigitBatch b) {
  const DigitItem &it = b.it[blockIdx.y];
  if (it.ksign > 0) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto e = [](double x) {
    const int ex = term_exp(x);
    return ex == DG_INF ? DG_NONE : ex;
  };
  if (it.mode == 0) {  // a column of op(A) is contiguous
    for (int k = blockIdx.x * 8 + warp; k < it.k; k += gridDim.x * 8) {
      const double *s = it.src + (long long)k * it.ld;
      int m = DG_NONE;
      for (int v = lane; v < it.nv; v += 32) m = max(m, e(s[v]));
      m = __reduce_max_sync(0xffffffffu, m);
      if (lane == 0) it.kexp[k] = m;
    }
    return;
  }
  // 32 columns x 256 rows per block step
  const int nkb = (it.k + 31) / 32, nvb = (it.nv + 255) / 256;
  for (int u = blockIdx.x; u < nkb * nvb; u += gridDim.x) {
    const int k = (u % nkb) * 32 + lane, v0 = (u / nkb) * 256 + warp;
    int m = DG_NONE;
    if (k < it.k)
#pragma unroll 8
      for (int q = 0; q < 32; ++q) {
        const int v = v0 + 8 * q;
        if (v < it.nv) m = max(m, e(it.src[(long long)v * it.ld + k]));
      }
    if (m != DG_NONE) atomicMax(it.kexp + k, m);
  }
}

// Largest scaled exponent of every vector, into emax (DG_NONE before).
__global__ void __launch_bounds__(256) digit_emax_kernel(const __grid_constant__ DigitBatch b) {
  const DigitItem &it = b.it[blockIdx.y];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (it.mode == 1) {
    for (int v = blockIdx.x * 8 + warp; v < it.nv; v += gridDim.x * 8) {
      const double *s = it.src + (long long)v * it.ld;
      int m = DG_NONE;
      for (int k = lane; k < it.k; k += 32) m = max(m, term_exp(s[k], it.ksign * it.kexp[k]));
      m = __reduce_max_sync(0xffffffffu, m);
      if (lane == 0) it.emax[v] = m;
    }
    return;
  }
  // 32 columns (of doubles or of complex pairs) x 256 rows per block step
  const int f = it.mode == 2 ? 2 : 1;
  const int nc = it.nv / f, kr = it.k / f;
  const int nvb = (nc + 31) / 32, nkb = (kr + 255) / 256;
  for (int u = blockIdx.x; u < nvb * nkb; u += gridDim.x) {
    const int v = (u % nvb) * 32 + lane, k0 = (u / nvb) * 256 + warp;
    int m = DG_NONE, m1 = DG_NONE;
    if (v < nc)
#pragma unroll 8
      for (int q = 0; q < 32; ++q) {
        const int k = k0 + 8 * q;
        if (k < kr) {
          const double *s = it.src + ((long long)k * it.ld + v) * f;
          if (f == 1) {
            m = max(m, term_exp(s[0], it.ksign * it.kexp[k]));
          } else {  // column 2 v: re, -im; column 2 v + 1: im, re
            const int o0 = it.ksign * it.kexp[2 * k], o1 = it.ksign * it.kexp[2 * k + 1];
            m = max(m, max(term_exp(s[0], o0), term_exp(s[1], o1)));
            m1 = max(m1, max(term_exp(s[1], o0), term_exp(s[0], o1)));
          }
        }
      }
    if (m != DG_NONE) atomicMax(it.emax + v * f, m);
    if (m1 != DG_NONE) atomicMax(it.emax + 2 * v + 1, m1);
  }
}

// Fixed point of x, its exponent shifted by off, for a vector whose largest such exponent is em: the integer nearest to
// x 2^(off + 1084 - em), |q| < 2^62.
__device__ __forceinline__ long long fixed63(double x, int off, int em) {
  const long long bits = __double_as_longlong(x);
  const int ex = (int)((bits >> 52) & 0x7ff);
  long long m = bits & 0xfffffffffffffll;
  if (ex > 0) m |= 1ll << 52;
  if (em == DG_INF || ex == 0x7ff || m == 0) return 0;  // infinities and NaN: the vector's products are NaN
  // m < 2^53; the largest entry becomes m * 2^9, smaller exponents shift right
  const int sh = em - (max(ex, 1) + off) - 9;
  long long q;
  if (sh <= 0) q = m << -sh;
  else if (sh > 54) q = 0;
  else q = (m + (1ll << (sh - 1))) >> sh;
  return bits < 0 ? -q : q;
}

// v 2^e: by the exponent field where the result is normal (the FP64 pipe is slow), else by scalbn
__device__ __forceinline__ double scale_exp(double v, int e) {
  const int ex = (__double2hiint(v) >> 20) & 0x7ff;
  if (ex == 0) return v;  // zero (|v| is an integer)
  if (ex + e >= 1 && ex + e <= 2046) return __hiloint2double(__double2hiint(v) + (e << 20), __double2loint(v));
  return scalbn(v, e);
}

// Digits of every operand into swizzled tiles: tile (v / vb, k / 32), four plane pairs of vb rows x 128 bytes;
// 16-byte chunk c of a row holds plane 2 * pair + c / 4, K-values 8 (c % 4) .. + 7, at chunk c ^ (row & 7).  A
// block stages 64 vectors x 32 K-values.
__global__ void __launch_bounds__(256) digit_pack_kernel(const __grid_constant__ DigitBatch b) {
  const DigitItem &it = b.it[blockIdx.y];
  __shared__ double sx[64][33];
  __shared__ int soff[DG_KT];
  const int tid = threadIdx.x;
  const int nvb = (it.nv + 63) / 64, total = nvb * it.nkt;
  for (int u = blockIdx.x; u < total; u += gridDim.x) {
    const int v0 = (u / it.nkt) * 64, kt = u % it.nkt, k0 = kt * DG_KT;
    __syncthreads();
    if (tid < DG_KT) soff[tid] = k0 + tid < it.k ? it.ksign * it.kexp[k0 + tid] : 0;
    if (it.mode == 2) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int id = tid + 256 * q, j = id & 31, p = id >> 5;
        double re = 0.0, im = 0.0;
        if (v0 + 2 * j < it.nv && k0 + 2 * p < it.k) {
          const double *s = it.src + 2 * ((long long)(k0 / 2 + p) * it.ld + v0 / 2 + j);
          re = s[0];
          im = s[1];
        }
        sx[2 * j][2 * p] = re;
        sx[2 * j][2 * p + 1] = -im;
        sx[2 * j + 1][2 * p] = im;
        sx[2 * j + 1][2 * p + 1] = re;
      }
    } else {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int id = tid + 256 * q;
        const int v = it.mode ? id >> 5 : id & 63, k = it.mode ? id & 31 : id >> 6;
        double x = 0.0;
        if (v0 + v < it.nv && k0 + k < it.k)
          x = it.mode ? it.src[(long long)(v0 + v) * it.ld + k0 + k] : it.src[(long long)(k0 + k) * it.ld + v0 + v];
        sx[v][k] = x;
      }
    }
    __syncthreads();
    const int v = tid >> 2, g = tid & 3;  // 8 K-values of one vector
    const int em = v0 + v < it.nv ? it.emax[v0 + v] : DG_NONE;
    uint32_t w[DG_PLANES][4];
#pragma unroll
    for (int e = 0; e < 8; e += 2) {
      // q + sum_s 128 * 256^s has the digits plus 128 as its bytes
      constexpr unsigned long long off = 0x8080808080808080ull;
      const unsigned long long a = (unsigned long long)fixed63(sx[v][g * 8 + e], soff[g * 8 + e], em) + off;
      const unsigned long long c = (unsigned long long)fixed63(sx[v][g * 8 + e + 1], soff[g * 8 + e + 1], em) + off;
#pragma unroll
      for (int s = 0; s < DG_PLANES; ++s) {
        const int shift = DG_BITS * (DG_PLANES - 1 - s);  // plane 0 is the leading digit
        const uint32_t d = ((uint32_t)(a >> shift) & 255u) | (((uint32_t)(c >> shift) & 255u) << 16);
        // fp16(1024 + u) - 1152 = u - 128, exactly
        const uint32_t h = d | 0x64006400u;
        __half2 x = *reinterpret_cast<const __half2 *>(&h);
        x = __hsub2(x, __half2half2(__ushort_as_half(0x6480)));
        w[s][e >> 1] = *reinterpret_cast<uint32_t *>(&x);
      }
    }
    const int vv = v0 + v, r = vv % it.vb;
    uint8_t *t = it.dst + ((long long)(vv / it.vb) * it.nkt + kt) * DG_PAIRS * it.vb * 128 + r * 128;
#pragma unroll
    for (int s = 0; s < DG_PLANES; ++s) {
      const int c = (s & 1) * 4 + g;
      *reinterpret_cast<uint4 *>(t + (s >> 1) * it.vb * 128 + ((c ^ (r & 7)) << 4)) =
          make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
    }
  }
}

struct DgItem {
  const uint8_t *A, *B;
  const int *ea, *eb;
  double *C, *ws;      // ws: partial sums (split K), nsplit slabs of m x n
  long long ldc;
  int m, n, nkt, ntc;  // ntc: 64-wide tiles per row of tiles
  int nsplit, kper;    // K splits and stages per split
  int sym, unit0;      // first work unit (tile, split)
};
struct DgBatch {
  DgItem it[DG_MAXB];
  int count, units;
  int *err;
};

// Work unit -> tile row, tile column, split.  A symmetric product keeps the tiles that reach the upper
// triangle: tile row mt has the columns from 2 mt on.
__device__ __forceinline__ void dg_unit(const DgItem &it, int u, int &mt, int &nt, int &sp) {
  sp = u % it.nsplit;
  int t = u / it.nsplit;
  if (!it.sym) {
    mt = t / it.ntc;
    nt = t % it.ntc;
    return;
  }
  mt = 0;
  while (t >= it.ntc - 2 * mt) {
    t -= it.ntc - 2 * mt;
    ++mt;
  }
  nt = 2 * mt + t;
}

__global__ void __launch_bounds__(DG_THREADS, 1) tc_dgemm_kernel(const __grid_constant__ DgBatch b, double alpha,
                                                                 double beta) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full_bar[DG_STAGES], empty_bar[DG_STAGES], tfull_bar, tempty_bar, drain_bar;
  __shared__ uint32_t tmem_s;
  __shared__ volatile int abort_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < DG_STAGES; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    mbar_init(smem_u32(&tfull_bar), 1);
    mbar_init(smem_u32(&drain_bar), 1);
    mbar_init(smem_u32(&tempty_bar), 32 * DG_EPI_WARPS);
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_s)),
                 "r"(DG_PLANES * DG_BN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_s;
  auto find = [&](int u) {
    int lo = 0, hi = b.count;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (b.it[mid].unit0 <= u) lo = mid;
      else hi = mid;
    }
    return lo;
  };
  if (warp == 0) {
    if (lane == 0) {  // producer: 96 KB of digits per stage
      long long g = 0;
      for (int u = blockIdx.x; u < b.units && !abort_s; u += gridDim.x) {
        const DgItem &it = b.it[find(u)];
        int mt, nt, sp;
        dg_unit(it, u - it.unit0, mt, nt, sp);
        const int kb = sp * it.kper, ke = min(it.nkt, kb + it.kper);
        const uint8_t *A = it.A + (long long)mt * it.nkt * DG_ABYTES, *B = it.B + (long long)nt * it.nkt * DG_BBYTES;
        for (int kt = kb; kt < ke; ++kt, ++g) {
          const int s = (int)(g % DG_STAGES);
          const long long r = g / DG_STAGES;
          if (r >= 1 && !mbar_wait(smem_u32(&empty_bar[s]), (uint32_t)((r - 1) & 1), &abort_s)) {
            atomicOr(b.err, DS_WAIT_TIMEOUT);
            abort_s = 1;
            break;
          }
          const uint32_t fb = smem_u32(&full_bar[s]), dst = smem_u32(base + s * DG_STAGE);
          mbar_expect_tx(fb, DG_STAGE);
          bulk_g2s(dst, A + (long long)kt * DG_ABYTES, DG_ABYTES, fb);
          bulk_g2s(dst + DG_ABYTES, B + (long long)kt * DG_BBYTES, DG_BBYTES, fb);
        }
      }
      // every issued copy lands before the CTA can exit, after an abort too
      for (long long q = (g > DG_STAGES ? g - DG_STAGES : 0); q < g; ++q)
        mbar_drain(smem_u32(&full_bar[q % DG_STAGES]), (uint32_t)((q / DG_STAGES) & 1));
    }
  } else if (warp == 1) {
    if (lane == 0) {  // MMA issuer
      const uint32_t idesc = (1u << 4) | ((uint32_t)(DG_BN >> 3) << 17) | ((uint32_t)(DG_BM >> 4) << 24);
      long long g = 0, ch = 0;  // stages, read-backs
      bool ok = true;
      for (int u = blockIdx.x; u < b.units && ok && !abort_s; u += gridDim.x) {
        const DgItem &it = b.it[find(u)];
        int mt, nt, sp;
        dg_unit(it, u - it.unit0, mt, nt, sp);
        const int kb = sp * it.kper, ke = min(it.nkt, kb + it.kper);
        for (int k0 = kb; k0 < ke && ok; k0 += DG_CHUNK, ++ch) {
          if (ch >= 1 && !mbar_wait(smem_u32(&tempty_bar), (uint32_t)((ch - 1) & 1), &abort_s)) {
            ok = false;
            break;
          }
          fence_after();
          const int k1 = min(ke, k0 + DG_CHUNK);
          const bool second = ((k0 - kb) / DG_CHUNK & 1) != 0;  // the upper accumulators go on
          for (int kt = k0; kt < k1; ++kt, ++g) {
            const int s = (int)(g % DG_STAGES);
            if (!mbar_wait(smem_u32(&full_bar[s]), (uint32_t)((g / DG_STAGES) & 1), &abort_s)) {
              ok = false;
              break;
            }
            fence_after();
            const uint32_t sa = smem_u32(base + s * DG_STAGE), sb = sa + DG_ABYTES;
#pragma unroll 1
            for (int kk = 0; kk < 2; ++kk) {
#pragma unroll
              for (int i = 0; i < DG_PLANES; ++i) {
                const uint64_t da = sdesc(sa + (i >> 1) * DG_ATILE + (i & 1) * 64 + kk * 32);
#pragma unroll
                for (int j = 0; j < DG_PLANES - i; ++j)
                  mma_f16(tmem + (uint32_t)((i + j) * DG_BN), da, sdesc(sb + (j >> 1) * DG_BTILE + (j & 1) * 64 + kk * 32),
                          idesc, (kt > k0 || kk > 0 || i > 0 || (second && i + j < DG_PLANES / 2)) ? 1u : 0u);
              }
            }
            mma_commit(smem_u32(&empty_bar[s]));
          }
          if (ok) mma_commit(smem_u32(&tfull_bar));
        }
      }
      if (!ok) {
        atomicOr(b.err, DS_WAIT_TIMEOUT);
        abort_s = 1;
      }
      // every issued MMA ends before the tensor memory is freed, after an abort too
      mma_commit(smem_u32(&drain_bar));
      mbar_drain(smem_u32(&drain_bar), 0);
    }
  } else {
    // read-back: warp w takes accumulator lanes 32 (w % 4) .. (its rows) and a quarter of the columns
    const int q = warp & 3, part = (warp - 2) >> 2;
    long long ch = 0;
    bool ok = true;
    for (int u = blockIdx.x; u < b.units && ok; u += gridDim.x) {
      const DgItem &it = b.it[find(u)];
      int mt, nt, sp;
      dg_unit(it, u - it.unit0, mt, nt, sp);
      const int kb = sp * it.kper, ke = min(it.nkt, kb + it.kper);
      long long hi[DG_EC], lo[DG_EC];
#pragma unroll
      for (int j = 0; j < DG_EC; ++j) hi[j] = lo[j] = 0;
      for (int k0 = kb; k0 < ke; k0 += DG_CHUNK, ++ch) {
        const bool ready = mbar_wait(smem_u32(&tfull_bar), (uint32_t)(ch & 1), &abort_s);
        if (!__all_sync(0xffffffffu, ready && !abort_s)) {
          if (lane == 0) atomicOr(b.err, DS_WAIT_TIMEOUT);
          abort_s = 1;
          ok = false;
          break;
        }
        fence_after();
        const uint32_t t0 = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(part * DG_EC);
        const bool all = ((k0 - kb) / DG_CHUNK & 1) != 0 || k0 + DG_CHUNK >= ke;
#pragma unroll
        for (int g = 0; g < DG_PLANES; ++g) {
          if (g < DG_PLANES / 2 && !all) continue;
          uint32_t v[DG_EC];
          TC_LD16(t0 + (uint32_t)(g * DG_BN), v);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (g == DG_PLANES - 1) {
            fence_before();
            mbar_arrive(smem_u32(&tempty_bar));
          }
#pragma unroll
          for (int j = 0; j < DG_EC; ++j) {
            const int x = __float2int_rn(__uint_as_float(v[j]));
            if (g < 4) hi[j] += (long long)x * (1 << (DG_BITS * (3 - g)));
            else lo[j] += (long long)x * (1 << (DG_BITS * (7 - g)));
          }
        }
      }
      if (!ok) break;
      // planes 0 and 0 weigh 2^112 in units of the two integers; hi counts 2^88, lo 2^56
      const int i = mt * DG_BM + q * 32 + lane;
      if (i < it.m) {
        const int eai = it.ea[i];
        const int xa = eai - 2 * 1084 + 56;  // one unit of a product of two integers is 2^(ea + eb - 2 * 1084)
        const int j0 = nt * DG_BN + part * DG_EC;
#pragma unroll
        for (int j = 0; j < DG_EC; ++j) {
          const int c = j0 + j;
          if (c >= it.n) continue;
          const int ebj = it.eb[c];
          double v = fma((double)hi[j], 4294967296.0, (double)lo[j]);
          v = scale_exp(v, xa + ebj);
          if (eai == DG_INF || ebj == DG_INF) v = __longlong_as_double(0x7ff8000000000000ll);
          if (it.nsplit > 1) {
            it.ws[((long long)sp * it.m + i) * it.n + c] = v;
            continue;
          }
          if (it.sym && i > c) continue;
          v *= alpha;
          double *p = it.C + (long long)i * it.ldc + c;
          *p = beta != 0.0 ? fma(beta, *p, v) : v;
          if (it.sym && i != c) {
            double *pm = it.C + (long long)c * it.ldc + i;
            *pm = beta != 0.0 ? fma(beta, *pm, v) : v;
          }
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(DG_PLANES * DG_BN) : "memory");
}

// Split K: the partial sums of every entry, in order
__global__ void __launch_bounds__(256) tc_dgemm_reduce_kernel(const __grid_constant__ DgBatch b, double alpha,
                                                              double beta) {
  const DgItem &it = b.it[blockIdx.y];
  if (it.nsplit <= 1) return;
  const long long mn = (long long)it.m * it.n;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < mn; e += (long long)gridDim.x * blockDim.x) {
    const long long i = e / it.n, j = e % it.n;
    const long long src = it.sym && i > j ? j * it.n + i : e;  // exactly symmetric result
    double v = it.ws[src];
    for (int s = 1; s < it.nsplit; ++s) v += it.ws[s * mn + src];
    v *= alpha;
    double *p = it.C + i * it.ldc + j;
    *p = beta != 0.0 ? fma(beta, *p, v) : v;
  }
}

}  // namespace

// C = beta*C + alpha*op(A)*op(B) on real sizes; amode, bmode: how the operands are read (DigitItem::mode)
struct DgGemm {
  const double *A, *B;
  double *C;
  int m, n, k, lda, ldb;
  long long ldc;
  int amode, bmode, sym;
};

// bytes of digits of both operands per unit of K: 8 planes of 2 bytes, rows padded to tiles
static double digit_bytes_per_k(int64_t m, int64_t n) {
  return 16.0 * ((m + DG_BM - 1) / DG_BM * DG_BM + (n + DG_BN - 1) / DG_BN * DG_BN);
}
// whether 512 terms of an m x n x k product (or all of them) fit in the scope's bytes
static bool digits_fit(int64_t m, int64_t n, int64_t k) {
  const double kp = std::min<double>(512.0, (k + DG_KT - 1) / DG_KT * DG_KT);
  return digit_bytes_per_k(m, n) * kp <= (double)tc_digit_rule().bytes;
}

static void dgemm_run(cudaStream_t st, const std::vector<DgGemm> &items, double alpha, double beta) {
  const double cap = (double)tc_digit_rule().bytes;
  RFDD_REQUIRE(tc_status_word() != nullptr, RFDD_ESTATE, "tensor-core GEMM launched without a status word");
  const int nsm = sm_count();
  RFDD_CUDA(cudaFuncSetAttribute(tc_dgemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, DG_SMEM));
  for (size_t s0 = 0, cnt = 0; s0 < items.size(); s0 += cnt) {
    // as many items as keep the digits of 512 terms within the scope's bytes (one does, see the takes functions)
    int kmax = 0;
    double per_k = 0.0;  // bytes of digits per unit of K
    for (cnt = 0; cnt < (size_t)DG_MAXB && s0 + cnt < items.size(); ++cnt) {
      const auto &g = items[s0 + cnt];
      const double b = digit_bytes_per_k(g.m, g.n);
      if (cnt > 0 && (per_k + b) * std::min(512, std::max(kmax, g.k)) > cap) break;
      kmax = std::max(kmax, g.k);
      per_k += b;
    }
    // K in passes whose digits fit; every pass but the first adds to C
    const int kpass = std::min<double>(kmax, std::max(512.0, std::floor(cap / per_k / 512.0) * 512.0));
    for (int kp = 0; kp < kmax; kp += kpass) {
      DigitBatch db;
      DgBatch gb;
      memset(&db, 0, sizeof(db));
      memset(&gb, 0, sizeof(gb));
      size_t bytes = 0, vecs = 0, wsum = 0;
      struct Src { const double *p; int ld, nv, k, mode, vb, with; size_t off, ev, kv; };
      // operands, each packed once even when several items use it; with: -1 for an op(A), which sets the powers of two
      // along K, else the op(A) that the operand is scaled for
      std::vector<Src> srcs;
      auto operand = [&](const double *p, int ld, int nv, int k, int mode, int vb, int with) {
        for (size_t q = 0; q < srcs.size(); ++q)
          if (srcs[q].p == p && srcs[q].ld == ld && srcs[q].nv == nv && srcs[q].k == k && srcs[q].mode == mode && srcs[q].vb == vb &&
              srcs[q].with == with)
            return (int)q;
        const size_t nkt = (k + DG_KT - 1) / DG_KT, tiles = (nv + vb - 1) / vb;
        srcs.push_back({p, ld, nv, k, mode, vb, with, bytes, vecs, with < 0 ? vecs + (size_t)(nv + 63) / 64 * 64 : srcs[with].kv});
        bytes += tiles * nkt * DG_PAIRS * vb * 128;
        vecs += (size_t)(nv + 63) / 64 * 64 + (with < 0 ? (size_t)(k + 63) / 64 * 64 : 0);
        return (int)srcs.size() - 1;
      };
      std::vector<int> ia, ib;
      double work = 0.0;
      for (int i = 0; i < (int)cnt; ++i) {
        const auto &g = items[s0 + i];
        const int k = std::min(kpass, g.k - kp);
        ia.push_back(-1);
        ib.push_back(-1);
        if (k <= 0) continue;
        // rows kp .. of the operand (a complex row holds two real ones, each of two doubles)
        auto from = [&](const double *p, int ld, int mode) { return p + (mode == 1 ? (int64_t)kp : (int64_t)kp * ld); };
        ia[i] = operand(from(g.A, g.lda, g.amode), g.lda, g.m, k, g.amode, DG_BM, -1);
        ib[i] = operand(from(g.B, g.ldb, g.bmode), g.ldb, g.n, k, g.bmode, DG_BN, ia[i]);
        DgItem &x = gb.it[gb.count];
        x.m = g.m;
        x.n = g.n;
        x.C = g.C;
        x.ldc = g.ldc;
        x.nkt = (k + DG_KT - 1) / DG_KT;
        x.ntc = (g.n + DG_BN - 1) / DG_BN;
        x.sym = g.sym;
        const int mtc = (g.m + DG_BM - 1) / DG_BM;
        int tiles = 0;
        for (int m = 0; m < mtc; ++m) tiles += x.sym ? std::max(0, x.ntc - 2 * m) : x.ntc;
        x.unit0 = tiles;  // until the splits are known
        work += (double)tiles * x.nkt;
        ++gb.count;
      }
      // splits: about three units of work per SM, none shallower than 512 terms
      const double target = std::max<double>(DG_SPLIT, std::ceil(work / (3.0 * nsm) / DG_SPLIT) * DG_SPLIT);
      int units = 0, splits = 1;
      for (int q = 0; q < gb.count; ++q) {
        DgItem &x = gb.it[q];
        const int tiles = x.unit0;
        x.nsplit = std::min(32, std::max(1, (int)std::floor(x.nkt / target)));
        x.kper = (x.nkt + x.nsplit - 1) / x.nsplit;
        x.kper = (x.kper + DG_SPLIT - 1) / DG_SPLIT * DG_SPLIT;
        x.nsplit = (x.nkt + x.kper - 1) / x.kper;
        x.unit0 = units;
        units += tiles * x.nsplit;
        splits = std::max(splits, x.nsplit);
        if (x.nsplit > 1) wsum += (size_t)x.nsplit * x.m * x.n;
      }
      gb.units = units;
      gb.err = tc_status_word();
      uint8_t *ws = nullptr;
      const size_t ebytes = (vecs * sizeof(int) + 255) / 256 * 256;
      RFDD_CUDA(cudaMallocAsync((void **)&ws, ebytes + bytes + wsum * sizeof(double), st));
      int *emax = reinterpret_cast<int *>(ws);
      double *part = reinterpret_cast<double *>(ws + ebytes + bytes);
      RFDD_CUDA(cudaMemsetAsync(emax, DG_NONE_BYTE, ebytes, st));
      long long be = 1, bp = 1, bk = 1;
      for (const Src &s : srcs) {
        const int nkt = (s.k + DG_KT - 1) / DG_KT;
        db.it[db.count++] = {s.p, s.ld, s.nv, s.k, s.mode, s.vb, nkt, ws + ebytes + s.off, emax + s.ev, emax + s.kv, s.with < 0 ? -1 : 1};
        if (s.with < 0)
          bk = std::max<long long>(bk, s.mode == 0 ? (s.k + 7) / 8 : (long long)((s.k + 31) / 32) * ((s.nv + 255) / 256));
        be = std::max<long long>(be, s.mode == 1 ? (s.nv + 7) / 8 : (long long)((s.nv + 31) / 32) * ((s.k + 255) / 256));
        bp = std::max<long long>(bp, (long long)((s.nv + 63) / 64) * nkt);
      }
      for (int i = 0, q = 0; i < (int)cnt; ++i) {
        if (ia[i] < 0) continue;
        DgItem &x = gb.it[q++];
        const Src &a = srcs[ia[i]], &c = srcs[ib[i]];
        x.A = ws + ebytes + a.off;
        x.B = ws + ebytes + c.off;
        x.ea = emax + a.ev;
        x.eb = emax + c.ev;
        if (x.nsplit > 1) {
          x.ws = part;
          part += (size_t)x.nsplit * x.m * x.n;
        }
      }
      digit_kexp_kernel<<<dim3((unsigned)std::min<long long>(bk, 2048), db.count), 256, 0, st>>>(db);
      RFDD_CHECK_LAUNCH();
      digit_emax_kernel<<<dim3((unsigned)std::min<long long>(be, 2048), db.count), 256, 0, st>>>(db);
      RFDD_CHECK_LAUNCH();
      digit_pack_kernel<<<dim3((unsigned)std::min<long long>(bp, 4096), db.count), 256, 0, st>>>(db);
      RFDD_CHECK_LAUNCH();
      const double bt = kp == 0 ? beta : 1.0;
      cudaEvent_t e0 = nullptr, e1 = nullptr;
      if (profiling_enabled()) {
        e0 = profile_event();
        e1 = profile_event();
        cudaEventRecord(e0, st);
      }
      tc_dgemm_kernel<<<std::max(1, std::min(units, nsm)), DG_THREADS, DG_SMEM, st>>>(gb, alpha, bt);
      RFDD_CHECK_LAUNCH();
      if (splits > 1) {
        tc_dgemm_reduce_kernel<<<dim3(512, gb.count), 256, 0, st>>>(gb, alpha, bt);
        RFDD_CHECK_LAUNCH();
      }
      if (e0) {
        double flops = 0.0;
        for (int i = 0; i < (int)cnt; ++i) {
          const auto &g = items[s0 + i];
          flops += 2.0 * g.m * (double)g.n * std::max(0, std::min(kpass, g.k - kp));
        }
        cudaEventRecord(e1, st);
        profile_push(e0, e1, flops, 0);
      }
      RFDD_CUDA(cudaFreeAsync(ws, st));
    }
  }
}

// Digit products pay where the batch has enough work for their four launches and every item fills a good part
// of a 128 x 64 tile.  Against double-FP32 (12 FP32 operations per product) the line lies at about 6e7
// products an item; against the FP64 pipes (two products per cycle and SM) at 3e7 in the whole batch.
bool tc_dgemm_takes(const GemmItem<double> &g) {
  return g.m >= 48 && g.n >= 48 && g.k >= 48 && (double)g.m * g.n * g.k >= 6.4e7 && digits_fit(g.m, g.n, g.k);
}

void tc_dgemm_batched(cudaStream_t st, const std::vector<GemmItem<double>> &items, bool ta, bool tb, double alpha,
                      double beta, const std::vector<char> &sym) {
  std::vector<DgGemm> v;
  for (size_t i = 0; i < items.size(); ++i) {
    const auto &g = items[i];
    v.push_back({g.A, g.B, g.C, g.m, g.n, g.k, g.lda, g.ldb, g.ldc, ta ? 0 : 1, tb ? 1 : 0,
                 !sym.empty() && sym[i] ? 1 : 0});
  }
  dgemm_run(st, v, alpha, beta);
}

template <typename T>
bool tc_fp64_takes(const std::vector<GemmItem<T>> &items) {
  constexpr double F = ST<T>::is_complex ? 2.0 : 1.0;
  double work = 0.0;
  for (const auto &g : items) {
    if (g.m < 32 || F * g.n < 32 || F * g.k < 32 || !digits_fit(g.m, (int64_t)F * g.n, (int64_t)F * g.k)) return false;
    work += F * F * g.m * g.n * (double)g.k;
  }
  return work >= 3.2e7;
}

template <typename T>
void tc_fp64_batched(cudaStream_t st, const std::vector<GemmItem<T>> &items, double alpha, double beta) {
  constexpr int F = ST<T>::is_complex ? 2 : 1;
  std::vector<DgGemm> v;
  for (const auto &g : items)
    v.push_back({reinterpret_cast<const double *>(g.A), reinterpret_cast<const double *>(g.B),
                 reinterpret_cast<double *>(g.C), g.m, F * g.n, F * g.k, F * g.lda, g.ldb, (long long)F * g.ldc, 1,
                 F == 2 ? 2 : 0, 0});
  dgemm_run(st, v, alpha, beta);
}
template bool tc_fp64_takes<double>(const std::vector<GemmItem<double>> &);
template bool tc_fp64_takes<cx<double>>(const std::vector<GemmItem<cx<double>>> &);
template void tc_fp64_batched<double>(cudaStream_t, const std::vector<GemmItem<double>> &, double, double);
template void tc_fp64_batched<cx<double>>(cudaStream_t, const std::vector<GemmItem<cx<double>>> &, double, double);

}  // namespace rfdd
