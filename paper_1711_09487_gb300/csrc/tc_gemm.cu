// Complex-FP32 GEMM on the 5th-generation tensor cores (tcgen05, kind::f16) for sm_103a.
//
// C = beta*C + alpha*A*B with complex A (m x k), B (k x n), C (m x n), interleaved (re, im),
// row-major.  The complex product is computed in real ("4M", realified) form:
//   Cr (m x 2n) = Ar (m x 2k) * Br (2k x 2n),
// where Ar and Cr are the interleaved storage read as real matrices and each complex B[p][j]
// becomes the 2x2 real block [[re, im], [-im, re]] of Br.  FP32 accuracy comes from a two-way split
// of scaled operands: every row of Ar and every column of Br is scaled by a power of two that puts
// its largest entry in [2^13, 2^14), and x = hi + lo with hi = fp16(x), lo = fp16(x - hi), rounded to
// nearest in both halves: an entry has an error of 2^-23 of itself or 2^-38 of the largest one of its row (column), whichever
// is more.  That is FP32 for entries down to 2^-15 of the largest; smaller ones keep fewer bits of their own (a split
// with an exponent of its own per entry, as TF32 has, keeps 22) and those below 2^-38 are gone.  The solves do not
// notice: the 12^3 pencil as D A D, D powers of two within 2^-e and 2^e, reaches the same residuals in the same
// passes with either split (e = 5: 2 passes, 1e-11; e = 9: 1e-8, the limit of FP32 factors), and 7-point pencils of contrasts
// up to 5e9 as well.
// A*B ~ Ahi*Bhi + Ahi*Blo + Alo*Bhi, accumulated in FP32 in tensor memory and scaled back in the
// epilogue.  Against the TF32 split of the same depth the operands take half the bytes, the MMAs
// run at twice the rate, and the lower half is rounded instead of truncated.
//
// Operands are first packed (and split) into tiles already laid out in the UMMA K-major
// 128-byte-swizzled shared-memory format: A tiles of 128 rows x 64 halves (16 KB), B tiles of
// 256 rows x 64 halves (32 KB).  A CTA computes one 128 x BN tile of Cr: one thread streams the
// tiles into shared memory with 1-D bulk copies (cp.async.bulk, completion on an mbarrier), one
// thread issues tcgen05.mma into a BN-column TMEM accumulator, and eight warps read the
// accumulator back with tcgen05.ld for the epilogue.  Every mbarrier wait is bounded; on time-out
// the kernel records DS_WAIT_TIMEOUT and skips its output.  The kernel is persistent: one CTA per
// SM walks a static round-robin list of all output tiles of all batch items, with two TMEM
// accumulators so that draining tile i overlaps the MMAs of tile i+1.
#include "dense.cuh"
#include "tc_common.cuh"
#include "tc_gemm.cuh"
#include "tc_tune.h"

#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <mutex>

namespace rfdd {

constexpr int TC_BM = 128;
constexpr int TC_BN = 256;
constexpr int TC_BK = 64;            // 16-bit values of K in a tile row (128 bytes)
constexpr int TC_BK32 = 32;          // FP32 values of K in a tile row (plain TF32 probe)
constexpr int ROW_B = 128;           // bytes of a tile row
constexpr int A_TILE = TC_BM * ROW_B;  // bytes
constexpr int B_TILE = TC_BN * ROW_B;  // bytes
// ring of operand stages of the one-CTA kernel: 2 x 96 KB for 256-wide tiles, 4 x 48 KB for 64-wide
template <int BN>
struct TcRing {
  static constexpr int STAGES = BN == 256 ? 2 : 4;
  static constexpr int BYTES = 2 * A_TILE + 2 * BN * ROW_B;
};
constexpr int TC_RING_BYTES = 2 * (2 * A_TILE + 2 * B_TILE);
static_assert(TcRing<64>::STAGES * TcRing<64>::BYTES == TC_RING_BYTES, "both rings fill the same shared memory");
constexpr int EPI_WARPS = 8;  // two per TMEM lane quarter, each drains half of the columns
constexpr int EPI_TILE = 32 * 32;  // floats a warp stages: 32 rows of 32 columns
constexpr int EPI_BYTES = EPI_WARPS * EPI_TILE * 4;
constexpr int TC_THREADS = 64 + 32 * EPI_WARPS;  // producer warp, MMA warp, epilogue warps
constexpr int TC_SMEM = TC_RING_BYTES + EPI_BYTES + 1024;

// Status word of the launches issued by the calling host thread (TcStatusScope): a kernel whose
// bounded wait ran out ORs DS_WAIT_TIMEOUT into it.  Each handle passes its own word, so a
// failure is reported by the solve that met it and by no other.
thread_local int *g_tc_status = nullptr;

thread_local TcDigitRule g_tc_digits;

TcStatusScope::TcStatusScope(int *w, TcDigitRule digits) : prev(g_tc_status), prev_digits(g_tc_digits) {
  g_tc_status = w;
  g_tc_digits = digits;
}
TcStatusScope::~TcStatusScope() {
  g_tc_status = prev;
  g_tc_digits = prev_digits;
}
int *tc_status_word() { return g_tc_status; }
TcDigitRule tc_digit_rule() { return g_tc_digits; }

// Events recorded around the tensor-core kernel launches of the calling host thread (probes).
thread_local const cudaEvent_t *g_tc_events = nullptr;
TcKernelEvents::TcKernelEvents(const cudaEvent_t *ab) : prev(g_tc_events) { g_tc_events = ab; }
TcKernelEvents::~TcKernelEvents() { g_tc_events = prev; }

struct TcItem {
  const uint8_t *Ahi, *Alo, *Bhi, *Blo;
  const float *sA, *sB;  // scale of every packed row of A and of B (16-bit split)
  float *C;
  long long ldc;  // real leading dimension of C
  int m, n2, nkt, mtc, ntc, tile0;  // tile0: first global tile index of this item
  long long amts;  // A tiles between consecutive 128-row tiles (0: nkt, a packed A of its own)
  int colmajor;    // 1: tiles walk down the columns (mt fastest), 0: along the rows (nt fastest)
  int vec;         // floats per access to C: 4 when every row of C is so aligned, else 1
};

// Position of tile `local` of an item.  Along the rows, the CTAs running at once share one row of
// A tiles and sweep all of B; down the columns they share one column of B tiles and sweep all of A.
// Down the columns is chosen when the item's packed A fits comfortably in L2 and B is wide, so that
// A stays cached while each B column is read once (tc_tile_order).
__device__ __forceinline__ void tile_pos(const TcItem &it, int local, int &mt, int &nt) {
  if (it.colmajor) {
    mt = local % it.mtc;
    nt = local / it.mtc;
  } else {
    mt = local / it.ntc;
    nt = local % it.ntc;
  }
}
constexpr int TC_MAXB = 64;
struct TcBatchP {
  TcItem it[TC_MAXB];
  int count, total_tiles;
  int *err;    // status words of the launch (DS_WAIT_TIMEOUT on a wait that ran out; far scales, see far_launch)
};

__device__ __forceinline__ int find_item(const TcBatchP &b, int tile) {
  int lo = 0, hi = b.count;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (b.it[mid].tile0 <= tile) lo = mid; else hi = mid;
  }
  return lo;
}

// Access to one 32 x 32 chunk of C by a warp, V floats per lane and row: 32 / V lanes cover a row, so
// access i takes rows i * V .. i * V + V - 1.  All loads of a chunk are independent (32 values per lane).
template <int V>
struct ChunkC {
  static constexpr int ROWS = V;         // rows per access
  static constexpr int NACC = 32 / V;    // accesses per chunk
  __device__ __forceinline__ static int row(int i, int lane) { return i * V + lane / (32 / V); }
  __device__ __forceinline__ static int col(int lane) { return (lane % (32 / V)) * V; }
  __device__ __forceinline__ static void load(const TcItem &it, int row0, int nrows, int col0, int lane, float beta,
                                              float (&cv)[32]) {
    const int c = col0 + col(lane);
    const float *p = it.C + (long long)(row0 + row(0, lane)) * it.ldc + c;
    const long long step = (long long)V * it.ldc;
    const bool on = beta != 0.f;
#pragma unroll
    for (int i = 0; i < NACC; ++i, p += step) {
      float *d = cv + i * V;
#pragma unroll
      for (int t = 0; t < V; ++t) d[t] = 0.f;
      if (on && row(i, lane) < nrows) {
        if (c + V <= it.n2) {
          if (V == 4) *reinterpret_cast<float4 *>(d) = *reinterpret_cast<const float4 *>(p);
          else d[0] = *p;
        } else {
#pragma unroll
          for (int t = 0; t < V; ++t)
            if (c + t < it.n2) d[t] = p[t];
        }
      }
    }
  }
  __device__ __forceinline__ static void store(const TcItem &it, float *p, int c, const float *d) {
    if (c + V <= it.n2) {
      if (V == 4) *reinterpret_cast<float4 *>(p) = *reinterpret_cast<const float4 *>(d);
      else *p = d[0];
    } else {
#pragma unroll
      for (int t = 0; t < V; ++t)
        if (c + t < it.n2) p[t] = d[t];
    }
  }
};

// Scales that the usual order of the read-back (drain_tile: (x rr) (alpha rb)) cannot take: an accumulator is below 2^45 and
// scales lie between 2^-126 and 2^114, so x rr stays in range up to rr = 2^80, and alpha rb is exact for an alpha that is a
// power of two within 2^13 of 1 (the solver's are 1 and -1), for others where the column is within 2^100 and alpha within
// 2^20 of 1.  The packing records other rows and columns in the word after the status word; launches that they concern
// read back by drain_far.  (Columns below 2^-87 are ordinary: factors of wide 2-D subdomains decay that far.  Rows beyond
// 2^93 are not.)  Looked at tile by tile the check cost more than the read-back
// gained, and with both orders in one body it spilled: K = 32 update of 8192 x 8192 0.27 ms, 0.30 and 0.36 with these.
__device__ __forceinline__ bool far_row(float s) { return s > 0x1p80f; }
__device__ __forceinline__ bool far_col(float s) { return !(s >= 0x1p-100f && s <= 0x1p100f); }
constexpr int FAR_ROW = 1, FAR_COL = 2;
__device__ __forceinline__ bool far_launch(const int *err, float alpha) {
  const float a = fabsf(alpha);
  const bool plain = (__float_as_uint(a) & 0x7fffffu) == 0 && a >= 0x1p-13f && a <= 0x1p13f;
  const int far = __ldcg(err + 1);
  return (far & FAR_ROW) || (!plain && (far || !(a >= 0x1p-20f && a <= 0x1p20f)));
}

// Read-back of such launches: scales on one side of 1 one after the other, scales on different sides by their
// product, then alpha.
template <int NCH, typename W, typename F>
__device__ __forceinline__ bool drain_far(const TcItem &it, uint32_t tacc, int mt, int col0, int q, int c0, int lane,
                                          float *stg, float alpha, float beta, W &&wait, F &&done) {
  const int row0 = mt * TC_BM + q * 32, nrows = min(32, it.m - row0);
  if (!wait()) return false;
#pragma unroll 1
  for (int c = c0; c < c0 + NCH; ++c) {
    uint32_t v[32];
    TC_LD32(tacc + ((uint32_t)(q * 32) << 16) + (uint32_t)(c * 32), v);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    if (c == c0 + NCH - 1) done();
#pragma unroll
    for (int j = 0; j < 32; ++j) stg[lane * 32 + (j ^ lane)] = __uint_as_float(v[j]);
    __syncwarp();
    const int j = col0 + c * 32 + lane;
    if (j < it.n2) {
      const float rb = it.sB[j];
#pragma unroll 1
      for (int r = 0; r < nrows; ++r) {
        const float rr = it.sA[row0 + r], x = stg[r * 32 + (lane ^ r)];
        const float y = (rr >= 1.f) == (rb >= 1.f) ? (x * rr) * rb : x * (rr * rb);
        float *p = it.C + (long long)(row0 + r) * it.ldc + j;
        *p = fmaf(alpha, y, beta != 0.f ? beta * *p : 0.f);
      }
    }
    __syncwarp();
  }
  return true;
}

// Epilogue of one output tile by one warp: TMEM lanes 32q..32q+31 (rows mt*128 + 32q ..), NCH column
// chunks of 32 accumulator columns from chunk c0 on; C = alpha * scaled acc + beta * C, rows and columns
// masked.  The accumulator's rows are turned into C's through shared memory (16-byte pieces of row r at
// piece ^ (r & 7): no bank conflicts either way).  What bounds it is the latency of C: two chunks of C are in
// flight from before the accumulator is ready (`wait` returns false if it never is), and each is
// replaced by the chunk after the next as soon as it has been used.  `done` runs once the
// accumulator has been read.  Measured, 8192 x 8192 complex, C rows on 32 bytes, the best of four launches each: K = 32
// 0.27 ms (0.35 with one chunk in flight and one float per access), K = 256 0.296 ms = 465 TFLOP/s (0.37 so; 0.49 with the
// TF32 split).
template <int NCH, bool SCALED, int V, typename W, typename F>
__device__ __forceinline__ bool drain_tile(const TcItem &it, uint32_t tacc, int mt, int col0, int q, int c0, int lane,
                                           float *stg, float alpha, float beta, W &&wait, F &&done) {
  using CC = ChunkC<V>;
  const int row0 = mt * TC_BM + q * 32;
  const int nrows = min(32, it.m - row0);
  float cb[NCH > 1 ? 2 : 1][32];
  CC::load(it, row0, nrows, col0 + c0 * 32, lane, beta, cb[0]);
  if (NCH > 1) CC::load(it, row0, nrows, col0 + c0 * 32 + 32, lane, beta, cb[NCH > 1 ? 1 : 0]);
  // scale of the row this lane takes from the accumulator
  const float ra = SCALED && lane < nrows ? it.sA[row0 + lane] : 1.f;
  if (!wait()) return false;
#pragma unroll
  for (int ci = 0; ci < NCH; ++ci) {
    const int c = c0 + ci, cc = col0 + c * 32;
    float rb[V];
#pragma unroll
    for (int t = 0; t < V; ++t) {
      const int j = cc + CC::col(lane) + t;
      rb[t] = (SCALED && j < it.n2 ? it.sB[j] : 1.f) * alpha;
    }
    uint32_t v[32];
    TC_LD32(tacc + ((uint32_t)(q * 32) << 16) + (uint32_t)(c * 32), v);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    if (ci == NCH - 1) done();
#pragma unroll
    for (int j = 0; j < 8; ++j)
      *reinterpret_cast<float4 *>(stg + lane * 32 + ((j ^ (lane & 7)) << 2)) =
          make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]), __uint_as_float(v[4 * j + 2]),
                      __uint_as_float(v[4 * j + 3]));
    __syncwarp();
    const int cl = CC::col(lane);
    float *p = it.C + (long long)(row0 + CC::row(0, lane)) * it.ldc + cc + cl;
    const long long step = (long long)V * it.ldc;
    float(&cv)[32] = cb[NCH > 1 ? ci & 1 : 0];
#pragma unroll
    for (int i = 0; i < CC::NACC; ++i, p += step) {
      const int r = CC::row(i, lane);
      const float *sp = stg + r * 32 + (((cl >> 2) ^ (r & 7)) << 2) + (cl & 3);
      float x[V];
      if (V == 4) *reinterpret_cast<float4 *>(x) = *reinterpret_cast<const float4 *>(sp);
      else x[0] = *sp;
      const float rr = SCALED ? __shfl_sync(0xffffffffu, ra, r) : 1.f;
      // the row's scale, then alpha times the column's: the product of the two scales may leave the range of a float
      // where the result does not (sums near 2^-126, huge rows and columns without common entries)
#pragma unroll
      for (int t = 0; t < V; ++t) x[t] = fmaf(rb[t], SCALED ? x[t] * rr : x[t], beta * cv[i * V + t]);
      if (r < nrows) CC::store(it, p, cc + cl, x);
    }
    __syncwarp();
    if (ci + 2 < NCH) CC::load(it, row0, nrows, cc + 64, lane, beta, cv);
  }
  return true;
}
template <int NCH, bool SCALED, typename W, typename F>
__device__ __forceinline__ bool drain_tile_vec(const TcItem &it, uint32_t tacc, int mt, int col0, int q, int c0,
                                               int lane, float *stg, float alpha, float beta, bool far, W &&wait,
                                               F &&done) {
  if (SCALED && far)
    return drain_far<NCH>(it, tacc, mt, col0, q, c0, lane, stg, alpha, beta, wait, done);
  if (it.vec == 4) return drain_tile<NCH, SCALED, 4>(it, tacc, mt, col0, q, c0, lane, stg, alpha, beta, wait, done);
  return drain_tile<NCH, SCALED, 1>(it, tacc, mt, col0, q, c0, lane, stg, alpha, beta, wait, done);
}

// Real columns of a tile that the MMAs compute: those of C, in steps of 16 (the MMA's N)
template <int BN>
__device__ __forceinline__ int tile_cols(const TcItem &it, int nt) {
  return min(BN, (it.n2 - nt * BN + 15) & ~15);
}

// Persistent, warp-specialised: warp 0 streams operand tiles, warp 1 issues the MMAs into one of
// two TMEM accumulators (BN columns each), warps 2..9 drain the other accumulator to C.
// F16: the scaled 16-bit split, three products; otherwise plain TF32 (peak probe).
// BN = 64 takes a quarter of a packed B tile per output tile, for launches that have too few 256-wide
// tiles to fill the chip or whose C has at most 64 real columns.
template <bool F16, int BN>
__global__ void __launch_bounds__(TC_THREADS, 1) tc_gemm_kernel(const __grid_constant__ TcBatchP b, float alpha,
                                                                float beta) {
  constexpr int STAGES = TcRing<BN>::STAGES, STAGE_BYTES = TcRing<BN>::BYTES;
  constexpr int SUB = TC_BN / BN;  // output tiles per packed B tile
  int *err = b.err;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  float *epi = reinterpret_cast<float *>(base + TC_RING_BYTES);
  __shared__ __align__(8) uint64_t full_bar[STAGES], empty_bar[STAGES], tfull_bar[2], tempty_bar[2],
      drain_bar;
  __shared__ uint32_t tmem_s;
  __shared__ volatile int abort_s, far_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&tfull_bar[a]), 1);
      mbar_init(smem_u32(&tempty_bar[a]), 32 * EPI_WARPS);
    }
    mbar_init(smem_u32(&drain_bar), 1);
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (threadIdx.x == 64) far_s = F16 && far_launch(err, alpha);  // in shared memory: the epilogue has no register to spare
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_s)),
                 "r"(2 * BN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_s;
  auto stage_addr = [&](int s, int which) -> uint32_t {  // which: 0 Ahi, 1 Alo, 2 Bhi, 3 Blo
    const uint32_t off = (uint32_t)s * STAGE_BYTES +
                         (which == 0 ? 0u : which == 1 ? (uint32_t)A_TILE : which == 2 ? 2u * A_TILE
                                                                                       : 2u * A_TILE + BN * ROW_B);
    return smem_u32(base + off);
  };
  if (warp == 0) {
    if (lane == 0) {  // producer
      long long g = 0;  // global k-tile counter (stage ring position)
      for (int tile = blockIdx.x; tile < b.total_tiles && !abort_s; tile += gridDim.x) {
        const TcItem &it = b.it[find_item(b, tile)];
        const int local = tile - it.tile0;
        int mt, nt;
        tile_pos(it, local, mt, nt);
        const long long ams = it.amts ? it.amts : it.nkt;
        const uint8_t *Ahi = it.Ahi + (long long)mt * ams * A_TILE, *Alo = it.Alo + (long long)mt * ams * A_TILE;
        const long long bo = (long long)(nt / SUB) * it.nkt * B_TILE + (nt % SUB) * (BN * ROW_B);
        const uint8_t *Bhi = it.Bhi + bo, *Blo = it.Blo + bo;
        const uint32_t nb = (uint32_t)tile_cols<BN>(it, nt) * ROW_B;
        for (int kt = 0; kt < it.nkt; ++kt, ++g) {
          const int s = (int)(g % STAGES);
          const long long u = g / STAGES;
          if (u >= 1 && !mbar_wait(smem_u32(&empty_bar[s]), (uint32_t)((u - 1) & 1), &abort_s)) {
            atomicOr(err, DS_WAIT_TIMEOUT);
            abort_s = 1;
            break;
          }
          const uint32_t fb = smem_u32(&full_bar[s]);
          mbar_expect_tx(fb, (F16 ? 2 : 1) * (A_TILE + nb));
          bulk_g2s(stage_addr(s, 0), Ahi + (long long)kt * A_TILE, A_TILE, fb);
          bulk_g2s(stage_addr(s, 2), Bhi + (long long)kt * B_TILE, nb, fb);
          if (F16) {
            bulk_g2s(stage_addr(s, 1), Alo + (long long)kt * A_TILE, A_TILE, fb);
            bulk_g2s(stage_addr(s, 3), Blo + (long long)kt * B_TILE, nb, fb);
          }
        }
      }
      // every issued copy must land before the CTA can exit, after an abort too
      for (long long q = (g > STAGES ? g - STAGES : 0); q < g; ++q)
        mbar_drain(smem_u32(&full_bar[q % STAGES]), (uint32_t)((q / STAGES) & 1));
    }
  } else if (warp == 1) {
    if (lane == 0) {  // MMA issuer
      const uint32_t idesc0 = (1u << 4) | (F16 ? 0u : (2u << 7) | (2u << 10)) | ((uint32_t)(TC_BM >> 4) << 24);
      long long g = 0;
      int lt = 0;
      for (int tile = blockIdx.x; tile < b.total_tiles && !abort_s; tile += gridDim.x, ++lt) {
        const TcItem &it = b.it[find_item(b, tile)];
        int mt, nt;
        tile_pos(it, tile - it.tile0, mt, nt);
        const uint32_t idesc = idesc0 | ((uint32_t)(tile_cols<BN>(it, nt) >> 3) << 17);
        const int acc = lt & 1;
        if (lt >= 2 && !mbar_wait(smem_u32(&tempty_bar[acc]), (uint32_t)(((lt >> 1) - 1) & 1), &abort_s)) {
          atomicOr(err, DS_WAIT_TIMEOUT);
          abort_s = 1;
          break;
        }
        fence_after();
        const uint32_t dacc = tmem + (uint32_t)(acc * BN);
        bool ok = true;
        for (int kt = 0; kt < it.nkt; ++kt, ++g) {
          const int s = (int)(g % STAGES);
          if (!mbar_wait(smem_u32(&full_bar[s]), (uint32_t)((g / STAGES) & 1), &abort_s)) {
            atomicOr(err, DS_WAIT_TIMEOUT);
            abort_s = 1;
            ok = false;
            break;
          }
          fence_after();
          const uint32_t ah = stage_addr(s, 0), al = stage_addr(s, 1), bh = stage_addr(s, 2), bl = stage_addr(s, 3);
#pragma unroll
          for (int kk = 0; kk < ROW_B / 32; ++kk) {
            const uint32_t o = kk * 32;  // 16 16-bit (8 TF32) values = 32 bytes along K inside the swizzle row
            if (F16) {
              mma_f16(dacc, sdesc(ah + o), sdesc(bh + o), idesc, (kt > 0 || kk > 0) ? 1u : 0u);
              mma_f16(dacc, sdesc(ah + o), sdesc(bl + o), idesc, 1u);
              mma_f16(dacc, sdesc(al + o), sdesc(bh + o), idesc, 1u);
            } else {
              mma_tf32(dacc, sdesc(ah + o), sdesc(bh + o), idesc, (kt > 0 || kk > 0) ? 1u : 0u);
            }
          }
          mma_commit(smem_u32(&empty_bar[s]));
        }
        if (!ok) break;
        mma_commit(smem_u32(&tfull_bar[acc]));
      }
      // every issued MMA ends before the tensor memory is freed, after an abort too
      mma_commit(smem_u32(&drain_bar));
      mbar_drain(smem_u32(&drain_bar), 0);
    }
  } else {
    // epilogue warps: warp w reads accumulator lanes 32*(w % 4) .. +31 (its TMEM sub-partition);
    // warps 2..5 take the first half of the column chunks, warps 6..9 the second
    constexpr int NCH = BN / 64;
    const int q = warp & 3;
    const int c0 = ((warp - 2) >> 2) * NCH;
    float *stg = epi + (warp - 2) * EPI_TILE;
    int lt = 0;
    for (int tile = blockIdx.x; tile < b.total_tiles; tile += gridDim.x, ++lt) {
      const TcItem &it = b.it[find_item(b, tile)];
      const int local = tile - it.tile0;
      int mt, nt;
      tile_pos(it, local, mt, nt);
      const int acc = lt & 1;
      const bool ok = drain_tile_vec<NCH, F16>(
          it, tmem + (uint32_t)(acc * BN), mt, nt * BN, q, c0, lane, stg, alpha, beta, far_s != 0,
          [&] {
            const bool ready = mbar_wait(smem_u32(&tfull_bar[acc]), (uint32_t)((lt >> 1) & 1), &abort_s);
            // the whole warp takes the same branch (tcgen05.ld is a warp-collective)
            const bool go = __all_sync(0xffffffffu, ready && !abort_s);
            fence_after();
            return go;
          },
          [&] {
            fence_before();
            mbar_arrive(smem_u32(&tempty_bar[acc]));
          });
      if (!ok) {
        if (lane == 0) atomicOr(err, DS_WAIT_TIMEOUT);
        abort_s = 1;
        break;
      }
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BN) : "memory");
  }
}

// ---------------------------------------------------------------------------------------
// Two-CTA variant (cta_group::2): a cluster of two CTAs on two SMs computes a 256 x 256 tile of
// Cr with one MMA stream.  Each CTA holds its own 128 rows of A and its half (128 packed rows) of
// the B tile in shared memory; the MMAs, issued by the leader CTA (rank 0), read A and B from both
// CTAs and leave rows 0..127 of the accumulator in the leader's TMEM and rows 128..255 in the
// peer's.  Per 64-deep K tile an SM so takes in 64 KB instead of the 96 KB of the one-CTA kernel
// (whose 128 x 256 tile needs all of B), which is what limits that kernel (operand feed, not the
// tensor pipe).
//
// Synchronisation (all waits bounded; DS_WAIT_TIMEOUT into *err on time-out):
//  - each CTA's producer loads its halves into its own stage and completes its own full_bar;
//  - the peer's warp 1 forwards: it waits on its own full_bar and arrives on the leader's pfull_bar;
//  - the leader waits on full_bar and pfull_bar, issues the MMAs, and commits to empty_bar of both
//    CTAs (stage reusable) and, per tile, to tfull_bar of both CTAs (accumulator ready);
//  - every epilogue warp of both CTAs drains its TMEM lanes and arrives on the leader's tempty_bar.
// ---------------------------------------------------------------------------------------
constexpr int T2_STAGES = 3;
constexpr int T2_BHALF = B_TILE / 2;                         // bytes of one CTA's B half
constexpr int T2_STAGE_BYTES = 2 * A_TILE + 2 * T2_BHALF;    // 64 KB
constexpr int T2_SMEM = T2_STAGES * T2_STAGE_BYTES + EPI_BYTES + 1024;

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// bounded wait with cluster-scope acquire (the barrier may be completed from the peer CTA)
__device__ __forceinline__ bool mbar_wait_cl(uint32_t bar, uint32_t parity, volatile int *abort_flag) {
  for (long long i = 0; i < WAIT_LIMIT; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((i & 1023) == 1023 && *abort_flag) return false;
  }
  return false;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mma2_f16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(da), "l"(db), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void mma2_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mma2_commit_both(uint32_t bar) {
  const uint16_t mask = 0x3;
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"(mask)
      : "memory");
}

// pair tile `local` of an item -> (pair row mp, tile column nt); two CTAs take rows 2 mp, 2 mp + 1
__device__ __forceinline__ void pair_pos(const TcItem &it, int local, int &mp, int &nt) {
  const int mpc = (it.mtc + 1) >> 1;
  if (it.colmajor) {
    mp = local % mpc;
    nt = local / mpc;
  } else {
    mp = local / it.ntc;
    nt = local % it.ntc;
  }
}

__global__ void __launch_bounds__(TC_THREADS, 1) tc_gemm2_kernel(const __grid_constant__ TcBatchP b, float alpha,
                                                                 float beta) {
  int *err = b.err;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  float *epi = reinterpret_cast<float *>(base + T2_STAGES * T2_STAGE_BYTES);
  __shared__ __align__(8) uint64_t full_bar[T2_STAGES], pfull_bar[T2_STAGES], empty_bar[T2_STAGES], tfull_bar[2],
      tempty_bar[2], drain_bar;
  __shared__ uint32_t tmem_s;
  __shared__ volatile int abort_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int cl = (int)(blockIdx.x >> 1), ncl = (int)(gridDim.x >> 1);
  if (threadIdx.x == 0) {
    for (int s = 0; s < T2_STAGES; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&pfull_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&tfull_bar[a]), 1);
      mbar_init(smem_u32(&tempty_bar[a]), 2 * EPI_WARPS);  // one arrival per epilogue warp of each CTA
    }
    mbar_init(smem_u32(&drain_bar), 1);
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {  // both CTAs of the pair allocate together
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_s)),
                 "r"(2 * TC_BN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  fence_before();
  cluster_sync_all();  // both CTAs' barriers initialised and TMEM allocated before any remote use
  fence_after();
  const uint32_t tmem = tmem_s;
  auto stage_addr = [&](int s, int which) -> uint32_t {  // which: 0 Ahi, 1 Alo, 2 Bhi half, 3 Blo half
    const uint32_t off = (uint32_t)s * T2_STAGE_BYTES +
                         (which == 0 ? 0u : which == 1 ? (uint32_t)A_TILE : which == 2 ? 2u * A_TILE
                                                                                       : 2u * A_TILE + T2_BHALF);
    return smem_u32(base + off);
  };
  if (warp == 0) {
    if (lane == 0) {  // producer (both CTAs): this CTA's A rows and B half
      long long g = 0;
      for (int pt = cl; pt < b.total_tiles && !abort_s; pt += ncl) {
        const TcItem &it = b.it[find_item(b, pt)];
        int mp, nt;
        pair_pos(it, pt - it.tile0, mp, nt);
        const int mt = min(2 * mp + (int)rank, it.mtc - 1);  // a missing second row re-reads the last one
        const long long ams = it.amts ? it.amts : it.nkt;
        const uint8_t *Ahi = it.Ahi + (long long)mt * ams * A_TILE, *Alo = it.Alo + (long long)mt * ams * A_TILE;
        const long long boff = (long long)nt * it.nkt * B_TILE + (long long)rank * T2_BHALF;
        const uint8_t *Bhi = it.Bhi + boff, *Blo = it.Blo + boff;
        for (int kt = 0; kt < it.nkt; ++kt, ++g) {
          const int s = (int)(g % T2_STAGES);
          const long long u = g / T2_STAGES;
          if (u >= 1 && !mbar_wait_cl(smem_u32(&empty_bar[s]), (uint32_t)((u - 1) & 1), &abort_s)) {
            atomicOr(err, DS_WAIT_TIMEOUT);
            abort_s = 1;
            break;
          }
          const uint32_t fb = smem_u32(&full_bar[s]);
          mbar_expect_tx(fb, T2_STAGE_BYTES);
          bulk_g2s(stage_addr(s, 0), Ahi + (long long)kt * A_TILE, A_TILE, fb);
          bulk_g2s(stage_addr(s, 1), Alo + (long long)kt * A_TILE, A_TILE, fb);
          bulk_g2s(stage_addr(s, 2), Bhi + (long long)kt * B_TILE, T2_BHALF, fb);
          bulk_g2s(stage_addr(s, 3), Blo + (long long)kt * B_TILE, T2_BHALF, fb);
        }
      }
      // every issued copy lands (after an abort too), and every stage's last consumption is signalled here (the
      // leader's commits arrive on this CTA's empty barriers), before the CTA leaves
      for (long long q = (g > T2_STAGES ? g - T2_STAGES : 0); q < g; ++q) {
        mbar_drain(smem_u32(&full_bar[q % T2_STAGES]), (uint32_t)((q / T2_STAGES) & 1));
        mbar_wait_cl(smem_u32(&empty_bar[q % T2_STAGES]), (uint32_t)((q / T2_STAGES) & 1), &abort_s);
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 1) {  // peer: forward "my halves of stage s are in" to the leader
      long long g = 0;
      for (int pt = cl; pt < b.total_tiles && !abort_s; pt += ncl) {
        const TcItem &it = b.it[find_item(b, pt)];
        bool ok = true;
        for (int kt = 0; kt < it.nkt; ++kt, ++g) {
          const int s = (int)(g % T2_STAGES);
          if (!mbar_wait_cl(smem_u32(&full_bar[s]), (uint32_t)((g / T2_STAGES) & 1), &abort_s)) {
            atomicOr(err, DS_WAIT_TIMEOUT);
            abort_s = 1;
            ok = false;
            break;
          }
          mbar_arrive_cluster(map_to_rank(smem_u32(&pfull_bar[s]), 0));
        }
        if (!ok) break;
      }
    } else if (lane == 0 && rank == 0) {  // leader: MMA issuer for the pair
      const uint32_t idesc = (1u << 4) | ((uint32_t)(TC_BN >> 3) << 17) |
                             ((uint32_t)((2 * TC_BM) >> 4) << 24);
      long long g = 0;
      int lt = 0;
      for (int pt = cl; pt < b.total_tiles && !abort_s; pt += ncl, ++lt) {
        const TcItem &it = b.it[find_item(b, pt)];
        const int acc = lt & 1;
        if (lt >= 2 && !mbar_wait_cl(smem_u32(&tempty_bar[acc]), (uint32_t)(((lt >> 1) - 1) & 1), &abort_s)) {
          atomicOr(err, DS_WAIT_TIMEOUT);
          abort_s = 1;
          break;
        }
        fence_after();
        const uint32_t dacc = tmem + (uint32_t)(acc * TC_BN);
        bool ok = true;
        for (int kt = 0; kt < it.nkt; ++kt, ++g) {
          const int s = (int)(g % T2_STAGES);
          const uint32_t par = (uint32_t)((g / T2_STAGES) & 1);
          if (!mbar_wait_cl(smem_u32(&full_bar[s]), par, &abort_s) ||
              !mbar_wait_cl(smem_u32(&pfull_bar[s]), par, &abort_s)) {
            atomicOr(err, DS_WAIT_TIMEOUT);
            abort_s = 1;
            ok = false;
            break;
          }
          fence_after();
          const uint32_t ah = stage_addr(s, 0), al = stage_addr(s, 1), bh = stage_addr(s, 2), bl = stage_addr(s, 3);
#pragma unroll
          for (int kk = 0; kk < ROW_B / 32; ++kk) {
            const uint32_t o = kk * 32;
            mma2_f16(dacc, sdesc(ah + o), sdesc(bh + o), idesc, (kt > 0 || kk > 0) ? 1u : 0u);
            mma2_f16(dacc, sdesc(ah + o), sdesc(bl + o), idesc, 1u);
            mma2_f16(dacc, sdesc(al + o), sdesc(bh + o), idesc, 1u);
          }
          mma2_commit_both(smem_u32(&empty_bar[s]));
        }
        if (!ok) break;
        mma2_commit_both(smem_u32(&tfull_bar[acc]));
      }
      // every issued MMA ends before either CTA frees its tensor memory (the cluster barrier below), after an abort too
      mma2_commit(smem_u32(&drain_bar));
      mbar_drain(smem_u32(&drain_bar), 0);
    }
  } else {
    // epilogue warps of both CTAs: this CTA's 128 accumulator rows of the pair tile
    const int q = warp & 3;
    constexpr int NCH = TC_BN / 64;
    const int c0 = ((warp - 2) >> 2) * NCH;
    float *stg = epi + (warp - 2) * EPI_TILE;
    const bool far = far_launch(err, alpha);
    const uint32_t tempty_leader0 = map_to_rank(smem_u32(&tempty_bar[0]), 0);
    const uint32_t tempty_leader1 = map_to_rank(smem_u32(&tempty_bar[1]), 0);
    int lt = 0;
    for (int pt = cl; pt < b.total_tiles; pt += ncl, ++lt) {
      const TcItem &it = b.it[find_item(b, pt)];
      int mp, nt;
      pair_pos(it, pt - it.tile0, mp, nt);
      const int mt = 2 * mp + (int)rank;  // rows beyond m (a missing second row) are masked
      const int acc = lt & 1;
      const bool ok = drain_tile_vec<NCH, true>(
          it, tmem + (uint32_t)(acc * TC_BN), mt, nt * TC_BN, q, c0, lane, stg, alpha, beta, far,
          [&] {
            const bool ready = mbar_wait_cl(smem_u32(&tfull_bar[acc]), (uint32_t)((lt >> 1) & 1), &abort_s);
            const bool go = __all_sync(0xffffffffu, ready && !abort_s);
            fence_after();
            return go;
          },
          [&] {
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(acc ? tempty_leader1 : tempty_leader0);
          });
      if (!ok) {
        if (lane == 0) atomicOr(err, DS_WAIT_TIMEOUT);
        abort_s = 1;
        break;
      }
    }
  }
  fence_before();
  cluster_sync_all();  // no CTA leaves while its peer may still signal it or read its shared memory
  fence_after();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * TC_BN) : "memory");
  }
}

// ---------------------------------------------------------------------------------------
// Tensor-pipe throughput probe: one CTA per SM issues `iters` x 4 MMAs, kind::tf32 of 128 x 256 x 8 or (F16)
// kind::f16 of 128 x 256 x 16, from operand tiles that stay in shared memory (no loads), into one TMEM
// accumulator, then waits for their completion on an mbarrier (bounded; DS_WAIT_TIMEOUT into *err
// on time-out).  Measures the MMA issue rate alone, not the operand feed.
// ---------------------------------------------------------------------------------------
template <bool F16>
__global__ void __launch_bounds__(128, 1) mma_probe_kernel(int iters, int *err) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t done_bar;
  __shared__ uint32_t tmem_s;
  __shared__ volatile int abort_s;
  const int warp = threadIdx.x >> 5;
  // operand tiles: zeros (the rate does not depend on the values)
  for (int i = threadIdx.x; i < (A_TILE + B_TILE) / 4; i += blockDim.x) reinterpret_cast<float *>(base)[i] = 0.f;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&done_bar), 1);
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_s)),
                 "r"(TC_BN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_s;
  if (threadIdx.x == 0) {
    const uint32_t idesc = (1u << 4) | (F16 ? 0u : (2u << 7) | (2u << 10)) | ((uint32_t)(TC_BN >> 3) << 17) |
                           ((uint32_t)(TC_BM >> 4) << 24);
    const uint32_t a = smem_u32(base), b = smem_u32(base + A_TILE);
    for (int it = 0; it < iters; ++it) {
#pragma unroll
      for (int kk = 0; kk < ROW_B / 32; ++kk) {
        const uint32_t acc = (it > 0 || kk > 0) ? 1u : 0u;
        if (F16) mma_f16(tmem, sdesc(a + kk * 32), sdesc(b + kk * 32), idesc, acc);
        else mma_tf32(tmem, sdesc(a + kk * 32), sdesc(b + kk * 32), idesc, acc);
      }
    }
    mma_commit(smem_u32(&done_bar));
    if (!mbar_wait(smem_u32(&done_bar), 0, &abort_s)) atomicOr(err, DS_WAIT_TIMEOUT);
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_BN) : "memory");
  }
}

double tc_mma_probe_tflops(cudaStream_t st, int *dev_status, bool f16) {
  const auto kernel = f16 ? mma_probe_kernel<true> : mma_probe_kernel<false>;
  int dev = 0, nsm = 0;
  RFDD_CUDA(cudaGetDevice(&dev));
  RFDD_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  const int smem = A_TILE + B_TILE + 1024;
  RFDD_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  cudaEvent_t e0, e1;
  RFDD_CUDA(cudaEventCreate(&e0));
  RFDD_CUDA(cudaEventCreate(&e1));
  const int iters = 4096;
  double best = 0.0;
  for (int rep = 0; rep < 4; ++rep) {  // the first launch is a warm-up
    RFDD_CUDA(cudaEventRecord(e0, st));
    kernel<<<nsm, 128, smem, st>>>(iters, dev_status);
    RFDD_CHECK_LAUNCH();
    RFDD_CUDA(cudaEventRecord(e1, st));
    RFDD_CUDA(cudaEventSynchronize(e1));
    float ms = 0.f;
    RFDD_CUDA(cudaEventElapsedTime(&ms, e0, e1));
    const double fl = 2.0 * TC_BM * TC_BN * (double)(f16 ? TC_BK : TC_BK32) * (double)iters * nsm;
    if (rep > 0 && ms > 0.f) best = std::max(best, fl / (ms * 1e-3) / 1e12);
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return best;
}

// ---------------------------------------------------------------------------------------
// packing: scale, split into 16-bit halves and write swizzled tiles
// ---------------------------------------------------------------------------------------
// Power of two that brings a row whose largest magnitude is m into [2^13, 2^14), and its inverse.
// 0, infinities and NaN: 1.  Below 2^-113 the factor stays at 2^126 (its inverse is still normal).
__device__ __forceinline__ void row_scale(float m, float &mul, float &inv) {
  const int ex = (int)(__float_as_uint(m) >> 23) & 255;
  const int f = (m == 0.f || ex == 255) ? 127 : min(267 - ex, 253);
  mul = __uint_as_float((uint32_t)f << 23);
  inv = __uint_as_float((uint32_t)(254 - f) << 23);
}
// x = hi + lo, both rounded to nearest
__device__ __forceinline__ void split_f16(float x, uint16_t &hi, uint16_t &lo) {
  const __half h = __float2half_rn(x);
  hi = __half_as_ushort(h);
  lo = __half_as_ushort(__float2half_rn(x - __half2float(h)));
}
__device__ __forceinline__ uint32_t pair16(uint16_t a, uint16_t b) { return (uint32_t)a | ((uint32_t)b << 16); }

struct PackItem {
  const float *src;   // interleaved complex source (as floats), or real
  long long ld;       // leading dimension in elements of the source
  int rows, k;        // A: rows x k; B: k x rows (elements)
  uint8_t *hi, *lo;   // tile buffers
  float *scale;       // inverse scale of every packed row (A: padded rows; B: 64-row blocks)
  int nblk;           // A: 128-row tiles; B: blocks of 64 packed rows
  int nkt;
  int side;           // A: > 0: columns left of the diagonal block of `side` rows have a scale of their own,
                      // the others' scales follow at scale + nblk * 128 (L and U of one factor)
};
struct PackBatchP {
  PackItem a[TC_MAXB], b[TC_MAXB];
  int na, nb;
  int *far;  // set where a scale is far (far_launch)
};

// A tiles: [mt][kt] 128 rows x 64 halves; 16-byte chunk c of row r stored at chunk c ^ (r & 7).  A row takes 32
// lanes, or 8 or 16 when it has no more chunks than that (the 32-deep panel updates): its largest magnitude
// first, then the split (the second read of the row comes from L1 / L2).
template <bool CPLX, int NW, bool AL8>
__device__ __forceinline__ void pack_a_rows(const PackItem &it, int *far) {
  constexpr int F = CPLX ? 2 : 1;
  const int kf = F * it.k, nq = it.nkt * 8, rows_pad = it.nblk * TC_BM;
  const int lpr = nq >= 32 ? 32 : nq >= 16 ? 16 : 8, per = 32 * NW / lpr, lane = threadIdx.x % lpr;
  // rows_pad is a multiple of per, so the lanes of a warp stay together
  for (int row = blockIdx.x * per + (int)threadIdx.x / lpr; row < rows_pad; row += gridDim.x * per) {
    const float *src = it.src + (long long)row * F * it.ld;
    const bool live = row < it.rows;
    auto load8 = [&](int q, float (&x)[8]) {
      const int k0 = q * 8;
      if (AL8) {
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const float2 v = (live && k0 + 2 * t < kf) ? *reinterpret_cast<const float2 *>(src + k0 + 2 * t)
                                                      : make_float2(0.f, 0.f);
          x[2 * t] = v.x;
          x[2 * t + 1] = v.y;
        }
      } else {
#pragma unroll
        for (int t = 0; t < 8; ++t) x[t] = (live && k0 + t < kf) ? src[k0 + t] : 0.f;
      }
    };
    // chunks left of the row's diagonal block (a multiple of eight values per block)
    const int ql = it.side > 0 ? (row / it.side) * it.side * F / 8 : 0;
    float ml = 0.f, mr = 0.f;
    for (int q = lane; q < nq; q += lpr) {
      float x[8];
      load8(q, x);
      float m = 0.f;
#pragma unroll
      for (int t = 0; t < 8; ++t) m = fmaxf(m, fabsf(x[t]));
      if (q < ql) ml = fmaxf(ml, m);
      else mr = fmaxf(mr, m);
    }
    for (int o = lpr >> 1; o > 0; o >>= 1) {
      ml = fmaxf(ml, __shfl_xor_sync(0xffffffffu, ml, o));
      mr = fmaxf(mr, __shfl_xor_sync(0xffffffffu, mr, o));
    }
    float fl, il, fr, ir;
    row_scale(ml, fl, il);
    row_scale(mr, fr, ir);
    if (lane == 0) {
      if (far_row(il) || far_row(ir)) atomicOr(far, FAR_ROW);
      if (it.side > 0) {
        it.scale[row] = il;
        it.scale[rows_pad + row] = ir;
      } else {
        it.scale[row] = ir;
      }
    }
    const int mt = row / TC_BM, r = row % TC_BM;
    for (int q = lane; q < nq; q += lpr) {
      float x[8];
      load8(q, x);
      const float f = q < ql ? fl : fr;
      uint16_t h[8], l[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) split_f16(x[t] * f, h[t], l[t]);
      const long long off = ((long long)mt * it.nkt + (q >> 3)) * A_TILE + r * ROW_B + (((q & 7) ^ (r & 7)) << 4);
      *reinterpret_cast<uint4 *>(it.hi + off) = make_uint4(pair16(h[0], h[1]), pair16(h[2], h[3]), pair16(h[4], h[5]), pair16(h[6], h[7]));
      *reinterpret_cast<uint4 *>(it.lo + off) = make_uint4(pair16(l[0], l[1]), pair16(l[2], l[3]), pair16(l[4], l[5]), pair16(l[6], l[7]));
    }
  }
}

// B tiles: the rows of Br^T.  Complex: rows n' = 2j + t (t: 0 real part column, 1 imaginary), K index k' = 2p + u:
//   Br^T[2j][2p] = re B[p][j], Br^T[2j][2p+1] = -im B[p][j], Br^T[2j+1][2p] = im, Br^T[2j+1][2p+1] = re.
// A block owns 64 packed rows (32 complex or 64 real columns of B): it stages up to PACK_KC rows of B
// in shared memory with reads along B's rows, takes the largest magnitude of every column, and writes
// the packed rows with coalesced 16-byte stores.  Deeper B is staged twice, chunk by chunk.
constexpr int PACK_KC = 256;
template <bool CPLX, int NW, bool AL8>
__device__ __forceinline__ void pack_b_rows(const PackItem &it, float *sb, int *far) {
  constexpr int F = CPLX ? 2 : 1;
  constexpr int CW = 64 / F;            // columns of B per block
  constexpr int PITCH = CPLX ? 66 : 65;  // floats per staged row
  __shared__ float smax[NW][64];
  __shared__ float mul_s[64];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nch = (it.k + PACK_KC - 1) / PACK_KC;
  for (int jb = blockIdx.x; jb < it.nblk; jb += gridDim.x) {
    const long long j0 = (long long)jb * CW;
    auto stage = [&](int p0, int pn, float &m0, float &m1) {
      if (CPLX) {
        const bool on = j0 + lane < it.rows;
#pragma unroll 8
        for (int p = warp; p < pn; p += NW) {
          const float *s = it.src + 2 * ((long long)(p0 + p) * it.ld + j0 + lane);
          float2 v = make_float2(0.f, 0.f);
          if (on) {
            if (AL8) v = *reinterpret_cast<const float2 *>(s);
            else v = make_float2(s[0], s[1]);
          }
          *reinterpret_cast<float2 *>(sb + p * PITCH + 2 * lane) = v;
          m0 = fmaxf(m0, fmaxf(fabsf(v.x), fabsf(v.y)));
        }
      } else {
        const bool on0 = j0 + lane < it.rows, on1 = j0 + lane + 32 < it.rows;
#pragma unroll 4
        for (int p = warp; p < pn; p += NW) {
          const float *r = it.src + (long long)(p0 + p) * it.ld + j0 + lane;
          const float v0 = on0 ? r[0] : 0.f, v1 = on1 ? r[32] : 0.f;
          sb[p * PITCH + lane] = v0;
          sb[p * PITCH + lane + 32] = v1;
          m0 = fmaxf(m0, fabsf(v0));
          m1 = fmaxf(m1, fabsf(v1));
        }
      }
    };
    float m0 = 0.f, m1 = 0.f;
    for (int ch = 0; ch < nch; ++ch) {
      __syncthreads();
      stage(ch * PACK_KC, min(PACK_KC, it.k - ch * PACK_KC), m0, m1);
    }
    smax[warp][lane] = m0;
    if (!CPLX) smax[warp][lane + 32] = m1;
    __syncthreads();
    if (tid < 64) {
      const int c = CPLX ? tid >> 1 : tid;
      float m = smax[0][c];
#pragma unroll
      for (int w = 1; w < NW; ++w) m = fmaxf(m, smax[w][c]);
      float mul, inv;
      row_scale(m, mul, inv);
      mul_s[tid] = mul;
      if (far_col(inv) && (__ldcg(far) & FAR_COL) == 0) atomicOr(far, FAR_COL);
      it.scale[(long long)jb * 64 + tid] = inv;
    }
    __syncthreads();
    for (int ch = 0; ch < nch; ++ch) {
      const int p0 = ch * PACK_KC, pn = min(PACK_KC, it.k - p0);
      if (nch > 1) {
        __syncthreads();
        stage(p0, pn, m0, m1);
        __syncthreads();
      }
      const int kt0 = p0 * F / TC_BK, tiles = (pn * F + TC_BK - 1) / TC_BK;
      for (int id = tid; id < tiles * 512; id += 32 * NW) {
        const int c = id & 7, rl = (id >> 3) & 63, kt = id >> 9;
        const float mul = mul_s[rl];
        uint16_t h[8], l[8];
        if (CPLX) {
          const int t = rl & 1;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int p = kt * 32 + c * 4 + e;
            const float2 v = p < pn ? *reinterpret_cast<const float2 *>(sb + p * PITCH + (rl & ~1))
                                    : make_float2(0.f, 0.f);
            split_f16((t == 0 ? v.x : v.y) * mul, h[2 * e], l[2 * e]);           // coefficient of Re A
            split_f16((t == 0 ? -v.y : v.x) * mul, h[2 * e + 1], l[2 * e + 1]);  // coefficient of Im A
          }
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const int p = kt * 64 + c * 8 + e;
            split_f16((p < pn ? sb[p * PITCH + rl] : 0.f) * mul, h[e], l[e]);
          }
        }
        const long long row = (long long)jb * 64 + rl;
        const int nt = (int)(row / TC_BN), r = (int)(row % TC_BN);
        const long long off = ((long long)nt * it.nkt + kt0 + kt) * B_TILE + r * ROW_B + ((c ^ (r & 7)) << 4);
        *reinterpret_cast<uint4 *>(it.hi + off) = make_uint4(pair16(h[0], h[1]), pair16(h[2], h[3]), pair16(h[4], h[5]), pair16(h[6], h[7]));
        *reinterpret_cast<uint4 *>(it.lo + off) = make_uint4(pair16(l[0], l[1]), pair16(l[2], l[3]), pair16(l[4], l[5]), pair16(l[6], l[7]));
      }
    }
    __syncthreads();
  }
}

// Both operands of every item in one launch (blockIdx.y: the A operands, then the B operands); zero, when
// given, is a status word cleared for the GEMM that follows.  NW warps a block.
template <bool CPLX, int NW>
__global__ void __launch_bounds__(32 * NW) pack_f16_kernel(const __grid_constant__ PackBatchP pb, int *zero) {
  extern __shared__ float pack_sb[];
  if (zero && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *zero = 0;
  // complex entries are read in one access where they lie on 8 bytes (the caller's pointer is one to floats)
  const bool is_a = (int)blockIdx.y < pb.na;
  const PackItem &it = is_a ? pb.a[blockIdx.y] : pb.b[blockIdx.y - pb.na];
  if (CPLX && (uintptr_t)it.src % 8 == 0) {
    if (is_a) pack_a_rows<CPLX, NW, true>(it, pb.far);
    else pack_b_rows<CPLX, NW, true>(it, pack_sb, pb.far);
  } else {
    if (is_a) pack_a_rows<CPLX, NW, false>(it, pb.far);
    else pack_b_rows<CPLX, NW, false>(it, pack_sb, pb.far);
  }
}

template <bool CPLX>
static void launch_pack(cudaStream_t st, PackBatchP &pb, int *words, int *zero = nullptr) {
  pb.far = words + 1;
  if (pb.na + pb.nb == 0) return;
  long long blocks = 1, all = 0;
  int kmax = 0;
  for (int i = 0; i < pb.na; ++i) {
    // 256 threads pack 8 to 32 rows at a time (pack_a_rows); whole blocks per 128-row tile either way
    const int rows = 256 / (pb.a[i].nkt >= 4 ? 32 : pb.a[i].nkt >= 2 ? 16 : 8);
    blocks = std::max(blocks, (long long)pb.a[i].nblk * (TC_BM / rows));
    all += (long long)pb.a[i].nblk * (TC_BM / rows);
  }
  for (int i = 0; i < pb.nb; ++i) {
    blocks = std::max(blocks, (long long)pb.b[i].nblk);
    all += pb.b[i].nblk;
    kmax = std::max(kmax, std::min(pb.b[i].k, PACK_KC));
  }
  // a launch with less than a block per SM (right-hand sides of a few columns) is a chain of memory latencies:
  // 32 warps a block shorten it four times
  const size_t smem = (size_t)kmax * (CPLX ? 66 : 65) * sizeof(float);
  const dim3 grid((unsigned)std::min<long long>(blocks, 2048), pb.na + pb.nb);
  if (all < sm_count()) pack_f16_kernel<CPLX, 32><<<grid, 1024, smem, st>>>(pb, zero);
  else pack_f16_kernel<CPLX, 8><<<grid, 256, smem, st>>>(pb, zero);
  RFDD_CHECK_LAUNCH();
}

// ---------------------------------------------------------------------------------------
// operands of the plain TF32 probe: real, rounded to TF32, tiles of 32 floats of K
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ float round_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}
struct Tf32PackItem {
  const float *src;
  long long ld;
  int m, n, k;
  float *dst;
  int mtc, ntc, nkt;
};
struct Tf32PackP {
  Tf32PackItem it;
};
// real B of the plain TF32 probe, staged through shared memory: a 32 (K) x 128 (N) slab, half a packed
// tile (128 rows x 32 K-values)
__global__ void __launch_bounds__(256) pack_b_real_t_kernel(Tf32PackP pb) {
  const Tf32PackItem it = pb.it;
  const int jblocks = it.ntc * 2;  // 128 columns per block
  const int nblk = jblocks * it.nkt;
  __shared__ float sb[32][129];
  for (int bid = blockIdx.x; bid < nblk; bid += gridDim.x) {
    const int kt = bid % it.nkt, jb = bid / it.nkt;
    const long long j0 = (long long)jb * 128;
    const int p0 = kt * TC_BK32;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int idx = threadIdx.x + 256 * i;
      const int pl = idx >> 7, jl = idx & 127;
      const long long j = j0 + jl;
      const int pp = p0 + pl;
      sb[pl][jl] = (j < it.n && pp < it.k) ? it.src[(long long)pp * it.ld + j] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int id = threadIdx.x + 256 * i;
      const int rl = id >> 3, c = id & 7;
      float h[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) h[t] = round_tf32(sb[c * 4 + t][rl]);
      const long long row = j0 + rl;
      const int nt = (int)(row / TC_BN), r = (int)(row % TC_BN);
      const long long off = ((long long)nt * it.nkt + kt) * (B_TILE / 4) + r * TC_BK32 + ((c ^ (r & 7)) << 2);
      *reinterpret_cast<float4 *>(it.dst + off) = make_float4(h[0], h[1], h[2], h[3]);
    }
  }
}

// real A of the plain TF32 probe
__global__ void pack_a_real_kernel(Tf32PackP pb) {
  const Tf32PackItem it = pb.it;
  const long long chunks = (long long)it.mtc * TC_BM * it.nkt * 8;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < chunks; e += (long long)gridDim.x * blockDim.x) {
    const long long row = e / (it.nkt * 8);
    const int q = (int)(e % (it.nkt * 8));
    const int kt = q >> 3, c = q & 7;
    const int mt = (int)(row / TC_BM), r = (int)(row % TC_BM);
    float h[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int kr = kt * TC_BK32 + c * 4 + t;
      h[t] = (row < it.m && kr < it.k) ? round_tf32(it.src[row * it.ld + kr]) : 0.f;
    }
    const long long off = ((long long)mt * it.nkt + kt) * (A_TILE / 4) + r * TC_BK32 + ((c ^ (r & 7)) << 2);
    *reinterpret_cast<float4 *>(it.dst + off) = make_float4(h[0], h[1], h[2], h[3]);
  }
}
// Per-device launch set-up of the tensor-core kernel: its dynamic shared-memory limit is raised
// once on every device it runs on, and the device's SM count sizes the persistent grid.
struct TcDevInfo {
  bool attr = false;
  int nsm = 0;
  int clusters2 = 0;  // two-CTA clusters of tc_gemm2_kernel that can be resident at once
};
static TcDevInfo tc_device_info() {
  static std::mutex mu;
  static std::vector<TcDevInfo> info;
  int dev = 0;
  RFDD_CUDA(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(mu);
  if ((int)info.size() <= dev) info.resize(dev + 1);
  TcDevInfo &d = info[dev];
  if (!d.attr) {
    const void *ones[] = {(const void *)tc_gemm_kernel<true, 256>, (const void *)tc_gemm_kernel<true, 64>,
                          (const void *)tc_gemm_kernel<false, 256>};
    for (const void *f : ones) RFDD_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM));
    const void *packs[] = {(const void *)pack_f16_kernel<true, 8>, (const void *)pack_f16_kernel<true, 32>,
                           (const void *)pack_f16_kernel<false, 8>, (const void *)pack_f16_kernel<false, 32>};
    for (const void *f : packs)
      RFDD_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, PACK_KC * 66 * (int)sizeof(float)));
    RFDD_CUDA(cudaFuncSetAttribute(tc_gemm2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, T2_SMEM));
    RFDD_CUDA(cudaDeviceGetAttribute(&d.nsm, cudaDevAttrMultiProcessorCount, dev));
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 2;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.gridDim = dim3(2, 1, 1);
    cfg.blockDim = dim3(TC_THREADS, 1, 1);
    cfg.dynamicSmemBytes = T2_SMEM;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int nc = 0;
    if (cudaOccupancyMaxActiveClusters(&nc, (void *)tc_gemm2_kernel, &cfg) != cudaSuccess) {
      cudaGetLastError();
      nc = 0;
    }
    d.clusters2 = nc;
    d.attr = true;
  }
  return d;
}
static int tc_device_setup() { return std::max(1, tc_device_info().nsm); }

// Kernel choice for a launch (g_tc_engine_override lets rfdd_cgemm force one for tests):
// the two-CTA kernel when it has work for every resident cluster and few of its pair tiles are
// half empty (an odd number of row tiles leaves the second CTA of the last pair without rows).
thread_local int g_tc_engine_override = 0;  // 0 automatic, 1 one-CTA kernel, 2 two-CTA kernel
TcEngineScope::TcEngineScope(int e) : prev(g_tc_engine_override) { g_tc_engine_override = e; }
TcEngineScope::~TcEngineScope() { g_tc_engine_override = prev; }

// The tile-shape autotuner (tc_tune.h) and the timings it is waiting for.  Launches it asks to
// measure are bracketed by events on their own stream; the events are polled without blocking at
// the next launch and when the table is read.
namespace {
struct TunePending {
  tune::Key key;
  int cand;
  double gflop;
  cudaEvent_t e0, e1;
};
std::mutex g_tune_mu;
tune::Tuner g_tuner;
std::vector<TunePending> g_tune_pending;

void tune_poll_locked() {
  for (size_t i = 0; i < g_tune_pending.size();) {
    TunePending &q = g_tune_pending[i];
    const cudaError_t r = cudaEventQuery(q.e1);
    if (r == cudaErrorNotReady) {
      ++i;
      continue;
    }
    float ms = 0.0f;
    if (r == cudaSuccess && cudaEventElapsedTime(&ms, q.e0, q.e1) == cudaSuccess && q.gflop > 0.0)
      g_tuner.record(q.key, q.cand, ms / q.gflop);
    else
      g_tuner.forget(q.key, q.cand);
    if (r != cudaSuccess) cudaGetLastError();
    cudaEventDestroy(q.e0);
    cudaEventDestroy(q.e1);
    g_tune_pending.erase(g_tune_pending.begin() + i);
  }
}
}  // namespace

int tc_autotune(int mode) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  const int prev = g_tuner.enabled ? 1 : 0;
  if (mode == 2) {
    tune_poll_locked();
    g_tuner.clear();
  } else {
    g_tuner.enabled = mode != 0;
  }
  return prev;
}

std::string tc_autotune_table() {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  tune_poll_locked();
  return g_tuner.dump();
}

// Tile walk of one item: down the columns when B spans at least 8 tile columns and the item's
// packed A (hi + lo) takes at most 48 MB of the 129 MB L2, else along the rows.
int tc_tile_order(int mtc, int ntc, int nkt) {
  const double a_bytes = 2.0 * mtc * nkt * (double)A_TILE;
  return (ntc >= 8 && mtc >= 2 && a_bytes <= 48e6) ? 1 : 0;
}

// Bytes of one packed operand: hi and lo tiles, then the scales (a multiple of 256 bytes)
static size_t packed_bytes(size_t tiles, size_t tile_bytes, size_t scales) {
  return 2 * tiles * tile_bytes + (scales * sizeof(float) + 255) / 256 * 256;
}

// Output tiles of the launch when they are BN wide: sets each item's tile counts, first tile and width of
// access to C
static int set_tiles(TcBatchP &tb, int BN) {
  int tiles = 0;
  for (int i = 0; i < tb.count; ++i) {
    TcItem &it = tb.it[i];
    it.ntc = ceil_div(it.n2, BN);
    it.vec = it.ldc % 4 == 0 && (uintptr_t)it.C % 16 == 0 ? 4 : 1;
    it.colmajor = tc_tile_order(it.mtc, it.ntc, it.nkt);
    it.tile0 = tiles;
    tiles += it.mtc * it.ntc;
  }
  tb.total_tiles = tiles;
  return tiles;
}

// One-CTA launch.  64-wide tiles when the 256-wide ones leave SMs without work (four times the tiles,
// and a ring four stages deep) or are at most a quarter full.
static void launch_one_cta(cudaStream_t st, TcBatchP &tb, int nsm, double alpha, double beta) {
  int n2max = 0;
  for (int i = 0; i < tb.count; ++i) n2max = std::max(n2max, tb.it[i].n2);
  const bool narrow = n2max <= 64 || set_tiles(tb, TC_BN) < nsm;
  const int tiles = set_tiles(tb, narrow ? 64 : TC_BN);
  const int grid = std::max(1, std::min(tiles, nsm));
  if (narrow) tc_gemm_kernel<true, 64><<<grid, TC_THREADS, TC_SMEM, st>>>(tb, (float)alpha, (float)beta);
  else tc_gemm_kernel<true, 256><<<grid, TC_THREADS, TC_SMEM, st>>>(tb, (float)alpha, (float)beta);
  RFDD_CHECK_LAUNCH();
}

template <bool CPLX, typename T>
static void tc_gemm_run(cudaStream_t st, const std::vector<GemmItem<T>> &items, double alpha, double beta,
                        const std::vector<TcPackedA> *pre = nullptr) {
  constexpr int F = CPLX ? 2 : 1;  // real columns / K entries per element
  RFDD_REQUIRE(g_tc_status != nullptr, RFDD_ESTATE, "tensor-core GEMM launched without a status word");
  const int nsm = tc_device_setup();
  for (size_t s0 = 0; s0 < items.size(); s0 += TC_MAXB) {
    const int cnt = (int)std::min<size_t>(TC_MAXB, items.size() - s0);
    PackBatchP pk;
    TcBatchP tb;
    memset(&pk, 0, sizeof(pk));
    memset(&tb, 0, sizeof(tb));
    size_t total = 0;
    std::vector<size_t> offA(cnt), offB(cnt);
    double flops = 0.0, cbytes = 0.0;
    for (int i = 0; i < cnt; ++i) {
      const auto &g = items[s0 + i];
      const size_t mtc = ceil_div(g.m, TC_BM), ntc = ceil_div((int64_t)F * g.n, TC_BN), nkt = ceil_div((int64_t)F * g.k, TC_BK);
      const bool packed = pre && (*pre)[s0 + i].hi;
      offA[i] = total;
      if (!packed) total += packed_bytes(mtc * nkt, A_TILE, mtc * TC_BM);
      offB[i] = total;
      total += packed_bytes(ntc * nkt, B_TILE, ntc * TC_BN);
      flops += (CPLX ? 8.0 : 2.0) * g.m * (double)g.n * g.k;
      // compulsory DRAM bytes: C read (beta != 0) and written, packed hi/lo operands read once
      cbytes += (beta != 0.0 ? 2.0 : 1.0) * 4.0 * F * g.m * (double)g.n +
                2.0 * ((double)mtc * nkt * A_TILE + (double)ntc * nkt * B_TILE);
    }
    uint8_t *ws = nullptr;
    RFDD_CUDA(cudaMallocAsync((void **)&ws, total, st));
    tb.count = cnt;
    for (int i = 0; i < cnt; ++i) {
      const auto &g = items[s0 + i];
      const int mtc = ceil_div(g.m, TC_BM), ntc = ceil_div((int64_t)F * g.n, TC_BN), nkt = ceil_div((int64_t)F * g.k, TC_BK);
      TcItem &it = tb.it[i];
      uint8_t *Bh = ws + offB[i], *Bl = Bh + (size_t)ntc * nkt * B_TILE;
      float *sB = reinterpret_cast<float *>(Bl + (size_t)ntc * nkt * B_TILE);
      pk.b[pk.nb++] = {reinterpret_cast<const float *>(g.B), g.ldb, g.n, g.k, Bh, Bl, sB, ceil_div((int64_t)F * g.n, 64), nkt, 0};
      it.Bhi = Bh;
      it.Blo = Bl;
      it.sB = sB;
      if (pre && (*pre)[s0 + i].hi) {
        const TcPackedA &p = (*pre)[s0 + i];
        it.Ahi = p.hi;
        it.Alo = p.lo;
        it.sA = p.scale;
        it.amts = p.mt_stride;
      } else {
        uint8_t *Ah = ws + offA[i], *Al = Ah + (size_t)mtc * nkt * A_TILE;
        float *sA = reinterpret_cast<float *>(Al + (size_t)mtc * nkt * A_TILE);
        pk.a[pk.na++] = {reinterpret_cast<const float *>(g.A), g.lda, g.m, g.k, Ah, Al, sA, mtc, nkt, 0};
        it.Ahi = Ah;
        it.Alo = Al;
        it.sA = sA;
        it.amts = 0;
      }
      it.C = reinterpret_cast<float *>(g.C);
      it.ldc = (long long)F * g.ldc;
      it.m = g.m;
      it.n2 = F * g.n;
      it.nkt = nkt;
      it.mtc = mtc;
    }
    const int tiles = set_tiles(tb, TC_BN);
    tb.err = g_tc_status;
    launch_pack<CPLX>(st, pk, g_tc_status);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (profiling_enabled()) {
      e0 = profile_event();
      e1 = profile_event();
      cudaEventRecord(e0, st);
    }
    // pair tiles of the two-CTA kernel
    long long pairs = 0, ghosts = 0;
    for (int i = 0; i < cnt; ++i) {
      pairs += (long long)((tb.it[i].mtc + 1) / 2) * tb.it[i].ntc;
      ghosts += (long long)(tb.it[i].mtc & 1) * tb.it[i].ntc;
    }
    const TcDevInfo dinfo = tc_device_info();
    // measured on 8192 x 8192 products: the two-CTA kernel gains from K = 256 (complex) on (4 %
    // there, 1.5 % at K = 1024) and loses at K = 128, where the epilogue, not the operand feed,
    // bounds both kernels
    int64_t k32_min = 1 << 30;  // K in units of 32 real entries
    for (int i = 0; i < cnt; ++i) k32_min = std::min<int64_t>(k32_min, ceil_div((int64_t)F * items[s0 + i].k, 32));
    const bool two_ok = dinfo.clusters2 > 0 && pairs >= dinfo.clusters2 && 8 * ghosts <= pairs;
    bool two = two_ok && (CPLX ? k32_min >= 16 : k32_min >= 8);
    // the autotuner decides where both kernels can run, outside stream capture
    tune::Key tkey;
    bool tmeasure = false;
    if (two_ok && g_tc_engine_override == 0) {
      cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
      RFDD_CUDA(cudaStreamIsCapturing(st, &cs));
      RFDD_CUDA(cudaGetDevice(&tkey.device));
      tkey.cplx = CPLX ? 1 : 0;
      tkey.splits = 3;
      tkey.kbucket = tune::k_bucket(k32_min);
      tkey.tbucket = tune::t_bucket(tiles, nsm);
      std::lock_guard<std::mutex> lk(g_tune_mu);
      tune_poll_locked();
      if (cs == cudaStreamCaptureStatusNone) {
        const tune::Choice ch = g_tuner.choose(tkey, two ? 1 : 0);
        two = ch.cand == 1;
        tmeasure = ch.measure;
      } else {
        const auto &t = g_tuner.table();
        const auto it = t.find(tkey);
        if (it != t.end() && it->second.winner >= 0) two = it->second.winner == 1;
      }
    }
    if (g_tc_engine_override == 1) two = false;
    if (g_tc_engine_override == 2) two = dinfo.clusters2 > 0;
    cudaEvent_t te0 = nullptr, te1 = nullptr;
    if (tmeasure) {
      if (cudaEventCreate(&te0) != cudaSuccess || cudaEventCreate(&te1) != cudaSuccess) {
        cudaGetLastError();
        if (te0) cudaEventDestroy(te0);
        te0 = te1 = nullptr;
        std::lock_guard<std::mutex> lk(g_tune_mu);
        g_tuner.forget(tkey, two ? 1 : 0);
      } else {
        RFDD_CUDA(cudaEventRecord(te0, st));
      }
    }
    if (g_tc_events) RFDD_CUDA(cudaEventRecord(g_tc_events[0], st));
    if (two) {
      TcBatchP t2 = tb;
      int p0 = 0;
      for (int i = 0; i < cnt; ++i) {
        t2.it[i].tile0 = p0;
        p0 += ((t2.it[i].mtc + 1) / 2) * t2.it[i].ntc;
      }
      t2.total_tiles = p0;
      const int ncl = std::max(1, std::min(p0, dinfo.clusters2));
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute attr;
      attr.id = cudaLaunchAttributeClusterDimension;
      attr.val.clusterDim.x = 2;
      attr.val.clusterDim.y = 1;
      attr.val.clusterDim.z = 1;
      cfg.gridDim = dim3(2 * ncl, 1, 1);
      cfg.blockDim = dim3(TC_THREADS, 1, 1);
      cfg.dynamicSmemBytes = T2_SMEM;
      cfg.stream = st;
      cfg.attrs = &attr;
      cfg.numAttrs = 1;
      RFDD_CUDA(cudaLaunchKernelEx(&cfg, tc_gemm2_kernel, t2, (float)alpha, (float)beta));
      RFDD_CHECK_LAUNCH();
    } else {
      launch_one_cta(st, tb, nsm, alpha, beta);
    }
    if (g_tc_events) RFDD_CUDA(cudaEventRecord(g_tc_events[1], st));
    if (te1) {
      RFDD_CUDA(cudaEventRecord(te1, st));
      std::lock_guard<std::mutex> lk(g_tune_mu);
      g_tune_pending.push_back({tkey, two ? 1 : 0, flops * 1e-9, te0, te1});
    }
    if (e0) {
      cudaEventRecord(e1, st);
      profile_push(e0, e1, flops, 1, cbytes);
    }
    RFDD_CUDA(cudaFreeAsync(ws, st));
  }
}


void tc_gemm_complex(cudaStream_t st, const std::vector<GemmItem<cx<float>>> &items, double alpha, double beta) {
  tc_gemm_run<true>(st, items, alpha, beta);
}

void tc_gemm_complex_pa(cudaStream_t st, const std::vector<GemmItem<cx<float>>> &items,
                        const std::vector<TcPackedA> &pa, double alpha, double beta) {
  RFDD_REQUIRE(pa.size() == items.size(), RFDD_EINVAL, "tc_gemm: one packed-A entry per item");
  std::vector<GemmItem<cx<float>>> live;
  std::vector<TcPackedA> lpa;
  for (size_t i = 0; i < items.size(); ++i)
    if (items[i].m > 0 && items[i].n > 0 && items[i].k > 0) {
      live.push_back(items[i]);
      lpa.push_back(pa[i]);
    }
  if (!live.empty()) tc_gemm_run<true>(st, live, alpha, beta, &lpa);
}

static int64_t packed_a_ktiles(int64_t k) { return ceil_div(2 * k, TC_BK); }
int64_t tc_packed_a_bytes(int64_t m, int64_t k, bool sides) {
  const size_t mtc = ceil_div(m, TC_BM);
  return (int64_t)packed_bytes(mtc * packed_a_ktiles(k), A_TILE, mtc * TC_BM * (sides ? 2 : 1));
}

TcPackedA tc_packed_view(const void *op, int64_t m, int64_t k_full, int64_t r0, int64_t c0, int side) {
  RFDD_REQUIRE(r0 % TC_BM == 0 && (2 * c0) % TC_BK == 0, RFDD_EINVAL, "packed view must start on a tile");
  const int64_t kt = packed_a_ktiles(k_full), mtc = ceil_div(m, TC_BM);
  const uint8_t *hi = static_cast<const uint8_t *>(op), *lo = hi + mtc * kt * A_TILE;
  const float *scale = reinterpret_cast<const float *>(lo + mtc * kt * A_TILE) + side * mtc * TC_BM;
  const int64_t off = ((r0 / TC_BM) * kt + (2 * c0) / TC_BK) * A_TILE;
  return TcPackedA{hi + off, lo + off, scale + r0, kt};
}

void tc_pack_a_batched(cudaStream_t st, const std::vector<TcPackJob> &jobs) {
  RFDD_REQUIRE(g_tc_status != nullptr, RFDD_ESTATE, "operands packed without a status word");
  tc_device_setup();
  for (size_t s0 = 0; s0 < jobs.size(); s0 += TC_MAXB) {
    const int cnt = (int)std::min<size_t>(TC_MAXB, jobs.size() - s0);
    PackBatchP pk;
    memset(&pk, 0, sizeof(pk));
    for (int i = 0; i < cnt; ++i) {
      const TcPackJob &j = jobs[s0 + i];
      if (j.m <= 0 || j.k <= 0) continue;
      const int64_t mtc = ceil_div(j.m, TC_BM), nkt = packed_a_ktiles(j.k);
      uint8_t *hi = static_cast<uint8_t *>(j.dst), *lo = hi + mtc * nkt * A_TILE;
      pk.a[pk.na++] = {reinterpret_cast<const float *>(j.A), j.lda, (int)j.m, (int)j.k, hi, lo,
                       reinterpret_cast<float *>(lo + mtc * nkt * A_TILE), (int)mtc, (int)nkt, j.side};
    }
    launch_pack<true>(st, pk, g_tc_status);
  }
}

void tc_gemm_real(cudaStream_t st, const std::vector<GemmItem<float>> &items, double alpha, double beta) {
  tc_gemm_run<false>(st, items, alpha, beta);
}

void tc_gemm_real_tf32(cudaStream_t st, const GemmItem<float> &g, double alpha, double beta) {
  RFDD_REQUIRE(g_tc_status != nullptr, RFDD_ESTATE, "tensor-core GEMM launched without a status word");
  const int nsm = tc_device_setup();
  const int mtc = ceil_div(g.m, TC_BM), ntc = ceil_div(g.n, TC_BN), nkt = ceil_div(g.k, TC_BK32);
  const size_t a_bytes = (size_t)mtc * nkt * A_TILE, b_bytes = (size_t)ntc * nkt * B_TILE;
  uint8_t *ws = nullptr;
  RFDD_CUDA(cudaMallocAsync((void **)&ws, a_bytes + b_bytes, st));
  uint8_t *Bt = ws + a_bytes;
  Tf32PackP pa{{g.A, g.lda, g.m, g.n, g.k, reinterpret_cast<float *>(ws), mtc, ntc, nkt}};
  Tf32PackP pb{{g.B, g.ldb, g.m, g.n, g.k, reinterpret_cast<float *>(Bt), mtc, ntc, nkt}};
  pack_a_real_kernel<<<4096, 256, 0, st>>>(pa);
  RFDD_CHECK_LAUNCH();
  pack_b_real_t_kernel<<<8192, 256, 0, st>>>(pb);
  RFDD_CHECK_LAUNCH();
  TcBatchP tb;
  memset(&tb, 0, sizeof(tb));
  tb.count = 1;
  tb.err = g_tc_status;
  TcItem &it = tb.it[0];
  it.Ahi = ws;
  it.Bhi = Bt;
  it.C = g.C;
  it.ldc = g.ldc;
  it.m = g.m;
  it.n2 = g.n;
  it.nkt = nkt;
  it.mtc = mtc;
  const int tiles = set_tiles(tb, TC_BN);
  if (g_tc_events) RFDD_CUDA(cudaEventRecord(g_tc_events[0], st));
  tc_gemm_kernel<false, 256><<<std::max(1, std::min(tiles, nsm)), TC_THREADS, TC_SMEM, st>>>(tb, (float)alpha, (float)beta);
  RFDD_CHECK_LAUNCH();
  if (g_tc_events) RFDD_CUDA(cudaEventRecord(g_tc_events[1], st));
  RFDD_CUDA(cudaFreeAsync(ws, st));
}

// =========================================================================================
// Allocation-free variant of the tensor-core complex GEMM.
//
// Some callers cannot call cudaMalloc: code running inside a memory-capped process or allocator
// arena, real-time loops that must not touch the allocator, or host code that must not
// synchronise with other streams the way allocation can.  For them the packed operand tiles
// live in the file-scope array below instead of a per-call workspace.  The array's host-side
// name is only a stand-in: its device address is looked up with cudaGetSymbolAddress once per
// device (on that device's first call, with the device current) and passed to the kernels.
// =========================================================================================
constexpr int NOALLOC_MAX_M = 1024;   // complex rows of A and C
constexpr int NOALLOC_MAX_N = 1024;   // complex columns of B and C
constexpr int NOALLOC_MAX_K = 128;    // complex inner dimension
constexpr size_t noalloc_bytes(size_t tiles, size_t tile_bytes, size_t scales) {
  return 2 * tiles * tile_bytes + (scales * sizeof(float) + 255) / 256 * 256;
}
constexpr size_t NOALLOC_KT = (2 * NOALLOC_MAX_K + TC_BK - 1) / TC_BK;
constexpr size_t NOALLOC_MT = (NOALLOC_MAX_M + TC_BM - 1) / TC_BM, NOALLOC_NT = (2 * NOALLOC_MAX_N + TC_BN - 1) / TC_BN;
constexpr size_t NOALLOC_A_BYTES = noalloc_bytes(NOALLOC_MT * NOALLOC_KT, A_TILE, NOALLOC_MT * TC_BM);
constexpr size_t NOALLOC_B_BYTES = noalloc_bytes(NOALLOC_NT * NOALLOC_KT, B_TILE, NOALLOC_NT * TC_BN);

static __device__ __align__(256) uint8_t g_noalloc_scratch[NOALLOC_A_BYTES + NOALLOC_B_BYTES];  // 3 MiB
// status words of the allocation-free launches, beside the scratch
static __device__ int g_noalloc_status[STATUS_WORDS];

struct NoallocAddr {
  uint8_t *scratch = nullptr;
  int *status = nullptr;
};
// Device addresses of the array and of its status word on the current device, looked up once per
// device with that device current (the host-side names are only stand-ins).
static NoallocAddr noalloc_addresses() {
  static std::mutex mu;
  static std::vector<NoallocAddr> addr;
  int dev = 0;
  RFDD_CUDA(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(mu);
  if ((int)addr.size() <= dev) addr.resize(dev + 1);
  if (!addr[dev].scratch) {
    void *p = nullptr, *q = nullptr;
    RFDD_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
    RFDD_CUDA(cudaGetSymbolAddress(&q, g_noalloc_status));
    addr[dev].scratch = reinterpret_cast<uint8_t *>(p);
    addr[dev].status = reinterpret_cast<int *>(q);
  }
  return addr[dev];
}

int tc_gemm_complex_noalloc(cudaStream_t st, const cx<float> *A, int64_t lda, const cx<float> *B, int64_t ldb,
                            cx<float> *C, int64_t ldc, int m, int n, int k, double alpha, double beta) {
  RFDD_REQUIRE(m >= 1 && n >= 1 && k >= 1, RFDD_EINVAL, "cgemm_noalloc: sizes must be positive");
  RFDD_REQUIRE(m <= NOALLOC_MAX_M && n <= NOALLOC_MAX_N && k <= NOALLOC_MAX_K, RFDD_EINVAL,
               "cgemm_noalloc: m, n must be <= 1024 and k <= 128 (size of the static scratch)");
  const NoallocAddr na = noalloc_addresses();
  const int nsm = tc_device_setup();
  const int mtc = ceil_div(m, TC_BM), ntc = ceil_div(2 * (int64_t)n, TC_BN), nkt = ceil_div(2 * (int64_t)k, TC_BK);
  uint8_t *Ah = na.scratch, *Al = Ah + (size_t)mtc * nkt * A_TILE;
  uint8_t *Bh = na.scratch + NOALLOC_A_BYTES, *Bl = Bh + (size_t)ntc * nkt * B_TILE;
  float *sA = reinterpret_cast<float *>(Al + (size_t)mtc * nkt * A_TILE);
  float *sB = reinterpret_cast<float *>(Bl + (size_t)ntc * nkt * B_TILE);
  PackBatchP pk;
  TcBatchP tb;
  memset(&pk, 0, sizeof(pk));
  memset(&tb, 0, sizeof(tb));
  pk.na = pk.nb = 1;
  pk.a[0] = {reinterpret_cast<const float *>(A), lda, m, k, Ah, Al, sA, mtc, nkt, 0};
  pk.b[0] = {reinterpret_cast<const float *>(B), ldb, n, k, Bh, Bl, sB, ceil_div(2 * (int64_t)n, 64), nkt, 0};
  TcItem &it = tb.it[0];
  it.Ahi = Ah;
  it.Alo = Al;
  it.Bhi = Bh;
  it.Blo = Bl;
  it.sA = sA;
  it.sB = sB;
  it.C = reinterpret_cast<float *>(C);
  it.ldc = 2ll * ldc;
  it.m = m;
  it.n2 = 2 * n;
  it.nkt = nkt;
  it.mtc = mtc;
  tb.count = 1;
  tb.err = na.status;
  // the status word keeps the last call's value: the packing launch clears it; that of the far scales is cleared here
  launch_pack<true>(st, pk, na.status, na.status);
  launch_one_cta(st, tb, nsm, alpha, beta);
  int status[STATUS_WORDS] = {};
  RFDD_CUDA(cudaMemcpyAsync(status, na.status, sizeof(status), cudaMemcpyDeviceToHost, st));
  RFDD_CUDA(cudaStreamSynchronize(st));
  if (status[1]) {  // cleared before this call returns: the next one may come on another stream
    RFDD_CUDA(cudaMemsetAsync(na.status + 1, 0, sizeof(int), st));
    RFDD_CUDA(cudaStreamSynchronize(st));
  }
  return status[0];
}

}  // namespace rfdd
