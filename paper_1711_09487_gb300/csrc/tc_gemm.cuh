// Tensor-core (tcgen05, two-way 16-bit split) complex-FP32 GEMM; host launcher.
#pragma once
#include "dense.cuh"

#include <string>

namespace rfdd {
// Status words (STATUS_WORDS device ints) that the tensor-core launches issued by the calling host thread record
// a failed wait in (DS_WAIT_TIMEOUT), for the lifetime of the scope.  A launch outside any scope is
// refused with RFDD_ESTATE.  digits: what the digit products of the scope may be used for and hold.
struct TcDigitRule {
  bool updates = true;                   // FP64 factorisation and solve updates (tc_fp64_takes)
  size_t bytes = digit_bytes_cap(0);     // device bytes of the digits of one launch
};
struct TcStatusScope {
  int *prev;
  TcDigitRule prev_digits;
  explicit TcStatusScope(int *word, TcDigitRule digits = {});
  ~TcStatusScope();
  TcStatusScope(const TcStatusScope &) = delete;
  TcStatusScope &operator=(const TcStatusScope &) = delete;
};
// the calling thread's status word (nullptr outside any scope)
int *tc_status_word();
// the rule of the calling thread's scope
TcDigitRule tc_digit_rule();
// While alive, the tensor-core kernel launches of the calling host thread record ab[0] just before
// and ab[1] just after the kernel (not the operand packing): the probes time the MMA kernel alone.
struct TcKernelEvents {
  const cudaEvent_t *prev;
  explicit TcKernelEvents(const cudaEvent_t *ab);
  ~TcKernelEvents();
  TcKernelEvents(const TcKernelEvents &) = delete;
  TcKernelEvents &operator=(const TcKernelEvents &) = delete;
};
// While alive, the tensor-core launches of the calling host thread use one kernel: 1 the one-CTA
// kernel (128 x 256 tiles), 2 the two-CTA kernel (256 x 256 tiles on SM pairs), 0 the automatic
// choice.  For tests that check both kernels.
struct TcEngineScope {
  int prev;
  explicit TcEngineScope(int engine);
  ~TcEngineScope();
  TcEngineScope(const TcEngineScope &) = delete;
  TcEngineScope &operator=(const TcEngineScope &) = delete;
};
// C = beta*C + alpha*A*B for every item (complex, row-major, no transposes)
void tc_gemm_complex(cudaStream_t st, const std::vector<GemmItem<cx<float>>> &items, double alpha, double beta);
// C = beta*C + alpha*A*B for real FP32 items (same kernel)
void tc_gemm_real(cudaStream_t st, const std::vector<GemmItem<float>> &items, double alpha, double beta);
// the same with one TF32 product per multiply (operands rounded to TF32): the throughput probe of
// the plain TF32 tensor path, not used by the solver
void tc_gemm_real_tf32(cudaStream_t st, const GemmItem<float> &item, double alpha, double beta);

// FP64 products by exact digit products on the tensor cores (tc_dgemm.cu): C = beta*C + alpha*op(A)*op(B), op as
// in gemm_batched, sym as in gemm_f64x2_batched.  tc_dgemm_takes: whether an item is large enough to gain and its
// digits fit.
bool tc_dgemm_takes(const GemmItem<double> &g);
void tc_dgemm_batched(cudaStream_t st, const std::vector<GemmItem<double>> &items, bool ta, bool tb, double alpha,
                      double beta, const std::vector<char> &sym);

// The same for products without transposes in real or complex FP64: the trailing and triangular-solve updates
// of the FP64 factorisations.  tc_fp64_takes: whether the batch as a whole gains over the FP64 pipes.
template <typename T>
bool tc_fp64_takes(const std::vector<GemmItem<T>> &items);
template <typename T>
void tc_fp64_batched(cudaStream_t st, const std::vector<GemmItem<T>> &items, double alpha, double beta);

// The tile-shape autotuner: mode 0 off (fixed rule), 1 on, 2 forget every class (re-tune);
// returns whether it was on.  tc_autotune_table: one line per class (tc_tune.h, Tuner::dump).
int tc_autotune(int mode);
std::string tc_autotune_table();
// A operand already scaled, split into 16-bit hi/lo and laid out in the kernel's tiles
// (tc_pack_a_batched): tile (mt, kt) of the operand at hi/lo + (mt * mt_stride + kt) * tile size, the
// inverse scale of each row in scale.  Lets a factor that is multiplied many times
// (triangular-solve updates, border products) be packed once.
struct TcPackedA {
  const uint8_t *hi = nullptr, *lo = nullptr;
  const float *scale = nullptr;
  int64_t mt_stride = 0;
};
// items[i] uses pa[i] as its A operand when pa[i].hi is set (items[i].A is then not read)
void tc_gemm_complex_pa(cudaStream_t st, const std::vector<GemmItem<cx<float>>> &items,
                        const std::vector<TcPackedA> &pa, double alpha, double beta);
// Packing of complex m x k matrices (row-major, leading dimension lda) into operands of
// tc_packed_a_bytes(m, k, side > 0) bytes each at dst: hi tiles, lo tiles, scales (rows and K padded
// with zeros to whole tiles).  side > 0: an L\U factor whose products use the part left of the
// diagonal blocks of `side` rows (L) or the rest (U), never both: each part of a row has its own scale.
struct TcPackJob {
  const cx<float> *A;
  int64_t lda, m, k;
  void *dst;
  int side = 0;
};
int64_t tc_packed_a_bytes(int64_t m, int64_t k, bool sides = false);
void tc_pack_a_batched(cudaStream_t st, const std::vector<TcPackJob> &jobs);
// the sub-matrix of a packed m x k_full operand starting at row r0 (a multiple of 128) and complex
// column c0 (a multiple of 32); side: 0 the only scale, or that of the left part; 1 the right part's
TcPackedA tc_packed_view(const void *op, int64_t m, int64_t k_full, int64_t r0 = 0, int64_t c0 = 0, int side = 0);
// TFLOP/s of kind::tf32 or kind::f16 MMAs issued back to back from operand tiles resident in shared memory
// (one CTA per SM, no operand loads): the tensor pipe's own rate.  Time-outs go to *dev_status.
double tc_mma_probe_tflops(cudaStream_t st, int *dev_status, bool f16);
// tile walk of a GEMM item with mtc x ntc output tiles and nkt K tiles: 1 down the columns, 0
// along the rows (see tc_gemm.cu)
int tc_tile_order(int mtc, int ntc, int nkt);
// allocation-free variant: packed operands in a static device array (m, n <= 1024, k <= 128);
// waits for `st` and returns the launch's DS_* status bits (0 = ok)
int tc_gemm_complex_noalloc(cudaStream_t st, const cx<float> *A, int64_t lda, const cx<float> *B, int64_t ldb,
                             cx<float> *C, int64_t ldc, int m, int n, int k, double alpha, double beta);
}  // namespace rfdd
