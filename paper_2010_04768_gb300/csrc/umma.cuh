// Tensor-core (tcgen05) contractions.
#pragma once
#include <cuda_bf16.h>

#include "common.cuh"

namespace gfcc {

// Entries of a digit-plane product that are to be summed in FP64 instead: (row, column) of the first min(count, cap).
// With more than cap of them the whole product is (kernels of the other way then return at once).
struct GuardList {
  unsigned *count = nullptr;
  int2 *at = nullptr;
  double *value = nullptr;
  unsigned cap = 0;
};

// D[m][n] = alpha * sum_k A[m][k] B[n][k] + beta * D[m][n]; A: M x K, B: N x K (BF16, K-major,
// row strides lda / ldb multiples of 8 elements, 16-byte aligned), D: FP32 row-major.
// nsplit > 1 splits K: partial sum z goes to D + z * split_stride (with beta != 0 each partial
// accumulates onto its own previous contents); the caller reduces the partials.  The split count actually used is returned through *nsplit_used if given.
int gemm_bf16_tn(cudaStream_t st, const __nv_bfloat16 *A, long long lda, const __nv_bfloat16 *B, long long ldb,
                 float *D, long long ldd, int M, int N, int K, float alpha, float beta, int nsplit = 1,
                 long long split_stride = 0);
// number of partial sums gemm_bf16_tn writes for a requested split of K
int umma_splits(int K, int nsplit);
// FP64-accurate product from digit planes with all digit pairs of a tile in one kernel (levels in
// TMEM): C(m, n0 + n) = alpha 2^(eA[m] + eB[n]) sum_{i+j<=P} 2^(-bits (i+j)) A_i B_j^T + beta C(m, n0 + n).
// A planes: Adig + i * plA (M x K, row stride ld), B planes: Bdig + j * plB (N x K), balanced digits of
// `bits` bits.  `work` holds emu_fused_work_bytes of FP64 partials (products whose K is split).
int emu_gemm_fused(cudaStream_t st, const __nv_bfloat16 *Adig, long long plA, int SA, const int *eA,
                   const __nv_bfloat16 *Bdig, long long plB, int SB, const int *eB, long long ld, int M, int N, int K,
                   int P, int bits, double alpha, double beta, double *C, IMap cm, IMap cn, long long n0,
                   double *work, long long m0 = 0, const GuardList *gate = nullptr);
// Appends to the list the entries (m0 + m, n0 + n) whose sum over k of A[m][k] B[n][k] (planes of magnitudes, row stride ld)
// is neither zero nor from theta up to a finite value.  `work` holds emu_guard_work_bytes.
int emu_guard(cudaStream_t st, const __nv_bfloat16 *A, const __nv_bfloat16 *B, long long ld, int M, int N, int K,
              float theta, const GuardList &list, long long m0, long long n0, float *work);
long long emu_guard_work_bytes(long long M, long long N, long long K);
long long emu_fused_work_bytes(long long M, long long N, long long K);
bool emu_fused_takes(int SA, int SB, int P);   // digit counts and level that emu_gemm_fused evaluates
// Tile autotuning (on by default): the first call of each GEMM shape with beta == 0 times the tiles that may win (one
// CTA, CTA pair, persistent, each in three widths), unless other calls share the GPU, and every later call of the shape
// uses the fastest.
void umma_set_autotune(bool on);
// CTA-pair tiles (cta_group::2, 256 rows x 128, 192 or 256 columns per pair): 0 timed by the autotuner beside the one-CTA
// tiles (default), 1 used whenever they apply, 2 never
void umma_set_pair_mode(int mode);
// persistent tile loop (one CTA per SM, two TMEM accumulators): 0 timed by the autotuner (default),
// 1 always, 2 never
void umma_set_persist_mode(int mode);
int umma_tuned_tile(int M, int N, int K, int nsplit);   // 0 if the shape was not tuned yet
// Limit of the bounded pipeline waits of the tensor-core kernels (process-wide; default 1 s) and a
// test-only switch under which their producers issue no loads (the wait then runs out with nothing
// in flight and the kernel returns the GFCC_ERR_TIMEOUT status).
void umma_set_wait(unsigned long long wait_ns, bool skip_loads);
// The error flag (one device word) of the calling thread's tensor-core kernels for the lifetime of the scope: a bounded
// wait that gives up sets it.  Each context has its own, and so has each call without one, so that neither a time-out nor
// a reset reaches another call.
struct UmmaScope {
  explicit UmmaScope(unsigned *flag);
  ~UmmaScope();
  UmmaScope(const UmmaScope &) = delete;
  UmmaScope &operator=(const UmmaScope &) = delete;
  unsigned *prev;
};
unsigned *umma_error_flag();             // the flag of the innermost scope
int umma_error_reset(cudaStream_t st);
int umma_error_check(cudaStream_t st);   // GFCC_ERR_TIMEOUT if a bounded wait gave up
int umma_timed_out();                    // records the message and returns GFCC_ERR_TIMEOUT

}  // namespace gfcc
