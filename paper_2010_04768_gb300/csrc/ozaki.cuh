// FP64-accurate products from BF16 digit planes on the tensor cores (ozaki.cu).
#pragma once
#include <cuda_bf16.h>

#include <cmath>

#include "common.cuh"
#include "umma.cuh"

namespace gfcc {

// Row stride of digit planes: whole 128-byte lines where a row has one (a K block of 64 digits that straddles two
// lines is fetched as both)
static inline long long emu_ld(long long K) { return K >= 64 ? (K + 63) / 64 * 64 : (K + 7) / 8 * 8; }


// An FP64 matrix (rows x K, K-major) split into S planes of balanced `bits`-bit digits (6: base 64) with
// a power-of-two scale per row: A[r][k] ~= 2^exp2[r] sum_i dig[i][r][k] 2^(-bits (i+1)).
struct EmuOperand {
  __nv_bfloat16 *dig = nullptr;   // [S][rows][ld]
  int *exp2 = nullptr;            // [rows]
  long long rows = 0, K = 0, ld = 0;
  int S = 0;
  int bits = 6;
  const __nv_bfloat16 *mag = nullptr;   // [rows][ld] magnitudes 2^-exp2[r] |A[r][k]| (guarded products), or nullptr
  // levels this operand's products may drop (as the A operand of emu_gemm) while keeping the error
  // bound of the level-P product of the operator with its Fock-like diagonal (set at setup: see
  // emu_level_drop)
  int drop = 0;
};
// Largest row scale exponent of an operand (max over rows of exp2[r]); host value, synchronises st.
int emu_max_exponent(cudaStream_t st, const EmuOperand &e, int *out);
// Levels an operand may drop: every product term of the operand is bounded by 2^-(6P-4) times its
// row scale (at most 2^e_max), while the bound of the level-P product of the ring operator with the
// diagonal folded in is at least 2^-(6P-4) times the smallest diagonal entry of its rows; one level
// (6 bits) may go when 2^(e_max + 6) <= min_diag.  At most one level is dropped.
static inline int emu_level_drop(int e_max, double min_diag) {
  return (min_diag > 0.0 && std::ldexp(1.0, e_max + 6) <= min_diag) ? 1 : 0;
}

long long emu_operand_bytes(long long rows, long long K, int S);
int emu_slice(cudaStream_t st, const double *A, long long rows, long long K, long long lda, int S, void *mem,
              EmuOperand &out, int bits = 6);
long long emu_gemm_work_bytes(long long M, long long N, long long K);
void emu_set_fused_max_n(long long n);   // widest product (columns) for the fused digit kernel
// C(m, n) = alpha * sum_k A[m][k] B[n][k] + beta * C(m, n) with digit pairs i + j <= P
// (the output row index of A's row m is m0 + m, the column index of B's row n is n0 + n)
int emu_gemm(cudaStream_t st, const EmuOperand &A, const EmuOperand &B, int P, double alpha, double beta, double *C,
             IMap cm, IMap cn, void *work, long long n0 = 0, long long m0 = 0, const GuardList *gate = nullptr);
// Digits of the contractions that take the place of FP64 ones: 8 digits of 7 bits hold 56 bits below the
// row scale (an FP64 sum keeps 53 below each of its partial sums), pairs to level 9.
constexpr int F64_DIGITS = 8, F64_BITS = 7, F64_LEVEL = 9;
// Sums of at most this many terms scale their rows to [1/2, 1) instead of [1/4, 1/2): one bit more, at the price of
// a first digit of up to 128, which leaves the levels exact for 6 K blocks of 64 (8 otherwise).
constexpr int F64_SHORT_K = 6 * 64;

// Split rows r0 .. r0 + rows - 1 of a strided matrix, X[rm(r) + km(k)], into digit planes and, with mag (F64_BITS
// digits only), a plane of magnitudes behind them.  `mem` holds emu_operand_bytes(rows, K, S), S + 1 planes with mag.
int emu_slice_strided(cudaStream_t st, const double *X, long long rows, long long K, IMap rm, IMap km, long long r0,
                      int S, int bits, void *mem, EmuOperand &out, bool mag = false);

// Workspace of the emulated contractions below: kept by its owner between calls, grown on demand.
struct EmuArena {
  void *p = nullptr;
  size_t cap = 0;
  int get(size_t bytes, void **out);   // GFCC_ERR_OOM (with no message kept) when it cannot grow
  void release();
  ~EmuArena() { release(); }
};
// the calling thread's arena (nullptr: a call allocates and frees its own)
extern thread_local EmuArena *g_emu_arena;

// A strided FP64 contraction (the index maps of gemm_f64) evaluated from digit planes (F64_DIGITS of
// F64_BITS): operands are gathered K-major and split, multiplied pairwise and combined with one rounding.
// Blocks of rows and columns keep the planes within EMU_BLOCK_BYTES each.  GFCC_ERR_OOM: nothing written.
//
// The digits hold 56 bits below the largest entry of a row, so an entry 2^-k below it keeps 56 - k where FP64 keeps 53,
// and an output far below the largest entries of its row and column may be less accurate than an FP64 sum (of Gaussian
// or evenly decaying entries it is more accurate).  `guarded`: outputs whose sum of magnitudes does not clear that error
// are summed in FP64 instead, or all of them if they are many; so are outputs with infinities or NaN.
int gemm_f64_emulated(cudaStream_t st, long long M, long long N, long long K, double alpha, const double *A, IMap am,
                      IMap ak, const double *B, IMap bk, IMap bn, double beta, double *C, IMap cm, IMap cn,
                      bool guarded);
// whether the (guarded) digit planes are faster than the FP64 units (time models of both; a_ready: A is split already)
bool emulation_pays(long long M, long long N, long long K, bool a_ready);

// The same with A already split into digit planes (rows x K, K-major, F64_DIGITS of F64_BITS, with magnitudes
// if guarded): only B (given through its index maps, N columns) is gathered and split per call; A, am, ak are the entries
// themselves, for the FP64 sums.
int gemm_f64_emulated_pre(cudaStream_t st, const EmuOperand &Ae, const double *A, IMap am, IMap ak, long long N,
                          const double *B, IMap bk, IMap bn, double alpha, double beta, double *C, IMap cm, IMap cn,
                          bool guarded);

}  // namespace gfcc
