// FP64-accurate matrix products on the BF16 tensor cores by exact digit splitting
// (the splitting scheme of Ozaki, Ogita, Oishi & Rump, Numer. Algorithms 59 (2012), with
// fixed-point digits per row).
//
// GB300 runs FP64 at about 1.1 TFLOP/s, three orders of magnitude below its BF16 tensor
// rate.  A row r of an FP64 operand is scaled by a power of two 2^-e_r so that its entries
// lie in (-1/2, 1/2), then written as S base-64 digits
//     a = 2^e_r * sum_{i=1..S} d_i 64^-i + rem,   d_i integer, |d_i| <= 32, |rem| <= 2^e_r 64^-S / 2.
// Digits are exact in BF16 (8 significant bits).  A digit product is an integer of magnitude
// <= 2^10, so a sum of up to 2^14 of them is an integer of magnitude <= 2^24 and the FP32
// accumulation of the tensor cores is exact.  The product of two operands is then
//     sum_k A[m][k] B[n][k] = 2^(e_m + f_n) sum_{i,j} 64^-(i+j) sum_k dA_i[m][k] dB_j[n][k]
// and the digit-pair products with i + j <= P are evaluated on the tensor cores, all of a tile in one kernel
// (umma_bf16.cu) or as one BF16 GEMM each (K split into chunks of 2^14 with separate FP32 partial sums), and
// combined with one rounding.  The truncation error per term is bounded by about 2^-(6P-4) of 2^(e_m + f_n);
// P = S + 1.  Contractions that take the place of FP64 sums use 8 digits of 7 bits instead.
#include <cuda_bf16.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "ozaki.cuh"
#include "umma.cuh"

namespace gfcc {

// products with at most this many columns take the fused kernel (all digit pairs of a tile in one
// CTA, levels in TMEM); wider ones, and digit counts it does not hold, one GEMM per digit pair
long long g_fused_max_n = 1LL << 40;

namespace {

constexpr int KCHUNK_BLOCKS = (1 << 14) / 64;   // K blocks (of 64) per exact partial sum

// Exact integer accumulation of digit-pair products: the FP32 partial sums are integers of
// magnitude <= 2^24, so they convert to int32 exactly; a pair of level L adds (sum_z part) shifted
// by 6 (Lhi - L) into the high accumulator (levels <= Lsplit) or by 6 (P - L) into the low one.
// The two int64 accumulators are separate planes, acc[t] = high and acc[tot + t] = low, so that a
// combine touches only its own; the first combine into a plane sets it.  No FP64 arithmetic.
__global__ void combine_int_kernel(const float *part, int nz, long long tot, int shift, int which, long long *acc,
                                   int first) {
  long long *a = acc + (which ? tot : 0);
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot; t += (long long)gridDim.x * blockDim.x) {
    long long s = 0;
    for (int z = 0; z < nz; z++) s += (long long)__float2int_rn(part[(long long)z * tot + t]);
    s <<= shift;
    a[t] = first ? s : a[t] + s;
  }
}
// C = alpha * (high 2^(ex - 6 Lhi) + low 2^(ex - 6 P)) + beta C, ex = eA[m] + eB[n].  Grid
// (cdiv(N, 256), rows): a block walks rows m = blockIdx.y, blockIdx.y + gridDim.y, ...
__global__ void finalize_kernel(const long long *acc, long long M, long long N, const int *eA, const int *eB,
                                int Lhi, int P, double alpha, double beta, double *C, IMap cm, IMap cn, long long n0) {
  const long long tot = M * N;
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  const int eb = eB[n];
  const long long offn = imap_apply(cn, n0 + n);
  for (long long m = blockIdx.y; m < M; m += gridDim.y) {
    const long long t = m * N + n;
    const int ex = eA[m] + eb;
    double val = scalbn((double)acc[t], ex - 6 * Lhi);
    if (P > Lhi) val += scalbn((double)acc[tot + t], ex - 6 * P);
    const long long off = imap_apply(cm, m) + offn;
    const double v = alpha * val;
    C[off] = beta != 0.0 ? v + beta * C[off] : v;
  }
}

}  // namespace

long long emu_operand_bytes(long long rows, long long K, int S) {
  const long long ld = emu_ld(K);
  return (long long)S * rows * ld * 2 + ((rows * 4 + 255) / 256) * 256 + 256;
}

int emu_slice(cudaStream_t st, const double *A, long long rows, long long K, long long lda, int S, void *mem,
              EmuOperand &out, int bits) {
  return emu_slice_strided(st, A, rows, K, imap1(lda), imap1(1), 0, S, bits, mem, out);
}

// The digit pairs of one level L = i + j share a weight, so several of them can accumulate in the
// same FP32 partial sums (beta = 1) while the sums stay exact integers: a partial over kbs K blocks
// of 64 holds up to KCHUNK_BLOCKS / kbs pairs (2^14 digit products of magnitude <= 2^10).  The K
// split is the one of a single pair; pairs are grouped within that bound, one integer combine per
// group.
long long emu_gemm_work_bytes(long long M, long long N, long long K) {
  const long long nk = (K + 63) / 64;
  const long long nz = (nk + KCHUNK_BLOCKS - 1) / KCHUNK_BLOCKS;
  return std::max(nz * M * N * 4 + M * N * 16 + 512, emu_fused_work_bytes(M, N, K));
}

void emu_set_fused_max_n(long long n) { g_fused_max_n = n; }

namespace {
__global__ void max_int_kernel(const int *x, long long n, int *out) {
  int m = -(1 << 30);
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    m = max(m, x[t]);
  for (int off = 16; off > 0; off >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, off));
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}
}  // namespace

int emu_max_exponent(cudaStream_t st, const EmuOperand &e, int *out) {
  int *d = nullptr;
  const int init = -(1 << 30);
  GFCC_CUDA(cudaMalloc(&d, sizeof(int)));
  GFCC_CUDA(cudaMemcpyAsync(d, &init, sizeof(int), cudaMemcpyHostToDevice, st));
  max_int_kernel<<<grid1d(e.rows), 256, 0, st>>>(e.exp2, e.rows, d);
  cudaError_t er = cudaGetLastError();
  count_launch();
  if (er == cudaSuccess) er = cudaMemcpyAsync(out, d, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (er == cudaSuccess) er = cudaStreamSynchronize(st);
  cudaFree(d);
  if (er != cudaSuccess) {
    set_error("emu_max_exponent: %s", cudaGetErrorString(er));
    return GFCC_ERR_CUDA;
  }
  return GFCC_OK;
}

int emu_gemm(cudaStream_t st, const EmuOperand &A, const EmuOperand &B, int P, double alpha, double beta, double *C,
             IMap cm, IMap cn, void *work, long long n0, long long m0, const GuardList *gate) {
  P = std::max(2, P - A.drop);
  const long long M = A.rows, N = B.rows, K = A.K;
  if (M <= 0 || N <= 0) return GFCC_OK;
  if (B.K != K || A.ld != B.ld || A.bits != B.bits) {
    set_error("emu_gemm: operands disagree in K (%lld vs %lld) or digits (%d vs %d bits)", A.K, B.K, A.bits, B.bits);
    return GFCC_ERR_ARG;
  }
  if ((N <= g_fused_max_n || A.bits != 6) && emu_fused_takes(A.S, B.S, P) && M <= (1LL << 31) - 256 && N <= (1LL << 31) - 256)
    return emu_gemm_fused(st, A.dig, A.rows * A.ld, A.S, A.exp2, B.dig, B.rows * B.ld, B.S, B.exp2, A.ld, (int)M,
                          (int)N, (int)K, P, A.bits, alpha, beta, C, cm, cn, n0, static_cast<double *>(work), m0, gate);
  if (A.bits != 6 || m0 != 0 || gate != nullptr) {
    set_error("emu_gemm: %d-bit digits to level %d are beyond the digit-pair products", A.bits, P);
    return GFCC_ERR_ARG;
  }
  const long long nk = (K + 63) / 64;
  const int nz = (int)((nk + KCHUNK_BLOCKS - 1) / KCHUNK_BLOCKS);
  const long long kbs = (nk + nz - 1) / nz;
  const int group = (int)std::max<long long>(1, KCHUNK_BLOCKS / kbs);   // pairs per exact partial
  float *part = static_cast<float *>(work);
  long long *acc =
      reinterpret_cast<long long *>(static_cast<unsigned char *>(work) + ((nz * M * N * 4 + 255) / 256) * 256);
  GFCC_TRY(check_extent_bytes(work, emu_gemm_work_bytes(M, N, K), "digit GEMM workspace"));
  GFCC_TRY(check_extent(C, 0, imap_max(cm, M) + imap_max(cn, n0 + N), "digit GEMM output"));
  const long long plA = A.rows * A.ld, plB = B.rows * B.ld;
  // two exact int64 accumulators: levels 2..Lhi (weights 64^(Lhi-L)) and Lhi+1..P (64^(P-L));
  // a group sum is below nz 2^24 < 2^33 (and a level holds at most S groups), so 4 levels of 6-bit
  // shifts stay below 2^63
  const int Lhi = std::min(P, 5);
  if (P - Lhi > 4 || nz > (1 << 16)) {
    set_error("emu_gemm: level %d or K %lld beyond the exact integer accumulation", P, K);
    return GFCC_ERR_ARG;
  }
  bool first = true, first_plane[2] = {true, true};
  for (int L = P; L >= 2; L--) {
    const int which = L <= Lhi ? 0 : 1;
    const int shift = which == 0 ? 6 * (Lhi - L) : 6 * (P - L);
    int in_group = 0;
    for (int i = 1; i <= A.S; i++) {
      const int j = L - i;
      if (j < 1 || j > B.S) continue;
      GFCC_TRY(gemm_bf16_tn(st, A.dig + (long long)(i - 1) * plA, A.ld, B.dig + (long long)(j - 1) * plB, B.ld, part,
                            N, (int)M, (int)N, (int)K, 1.0f, in_group == 0 ? 0.0f : 1.0f, nz, M * N));
      in_group++;
      // last pair of the level or a full group: fold the partials into the integer accumulators
      bool last = true;
      for (int i2 = i + 1; i2 <= A.S; i2++)
        if (L - i2 >= 1 && L - i2 <= B.S) last = false;
      if (in_group == group || last) {
        combine_int_kernel<<<grid1d(M * N), 256, 0, st>>>(part, umma_splits((int)K, nz), M * N, shift, which, acc,
                                                           first_plane[which] ? 1 : 0);
        GFCC_LAUNCH_CHECK();
        first = false;
        first_plane[which] = false;
        in_group = 0;
      }
    }
  }
  if (first) GFCC_CUDA(cudaMemsetAsync(acc, 0, sizeof(long long) * 2 * M * N, st));
  finalize_kernel<<<dim3(cdiv(N, 256), (unsigned)std::min<long long>(M, 8192)), 256, 0, st>>>(
      acc, M, N, A.exp2, B.exp2, Lhi, P, alpha, beta, C, cm, cn, n0);
  GFCC_LAUNCH_CHECK();
  return GFCC_OK;
}

// ---------------------------------------------------------------- strided operands
namespace {

constexpr int SL_ROWS = 32, SL_K = 64, SL_THREADS = 256;

// Both passes read a SL_ROWS x SL_K tile with the lanes along whichever index of X is contiguous
// (k_lanes: the K index), so that a transposed operand is read in whole sectors too.
template <typename F>
__device__ __forceinline__ void for_tile(bool k_lanes, F f) {
  for (int e = threadIdx.x; e < SL_ROWS * SL_K; e += SL_THREADS)
    if (k_lanes)
      f(e / SL_K, e % SL_K);
    else
      f(e % SL_ROWS, e / SL_ROWS);
}

// be[r] = largest biased exponent among the entries of row r0 + r (be zeroed by the caller); a block
// covers SL_ROWS rows and `span` K values, a tile with eight loads of every thread in flight at a time (41 million
// entries 66 us; 168 us with a 64-bit division and one load in flight per entry)
__global__ __launch_bounds__(SL_THREADS) void strided_exp_kernel(const double *X, long long rows, long long K, IMap rm,
                                                                 IMap km, long long r0, bool k_lanes, int span,
                                                                 unsigned gx, int *be) {
  constexpr int PER = SL_ROWS * SL_K / SL_THREADS;
  __shared__ int mx[SL_ROWS];
  __shared__ long long ro[SL_ROWS], ko[2][SL_K];   // the K offsets of a tile are formed while the one before is read
  const unsigned bx = blockIdx.x % gx, by = blockIdx.x / gx;
  const long long rb = (long long)bx * SL_ROWS;
  if (threadIdx.x < SL_ROWS) {
    mx[threadIdx.x] = 0;
    ro[threadIdx.x] = rb + threadIdx.x < rows ? imap_apply(rm, r0 + rb + threadIdx.x) : -1;
  }
  const long long kbeg = (long long)by * span, kend = min(K, kbeg + span);
  auto offsets = [&](long long k0, long long *dst) {
    if (threadIdx.x >= 64 && threadIdx.x < 64 + SL_K) {
      const int k = threadIdx.x - 64;
      dst[k] = k0 + k < kend ? imap_apply(km, k0 + k) : -1;
    }
  };
  int m[PER];
#pragma unroll
  for (int u = 0; u < PER; u++) m[u] = 0;
  offsets(kbeg, ko[0]);
  __syncthreads();
  int cur = 0;
  for (long long k0 = kbeg; k0 < kend; k0 += SL_K, cur ^= 1) {
    double v[PER];
#pragma unroll
    for (int u = 0; u < PER; u++) {
      const int e = threadIdx.x + u * SL_THREADS;
      const int r = k_lanes ? e / SL_K : e % SL_ROWS, k = k_lanes ? e % SL_K : e / SL_ROWS;
      v[u] = ro[r] >= 0 && ko[cur][k] >= 0 ? X[ro[r] + ko[cur][k]] : 0.0;
    }
    if (k0 + SL_K < kend) offsets(k0 + SL_K, ko[cur ^ 1]);
#pragma unroll
    for (int u = 0; u < PER; u++) m[u] = max(m[u], (__double2hiint(v[u]) >> 20) & 0x7ff);
    __syncthreads();
  }
  if (k_lanes) {
    // the lanes of a warp share the row of each element
#pragma unroll
    for (int u = 0; u < PER; u++) {
      const int w = __reduce_max_sync(0xffffffffu, m[u]);
      if ((threadIdx.x & 31) == 0) atomicMax(&mx[(threadIdx.x + u * SL_THREADS) / SL_K], w);
    }
  } else {
#pragma unroll
    for (int u = 1; u < PER; u++) m[0] = max(m[0], m[u]);
    atomicMax(&mx[threadIdx.x % SL_ROWS], m[0]);
  }
  __syncthreads();
  if (threadIdx.x < SL_ROWS && ro[threadIdx.x] >= 0 && mx[threadIdx.x] > 0) atomicMax(&be[rb + threadIdx.x], mx[threadIdx.x]);
}

// biased exponent -> e with max_k |X[r][k]| 2^-e in [1/4, 1/2) (less == 1021) or [1/2, 1) (1022); rows of zeros 0
__global__ void strided_exp_final_kernel(int *be, long long rows, int less) {
  const long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (r < rows) be[r] = be[r] > 0 ? be[r] - less : 0;
}

// |x| 2^-e in BF16, rounded down (infinities and NaN kept); what is not zero counts as 2^-60 at least, so that a sum of
// products of magnitudes is zero only where every product is
__device__ __forceinline__ unsigned magnitude_bf16(double x, int e) {
  const int hi = __double2hiint(x) & 0x7fffffff, E = hi >> 20;
  if (hi == 0 && __double2loint(x) == 0) return 0u;
  if (E == 0x7ff) return (hi & 0xfffff) != 0 || __double2loint(x) != 0 ? 0x7fc0u : 0x7f80u;
  const int f = E - 1023 - e + 127;
  return E == 0 || f < 127 - 60 ? (unsigned)(127 - 60) << 7 : (unsigned)f << 7 | ((hi >> 13) & 0x7f);
}

// dig[i][r][k] = i-th digit of X[rm(r0 + r) + km(k)] 2^-e[r] (k < K), 0 for K <= k < ld; mag: plane S of dig holds the
// magnitudes
__global__ __launch_bounds__(SL_THREADS) void strided_slice_kernel(const double *X, long long rows, long long K, IMap rm,
                                                                   IMap km, long long r0, bool k_lanes, const int *e,
                                                                   int S, int bits, unsigned gx, __nv_bfloat16 *dig,
                                                                   long long ld, bool mag) {
  __shared__ double tile[SL_ROWS][SL_K + 1];
  __shared__ long long ro[SL_ROWS], ko[SL_K];
  __shared__ int ex[SL_ROWS];
  const long long rb = (long long)(blockIdx.x % gx) * SL_ROWS, k0 = (long long)(blockIdx.x / gx) * SL_K;
  if (threadIdx.x < SL_ROWS) {
    const bool in = rb + threadIdx.x < rows;
    ro[threadIdx.x] = in ? imap_apply(rm, r0 + rb + threadIdx.x) : -1;
    ex[threadIdx.x] = in ? e[rb + threadIdx.x] : 0;
  } else if (threadIdx.x >= 64 && threadIdx.x < 64 + SL_K) {
    const int k = threadIdx.x - 64;
    ko[k] = k0 + k < K ? imap_apply(km, k0 + k) : -1;
  }
  __syncthreads();
  for_tile(k_lanes, [&](int r, int k) { tile[r][k] = (ro[r] >= 0 && ko[k] >= 0) ? X[ro[r] + ko[k]] : 0.0; });
  __syncthreads();
  const long long plane = rows * ld;
  for (int t = threadIdx.x; t < SL_ROWS * SL_K / 2; t += SL_THREADS) {
    const int r = t / (SL_K / 2), k = 2 * (t % (SL_K / 2));
    if (ro[r] < 0 || k0 + k >= ld) continue;
    if (bits != F64_BITS) {   // digits rounded one after the other (the levels these products drop keep their sums)
      long long Y0 = fixed_point(tile[r][k], ex[r], bits * S), Y1 = fixed_point(tile[r][k + 1], ex[r], bits * S);
      __nv_bfloat162 *dst = reinterpret_cast<__nv_bfloat162 *>(dig + (rb + r) * ld + k0 + k);
      for (int i = 0; i < S; i++) {
        const int sh = bits * (S - 1 - i);
        const long long d0 = sh > 0 ? (Y0 + (1LL << (sh - 1))) >> sh : Y0;
        const long long d1 = sh > 0 ? (Y1 + (1LL << (sh - 1))) >> sh : Y1;
        Y0 -= d0 << sh;
        Y1 -= d1 << sh;
        dst[i * (plane / 2)] = __floats2bfloat162_rn((float)(int)d0, (float)(int)d1);
      }
      continue;
    }
    // Half a place added to every digit (and a whole one more to the first, which then is not negative) makes the
    // digits plain bit fields; each is exact in BF16
    const unsigned long long bias = ((1ULL << (bits * S)) - 1) / ((1ULL << bits) - 1) << (bits - 1);
    const unsigned long long lift = 1ULL << (bits * S);   // 2^bits in the first place
    const unsigned long long Y0 = (unsigned long long)fixed_point(tile[r][k], ex[r], bits * S) + bias + lift,
                             Y1 = (unsigned long long)fixed_point(tile[r][k + 1], ex[r], bits * S) + bias + lift;
    unsigned *dst = reinterpret_cast<unsigned *>(dig + (rb + r) * ld + k0 + k);
    const unsigned mask = (1u << bits) - 1;
    const float half = 8388608.0f + (float)(1 << (bits - 1));
    for (int i = 0, sh = bits * (S - 1); i < S; i++, sh -= bits, dst += plane / 2) {
      const unsigned mi = i == 0 ? 1023u : mask;
      const float off = i == 0 ? half + (float)(1 << bits) : half;
      const unsigned f0 = __float_as_uint(__uint_as_float(0x4b000000u | ((unsigned)(Y0 >> sh) & mi)) - off);
      const unsigned f1 = __float_as_uint(__uint_as_float(0x4b000000u | ((unsigned)(Y1 >> sh) & mi)) - off);
      *dst = __byte_perm(f0, f1, 0x7632);
    }
    if (mag) *dst = magnitude_bf16(tile[r][k], ex[r]) | magnitude_bf16(tile[r][k + 1], ex[r]) << 16;
  }
}

}  // namespace

int emu_slice_strided(cudaStream_t st, const double *X, long long rows, long long K, IMap rm, IMap km, long long r0,
                      int S, int bits, void *mem, EmuOperand &out, bool mag) {
  out.rows = rows;
  out.K = K;
  out.ld = emu_ld(K);
  out.S = S;
  out.bits = bits;
  unsigned char *p = static_cast<unsigned char *>(mem);
  out.dig = reinterpret_cast<__nv_bfloat16 *>(p);
  out.mag = mag ? out.dig + S * rows * out.ld : nullptr;
  p += ((long long)(S + (mag ? 1 : 0)) * rows * out.ld * 2 + 255) / 256 * 256;
  out.exp2 = reinterpret_cast<int *>(p);
  if (rows <= 0 || K <= 0) return GFCC_OK;
  if (mag && bits != F64_BITS) {
    set_error("emu_slice_strided: magnitudes go with %d-bit digits", F64_BITS);
    return GFCC_ERR_ARG;
  }
  GFCC_TRY(check_extent(X, 0, imap_max(rm, r0 + rows) + imap_max(km, K), "digit split input"));
  GFCC_TRY(check_extent_bytes(mem, emu_operand_bytes(rows, K, S + (mag ? 1 : 0)), "digit split output"));
  const bool k_lanes = km.s0 == 1 || rm.s0 != 1;
  const long long gx = (rows + SL_ROWS - 1) / SL_ROWS, gy = (out.ld + SL_K - 1) / SL_K;
  // K values per block of the exponent pass: enough blocks for the chip, one tile at least
  long long span = SL_K;
  while (gx * ((K + span - 1) / span) > 152 * 16 && span < (1 << 20)) span *= 2;
  const long long gz = (K + span - 1) / span;
  if (gx * gy > 0x7fffffffLL || gx * gz > 0x7fffffffLL) {
    set_error("emu_slice_strided: grid too large (rows %lld, K %lld)", rows, K);
    return GFCC_ERR_ARG;
  }
  GFCC_CUDA(cudaMemsetAsync(out.exp2, 0, sizeof(int) * rows, st));
  strided_exp_kernel<<<(unsigned)(gx * gz), SL_THREADS, 0, st>>>(X, rows, K, rm, km, r0, k_lanes, (int)span, (unsigned)gx,
                                                                 out.exp2);
  GFCC_LAUNCH_CHECK();
  strided_exp_final_kernel<<<cdiv(rows, 256), 256, 0, st>>>(out.exp2, rows, bits == F64_BITS && K <= F64_SHORT_K ? 1022 : 1021);
  GFCC_LAUNCH_CHECK();
  strided_slice_kernel<<<(unsigned)(gx * gy), SL_THREADS, 0, st>>>(X, rows, K, rm, km, r0, k_lanes, out.exp2, S, bits,
                                                                   (unsigned)gx, out.dig, out.ld, mag);
  GFCC_LAUNCH_CHECK();
  return GFCC_OK;
}

thread_local EmuArena *g_emu_arena = nullptr;

int EmuArena::get(size_t bytes, void **out) {
  if (cap < bytes) {
    release();
    if (dmalloc(&p, bytes) != cudaSuccess) {
      cudaGetLastError();
      p = nullptr;
      return GFCC_ERR_OOM;
    }
    cap = bytes;
  }
  *out = p;
  return GFCC_OK;
}

void EmuArena::release() {
  if (p) dfree(p);   // cudaFree waits for the work that uses it
  p = nullptr;
  cap = 0;
}

namespace {
constexpr long long EMU_BLOCK_BYTES = 4LL << 30;

// rows (or columns) of a block whose planes (magnitudes among them) stay within EMU_BLOCK_BYTES
long long block_rows(long long rows, long long K) {
  const long long per = emu_ld(K) * 2 * (F64_DIGITS + 1) + 8;
  return std::min(rows, std::max<long long>(256, EMU_BLOCK_BYTES / per / 128 * 128));
}

long long up256(long long x) { return (x + 255) / 256 * 256; }

// The error of a digit-plane output in units of its row and column scales is, with remainders of both signs, about
// sqrt(K) 2^-58 (seven digit pairs of level 10 and above dropped from each product, each below 2^-58; both entries
// rounded to 2^-57), and the FP64 sum's bound K 2^-53 times the sum of magnitudes: 2^-5 / sqrt(K) is where one standard
// deviation meets it, GUARD_THETA / sqrt(K) asks for six.
constexpr float GUARD_THETA = 0.2f;
float guard_theta(long long K) { return GUARD_THETA / std::sqrt((float)K); }
// Listed outputs are summed at about 0.4 of the rate of the contraction: beyond an eighth of them it takes over
unsigned guard_cap(long long M, long long N) {
  return (unsigned)std::min<long long>(1LL << 26, std::max<long long>(1024, M * N / 8));
}
long long guard_bytes(unsigned cap) { return 256 + up256(8LL * cap) + 8LL * cap; }
GuardList guard_list(void *mem, unsigned cap) {
  GuardList g;
  unsigned char *p = static_cast<unsigned char *>(mem);
  g.count = reinterpret_cast<unsigned *>(p);
  g.at = reinterpret_cast<int2 *>(p + 256);
  g.value = reinterpret_cast<double *>(p + 256 + up256(8LL * cap));
  g.cap = cap;
  return g;
}

// value[i] = alpha sum_k A(m, k) B(k, n) + beta C(m, n) of the listed outputs, WARPS warps each
template <int WARPS>
__global__ __launch_bounds__(256) void guard_values_kernel(Contract c, GuardList g) {
  constexpr int PER = 8 / WARPS;   // outputs a block
  __shared__ double part[8];
  const unsigned count = *g.count;
  if (count > g.cap) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, first = threadIdx.x % (32 * WARPS);
  for (unsigned i0 = blockIdx.x * PER; i0 < count; i0 += gridDim.x * PER) {
    const unsigned i = i0 + warp / WARPS;
    double s = 0.0;
    int2 at = make_int2(0, 0);
    if (i < count) {
      at = g.at[i];
      const double *a = c.A + imap_apply(c.am, at.x), *b = c.B + imap_apply(c.bn, at.y);
#pragma unroll 4
      for (long long k = first; k < c.K; k += 32 * WARPS) s = fma(a[imap_apply(c.ak, k)], b[imap_apply(c.bk, k)], s);
    }
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (WARPS > 1) {
      if (lane == 0) part[warp] = s;
      __syncthreads();
      s = 0.0;
      for (int w = 0; w < WARPS; w++) s += part[warp / WARPS * WARPS + w];
      __syncthreads();
    }
    if (first == 0 && i < count) {
      s *= c.alpha;
      if (c.beta != 0.0) s += c.beta * c.C[imap_apply(c.cm, at.x) + imap_apply(c.cn, at.y)];
      g.value[i] = s;
    }
  }
}
// A guarded product in the order its kernels need: the list of all blocks, the listed values (from C as it was), the
// planes' product or the FP64 contraction, the listed values stored.
template <typename List, typename Product>
int guarded_product(cudaStream_t st, const Contract &p, const GuardList &g, List list, Product product) {
  GFCC_CUDA(cudaMemsetAsync(g.count, 0, sizeof(unsigned), st));
  GFCC_TRY(list());
  if (p.K >= 4096)
    guard_values_kernel<8><<<152 * 8, 256, 0, st>>>(p, g);
  else
    guard_values_kernel<1><<<152 * 8, 256, 0, st>>>(p, g);
  GFCC_LAUNCH_CHECK();
  GFCC_TRY(product());
  return contract_listed(p, g, st);
}
}  // namespace

// FP64 units: 1.1 TFLOP/s on 16 x 16 tiles.  Digit planes: 36 pairs of BF16 products and one of magnitudes at about 1.1e15
// flop/s on padded tiles, 4 ps an output for the ends of the tiles, the split of both operands (two reads of 8 bytes,
// nine planes of 2 bytes, at about 3 TB/s), and some 12 launches.  Error against quad sums (1e-16 relative): Gaussian
// entries, FP64 units 1.9, 2.1, 2.4, 3.0, 5.7, 14 at K = 32, 64, 160, 300, 1280, 6400; planes 0.6, 0.7, 0.7, 0.7, 2.4,
// 4.0; entries that decay along K as the Cholesky vectors do, 2.5, 2.6, 3.3, 3.9, 6.6, 7.0 and 0.7, 0.8, 1.1, 1.1, 3.5,
// 3.5.  What the guard costs: CCSD and Lambda at o=16 v=80 103 -> 114 ms, closed-shell solve at o=30 v=150 63 -> 69 ms,
// IP + EA set-up and solve at o=20 v=100 39 -> 41 ms.
bool emulation_pays(long long M, long long N, long long K, bool a_ready) {
  if (K < 32) return false;
  const double m16 = (double)((M + 15) / 16 * 16), n16 = (double)((N + 15) / 16 * 16);
  const double f64 = 2.0 * m16 * n16 * (double)K / 1.1e12;
  const double m128 = (double)((M + 127) / 128 * 128), n32 = (double)((N + 31) / 32 * 32);
  const double n128 = (double)((N + 127) / 128 * 128), m32 = (double)((M + 31) / 32 * 32);
  const double tile = std::min(m128 * n32, n128 * m32);
  const double emu = 37.0 * 2.0 * tile * (double)((K + 63) / 64 * 64) / 1.1e15 + 4e-12 * tile +
                     34.0 * ((a_ready ? 0.0 : (double)M) + (double)N) * (double)K / 3e12 + (a_ready ? 4e-5 : 5e-5);
  return emu < f64;
}

int gemm_f64_emulated_pre(cudaStream_t st, const EmuOperand &Ae, const double *A, IMap am, IMap ak, long long N,
                          const double *B, IMap bk, IMap bn, double alpha, double beta, double *C, IMap cm, IMap cn,
                          bool guarded) {
  const long long M = Ae.rows, K = Ae.K;
  if (M <= 0 || N <= 0) return GFCC_OK;
  GFCC_TRY(check_extent(B, 0, imap_max(bk, K) + imap_max(bn, N), "emulated contraction operand B"));
  GFCC_TRY(check_extent(C, 0, imap_max(cm, M) + imap_max(cn, N), "emulated contraction output C"));
  if (guarded && Ae.mag == nullptr) {
    set_error("emulated contraction: the sliced operand has no magnitudes");
    return GFCC_ERR_ARG;
  }
  const long long nb = block_rows(N, K);
  const unsigned cap = guarded ? guard_cap(M, N) : 0;
  const long long bbytes = up256(emu_operand_bytes(nb, K, F64_DIGITS + 1)), gbytes = guarded ? up256(guard_bytes(cap)) : 0;
  const long long wbytes = std::max(emu_fused_work_bytes(M, nb, K), guarded ? emu_guard_work_bytes(M, nb, K) : 0);
  EmuArena local;
  EmuArena *ar = g_emu_arena ? g_emu_arena : &local;
  void *mem = nullptr;
  if (ar->get((size_t)(bbytes + gbytes + wbytes), &mem) < 0) {
    set_error("emulated contraction: cannot allocate its temporaries (M=%lld N-block=%lld K=%lld)", M, nb, K);
    return GFCC_ERR_OOM;
  }
  void *gm = static_cast<unsigned char *>(mem) + bbytes, *gw = static_cast<unsigned char *>(gm) + gbytes;
  EmuOperand eb;
  long long sliced = -1;   // the first column of the block that eb holds
  auto slice = [&](long long n0) -> int {
    if (sliced == n0) return GFCC_OK;
    sliced = n0;
    return emu_slice_strided(st, B, std::min(nb, N - n0), K, bn, bk, n0, F64_DIGITS, F64_BITS, mem, eb, guarded);
  };
  const GuardList g = guarded ? guard_list(gm, cap) : GuardList();
  auto list = [&]() -> int {
    for (long long n0 = 0; n0 < N; n0 += nb) {
      GFCC_TRY(slice(n0));
      GFCC_TRY(emu_guard(st, Ae.mag, eb.mag, Ae.ld, (int)M, (int)eb.rows, (int)K, guard_theta(K), g, 0, n0,
                         static_cast<float *>(gw)));
    }
    return GFCC_OK;
  };
  auto product = [&]() -> int {
    for (long long n0 = 0; n0 < N; n0 += nb) {
      GFCC_TRY(slice(n0));
      GFCC_TRY(emu_gemm(st, Ae, eb, F64_LEVEL, alpha, beta, C, cm, cn, gw, n0, 0, guarded ? &g : nullptr));
    }
    return GFCC_OK;
  };
  if (!guarded) return product();
  Contract c;
  c.A = A; c.B = B; c.C = C;
  c.M = M; c.N = N; c.K = K;
  c.am = am; c.ak = ak; c.bk = bk; c.bn = bn; c.cm = cm; c.cn = cn;
  c.alpha = alpha; c.beta = beta;
  return guarded_product(st, c, g, list, product);
}

int gemm_f64_emulated(cudaStream_t st, long long M, long long N, long long K, double alpha, const double *A, IMap am,
                      IMap ak, const double *B, IMap bk, IMap bn, double beta, double *C, IMap cm, IMap cn,
                      bool guarded) {
  if (M <= 0 || N <= 0) return GFCC_OK;
  GFCC_TRY(check_extent(A, 0, imap_max(am, M) + imap_max(ak, K), "emulated contraction operand A"));
  GFCC_TRY(check_extent(B, 0, imap_max(bk, K) + imap_max(bn, N), "emulated contraction operand B"));
  GFCC_TRY(check_extent(C, 0, imap_max(cm, M) + imap_max(cn, N), "emulated contraction output C"));
  const long long mb = block_rows(M, K), nb = block_rows(N, K);
  const int planes = F64_DIGITS + (guarded ? 1 : 0);
  const unsigned cap = guarded ? guard_cap(M, N) : 0;
  const long long abytes = up256(emu_operand_bytes(mb, K, planes)), bbytes = up256(emu_operand_bytes(nb, K, planes));
  const long long gbytes = guarded ? up256(guard_bytes(cap)) : 0;
  const long long wbytes = std::max(emu_fused_work_bytes(mb, nb, K), guarded ? emu_guard_work_bytes(mb, nb, K) : 0);
  EmuArena local;
  EmuArena *ar = g_emu_arena ? g_emu_arena : &local;
  void *mem = nullptr;
  GFCC_TRY(ar->get((size_t)(abytes + bbytes + gbytes + wbytes), &mem));
  unsigned char *bm = static_cast<unsigned char *>(mem) + abytes, *gm = bm + bbytes;
  void *gw = gm + gbytes;
  EmuOperand ea, eb;
  long long am0 = -1, bn0 = -1;   // first row and column of the blocks that ea and eb hold
  auto slice = [&](long long m0, long long n0) -> int {
    if (am0 != m0)
      GFCC_TRY(emu_slice_strided(st, A, std::min(mb, M - m0), K, am, ak, m0, F64_DIGITS, F64_BITS, mem, ea, guarded));
    am0 = m0;
    if (bn0 != n0)
      GFCC_TRY(emu_slice_strided(st, B, std::min(nb, N - n0), K, bn, bk, n0, F64_DIGITS, F64_BITS, bm, eb, guarded));
    bn0 = n0;
    return GFCC_OK;
  };
  const GuardList g = guarded ? guard_list(gm, cap) : GuardList();
  auto list = [&]() -> int {
    for (long long m0 = 0; m0 < M; m0 += mb)
      for (long long n0 = 0; n0 < N; n0 += nb) {
        GFCC_TRY(slice(m0, n0));
        GFCC_TRY(emu_guard(st, ea.mag, eb.mag, ea.ld, (int)ea.rows, (int)eb.rows, (int)K, guard_theta(K), g, m0, n0,
                           static_cast<float *>(gw)));
      }
    return GFCC_OK;
  };
  auto product = [&]() -> int {
    for (long long m0 = 0; m0 < M; m0 += mb)
      for (long long n0 = 0; n0 < N; n0 += nb) {
        GFCC_TRY(slice(m0, n0));
        GFCC_TRY(emu_gemm(st, ea, eb, F64_LEVEL, alpha, beta, C, cm, cn, gw, n0, m0, guarded ? &g : nullptr));
      }
    return GFCC_OK;
  };
  if (!guarded) return product();
  Contract c;
  c.A = A; c.B = B; c.C = C;
  c.M = M; c.N = N; c.K = K;
  c.am = am; c.ak = ak; c.bk = bk; c.bn = bn; c.cm = cm; c.cn = cn;
  c.alpha = alpha; c.beta = beta;
  return guarded_product(st, c, g, list, product);
}

}  // namespace gfcc
