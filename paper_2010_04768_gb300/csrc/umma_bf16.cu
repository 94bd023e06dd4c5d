// BF16 x BF16 -> FP32 GEMM on the 5th-generation tensor cores (tcgen05, sm_103a).
//
//   D[m][n] = alpha * sum_k A[m][k] B[n][k] (+ beta * D[m][n])     (both operands K-major)
//
// This is the contraction engine of the mixed-precision sigma product: the ring
// matrix Wbar_ovvo (and the other Hbar blocks) are stored once in BF16, the Krylov
// vectors are rounded to BF16 when they are unpacked, products accumulate in FP32
// in tensor memory (TMEM).
//
// Structure (one 128 x 64, 128 x 128 or 128 x 256 output tile per CTA, 4 warps; here the last):
//   * warp 0, one lane: TMA producer.  A tile 128 x 64 and B tile 256 x 64 (BF16,
//     128-byte swizzle) per stage into a 4-stage shared-memory ring, completion
//     tracked by mbarrier transaction counts.
//   * warp 1: MMA issuer (the whole warp, one elected lane, so that descriptors stay in uniform registers).  Four
//     tcgen05.mma (M=128, N=256, K=16) per stage, accumulating in 256 TMEM columns; tcgen05.commit releases the stage.
//   * all 4 warps: epilogue.  tcgen05.ld of the warp's 32 TMEM lanes, scale, store along rows through shared memory.
// Every wait is bounded (about one second of %globaltimer); on time-out the CTA sets
// the error flag, stops issuing work, drains what it issued and frees its TMEM.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <tuple>
#include <utility>

#include "common.cuh"
#include "ozaki.cuh"
#include "umma.cuh"

namespace gfcc {

namespace {

constexpr int BM = 128, BK = 64, THREADS = 128;
constexpr int RASTER_GM = 16;   // row tiles per rasterisation group
// BN (the N extent of a tile and of the TMEM accumulator) is a template parameter: 256 for wide
// operands, 128 / 64 when the contraction has few columns (a tile wider than N wastes MMA work).
// ST: pipeline stages (0: the default for BN).  Contractions with only a K block or two per CTA use
// 2 stages, so that several CTAs fit an SM and the per-CTA set-up overlaps.
template <int BN, int ST = 0>
struct Tile {
  static constexpr int STAGES = ST > 0 ? ST : (BN == 256 ? 4 : 6);
  static constexpr int A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2, STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /* alignment */ + 256 /* barriers */;
};
// Bounded waits.  The limit of the pipeline waits is a launch parameter (default 1 s, settable
// process-wide so that a test can make a wait run out); the waits of the abort path, for work
// this CTA has already issued, always keep the fixed DRAIN_NS.
constexpr unsigned long long DRAIN_NS = 1000000000ULL;
// Launch-time control of the pipeline: wait limit, and (test only) a producer that issues no
// loads, so that the consumer's wait runs out with no asynchronous copy outstanding.
struct UmmaCtl {
  unsigned long long wait_ns;
  int skip_loads;
  unsigned *error;   // set by a wait that ran out (the flag of the call that launched the kernel)
};
unsigned long long g_wait_ns = 1000000000ULL;
bool g_skip_loads = false;
thread_local unsigned *t_error_flag = nullptr;

// The control block of a launch by the calling thread; a launch outside every UmmaScope is refused (its time-outs
// would go unreported).
int umma_ctl(UmmaCtl *ctl) {
  if (t_error_flag == nullptr) {
    set_error("internal: tensor-core product outside a call's error scope");
    return GFCC_ERR_STATE;
  }
  *ctl = UmmaCtl{g_wait_ns, g_skip_loads ? 1 : 0, t_error_flag};
  return GFCC_OK;
}

__device__ __forceinline__ unsigned smem_u32(const void *p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(unsigned addr, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(addr), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(unsigned addr, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(addr), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(unsigned addr, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(addr), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait (limit_ns of %globaltimer) for the phase of the given parity; false on time-out or
// abort.  Once a kernel of the call has timed out, the waits of the others give up after GIVE_UP_NS, so that a call
// whose waits run out ends after about one limit and not after one per product.
constexpr long long GIVE_UP_NS = 50000;
__device__ __forceinline__ bool mbar_wait(unsigned addr, unsigned parity, volatile int *abort_flag,
                                          unsigned long long limit_ns, unsigned *error) {
  if (mbar_try_wait(addr, parity)) return true;
  const unsigned long long t0 = globaltimer();
  while (true) {
    if (mbar_try_wait(addr, parity)) return true;
    if (*abort_flag) return false;
    const long long dt = (long long)(globaltimer() - t0);
    if (dt > (long long)limit_ns) {
      *abort_flag = 1;
      atomicOr(error, 1u);
      return false;
    }
    if (dt > GIVE_UP_NS && *reinterpret_cast<volatile unsigned *>(error) != 0) {
      *abort_flag = 1;
      return false;
    }
  }
}

// The waits of the abort path: for work this CTA has issued, always up to DRAIN_NS.
__device__ __forceinline__ void drain_wait(unsigned addr, unsigned parity, unsigned *error) {
  const unsigned long long t0 = globaltimer();
  while (!mbar_try_wait(addr, parity))
    if ((long long)(globaltimer() - t0) > (long long)DRAIN_NS) {
      atomicOr(error, 1u);
      return;
    }
}

__device__ __forceinline__ void tma_load_2d(unsigned dst, const CUtensorMap *map, unsigned mbar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(
          dst),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(mbar), "r"(x), "r"(y)
      : "memory");
}

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 bytes apart.
__device__ __forceinline__ unsigned long long smem_desc(unsigned addr) {
  unsigned long long d = 0;
  d |= (unsigned long long)((addr & 0x3FFFF) >> 4);       // start address
  d |= (unsigned long long)(16 >> 4) << 16;               // leading byte offset (unused for swizzled K-major)
  d |= (unsigned long long)(1024 >> 4) << 32;             // stride byte offset
  d |= 1ULL << 46;                                        // descriptor version
  d |= 2ULL << 61;                                        // 128-byte swizzle
  return d;
}

// Instruction descriptor of kind::f16: BF16 A and B, FP32 accumulator, K-major A and B, M x N.
__host__ __device__ constexpr unsigned idesc_bf16(int M, int N) {
  return (1u << 4)                      // D format: F32
         | (1u << 7)                    // A format: BF16
         | (1u << 10)                   // B format: BF16
         | ((unsigned)(N >> 3) << 17)   // N / 8
         | ((unsigned)(M >> 4) << 24);  // M / 16
}

__device__ __forceinline__ void umma_bf16(unsigned d_tmem, unsigned long long a, unsigned long long b, unsigned idesc,
                                          unsigned accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.u32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}

// One lane of a converged warp.  The MMA loops run in a whole warp and issue from the elected lane, so that
// descriptors and barrier addresses stay in uniform registers.
__device__ __forceinline__ bool elect_one() {
  unsigned p;
  asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(p));
  return p != 0;
}

__device__ __forceinline__ void umma_commit(unsigned mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ void tmem_ld_32(unsigned taddr, float (&v)[32]) {
  unsigned r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; i++) v[i] = __uint_as_float(r[i]);
}

// A warp's 32 x 32 block of an accumulator (v: its row `lane`) to D[row0 ..][col0 ..] through shared memory (buf: 32
// rows of STORE_LD floats of this warp), so that stores run along rows: eight lanes a row of four columns each, or a
// lane a column where D does not align.  Rows straight from the registers are 32 separate 16-byte pieces a store:
// 96957 x 60 outputs took 24 us whatever K.
constexpr int STORE_LD = 36, STORE_BYTES = 32 * STORE_LD * 4;
__device__ __forceinline__ void store_block(float *buf, const float (&v)[32], float alpha, float beta, float *D,
                                            long long ldd, int row0, int M, int col0, int N) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < 32; i += 4)
    *reinterpret_cast<float4 *>(buf + lane * STORE_LD + i) =
        make_float4(alpha * v[i], alpha * v[i + 1], alpha * v[i + 2], alpha * v[i + 3]);
  __syncwarp();
  const int ncols = min(32, N - col0), rows = min(32, M - row0);
  float *base = D + (long long)row0 * ldd + col0;
  if (((ldd | ncols) & 3) == 0 && (reinterpret_cast<uintptr_t>(base) & 15) == 0) {
    const int r0 = lane >> 3, c = (lane & 7) * 4;
    if (c < ncols) {
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const int r = r0 + 4 * i;
        if (r >= rows) break;
        float4 x = *reinterpret_cast<const float4 *>(buf + r * STORE_LD + c);
        float4 *dst = reinterpret_cast<float4 *>(base + r * ldd + c);
        if (beta != 0.0f) {
          const float4 d = *dst;
          x = make_float4(x.x + beta * d.x, x.y + beta * d.y, x.z + beta * d.z, x.w + beta * d.w);
        }
        *dst = x;
      }
    }
  } else if (lane < ncols) {
#pragma unroll 8
    for (int r = 0; r < rows; r++) {
      const float x = buf[r * STORE_LD + lane];
      float *dst = base + r * ldd + lane;
      *dst = beta != 0.0f ? x + beta * *dst : x;
    }
  }
  __syncwarp();
}

// GUARD: the outputs are not stored; those beside [theta, infinity) and not zero are listed (emu_guard)
struct GuardArgs {
  GuardList list;
  float theta = 0.0f;
  int m0 = 0, n0 = 0;
};

// mask: which of the 32 entries (row, col ..) go on the list
__device__ __forceinline__ void guard_append(const GuardArgs &g, unsigned mask, int row, int col) {
  const unsigned n = __popc(mask);
  if (n == 0 || *reinterpret_cast<volatile unsigned *>(g.list.count) > g.list.cap) return;
  unsigned i = atomicAdd(g.list.count, n);
  for (; mask != 0; mask &= mask - 1, i++)
    if (i < g.list.cap) g.list.at[i] = make_int2(g.m0 + row, g.n0 + col + __ffs(mask) - 1);
}

__device__ __forceinline__ bool guard_hit(float v, float theta) { return v != 0.0f && !(v >= theta && v < 1e30f); }

template <int BN, int ST, bool GUARD = false>
__global__ void __launch_bounds__(THREADS, 1)
    umma_bf16_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, float *D,
                          long long ldd, int M, int N, int K, float alpha, float beta, int kb_per_split,
                          long long split_stride, UmmaCtl ctl, GuardArgs guard) {
  chain_start();
  constexpr int STAGES = Tile<BN, ST>::STAGES, A_BYTES = Tile<BN, ST>::A_BYTES,
                STAGE_BYTES = Tile<BN, ST>::STAGE_BYTES;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned long long *bars = reinterpret_cast<unsigned long long *>(smem + STAGES * STAGE_BYTES);
  unsigned long long *full = bars, *empty = bars + STAGES, *done = bars + 2 * STAGES;
  unsigned *tmem_slot = reinterpret_cast<unsigned *>(bars + 2 * STAGES + 1);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  volatile int *issued = reinterpret_cast<volatile int *>(tmem_slot + 2);     // TMA stages issued
  volatile int *consumed = reinterpret_cast<volatile int *>(tmem_slot + 3);   // stages the MMA warp waited for

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // tile order: groups of RASTER_GM row tiles sweep all column tiles, row tile fastest, so the CTAs
  // in flight share a few A row panels and B column panels (L2 reuse on long-K products)
  int m_tile, n_tile;
  {
    const int nM = gridDim.x, nN = gridDim.y;
    const int id = blockIdx.y * nM + blockIdx.x;
    const int first_m = (id / (RASTER_GM * nN)) * RASTER_GM;
    const int gm = min(nM - first_m, RASTER_GM);
    const int r = id - first_m * nN;
    m_tile = first_m + r % gm;
    n_tile = r / gm;
  }
  const int m0 = m_tile * BM, n0 = n_tile * BN;
  // split-K: this CTA covers K blocks [kb0, kb1) and writes its partial sum to D + z * split_stride
  const int nk_all = (K + BK - 1) / BK;
  const int kb0 = blockIdx.z * kb_per_split;
  const int kb1 = min(nk_all, kb0 + kb_per_split);
  const int nk = kb1 - kb0;
  D += (long long)blockIdx.z * split_stride;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; s++) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    mbar_init(smem_u32(done), 1);
    *abort_flag = 0;
    *issued = 0;
    *consumed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {   // TMEM: BN FP32 columns x 128 lanes for the accumulator
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(BN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer
    for (int kb = 0; kb < nk && !ctl.skip_loads; kb++) {
      const int s = kb % STAGES;
      const unsigned ph = (kb / STAGES) & 1;
      if (!mbar_wait(smem_u32(&empty[s]), ph ^ 1, abort_flag, ctl.wait_ns, ctl.error)) break;
      unsigned char *sa = smem + s * STAGE_BYTES;
      unsigned char *sb = sa + A_BYTES;
      mbar_expect_tx(smem_u32(&full[s]), STAGE_BYTES);
      tma_load_2d(smem_u32(sa), &tmA, smem_u32(&full[s]), (kb0 + kb) * BK, m0);
      tma_load_2d(smem_u32(sb), &tmB, smem_u32(&full[s]), (kb0 + kb) * BK, n0);
      *issued = kb + 1;
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer
    const unsigned idesc = idesc_bf16(BM, BN);
    const unsigned long long d0 = smem_desc(smem_u32(smem));
    for (int kb = 0; kb < nk; kb++) {
      const int s = kb % STAGES;
      const unsigned ph = (kb / STAGES) & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&full[s]), ph, abort_flag, ctl.wait_ns, ctl.error))) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const unsigned long long da = d0 + s * (STAGE_BYTES >> 4), db = da + (A_BYTES >> 4);
      if (elect_one()) {
        *consumed = kb + 1;
#pragma unroll
        for (int k = 0; k < BK / 16; k++) {
          // advance 16 BF16 (32 bytes) along K inside the 128-byte swizzle atom
          umma_bf16(tmem, da + 2 * k, db + 2 * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
        }
        umma_commit(smem_u32(&empty[s]));
      }
      __syncwarp();
    }
    if (elect_one()) umma_commit(smem_u32(done));   // arrives when every MMA issued above has completed
  }
  __syncwarp();

  // ---------------- epilogue: all 4 warps
  const bool ready = mbar_wait(smem_u32(done), 0, abort_flag, ctl.wait_ns, ctl.error);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  // tcgen05.ld is warp-collective: take the decision per warp
  if (__all_sync(0xffffffffu, ready && !*abort_flag)) {
    // every load has landed and every MMA has completed: the stages hold the blocks on their way out
    float *buf = reinterpret_cast<float *>(smem + warp * STORE_BYTES);
    const int row0 = m0 + warp * 32;
#pragma unroll 1
    for (int c0 = 0; c0 < BN && n0 + c0 < N && row0 < M; c0 += 32) {
      float v[32];
      tmem_ld_32(tmem + ((unsigned)(warp * 32) << 16) + c0, v);
      if constexpr (GUARD) {
        unsigned mask = 0;
#pragma unroll
        for (int i = 0; i < 32; i++)
          if (row0 + lane < M && n0 + c0 + i < N && guard_hit(v[i], guard.theta)) mask |= 1u << i;
        guard_append(guard, mask, row0 + lane, n0 + c0);
        __syncwarp();
      } else {
        store_block(buf, v, alpha, beta, D, ldd, row0, M, n0 + c0, N);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) {
    // after a time-out: the MMA warp always commits `done` once its issued products have completed
    // (wait for it, so that no tcgen05.mma still reads shared memory or writes TMEM when the TMEM is
    // freed), then let the TMA copies this CTA issued land before its shared memory goes away.
    // These waits keep the fixed DRAIN_NS limit; if one of them runs out as well, the CTA exits with
    // that work in flight (the error flag is already set).
    drain_wait(smem_u32(done), 0, ctl.error);
    for (int kb = *consumed; kb < *issued; kb++)
      drain_wait(smem_u32(&full[kb % STAGES]), (kb / STAGES) & 1, ctl.error);
  }
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(BN));
  }
}

// ---------------------------------------------------------------------------------------------
// The same product with a persistent tile loop: one CTA per SM walks the output tiles (and K splits)
// of the launch; six warps: warp 0 the TMA producer, warp 1 the MMA issuer, warps 2-5 the epilogue
// (warp w reads TMEM lanes 32 (w mod 4) .. + 31).  Two accumulators of BN columns in TMEM (ping-pong):
// the epilogue of a tile overlaps the main loop of the next, and the load pipeline runs on across
// tiles, so products with few K blocks per tile (the long thin contractions of the sigma product)
// no longer pay a pipeline fill, a TMEM allocation and an unoverlapped epilogue per tile.
constexpr int PERSIST_THREADS = 192;
template <int BN>
struct PTile {
  static constexpr int STAGES = BN == 256 ? 4 : 6;
  static constexpr int A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2, STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 512 + 4 * STORE_BYTES;
};

template <int BN>
__global__ void __launch_bounds__(PERSIST_THREADS, 1)
    umma_persist_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                             float *D, long long ldd, int M, int N, int K, float alpha, float beta, int kb_per_split,
                             long long split_stride, int nM, int nN, int nsplit, UmmaCtl ctl) {
  chain_start();
  constexpr int STAGES = PTile<BN>::STAGES, A_BYTES = PTile<BN>::A_BYTES, STAGE_BYTES = PTile<BN>::STAGE_BYTES;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned long long *bars = reinterpret_cast<unsigned long long *>(smem + STAGES * STAGE_BYTES);
  unsigned long long *full = bars, *empty = bars + STAGES;
  unsigned long long *accf = bars + 2 * STAGES, *acce = accf + 2, *drain = acce + 2;
  unsigned *tmem_slot = reinterpret_cast<unsigned *>(drain + 1);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  volatile int *issued = reinterpret_cast<volatile int *>(tmem_slot + 2);
  volatile int *consumed = reinterpret_cast<volatile int *>(tmem_slot + 3);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nk_all = (K + BK - 1) / BK;
  const int tiles = nM * nN * nsplit;
  // tile t: split z = t / (nM nN); within a split, groups of RASTER_GM row tiles sweep the column tiles
  auto tile_of = [&](int t, int &m0, int &n0, int &kb0, int &nk, long long &zoff) {
    const int z = t / (nM * nN), id = t - z * (nM * nN);
    const int first_m = (id / (RASTER_GM * nN)) * RASTER_GM;
    const int gm = min(nM - first_m, RASTER_GM);
    const int r = id - first_m * nN;
    m0 = (first_m + r % gm) * BM;
    n0 = (r / gm) * BN;
    kb0 = z * kb_per_split;
    nk = min(nk_all, kb0 + kb_per_split) - kb0;
    zoff = (long long)z * split_stride;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; s++) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    for (int b = 0; b < 2; b++) {
      mbar_init(smem_u32(&accf[b]), 1);
      mbar_init(smem_u32(&acce[b]), 4);   // one arrive per epilogue warp
    }
    mbar_init(smem_u32(drain), 1);
    *abort_flag = 0;
    *issued = 0;
    *consumed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {   // TMEM: two accumulators of BN FP32 columns x 128 lanes
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(2 * BN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0 && !ctl.skip_loads) {
      // ---------------- TMA producer: K blocks of the CTA's tiles, one continuous pipeline
      int it = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
        int m0, n0, kb0, nk;
        long long zoff;
        tile_of(t, m0, n0, kb0, nk, zoff);
        for (int kb = 0; kb < nk; kb++, it++) {
          const int s = it % STAGES;
          const unsigned ph = (it / STAGES) & 1;
          if (!mbar_wait(smem_u32(&empty[s]), ph ^ 1, abort_flag, ctl.wait_ns, ctl.error)) {
            ok = false;
            break;
          }
          unsigned char *sa = smem + s * STAGE_BYTES;
          mbar_expect_tx(smem_u32(&full[s]), STAGE_BYTES);
          tma_load_2d(smem_u32(sa), &tmA, smem_u32(&full[s]), (kb0 + kb) * BK, m0);
          tma_load_2d(smem_u32(sa + A_BYTES), &tmB, smem_u32(&full[s]), (kb0 + kb) * BK, n0);
          *issued = it + 1;
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: accumulator lt & 1 of the CTA's lt-th tile
    const unsigned idesc = idesc_bf16(BM, BN);
    const unsigned long long d0 = smem_desc(smem_u32(smem));
    int it = 0, lt = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x, lt++) {
      int m0, n0, kb0, nk;
      long long zoff;
      tile_of(t, m0, n0, kb0, nk, zoff);
      const int buf = lt & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&acce[buf]), ((lt >> 1) & 1) ^ 1, abort_flag, ctl.wait_ns, ctl.error))) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const unsigned acc = tmem + (unsigned)(buf * BN);
      for (int kb = 0; kb < nk; kb++, it++) {
        const int s = it % STAGES;
        const unsigned ph = (it / STAGES) & 1;
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&full[s]), ph, abort_flag, ctl.wait_ns, ctl.error))) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const unsigned long long da = d0 + s * (STAGE_BYTES >> 4), db = da + (A_BYTES >> 4);
        if (elect_one()) {
          *consumed = it + 1;
#pragma unroll
          for (int k = 0; k < BK / 16; k++) umma_bf16(acc, da + 2 * k, db + 2 * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
          umma_commit(smem_u32(&empty[s]));
        }
        __syncwarp();
      }
      if (ok && elect_one()) umma_commit(smem_u32(&accf[buf]));
      __syncwarp();
    }
    if (elect_one()) umma_commit(smem_u32(drain));   // arrives once every MMA issued above has completed
  } else {
    // ---------------- epilogue warps 2..5: rows 32 (warp mod 4) + lane of each tile
    const int q = warp & 3;
    float *out = reinterpret_cast<float *>(smem + STAGES * STAGE_BYTES + 512 + q * STORE_BYTES);
    int lt = 0;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x, lt++) {
      int m0, n0, kb0, nk;
      long long zoff;
      tile_of(t, m0, n0, kb0, nk, zoff);
      const int buf = lt & 1;
      const bool ready = mbar_wait(smem_u32(&accf[buf]), (lt >> 1) & 1, abort_flag, ctl.wait_ns, ctl.error);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (!__all_sync(0xffffffffu, ready && !*abort_flag)) break;
      const int row0 = m0 + q * 32;
#pragma unroll 1
      for (int c0 = 0; c0 < BN && n0 + c0 < N && row0 < M; c0 += 32) {
        float v[32];
        tmem_ld_32(tmem + ((unsigned)(q * 32) << 16) + (unsigned)(buf * BN + c0), v);
        store_block(out, v, alpha, beta, D + zoff, ldd, row0, M, n0 + c0, N);
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&acce[buf])) : "memory");
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0) {
    // every MMA the issuer committed has completed (the drain barrier); after a time-out also the TMA
    // copies issued but not consumed land before the shared memory goes away (fixed DRAIN_NS limits)
    drain_wait(smem_u32(drain), 0, ctl.error);
    if (*abort_flag)
      for (int it = *consumed; it < *issued; it++)
        drain_wait(smem_u32(&full[it % STAGES]), (it / STAGES) & 1, ctl.error);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BN));
  }
}

// ---------------------------------------------------------------------------------------------
// The same product on CTA pairs (tcgen05 cta_group::2): a cluster of two CTAs on two SMs computes a
// 256 x 256 (192, 128) output tile with M = 256 MMAs.  Each CTA stages its own 128 rows of A and one half of
// the columns of the B tile, so per SM the shared memory holds and the tensor core reads half of the B
// tile of the one-CTA kernel: with a 128 x 256 tile per SM the operand traffic through shared
// memory (TMA writes plus MMA reads, about 1.5x the shared-memory bandwidth at the full MMA rate in
// the one-CTA kernel) drops to about the bandwidth.  The leader CTA (cluster rank 0) issues the MMAs
// for the pair; both CTAs' loads complete on the leader's barriers; the MMA commits arrive on the
// barriers of both CTAs (multicast); each CTA's TMEM holds its own 128 rows of the accumulator and
// each CTA writes them.  Same bounded waits and abort path as the one-CTA kernel; the pair meets at a
// cluster barrier before either frees its TMEM and exits.
// Tiles of 192 and 128 columns fill the chip where 256 would leave the last wave of its 76 pairs nearly empty.
template <int PBN>
struct PairTile {
  static constexpr int HALF = PBN / 2, STAGES = PBN == 256 ? 6 : (PBN == 192 ? 7 : 8);
  static constexpr int A_BYTES = BM * BK * 2, B_BYTES = HALF * BK * 2, STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
  static constexpr int TMEM_COLS = PBN > 128 ? 256 : 128;   // a power of two
};

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// shared::cluster address of a shared::cta address in CTA `rank` of the cluster
__device__ __forceinline__ unsigned map_to_rank(unsigned addr, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

// TMA tile load into this CTA's shared memory, completion on an mbarrier of either CTA of the pair
__device__ __forceinline__ void tma_load_2d_pair(unsigned dst, const CUtensorMap *map, unsigned mbar_cluster, int x,
                                                 int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, "
      "%4}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(mbar_cluster), "r"(x), "r"(y)
      : "memory");
}

__device__ __forceinline__ void umma_bf16_pair(unsigned d_tmem, unsigned long long a, unsigned long long b,
                                               unsigned idesc, unsigned accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.u32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}

// arrive (once all earlier MMAs of this thread have completed) on the mbarrier at this shared
// offset in both CTAs of the pair
__device__ __forceinline__ void umma_commit_pair(unsigned mbar) {
  const unsigned short mask = 0x3;
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(mbar),
      "h"(mask)
      : "memory");
}

template <int PBN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
    umma_pair_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, float *D,
                          long long ldd, int M, int N, int K, float alpha, float beta, int kb_per_split,
                          long long split_stride, UmmaCtl ctl) {
  chain_start();
  constexpr int STAGES = PairTile<PBN>::STAGES, A_BYTES = PairTile<PBN>::A_BYTES,
                STAGE_BYTES = PairTile<PBN>::STAGE_BYTES, TMEM_COLS = PairTile<PBN>::TMEM_COLS;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned long long *bars = reinterpret_cast<unsigned long long *>(smem + STAGES * STAGE_BYTES);
  unsigned long long *full = bars, *empty = bars + STAGES, *done = bars + 2 * STAGES;
  unsigned *tmem_slot = reinterpret_cast<unsigned *>(bars + 2 * STAGES + 1);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  volatile int *issued = reinterpret_cast<volatile int *>(tmem_slot + 2);
  volatile int *consumed = reinterpret_cast<volatile int *>(tmem_slot + 3);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned rank = cluster_rank();
  const bool leader = rank == 0;
  // pair tile order as in the one-CTA kernel, over 256-row pair tiles
  int mp_tile, n_tile;
  {
    const int nM = gridDim.x / 2, nN = gridDim.y;
    const int id = blockIdx.y * nM + (int)(blockIdx.x / 2);
    const int first_m = (id / (RASTER_GM * nN)) * RASTER_GM;
    const int gm = min(nM - first_m, RASTER_GM);
    const int r = id - first_m * nN;
    mp_tile = first_m + r % gm;
    n_tile = r / gm;
  }
  const int m0 = mp_tile * (2 * BM) + (int)rank * BM;        // this CTA's rows
  const int n0 = n_tile * PBN;                            // the pair's columns
  const int nb0 = n0 + (int)rank * PairTile<PBN>::HALF;                 // this CTA's half of the B tile
  const int nk_all = (K + BK - 1) / BK;
  const int kb0 = blockIdx.z * kb_per_split;
  const int kb1 = min(nk_all, kb0 + kb_per_split);
  const int nk = kb1 - kb0;
  D += (long long)blockIdx.z * split_stride;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; s++) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    mbar_init(smem_u32(done), 1);
    *abort_flag = 0;
    *issued = 0;
    *consumed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // The allocation reaches into the peer's SM, so both CTAs of the pair have to be running before either asks for it: a
  // CTA that asked while its peer's SM was still held by another stream's kernel waited without end, about once in 150
  // solves of four streams.
  cluster_sync_all();
  if (warp == 0) {   // TMEM of both CTAs: TMEM_COLS FP32 columns x 128 lanes each (one warp per CTA)
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  cluster_sync_all();   // both CTAs' barriers initialised and TMEM allocated before any remote arrive
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer (both CTAs): loads complete on the leader's full barriers
    for (int kb = 0; kb < nk && !ctl.skip_loads; kb++) {
      const int s = kb % STAGES;
      const unsigned ph = (kb / STAGES) & 1;
      if (!mbar_wait(smem_u32(&empty[s]), ph ^ 1, abort_flag, ctl.wait_ns, ctl.error)) break;
      unsigned char *sa = smem + s * STAGE_BYTES;
      unsigned char *sb = sa + A_BYTES;
      if (leader) mbar_expect_tx(smem_u32(&full[s]), 2 * STAGE_BYTES);
      const unsigned fb = map_to_rank(smem_u32(&full[s]), 0);
      tma_load_2d_pair(smem_u32(sa), &tmA, fb, (kb0 + kb) * BK, m0);
      tma_load_2d_pair(smem_u32(sb), &tmB, fb, (kb0 + kb) * BK, nb0);
      *issued = kb + 1;
    }
  } else if (warp == 1 && leader) {
    // ---------------- MMA issuer (leader only): M = 256 over the pair, N = PBN
    const unsigned idesc = idesc_bf16(2 * BM, PBN);
    const unsigned long long d0 = smem_desc(smem_u32(smem));
    for (int kb = 0; kb < nk; kb++) {
      const int s = kb % STAGES;
      const unsigned ph = (kb / STAGES) & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&full[s]), ph, abort_flag, ctl.wait_ns, ctl.error))) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const unsigned long long da = d0 + s * (STAGE_BYTES >> 4), db = da + (A_BYTES >> 4);
      if (elect_one()) {
        *consumed = kb + 1;
#pragma unroll
        for (int k = 0; k < BK / 16; k++)
          umma_bf16_pair(tmem, da + 2 * k, db + 2 * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
        umma_commit_pair(smem_u32(&empty[s]));
      }
      __syncwarp();
    }
    if (elect_one()) umma_commit_pair(smem_u32(done));   // both CTAs: every MMA issued above has completed
  }
  __syncwarp();

  // ---------------- epilogue: all 4 warps of each CTA, its own 128 rows (skipped once any CTA of the
  // call has given up, so that a pair whose leader aborted writes nothing)
  const bool ready = mbar_wait(smem_u32(done), 0, abort_flag, ctl.wait_ns, ctl.error);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const bool failed = *reinterpret_cast<volatile unsigned *>(ctl.error) != 0;
  if (__all_sync(0xffffffffu, ready && !*abort_flag && !failed) && nk > 0) {
    // the pair's MMAs have completed and all loads landed: the stages hold the blocks on their way out
    float *buf = reinterpret_cast<float *>(smem + warp * STORE_BYTES);
    const int row0 = m0 + warp * 32;
#pragma unroll 1
    for (int c0 = 0; c0 < PBN && n0 + c0 < N && row0 < M; c0 += 32) {
      float v[32];
      tmem_ld_32(tmem + ((unsigned)(warp * 32) << 16) + c0, v);
      store_block(buf, v, alpha, beta, D, ldd, row0, M, n0 + c0, N);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && leader && *abort_flag) {
    // leader after a time-out: the committed MMAs (done), then the loads it waited for of both CTAs
    // (the pair's copies complete on the leader's barriers), each with the fixed DRAIN_NS limit
    drain_wait(smem_u32(done), 0, ctl.error);
    for (int kb = *consumed; kb < *issued; kb++)
      drain_wait(smem_u32(&full[kb % STAGES]), (kb / STAGES) & 1, ctl.error);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  cluster_sync_all();   // neither CTA frees its TMEM or shared memory while the pair's work is in flight
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
  }
  // and stay until both have given it back
  cluster_sync_all();
}

// ---------------------------------------------------------------------------------------------
// FP64-accurate product from digit planes with every digit pair of a tile in one CTA:
//   C = alpha 2^(eA[m] + eB[n]) sum_L 2^(-bL) sum_{i+j=L, L<=P} A_i B_j^T + beta C   (b-bit digits).
// The accumulator of each level L = i + j lives in its own BN columns of TMEM (8 levels of 64 columns
// fill it).  The tensor cores read both operands from shared memory, so the work is arranged to
// read and load each byte as seldom as possible: the B planes of a K block lie one after the other, so one
// MMA multiplies an A plane with up to 256 / BN of them at once (N = 256) and adds the products to as
// many consecutive levels; per K block every plane is loaded once (A planes through a ring of slots, B
// planes double-buffered).  Persistent: one CTA per SM walks the tiles; a producer warp, an MMA warp and
// epilogue warps of 16 columns each.  A level is an exact integer while it holds at most 2^24 / 2^(2b-2) products:
// after kc K blocks the epilogue warps add the levels to two int64 accumulators per output (levels
// 2..5 and 6..9) and the MMA warp starts them anew.  The last step, integer to FP64 with one rounding, is
// integer arithmetic too (FP64 operations are issued at two per SM and clock).
// Bound by the tensor cores: 8000 x 3200 x 8000 at level 9 (36 pairs) 7.8 ms, 1.88 PFLOP/s of BF16 products.
// Before (one GEMM per pair with FP32 partial sums in global memory for wide products, one N = 64 MMA per
// pair for narrow ones): the residual's ring product of 40 systems at o=40 v=200 9.1 -> 5.4 ms, its other
// four products 7.3 -> 2.1 ms.
constexpr int EMU_MAXS = 8, EMU_A_SLOTS = 6, EMU_COLS = 16;   // EMU_COLS: columns of an epilogue thread
constexpr int EMU_A_BYTES = BM * BK * 2;
template <int BN>
struct EmuTile {
  static constexpr int B_PLANE = BN * BK * 2, B_BYTES = EMU_MAXS * B_PLANE, GROUP = 256 / BN, COLS = EMU_MAXS * BN;
  static constexpr int EPI_WARPS = 4 * BN / EMU_COLS, THREADS = 64 + 32 * EPI_WARPS;
  static constexpr int SMEM_BYTES = EMU_A_SLOTS * EMU_A_BYTES + 2 * B_BYTES + 1024 + 512;
};

struct EmuArgs {
  int SA, SB, P, bits;          // planes of A and B, highest level, bits of a digit
  int M, N, nM, nN, nz;         // output, tiles, K splits
  int nk, kb_per_split, kc;     // K blocks: all, of a split, between two drains
  const int *eA, *eB;
  int alpha_exp;                // alpha = alpha_mul 2^alpha_exp
  double alpha_mul, beta;
  double *C, *part;
  IMap rm, cm;                  // row / column maps of C
  long long r0g, c0g;           // first row / column index
  const unsigned *gate;         // nothing is done when *gate > gate_cap (nullptr: always)
  unsigned gate_cap;
  UmmaCtl ctl;
};

__device__ __forceinline__ void tma_load_3d(unsigned dst, const CUtensorMap *map, unsigned mbar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(
          dst),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(mbar), "r"(x), "r"(y), "r"(z)
      : "memory");
}

__device__ __forceinline__ void tmem_ld_8_nowait(unsigned taddr, unsigned (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

// (hi 2^sh + lo) 2^e2 rounded once to FP64 (round to nearest, ties to even) with integer operations
__device__ __forceinline__ double fixed_to_f64(long long hi, long long lo, int sh, int e2) {
  const __int128 t = ((__int128)hi << sh) + lo;
  if (t == 0) return 0.0;
  const bool neg = t < 0;
  unsigned __int128 u = neg ? -(unsigned __int128)t : (unsigned __int128)t;
  const unsigned long long uh = (unsigned long long)(u >> 64);
  const int lz = uh ? __clzll((long long)uh) : 64 + __clzll((long long)(unsigned long long)u);
  u <<= lz;
  const unsigned long long top = (unsigned long long)(u >> 64);
  unsigned long long mant = top >> 11;
  const unsigned long long rem = top & 0x7ffULL;
  const bool sticky = (unsigned long long)u != 0;
  if (rem > 0x400ULL || (rem == 0x400ULL && (sticky || (mant & 1)))) mant++;
  const int be = 127 - lz + e2 + 1023;   // biased exponent of the leading bit
  double v;
  if (be >= 1 && be <= 2045)
    v = __longlong_as_double((long long)(((unsigned long long)be << 52) + (mant - (1ULL << 52))));
  else
    v = scalbn((double)mant, 127 - lz + e2 - 52);
  return neg ? -v : v;
}

// The MMAs of one K block at level P, called by a whole warp so that the descriptors stay in uniform
// registers (built lane by lane, an MMA took about 130 clocks to issue, four times what N = 64 takes to
// execute); everything but the slot is a compile-time constant.  ita counts the A planes consumed.
template <int BN, int P>
__device__ __forceinline__ bool emu_issue_kblock(unsigned tmem, unsigned sa0, unsigned sb, unsigned long long *afull,
                                                 unsigned long long *aempty, int &ita, bool start,
                                                 volatile int *consumed_a, volatile int *abort_flag,
                                                 unsigned long long wait_ns, unsigned *error) {
  using T = EmuTile<BN>;
  const unsigned long long db = smem_desc(sb);
#pragma unroll
  for (int i = 1; i < P; i++, ita++) {
    const int s = ita % EMU_A_SLOTS;
    if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&afull[s]), (ita / EMU_A_SLOTS) & 1, abort_flag, wait_ns, error)))
      return false;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned long long da = smem_desc(sa0 + s * EMU_A_BYTES);
    if (elect_one()) {
      *consumed_a = ita + 1;
#pragma unroll
      for (int k = 0; k < BK / 16; k++)
#pragma unroll
        for (int j = 1; j <= P - i; j += T::GROUP) {
          // plane 1 meets every level first (there are P - 1 B planes), so it starts the accumulators
          const int g = T::GROUP < P - i - j + 1 ? T::GROUP : P - i - j + 1;
          const unsigned acc = (i > 1 || k > 0) ? 1u : (start ? 0u : 1u);
          umma_bf16(tmem + (unsigned)((i + j - 2) * BN), da + 2 * k, db + (j - 1) * (T::B_PLANE >> 4) + 2 * k,
                    idesc_bf16(BM, g * BN), acc);
        }
      umma_commit(smem_u32(&aempty[s]));
    }
    __syncwarp();
  }
  return true;
}

template <int BN>
__global__ void __launch_bounds__(EmuTile<BN>::THREADS, 1)
    umma_emu_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ EmuArgs a) {
  using T = EmuTile<BN>;
  if (a.gate != nullptr && *a.gate > a.gate_cap) return;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char *smA = smem, *smB = smem + EMU_A_SLOTS * EMU_A_BYTES;
  unsigned long long *bars = reinterpret_cast<unsigned long long *>(smB + 2 * T::B_BYTES);
  unsigned long long *afull = bars, *aempty = afull + EMU_A_SLOTS, *bfull = aempty + EMU_A_SLOTS, *bempty = bfull + 2;
  unsigned long long *accf = bempty + 2, *acce = accf + 1, *drain = acce + 1;
  unsigned *tmem_slot = reinterpret_cast<unsigned *>(drain + 1);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  volatile int *issued_a = reinterpret_cast<volatile int *>(tmem_slot + 2), *issued_b = issued_a + 1;
  volatile int *consumed_a = issued_a + 2, *consumed_b = issued_a + 3;
  volatile int *go = issued_a + 4;   // the epilogue group's decision per chunk (two in turn)

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tiles = a.nM * a.nN * a.nz;
  const int SAe = min(a.SA, a.P - 1);   // A planes with at least one partner
  const int SBe = min(a.SB, a.P - 1);
  const unsigned long long wait_ns = a.ctl.wait_ns;
  unsigned *error = a.ctl.error;
  // tile t: split z, then groups of RASTER_GM row tiles sweep the column tiles
  auto tile_of = [&](int t, int &m0, int &n0, int &z, int &kb0, int &nk) {
    z = t / (a.nM * a.nN);
    const int id = t - z * (a.nM * a.nN);
    const int first_m = (id / (RASTER_GM * a.nN)) * RASTER_GM;
    const int gm = min(a.nM - first_m, RASTER_GM);
    const int r = id - first_m * a.nN;
    m0 = (first_m + r % gm) * BM;
    n0 = (r / gm) * BN;
    kb0 = z * a.kb_per_split;
    nk = min(a.nk, kb0 + a.kb_per_split) - kb0;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < EMU_A_SLOTS; s++) {
      mbar_init(smem_u32(&afull[s]), 1);
      mbar_init(smem_u32(&aempty[s]), 1);
    }
    for (int s = 0; s < 2; s++) {
      mbar_init(smem_u32(&bfull[s]), 1);
      mbar_init(smem_u32(&bempty[s]), 1);
    }
    mbar_init(smem_u32(accf), 1);
    mbar_init(smem_u32(acce), T::EPI_WARPS);
    mbar_init(smem_u32(drain), 1);
    *abort_flag = 0;
    *issued_a = *issued_b = *consumed_a = *consumed_b = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(T::COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0 && !a.ctl.skip_loads) {
      // ---------------- TMA producer: per K block all B planes at once, then the A planes one by one
      int ita = 0, itb = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
        int m0, n0, z, kb0, nk;
        tile_of(t, m0, n0, z, kb0, nk);
        for (int kb = kb0; kb < kb0 + nk && ok; kb++) {
          const int sb = itb & 1;
          if (!mbar_wait(smem_u32(&bempty[sb]), ((itb >> 1) & 1) ^ 1, abort_flag, wait_ns, error)) {
            ok = false;
            break;
          }
          mbar_expect_tx(smem_u32(&bfull[sb]), SBe * T::B_PLANE);
          tma_load_3d(smem_u32(smB + sb * T::B_BYTES), &tmB, smem_u32(&bfull[sb]), kb * BK, n0, 0);
          *issued_b = ++itb;
          for (int i = 0; i < SAe; i++) {
            const int s = ita % EMU_A_SLOTS;
            if (!mbar_wait(smem_u32(&aempty[s]), ((ita / EMU_A_SLOTS) & 1) ^ 1, abort_flag, wait_ns, error)) {
              ok = false;
              break;
            }
            mbar_expect_tx(smem_u32(&afull[s]), EMU_A_BYTES);
            tma_load_3d(smem_u32(smA + s * EMU_A_BYTES), &tmA, smem_u32(&afull[s]), kb * BK, m0, i);
            *issued_a = ++ita;
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (the whole warp; one elected lane issues)
    int ita = 0, itb = 0, ch = 0;
    bool ok = true;
    const unsigned sa0 = smem_u32(smA);
    for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
      int m0, n0, z, kb0, nk;
      tile_of(t, m0, n0, z, kb0, nk);
      for (int c0 = 0; c0 < nk && ok; c0 += a.kc, ch++) {
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(acce), (ch & 1) ^ 1, abort_flag, wait_ns, error))) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int c1 = min(nk, c0 + a.kc);
        for (int kb = c0; kb < c1 && ok; kb++, itb++) {
          const int sbuf = itb & 1;
          if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bfull[sbuf]), (itb >> 1) & 1, abort_flag, wait_ns, error))) {
            ok = false;
            break;
          }
          if (lane == 0) *consumed_b = itb + 1;
          const unsigned sb = smem_u32(smB + sbuf * T::B_BYTES);
          const bool start = kb == c0;
          switch (a.P) {
#define GFCC_EMU_LEVEL(P)                                                                                       \
  case P:                                                                                                       \
    ok = emu_issue_kblock<BN, P>(tmem, sa0, sb, afull, aempty, ita, start, consumed_a, abort_flag, wait_ns, error); \
    break;
            GFCC_EMU_LEVEL(2)
            GFCC_EMU_LEVEL(3)
            GFCC_EMU_LEVEL(4)
            GFCC_EMU_LEVEL(5)
            GFCC_EMU_LEVEL(6)
            GFCC_EMU_LEVEL(7)
            GFCC_EMU_LEVEL(8)
            GFCC_EMU_LEVEL(9)
#undef GFCC_EMU_LEVEL
            default: ok = false; break;
          }
          if (ok && elect_one()) umma_commit(smem_u32(&bempty[sbuf]));
          __syncwarp();
        }
        if (ok && elect_one()) umma_commit(smem_u32(accf));
        __syncwarp();
      }
    }
    if (elect_one()) umma_commit(smem_u32(drain));   // arrives once every MMA issued above has completed
    __syncwarp();
  } else {
    // ---------------- epilogue: warp w reads TMEM lanes 32 (w mod 4) .. + 31, NC of the columns
    constexpr int NC = EMU_COLS;
    const int q = warp & 3, part = (warp - 2) >> 2;
    const int Lhi = min(a.P, 5), b = a.bits;
    const unsigned trow = tmem + ((unsigned)(q * 32) << 16) + (unsigned)(part * NC);
    long long hi[NC], lo[NC];
    int ch = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
      int m0, n0, z, kb0, nk;
      tile_of(t, m0, n0, z, kb0, nk);
#pragma unroll
      for (int c = 0; c < NC; c++) hi[c] = lo[c] = 0;
      for (int c0 = 0; c0 < nk; c0 += a.kc, ch++) {
        // one lane polls and decides for the group; the other warps block on a named barrier (polling by
        // all of them takes shared-memory cycles from the loads)
        if (warp == 2 && lane == 0) {
          const bool ready = mbar_wait(smem_u32(accf), ch & 1, abort_flag, wait_ns, error);
          go[ch & 1] = ready && !*abort_flag ? 1 : 0;
        }
        __syncwarp();
        asm volatile("bar.sync 1, %0;" ::"n"(32 * T::EPI_WARPS) : "memory");
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (!go[ch & 1]) {
          ok = false;
          break;
        }
#pragma unroll
        for (int g = 0; g < NC; g += 8) {
          // two levels at a time: hi takes levels 2..Lhi, lo the ones above
#pragma unroll
          for (int l = 0; l < EMU_MAXS; l += 2) {
            unsigned r[2][8];
            if (2 + l > a.P) break;
            tmem_ld_8_nowait(trow + (unsigned)(l * BN + g), r[0]);
            if (3 + l <= a.P) tmem_ld_8_nowait(trow + (unsigned)((l + 1) * BN + g), r[1]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int d = 0; d < 2; d++) {
              if (2 + l + d > a.P) break;
              const int sh = b * ((l < 4 ? Lhi : a.P) - 2 - l - d);
#pragma unroll
              for (int c = 0; c < 8; c++) {
                const long long x = (long long)__float2int_rn(__uint_as_float(r[d][c])) << sh;
                if (l < 4)
                  hi[g + c] += x;
                else
                  lo[g + c] += x;
              }
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(acce)) : "memory");
      }
      const int row = m0 + q * 32 + lane;
      const int c0 = n0 + part * NC;
      const int sh = b * (a.P - Lhi), e0 = -b * a.P;
      if (!ok || row >= a.M) {
        // nothing to store
      } else if (a.part != nullptr) {
        double *dst = a.part + ((long long)z * a.M + row) * a.N + c0;
#pragma unroll
        for (int c = 0; c < NC; c++)
          if (c0 + c < a.N) dst[c] = fixed_to_f64(hi[c], lo[c], sh, e0);
      } else {
        const int ea = a.eA[row] + a.alpha_exp + e0;
        double *base = a.C + imap_apply(a.rm, a.r0g + row);
        // the column offset walks without a division per column
        const long long x0 = a.c0g + c0;
        const bool two = a.cm.d0 > 0;
        long long rr = two ? x0 % a.cm.d0 : 0;
        long long off = imap_apply(a.cm, x0);
        const long long wrap = two ? a.cm.s1 - a.cm.d0 * a.cm.s0 : 0;
#pragma unroll
        for (int c = 0; c < NC; c++) {
          if (c0 + c < a.N) {
            double v = fixed_to_f64(hi[c], lo[c], sh, ea + a.eB[c0 + c]);
            if (a.alpha_mul != 1.0) v *= a.alpha_mul;
            if (a.beta != 0.0) v += a.beta * base[off];
            base[off] = v;
          }
          off += a.cm.s0;
          if (two && ++rr == a.cm.d0) {
            rr = 0;
            off += wrap;
          }
        }
      }
      __syncwarp();
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0) {
    // every MMA has completed (the drain barrier); after a time-out also the copies that were issued but
    // not consumed land before the shared memory goes away (fixed DRAIN_NS limits)
    drain_wait(smem_u32(drain), 0, error);
    if (*abort_flag) {
      for (int it = *consumed_a; it < *issued_a; it++)
        drain_wait(smem_u32(&afull[it % EMU_A_SLOTS]), (it / EMU_A_SLOTS) & 1, error);
      for (int it = *consumed_b; it < *issued_b; it++)
        drain_wait(smem_u32(&bfull[it & 1]), (it >> 1) & 1, error);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(T::COLS));
  }
}

// C = alpha 2^(eA + eB) sum_z part[z] + beta C (the K splits of umma_emu_kernel)
__global__ void emu_split_reduce_kernel(const double *part, int nz, int M, int N, const int *eA, const int *eB,
                                        double alpha, double beta, double *C, IMap cm, IMap cn, long long m0g,
                                        long long n0g, const unsigned *gate, unsigned gate_cap) {
  if (gate != nullptr && *gate > gate_cap) return;
  const long long tot = (long long)M * N;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot; t += (long long)gridDim.x * blockDim.x) {
    const int m = (int)(t / N), n = (int)(t - (long long)m * N);
    double s = 0.0;
    for (int z = 0; z < nz; z++) s += part[(long long)z * tot + t];
    const long long off = imap_apply(cm, m0g + m) + imap_apply(cn, n0g + n);
    const double val = alpha * ldexp(s, eA[m] + eB[n]);
    C[off] = beta != 0.0 ? val + beta * C[off] : val;
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (fn == nullptr) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    else
      cudaGetLastError();
  }
  return fn;
}

// 2-D K-major BF16 tensor map: rows x K (row stride ld elements), box 64 (K) x box_rows, 128-byte swizzle
int make_map(CUtensorMap *map, const void *base, long long rows, long long K, long long ld, int box_rows) {
  auto fn = encode_fn();
  if (fn == nullptr) {
    set_error("cuTensorMapEncodeTiled is not available from the driver");
    return GFCC_ERR_CUDA;
  }
  const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  const cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("cuTensorMapEncodeTiled failed (%d) for rows=%lld K=%lld ld=%lld", (int)r, rows, K, ld);
    return GFCC_ERR_ARG;
  }
  return GFCC_OK;
}

}  // namespace

int umma_splits(int K, int nsplit) {
  const int nk = (K + BK - 1) / BK;
  if (nsplit < 1) nsplit = 1;
  if (nsplit > nk) nsplit = nk;
  const int kbs = (nk + nsplit - 1) / nsplit;
  return (nk + kbs - 1) / kbs;
}

UmmaScope::UmmaScope(unsigned *flag) : prev(t_error_flag) { t_error_flag = flag; }
UmmaScope::~UmmaScope() { t_error_flag = prev; }
unsigned *umma_error_flag() { return t_error_flag; }

int umma_error_reset(cudaStream_t st) {
  GFCC_CUDA(cudaMemsetAsync(t_error_flag, 0, sizeof(unsigned), st));
  return GFCC_OK;
}

int umma_error_check(cudaStream_t st) {
  unsigned h = 0;
  GFCC_CUDA(cudaMemcpyAsync(&h, t_error_flag, sizeof(h), cudaMemcpyDeviceToHost, st));
  GFCC_CUDA(cudaStreamSynchronize(st));
  return h != 0 ? umma_timed_out() : GFCC_OK;
}

int umma_timed_out() {
  set_error("a tensor-core GEMM wait timed out on the device");
  return GFCC_ERR_TIMEOUT;
}

namespace {
// tile autotuner state: (device, M, N, K, split) -> tile width
bool g_autotune = true;
// 0: the autotuner also times the CTA-pair tile; 1: the pair tile whenever it applies; 2: never
int g_pair_mode = 0;
constexpr int TILE_PAIR = 512;   // autotuner key offset of the CTA-pair tiles (+ their width)
constexpr int TILE_PERSIST = 1024;   // autotuner key offset of the persistent kernel (+ its tile width)
// 0: the autotuner also times the persistent kernel; 1: always the persistent kernel; 2: never
int g_persist_mode = 0;
std::mutex g_tune_mu;
std::map<std::tuple<int, int, int, int, int>, int> g_tune;

template <int BN, int ST, bool GUARD = false>
int launch_umma_st(cudaStream_t st, const __nv_bfloat16 *A, long long lda, const __nv_bfloat16 *B, long long ldb,
                   float *D, long long ldd, int M, int N, int K, float alpha, float beta, int nsplit, int kbs,
                   long long split_stride, const GuardArgs &guard = GuardArgs()) {
  UmmaCtl ctl;
  GFCC_TRY(umma_ctl(&ctl));
  CUtensorMap ma, mb;
  GFCC_TRY(make_map(&ma, A, M, K, lda, BM));
  GFCC_TRY(make_map(&mb, B, N, K, ldb, BN));
  static bool attr[64] = {false};
  int dev = 0;
  GFCC_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64 || !attr[dev]) {
    GFCC_CUDA(cudaFuncSetAttribute(umma_bf16_gemm_kernel<BN, ST, GUARD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   Tile<BN, ST>::SMEM_BYTES));
    if (dev >= 0 && dev < 64) attr[dev] = true;
  }
  if ((N + BN - 1) / BN > 65535 || nsplit > 65535) {
    set_error("gemm_bf16_tn: grid too large (N=%d, nsplit=%d)", N, nsplit);
    return GFCC_ERR_ARG;
  }
  dim3 grid((M + BM - 1) / BM, (N + BN - 1) / BN, nsplit);
  GFCC_CUDA(launch_chained(umma_bf16_gemm_kernel<BN, ST, GUARD>, grid, THREADS, Tile<BN, ST>::SMEM_BYTES, st, ma, mb, D,
                           ldd, M, N, K, alpha, beta, kbs, split_stride, ctl, guard));
  GFCC_LAUNCH_CHECK();
  return GFCC_OK;
}

template <int BN>
int launch_umma_persist(cudaStream_t st, const __nv_bfloat16 *A, long long lda, const __nv_bfloat16 *B, long long ldb,
                        float *D, long long ldd, int M, int N, int K, float alpha, float beta, int nsplit, int kbs,
                        long long split_stride) {
  UmmaCtl ctl;
  GFCC_TRY(umma_ctl(&ctl));
  CUtensorMap ma, mb;
  GFCC_TRY(make_map(&ma, A, M, K, lda, BM));
  GFCC_TRY(make_map(&mb, B, N, K, ldb, BN));
  static bool attr[64] = {false};
  static int nsm[64] = {0};
  int dev = 0;
  GFCC_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64 || !attr[dev]) {
    GFCC_CUDA(cudaFuncSetAttribute(umma_persist_gemm_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   PTile<BN>::SMEM_BYTES));
    int sms = 0;
    GFCC_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (dev >= 0 && dev < 64) {
      attr[dev] = true;
      nsm[dev] = sms;
    }
  }
  const int sms = (dev >= 0 && dev < 64 && nsm[dev] > 0) ? nsm[dev] : 152;
  const long long nM = (M + BM - 1) / BM, nN = (N + BN - 1) / BN, tiles = nM * nN * nsplit;
  if (tiles > 0x7fffffffLL) {
    set_error("gemm_bf16_tn: too many tiles (M=%d, N=%d, nsplit=%d)", M, N, nsplit);
    return GFCC_ERR_ARG;
  }
  const unsigned grid = (unsigned)std::min<long long>(tiles, sms);
  GFCC_CUDA(launch_chained(umma_persist_gemm_kernel<BN>, grid, PERSIST_THREADS, PTile<BN>::SMEM_BYTES, st, 
      ma, mb, D, ldd, M, N, K, alpha, beta, kbs, split_stride, (int)nM, (int)nN, nsplit, ctl));
  GFCC_LAUNCH_CHECK();
  return GFCC_OK;
}

template <int PBN>
int launch_umma_pair(cudaStream_t st, const __nv_bfloat16 *A, long long lda, const __nv_bfloat16 *B, long long ldb,
                     float *D, long long ldd, int M, int N, int K, float alpha, float beta, int nsplit, int kbs,
                     long long split_stride) {
  UmmaCtl ctl;
  GFCC_TRY(umma_ctl(&ctl));
  CUtensorMap ma, mb;
  GFCC_TRY(make_map(&ma, A, M, K, lda, BM));
  GFCC_TRY(make_map(&mb, B, N, K, ldb, PairTile<PBN>::HALF));
  static bool attr[64] = {false};
  int dev = 0;
  GFCC_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64 || !attr[dev]) {
    GFCC_CUDA(cudaFuncSetAttribute(umma_pair_gemm_kernel<PBN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   PairTile<PBN>::SMEM_BYTES));
    if (dev >= 0 && dev < 64) attr[dev] = true;
  }
  const long long mp = (M + 2 * BM - 1) / (2 * BM);
  if ((N + PBN - 1) / PBN > 65535 || nsplit > 65535 || 2 * mp > 0x7fffffffLL) {
    set_error("gemm_bf16_tn: grid too large (M=%d, N=%d, nsplit=%d)", M, N, nsplit);
    return GFCC_ERR_ARG;
  }
  dim3 grid((unsigned)(2 * mp), (N + PBN - 1) / PBN, nsplit);
  GFCC_CUDA(launch_chained(umma_pair_gemm_kernel<PBN>, grid, THREADS, PairTile<PBN>::SMEM_BYTES, st, ma, mb, D, ldd, M, N, K, alpha, beta, kbs,
                                                                              split_stride, ctl));
  GFCC_LAUNCH_CHECK();
  return GFCC_OK;
}

// few K blocks per CTA: two stages
template <int BN>
int launch_umma(cudaStream_t st, const __nv_bfloat16 *A, long long lda, const __nv_bfloat16 *B, long long ldb,
                float *D, long long ldd, int M, int N, int K, float alpha, float beta, int nsplit, int kbs,
                long long split_stride) {
  if (kbs <= 2)
    return launch_umma_st<BN, 2>(st, A, lda, B, ldb, D, ldd, M, N, K, alpha, beta, nsplit, kbs, split_stride);
  return launch_umma_st<BN, 0>(st, A, lda, B, ldb, D, ldd, M, N, K, alpha, beta, nsplit, kbs, split_stride);
}
}  // namespace

int gemm_bf16_tn(cudaStream_t st, const __nv_bfloat16 *A, long long lda, const __nv_bfloat16 *B, long long ldb,
                 float *D, long long ldd, int M, int N, int K, float alpha, float beta, int nsplit,
                 long long split_stride) {
  if (M <= 0 || N <= 0) return GFCC_OK;
  const int nk = (K + BK - 1) / BK;
  if (nsplit < 1) nsplit = 1;
  if (nsplit > nk) nsplit = nk;
  const int kbs = (nk + nsplit - 1) / nsplit;
  nsplit = (nk + kbs - 1) / kbs;   // every split gets at least one K block
  if (nsplit > 1 && split_stride < (long long)(M - 1) * ldd + N) {
    set_error("gemm_bf16_tn: split-K writes separate partial sums (stride >= one output)");
    return GFCC_ERR_ARG;
  }
  if (K <= 0 || (lda % 8) || (ldb % 8) || lda < K || ldb < K || ldd < N ||
      (reinterpret_cast<uintptr_t>(A) & 15) || (reinterpret_cast<uintptr_t>(B) & 15)) {
    set_error("gemm_bf16_tn: need K > 0, 16-byte aligned operands and row strides that are multiples of 8 "
              "(M=%d N=%d K=%d lda=%lld ldb=%lld)", M, N, K, lda, ldb);
    return GFCC_ERR_ARG;
  }
  GFCC_TRY(check_extent_bytes(A, (long long)(M - 1) * lda * 2 + (long long)K * 2, "bf16 GEMM operand A"));
  GFCC_TRY(check_extent_bytes(B, (long long)(N - 1) * ldb * 2 + (long long)K * 2, "bf16 GEMM operand B"));
  GFCC_TRY(check_extent_bytes(D, ((long long)(M - 1) * ldd + N + (long long)(nsplit - 1) * split_stride) * 4,
                              "bf16 GEMM output D"));
  // tile widths: 64 / 128 / 256 columns per CTA, TILE_PAIR + 128 / 192 / 256 (256 rows over a CTA pair), or
  // TILE_PERSIST + 64 / 128 / 256 (the persistent kernel with that width)
  auto run = [&](int bn) -> int {
    if (bn == 64) return launch_umma<64>(st, A, lda, B, ldb, D, ldd, M, N, K, alpha, beta, nsplit, kbs, split_stride);
    if (bn == 128) return launch_umma<128>(st, A, lda, B, ldb, D, ldd, M, N, K, alpha, beta, nsplit, kbs, split_stride);
    if (bn == TILE_PAIR + 128)
      return launch_umma_pair<128>(st, A, lda, B, ldb, D, ldd, M, N, K, alpha, beta, nsplit, kbs, split_stride);
    if (bn == TILE_PAIR + 192)
      return launch_umma_pair<192>(st, A, lda, B, ldb, D, ldd, M, N, K, alpha, beta, nsplit, kbs, split_stride);
    if (bn == TILE_PAIR + 256)
      return launch_umma_pair<256>(st, A, lda, B, ldb, D, ldd, M, N, K, alpha, beta, nsplit, kbs, split_stride);
    if (bn == TILE_PERSIST + 64)
      return launch_umma_persist<64>(st, A, lda, B, ldb, D, ldd, M, N, K, alpha, beta, nsplit, kbs, split_stride);
    if (bn == TILE_PERSIST + 128)
      return launch_umma_persist<128>(st, A, lda, B, ldb, D, ldd, M, N, K, alpha, beta, nsplit, kbs, split_stride);
    if (bn == TILE_PERSIST + 256)
      return launch_umma_persist<256>(st, A, lda, B, ldb, D, ldd, M, N, K, alpha, beta, nsplit, kbs, split_stride);
    return launch_umma<256>(st, A, lda, B, ldb, D, ldd, M, N, K, alpha, beta, nsplit, kbs, split_stride);
  };
  // the pair kernel needs two row tiles and pays off on wide products with a long K loop; its widths by the waves of
  // 76 pairs (clocks of a tile: a K block's loads at 55 bytes a clock, some 16 a column and 6000 for its ends).
  // 3591 x 1620 x 3591: 192 columns 38 us, 256 columns 50 us; 8000 x 3200 x 8000: 256 columns 257 us, 128 348 us.
  const bool pair_ok = g_pair_mode != 2 && M > BM && N > 128 && kbs >= 8;
  auto pair_cost = [&](int w) {
    const long long tiles = ((M + 2 * BM - 1) / (2 * BM)) * ((N + w - 1LL) / w) * nsplit;
    return (double)((tiles + 75) / 76) * (kbs * (298.0 + 1.16 * w) + 16.0 * w + 6000.0);
  };
  const int pair_best = pair_cost(256) <= std::min(pair_cost(192), pair_cost(128)) ? 256
                        : pair_cost(192) <= pair_cost(128)                       ? 192
                                                                                 : 128;
  if (g_pair_mode == 1) return pair_ok ? run(TILE_PAIR + pair_best) : run(N <= 64 ? 64 : (N <= 128 ? 128 : 256));
  const int narrow = N <= 64 ? 64 : (N <= 128 ? 128 : 256);
  if (g_persist_mode == 1) return run(TILE_PERSIST + narrow);
  // the persistent kernel pays off once a launch has several waves of tiles
  const long long tiles_narrow = ((M + BM - 1) / BM) * ((N + narrow - 1) / narrow) * (long long)nsplit;
  const bool persist_ok = g_persist_mode != 2 && tiles_narrow > 2 * 152;
  // default: the narrowest tile that covers N (wide N keeps the 256-column tile)
  int bn = N <= 64 ? 64 : (N <= 128 ? 128 : 256);
  if (concurrent_calls()) {
    // beside other calls no launch is timed: a choice made alone, or the tile whose busiest SM has the least to do, by the
    // clocks of pair_cost (one-CTA tiles without the halved B tile)
    auto cost = [&](int w) {
      const long long tiles = ((M + BM - 1LL) / BM) * ((N + w - 1LL) / w) * nsplit;
      return (double)((tiles + 151) / 152) * (kbs * (298.0 + 2.33 * w) + 16.0 * w + 6000.0);
    };
    bn = 64;
    for (int w : {128, 256})
      if (w / 2 < N && cost(w) < cost(bn)) bn = w;
    if (pair_ok && pair_cost(pair_best) < cost(bn)) bn = TILE_PAIR + pair_best;
    const int t = umma_tuned_tile(M, N, K, nsplit);
    if (t) bn = t;
  } else if (g_autotune && beta != 0.0f) {
    // accumulating calls are not timed (they would change D); they reuse a tuned choice if any
    const int t = umma_tuned_tile(M, N, K, nsplit);
    if (t) bn = t;
  } else if (g_autotune) {
    int dev = 0;
    GFCC_CUDA(cudaGetDevice(&dev));
    const auto key = std::make_tuple(dev, M, N, K, nsplit);
    int best = 0;
    {
      std::lock_guard<std::mutex> lk(g_tune_mu);
      auto it = g_tune.find(key);
      if (it != g_tune.end()) best = it->second;
    }
    if (best == 0) {
      // first call of this shape: time every tile width that may win (the faster of two launches each, CUDA events on
      // the stream; beta == 0, so the repeated launches leave the same D) and keep the fastest
      struct Events {
        cudaEvent_t e[3] = {nullptr, nullptr, nullptr};
        ~Events() {
          for (cudaEvent_t x : e)
            if (x) cudaEventDestroy(x);
        }
      } events;
      cudaEvent_t *ev = events.e;
      for (cudaEvent_t &x : events.e) GFCC_CUDA(cudaEventCreate(&x));
      float best_ms = 0.0f;
      // 64 columns read the A rows four times as often as 256: not for wide products with a long K loop
      const bool wide = N >= 512 && K >= 512;
      for (int cand : {64, 128, 256, TILE_PAIR + 128, TILE_PAIR + 192, TILE_PAIR + 256, TILE_PERSIST + 64,
                       TILE_PERSIST + 128, TILE_PERSIST + 256}) {
        const int w = cand > TILE_PERSIST ? cand - TILE_PERSIST : cand > TILE_PAIR ? cand - TILE_PAIR : cand;
        if (cand > TILE_PAIR && cand < TILE_PERSIST
                ? !pair_ok || pair_cost(w) > 1.15 * pair_cost(pair_best)
                : ((cand > TILE_PERSIST) != persist_ok || (w > 64 && w / 2 >= N) || (w == 64 && wide)))
          continue;   // never better
        GFCC_CUDA(cudaEventRecord(ev[0], st));
        GFCC_TRY(run(cand));
        GFCC_CUDA(cudaEventRecord(ev[1], st));
        GFCC_TRY(run(cand));
        GFCC_CUDA(cudaEventRecord(ev[2], st));
        GFCC_CUDA(cudaEventSynchronize(ev[2]));
        float ms = 0.0f, ms2 = 0.0f;
        GFCC_CUDA(cudaEventElapsedTime(&ms, ev[0], ev[1]));
        GFCC_CUDA(cudaEventElapsedTime(&ms2, ev[1], ev[2]));
        ms = std::min(ms, ms2);
        if (best == 0 || ms < best_ms) {
          best = cand;
          best_ms = ms;
        }
      }
      GFCC_TRY(umma_error_check(st));   // no choice is kept from launches that gave up
      std::lock_guard<std::mutex> lk(g_tune_mu);
      g_tune[key] = best;
    }
    bn = best;
  }
  return run(bn);
}

namespace {
constexpr int EMU_SMS = 152;
constexpr int EMU_MAX_SPLIT_TILES = 8 * EMU_SMS;   // tiles x K splits of a split product: bounds its partial sums

// Tiling of a fused digit product: tile width, whether A and B change places, K splits.  The model (in
// clocks of an SM) weighs the MMAs of 36 digit pairs, the loads of 16 planes at about 55 bytes a clock,
// the drains and the last step of a tile, over the busiest SM.  It does not depend on the digits kept, so that
// a workspace sized for a shape serves every level.
struct EmuPlan {
  int bn = 64, nz = 1;
  bool swap = false;
};
EmuPlan emu_plan(long long M, long long N, long long K) {
  const long long nk = (K + BK - 1) / BK;
  EmuPlan best;
  double cost = 0.0;
  for (int sw = 0; sw < 2; sw++)
    for (int bn : {64, 32}) {
      const long long rows = sw ? N : M, cols = sw ? M : N;
      const double tiles = (double)((rows + BM - 1) / BM) * (double)((cols + bn - 1) / bn);
      const double kb = std::max(72.0 * bn, (8.0 * EMU_A_BYTES + 8.0 * bn * BK * 2) / 55.0);
      for (long long nz = 1; nz == 1 || (nz <= nk / 4 && tiles * nz <= EMU_MAX_SPLIT_TILES); nz = nz < 8 ? nz + 1 : nz * 5 / 4) {
        const double per = std::ceil((double)nk / nz);
        const double t = std::ceil(tiles * nz / EMU_SMS) * (per * kb + std::ceil(per / 8) * 64.0 * bn + 45.0 * bn + 2500.0) +
                         (nz > 1 ? 4000.0 + 8.0 * 2.0 * nz * M * N / 2500.0 : 0.0);
        if (cost == 0.0 || t < 0.98 * cost) {
          cost = t;
          best.bn = bn;
          best.nz = (int)nz;
          best.swap = sw != 0;
        }
      }
    }
  // every split gets at least one K block
  const long long per = (nk + best.nz - 1) / best.nz;
  best.nz = (int)((nk + per - 1) / per);
  return best;
}

// 3-D K-major BF16 tensor map over digit planes: planes x rows x K, box `planes` x box_rows x 64
int make_plane_map(CUtensorMap *map, const void *base, long long planes, long long rows, long long K, long long ld,
                   long long plane, int box_rows, int box_planes) {
  auto fn = encode_fn();
  if (fn == nullptr) {
    set_error("cuTensorMapEncodeTiled is not available from the driver");
    return GFCC_ERR_CUDA;
  }
  const cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)planes};
  const cuuint64_t strides[2] = {(cuuint64_t)ld * 2, (cuuint64_t)plane * 2};
  const cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)box_rows, (cuuint32_t)box_planes};
  const cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("cuTensorMapEncodeTiled failed (%d) for planes=%lld rows=%lld K=%lld ld=%lld", (int)r, planes, rows, K, ld);
    return GFCC_ERR_ARG;
  }
  return GFCC_OK;
}

template <int BN>
int launch_emu(cudaStream_t st, const CUtensorMap &ma, const CUtensorMap &mb, const EmuArgs &a) {
  static bool attr[64] = {false};
  int dev = 0;
  GFCC_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64 || !attr[dev]) {
    GFCC_CUDA(cudaFuncSetAttribute(umma_emu_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   EmuTile<BN>::SMEM_BYTES));
    if (dev >= 0 && dev < 64) attr[dev] = true;
  }
  const long long tiles = (long long)a.nM * a.nN * a.nz;
  umma_emu_kernel<BN><<<(unsigned)std::min<long long>(tiles, EMU_SMS), EmuTile<BN>::THREADS, EmuTile<BN>::SMEM_BYTES, st>>>(
      ma, mb, a);
  GFCC_LAUNCH_CHECK();
  return GFCC_OK;
}
}  // namespace

// (grows with N: a workspace sized for a shape serves fewer columns too)
long long emu_fused_work_bytes(long long M, long long N, long long K) {
  const long long nk = (K + BK - 1) / BK;
  return std::min<long long>(std::max<long long>(1, nk / 4) * M * N * 8, 8LL * EMU_MAX_SPLIT_TILES * BM * 64) + 256;
}

bool emu_fused_takes(int SA, int SB, int P) {
  return SA >= 1 && SB >= 1 && SA <= EMU_MAXS && SB <= EMU_MAXS && P >= 2 && P <= 9 && P - 1 <= SA && P - 1 <= SB;
}

int emu_gemm_fused(cudaStream_t st, const __nv_bfloat16 *Adig, long long plA, int SA, const int *eA,
                   const __nv_bfloat16 *Bdig, long long plB, int SB, const int *eB, long long ld, int M, int N, int K,
                   int P, int bits, double alpha, double beta, double *C, IMap cm, IMap cn, long long n0,
                   double *work, long long m0, const GuardList *gate) {
  if (M <= 0 || N <= 0) return GFCC_OK;
  if (!emu_fused_takes(SA, SB, P) || bits < 1 || bits > 7 || K <= 0 || (ld % 8) ||
      (reinterpret_cast<uintptr_t>(Adig) & 15) || (reinterpret_cast<uintptr_t>(Bdig) & 15) || (plA % 8) ||
      (plB % 8)) {
    set_error("emu_gemm_fused: unsupported digits (SA=%d SB=%d P=%d bits=%d) or alignment", SA, SB, P, bits);
    return GFCC_ERR_ARG;
  }
  const EmuPlan pl = emu_plan(M, N, K);
  EmuArgs a;
  a.SA = SA; a.SB = SB; a.P = P; a.bits = bits;
  a.M = M; a.N = N;
  a.eA = eA; a.eB = eB;
  a.C = C;
  a.rm = cm; a.cm = cn;
  a.r0g = m0; a.c0g = n0;
  if (pl.swap) {
    std::swap(Adig, Bdig);
    std::swap(plA, plB);
    std::swap(a.SA, a.SB);
    std::swap(a.M, a.N);
    std::swap(a.eA, a.eB);
    std::swap(a.rm, a.cm);
    std::swap(a.r0g, a.c0g);
  }
  a.nM = (a.M + BM - 1) / BM;
  a.nN = (a.N + pl.bn - 1) / pl.bn;
  a.nz = pl.nz;
  a.nk = (K + BK - 1) / BK;
  a.kb_per_split = (a.nk + a.nz - 1) / a.nz;
  // a level holds up to P - 1 pairs: (P - 1) kc 64 products of at most 2^(2 bits - 2) stay within 2^24.  The first of
  // the 7-bit digits of short sums (F64_SHORT_K) may be twice as large: two pairs of a level count twice and the pair of
  // first digits, a level of its own, four times, which 6 blocks allow for P <= 9.
  a.kc = (1 << (26 - 2 * bits)) / (BK * (P - 1));
  static_assert(F64_SHORT_K <= 6 * BK && (9 + 1) * 6 * BK <= 1 << (26 - 2 * F64_BITS), "short sums are exact");
  a.beta = beta;
  int ex = 0;
  const double fr = frexp(alpha, &ex);
  const bool pow2 = fr == 0.5;
  a.alpha_exp = pow2 ? ex - 1 : 0;
  a.alpha_mul = pow2 ? 1.0 : alpha;
  GFCC_TRY(umma_ctl(&a.ctl));
  a.part = a.nz > 1 ? work : nullptr;
  a.gate = gate != nullptr ? gate->count : nullptr;
  a.gate_cap = gate != nullptr ? gate->cap : 0;
  if ((long long)a.nM * a.nN * a.nz > 0x7fffffffLL || a.kc < 1) {
    set_error("emu_gemm_fused: too many tiles (M=%d, N=%d)", M, N);
    return GFCC_ERR_ARG;
  }
  if (a.nz > 1) GFCC_TRY(check_extent_bytes(work, emu_fused_work_bytes(M, N, K), "fused digit GEMM partials"));
  GFCC_TRY(check_extent(C, 0, imap_max(cm, m0 + M) + imap_max(cn, n0 + N), "fused digit GEMM output"));
  CUtensorMap ma, mb;
  GFCC_TRY(make_plane_map(&ma, Adig, a.SA, a.M, K, ld, plA, BM, 1));
  GFCC_TRY(make_plane_map(&mb, Bdig, a.SB, a.N, K, ld, plB, pl.bn, std::min(a.SB, P - 1)));
  GFCC_TRY(pl.bn == 64 ? launch_emu<64>(st, ma, mb, a) : launch_emu<32>(st, ma, mb, a));
  if (a.nz > 1) {
    emu_split_reduce_kernel<<<grid1d((long long)M * N), 256, 0, st>>>(work, a.nz, a.M, a.N, a.eA, a.eB, alpha, beta, C,
                                                                       a.rm, a.cm, a.r0g, a.c0g, a.gate, a.gate_cap);
    GFCC_LAUNCH_CHECK();
  }
  return GFCC_OK;
}

namespace {
// K splits of the sum of magnitudes: few tiles and a long K would leave SMs idle
int guard_splits(long long M, long long N, long long K) {
  const long long bn = N <= 64 ? 64 : (N <= 128 ? 128 : 256), nk = (K + BK - 1) / BK;
  const long long tiles = ((M + BM - 1) / BM) * ((N + bn - 1) / bn);
  return umma_splits((int)K, (int)std::max<long long>(1, std::min<long long>(nk / 4, 2 * EMU_SMS / tiles)));
}

__global__ void guard_sum_kernel(const float *part, int nsplit, int M, int N, GuardArgs g) {
  const long long tot = (long long)M * N;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot; t += (long long)gridDim.x * blockDim.x) {
    float v = 0.0f;
    for (int z = 0; z < nsplit; z++) v += part[z * tot + t];
    if (guard_hit(v, g.theta)) guard_append(g, 1u, (int)(t / N), (int)(t % N));
  }
}

template <int BN>
int launch_guard(cudaStream_t st, const __nv_bfloat16 *A, const __nv_bfloat16 *B, long long ld, int M, int N, int K,
                 int nsplit, int kbs, float *work, const GuardArgs &g) {
  if (nsplit > 1) return launch_umma<BN>(st, A, ld, B, ld, work, N, M, N, K, 1.0f, 0.0f, nsplit, kbs, (long long)M * N);
  if (kbs <= 2) return launch_umma_st<BN, 2, true>(st, A, ld, B, ld, nullptr, 0, M, N, K, 1.0f, 0.0f, 1, kbs, 0, g);
  return launch_umma_st<BN, 0, true>(st, A, ld, B, ld, nullptr, 0, M, N, K, 1.0f, 0.0f, 1, kbs, 0, g);
}
}  // namespace

long long emu_guard_work_bytes(long long M, long long N, long long K) {
  const int nsplit = guard_splits(M, N, K);
  return nsplit > 1 ? 4LL * nsplit * M * N : 0;
}

int emu_guard(cudaStream_t st, const __nv_bfloat16 *A, const __nv_bfloat16 *B, long long ld, int M, int N, int K,
              float theta, const GuardList &list, long long m0, long long n0, float *work) {
  if (M <= 0 || N <= 0) return GFCC_OK;
  if (K <= 0 || (ld % 8) || (reinterpret_cast<uintptr_t>(A) & 15) || (reinterpret_cast<uintptr_t>(B) & 15) ||
      m0 + M > (1LL << 31) - 1 || n0 + N > (1LL << 31) - 1) {
    set_error("emu_guard: unsupported shape or alignment (M=%d N=%d K=%d)", M, N, K);
    return GFCC_ERR_ARG;
  }
  GFCC_TRY(check_extent_bytes(A, (long long)(M - 1) * ld * 2 + (long long)K * 2, "magnitudes A"));
  GFCC_TRY(check_extent_bytes(B, (long long)(N - 1) * ld * 2 + (long long)K * 2, "magnitudes B"));
  const int nsplit = guard_splits(M, N, K), nk = (K + BK - 1) / BK, kbs = (nk + nsplit - 1) / nsplit;
  if (nsplit > 1) GFCC_TRY(check_extent_bytes(work, emu_guard_work_bytes(M, N, K), "partial sums of magnitudes"));
  GuardArgs g;
  g.list = list;
  g.theta = theta;
  g.m0 = (int)m0;
  g.n0 = (int)n0;
  GFCC_TRY(N <= 64    ? launch_guard<64>(st, A, B, ld, M, N, K, nsplit, kbs, work, g)
           : N <= 128 ? launch_guard<128>(st, A, B, ld, M, N, K, nsplit, kbs, work, g)
                      : launch_guard<256>(st, A, B, ld, M, N, K, nsplit, kbs, work, g));
  if (nsplit > 1) {
    guard_sum_kernel<<<grid1d((long long)M * N), 256, 0, st>>>(work, nsplit, M, N, g);
    GFCC_LAUNCH_CHECK();
  }
  return GFCC_OK;
}

void umma_set_autotune(bool on) { g_autotune = on; }

void umma_set_pair_mode(int mode) { g_pair_mode = mode; }
void umma_set_persist_mode(int mode) { g_persist_mode = mode; }

unsigned long long host_wait_limit() { return std::max(2000000000ULL, 60 * g_wait_ns); }

void umma_set_wait(unsigned long long wait_ns, bool skip_loads) {
  g_wait_ns = wait_ns;
  g_skip_loads = skip_loads;
}

int umma_tuned_tile(int M, int N, int K, int nsplit) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  std::lock_guard<std::mutex> lk(g_tune_mu);
  auto it = g_tune.find(std::make_tuple(dev, M, N, K, nsplit));
  return it == g_tune.end() ? 0 : it->second;
}

}  // namespace gfcc
