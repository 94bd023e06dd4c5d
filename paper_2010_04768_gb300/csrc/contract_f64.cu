// Generic strided FP64 tensor contraction on CUDA cores (DFMA).
//
//   C(m, n) = alpha * sum_k A(m, k) B(k, n) + beta * C(m, n),   batched over blockIdx.z
//
// Each GEMM index may fuse two tensor indices through an IMap, so the setup of the
// Hbar elements and the FP64 sigma product are written as plain contractions
// without explicit transposes.  GB300 has about 1.26 TFLOP/s of FP64 (two FMA per SM and clock), so
// the FP64 pipe bounds every tile, padding included: 16 x 16 x 16 products already keep an SM busy for
// 2048 clocks, long enough to hide the next K block's loads behind them.  What is left to gain is the
// balance over the SMs: small tiles, tile shapes that follow M and N, and the K range of a tile
// shared by a cluster.  Measured against one shape (64 x 64 tiles, single-buffered, a 64-bit division per
// element and index), with plain launches: sigma product of one vector at o=4 v=12 600 -> 107 us, the tiny workload's
// IP + EA solve 71 -> 13 ms, o=13 v=67 IP + EA 278 -> 74 ms (ring contraction at 1.11 TFLOP/s, 0.88 of the pipe), the
// Green's-function overlaps of 40 systems at o=40 v=200 4.0 -> 0.5 ms.  With chained launches, the last K step's padding
// skipped and the solver's shorter steps these take 63 us, 8 ms and 65 ms.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>

#include "common.cuh"

#include "kernels.cuh"
#include "ozaki.cuh"

namespace gfcc {

namespace cg = cooperative_groups;

namespace {

constexpr int BK = 16, KSTEP = 4, NT = 256;
constexpr int NUM_SM = 152;

// x / d by 32-bit division where both fit (the 64-bit one costs several times as many instructions)
__device__ __forceinline__ long long fast_div(long long x, long long d) {
  if ((((unsigned long long)x | (unsigned long long)d) >> 32) == 0) return (long long)((unsigned)x / (unsigned)d);
  return x / d;
}

__device__ __forceinline__ long long map_offset(const IMap &m, long long x) {
  if (m.d0 <= 0) return x * m.s0;
  const long long q = fast_div(x, m.d0);
  return (x - q * m.d0) * m.s0 + q * m.s1;
}

// A fused K index walked in steps of BK without a division per step: x = q d0 + r.
struct KWalk {
  long long d0, r, off, step, wrap;
  int dr;
  __device__ __forceinline__ void init(const IMap &m, long long x) {
    if (m.d0 <= 0) {
      d0 = 1LL << 62;
      r = x;
      off = x * m.s0;
      dr = BK;
      step = BK * m.s0;
      wrap = 0;
      return;
    }
    d0 = m.d0;
    const long long q = fast_div(x, d0), dq = fast_div(BK, d0);
    r = x - q * d0;
    off = r * m.s0 + q * m.s1;
    dr = (int)(BK - dq * d0);
    step = dr * m.s0 + dq * m.s1;
    wrap = m.s1 - d0 * m.s0;
  }
  __device__ __forceinline__ void next() {
    r += dr;
    off += step;
    if (r >= d0) {
      r -= d0;
      off += wrap;
    }
  }
};

// One BM x BN output tile per block, BM = TM RM and BN = (NT / TM) RN: thread (ty, tx) holds outputs
// (ty + TM i, tx + TN j).  The K loop is double-buffered: the next K block is on its way from global
// memory while this one is multiplied.  A cluster of gridDim.z / batch blocks (along z) may share
// the K range of a tile; its partial sums meet through distributed shared memory in rank order.
template <int TM, int RM, int RN>
__device__ __forceinline__ void contract_tile(const Contract &c, int kcluster, long long m0, long long n0) {
  constexpr int TN = NT / TM, BM = TM * RM, BN = TN * RN;
  constexpr int LA = (BM * BK + NT - 1) / NT, LB = (BN * BK + NT - 1) / NT;
  __shared__ double As[2][BK][BM + 1];
  __shared__ double Bs[2][BK][BN + 1];
  __shared__ double red[BM * BN];
  const int tx = threadIdx.x % TN, ty = threadIdx.x / TN;
  const long long b = blockIdx.z / c.nsplit;
  const long long z = blockIdx.z - b * c.nsplit;
  const double *A = c.A + b * c.sab;
  const double *B = c.B + b * c.sbb;
  double *C = c.C + b * c.scb + (kcluster > 1 ? 0 : z * c.scz);
  const long long kbeg = z * c.kchunk;
  const long long kend = min(c.K, kbeg + c.kchunk);

  // this thread's elements of the A and B tiles: lanes run along K where K is the contiguous index
  // of the operand, else along M (N)
  const bool a_k = c.ak.s0 == 1, b_k = c.bk.s0 == 1;
  int am[LA], akl[LA], bn[LB], bkl[LB];
  bool aok[LA], bok[LB];
  const double *ap[LA], *bp[LB];
  KWalk aw[LA], bw[LB];
#pragma unroll
  for (int r = 0; r < LA; r++) {
    const int e = threadIdx.x + NT * r;
    am[r] = a_k ? e / BK : e % BM;
    akl[r] = a_k ? e % BK : e / BM;
    aok[r] = e < BM * BK && m0 + am[r] < c.M;
    ap[r] = A + (aok[r] ? map_offset(c.am, m0 + am[r]) : 0);
    aw[r].init(c.ak, kbeg + akl[r]);
  }
#pragma unroll
  for (int r = 0; r < LB; r++) {
    const int e = threadIdx.x + NT * r;
    bn[r] = b_k ? e / BK : e % BN;
    bkl[r] = b_k ? e % BK : e / BN;
    bok[r] = e < BN * BK && n0 + bn[r] < c.N;
    bp[r] = B + (bok[r] ? map_offset(c.bn, n0 + bn[r]) : 0);
    bw[r].init(c.bk, kbeg + bkl[r]);
  }
  double va[LA], vb[LB];
  auto fetch = [&](long long k0) {
#pragma unroll
    for (int r = 0; r < LA; r++) {
      va[r] = (aok[r] && k0 + akl[r] < kend) ? ap[r][aw[r].off] : 0.0;
      aw[r].next();
    }
#pragma unroll
    for (int r = 0; r < LB; r++) {
      vb[r] = (bok[r] && k0 + bkl[r] < kend) ? bp[r][bw[r].off] : 0.0;
      bw[r].next();
    }
  };
  auto stage = [&](int buf) {
#pragma unroll
    for (int r = 0; r < LA; r++)
      if (BM * BK % NT == 0 || threadIdx.x + NT * r < BM * BK) As[buf][akl[r]][am[r]] = va[r];
#pragma unroll
    for (int r = 0; r < LB; r++)
      if (BN * BK % NT == 0 || threadIdx.x + NT * r < BN * BK) Bs[buf][bkl[r]][bn[r]] = vb[r];
  };
  double acc[RM][RN];
#pragma unroll
  for (int i = 0; i < RM; i++)
#pragma unroll
    for (int j = 0; j < RN; j++) acc[i][j] = 0.0;

  if (kbeg < kend) {
    fetch(kbeg);
    stage(0);
  }
  __syncthreads();
  int buf = 0;
  for (long long k0 = kbeg; k0 < kend; k0 += BK, buf ^= 1) {
    const bool more = k0 + BK < kend;
    if (more) fetch(k0 + BK);
    // the last step multiplies no more than its K values, to a multiple of four
    const int left = (int)min((long long)BK, kend - k0);
#pragma unroll
    for (int k4 = 0; k4 < BK; k4 += KSTEP) {
      if (k4 >= left) break;
#pragma unroll
      for (int kk = k4; kk < k4 + KSTEP; kk++) {
        double a[RM], bb[RN];
#pragma unroll
        for (int i = 0; i < RM; i++) a[i] = As[buf][kk][ty + TM * i];
#pragma unroll
        for (int j = 0; j < RN; j++) bb[j] = Bs[buf][kk][tx + TN * j];
#pragma unroll
        for (int i = 0; i < RM; i++)
#pragma unroll
          for (int j = 0; j < RN; j++) acc[i][j] = fma(a[i], bb[j], acc[i][j]);
      }
    }
    if (more) stage(buf ^ 1);
    __syncthreads();
  }
  auto store = [&](int ml, int nl, double v) {
    const long long m = m0 + ml, n = n0 + nl;
    if (m >= c.M || n >= c.N) return;
    const long long off = map_offset(c.cm, m) + map_offset(c.cn, n);
    double val = c.alpha * v;
    if (c.beta != 0.0) val += c.beta * C[off];
    C[off] = val;
  };
  if (kcluster > 1) {
    cg::cluster_group cl = cg::this_cluster();
#pragma unroll
    for (int i = 0; i < RM; i++)
#pragma unroll
      for (int j = 0; j < RN; j++) red[(ty + TM * i) * BN + tx + TN * j] = acc[i][j];
    cl.sync();
    // block z of the cluster adds up and stores its share of the tile
    const int share = (BM * BN + kcluster - 1) / kcluster;
    const int e1 = min(BM * BN, ((int)z + 1) * share);
    for (int e = (int)z * share + threadIdx.x; e < e1; e += NT) {
      double s = 0.0;
      for (int r = 0; r < kcluster; r++) s += cl.map_shared_rank(red, r)[e];
      store(e / BN, e % BN, s);
    }
    cl.sync();   // no block leaves while another reads its partial sums
    return;
  }
#pragma unroll
  for (int i = 0; i < RM; i++)
#pragma unroll
    for (int j = 0; j < RN; j++) store(ty + TM * i, tx + TN * j, acc[i][j]);
}

template <int TM, int RM, int RN>
__global__ __launch_bounds__(NT) void contract_f64_kernel(Contract c, int kcluster) {
  chain_start();
  contract_tile<TM, RM, RN>(c, kcluster, (long long)blockIdx.x * TM * RM, (long long)blockIdx.y * (NT / TM) * RN);
}

// One launch for both ends of a guarded digit-plane product: blocks of one wave store the listed values, or walk the
// 32 x 32 tiles if the list has overflowed (a block for each of 40 000 tiles took 30 us to find that it has not).
constexpr int LISTED_BLOCKS = NUM_SM * 4;
__global__ __launch_bounds__(NT) void contract_listed_kernel(Contract c, GuardList list, long long mt, long long tiles) {
  const unsigned count = *list.count;
  if (count <= list.cap) {
    for (unsigned i = blockIdx.x * NT + threadIdx.x; i < count; i += gridDim.x * NT)
      c.C[map_offset(c.cm, list.at[i].x) + map_offset(c.cn, list.at[i].y)] = list.value[i];
    return;
  }
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
    contract_tile<16, 2, 2>(c, 1, t % mt * 32, t / mt * 32);
    __syncthreads();
  }
}

struct Tiling {
  int bm, bn, kcluster;
};

// The FP64 pipe (two FMA per SM and clock) bounds every tile: a tile takes bm bn K / 2 clocks of an
// SM, padding included, so the best tiling is the one whose busiest SM has the fewest of them.
// Candidates: 32 x 32 tiles, and tiles of 256 outputs from 64 x 4 to 4 x 64 (no more than 1 output per
// thread, hence a few per cent slower on large products), each with the K range shared by up to 8 blocks.
Tiling choose_tiling(long long M, long long N, long long K, long long batch, bool cluster) {
  static const int shape[6][2] = {{32, 32}, {16, 16}, {64, 4}, {32, 8}, {8, 32}, {4, 64}};
  Tiling best{16, 16, 1};
  double cost = 0.0;
  for (const auto &s : shape) {
    const double tiles = (double)((M + s[0] - 1) / s[0]) * (double)((N + s[1] - 1) / s[1]) * (double)batch;
    if ((N + s[1] - 1) / s[1] > 65535) continue;
    for (int S = 1; S <= (cluster ? 8 : 1); S *= 2) {
      if (S > 1 && K < 2 * BK * S) break;
      const double ks = S == 1 ? std::ceil((double)K / KSTEP) * KSTEP : std::ceil(std::ceil((double)K / S) / BK) * BK;
      const double t = std::ceil(tiles * S / NUM_SM) * (ks * s[0] * s[1] / 2.0 * (s[0] == 32 && s[1] == 32 ? 1.0 : 1.04) +
                                                        1000.0 + (S > 1 ? 1500.0 : 0.0));
      if (cost == 0.0 || t < cost) {
        cost = t;
        best = Tiling{s[0], s[1], S};
      }
    }
  }
  return best;
}

template <int TM, int RM, int RN>
int launch_contract(const Contract &c, int kcluster, long long mt, long long nt, cudaStream_t st) {
  dim3 grid((unsigned)mt, (unsigned)nt, (unsigned)(c.batch * c.nsplit));
  if (kcluster <= 1) {
    GFCC_CUDA(launch_chained(contract_f64_kernel<TM, RM, RN>, grid, dim3(NT), 0, st, c, 1));
  } else {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(NT);
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // as launch_chained
    at[1].val.programmaticStreamSerializationAllowed = 1;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = (unsigned)kcluster;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    GFCC_CUDA(cudaLaunchKernelEx(&cfg, contract_f64_kernel<TM, RM, RN>, c, kcluster));
  }
  GFCC_LAUNCH_CHECK();
  return GFCC_OK;
}
}  // namespace

int contract_f64(const Contract &c, cudaStream_t st) {
  if (c.M <= 0 || c.N <= 0 || c.batch <= 0) return GFCC_OK;
  // K == 0 leaves acc = 0, so C = beta * C (the empty sum).
  Contract cc = c;
  if (cc.nsplit < 1) cc.nsplit = 1;
  if (cc.nsplit == 1) cc.kchunk = cc.K > 0 ? cc.K : 1;
  if (cc.kchunk < 1 || cc.kchunk * cc.nsplit < cc.K) {
    set_error("contract_f64: split-K chunk %lld x %lld does not cover K=%lld", cc.kchunk, cc.nsplit, cc.K);
    return GFCC_ERR_ARG;
  }
  Tiling t = choose_tiling(cc.M, cc.N, cc.nsplit > 1 ? cc.kchunk : cc.K, cc.batch * cc.nsplit, cc.nsplit == 1);
  const long long mt = (c.M + t.bm - 1) / t.bm, nt = (c.N + t.bn - 1) / t.bn;
  if (mt > 0x7fffffffLL || nt > 65535 || c.batch * cc.nsplit * t.kcluster > 65535) {
    if (t.kcluster > 1 && c.batch * cc.nsplit <= 65535) {
      t.kcluster = 1;
    } else {
      set_error("contract_f64: grid too large (M=%lld N=%lld batch=%lld)", c.M, c.N, c.batch);
      return GFCC_ERR_ARG;
    }
  }
  {
    const long long ka = imap_max(c.am, c.M) + imap_max(c.ak, c.K) + (c.batch - 1) * c.sab;
    const long long kb = imap_max(c.bk, c.K) + imap_max(c.bn, c.N) + (c.batch - 1) * c.sbb;
    const long long kc = imap_max(c.cm, c.M) + imap_max(c.cn, c.N) + (c.batch - 1) * c.scb + (cc.nsplit - 1) * cc.scz;
    if (c.K > 0) {
      GFCC_TRY(check_extent(c.A, 0, ka, "contraction operand A"));
      GFCC_TRY(check_extent(c.B, 0, kb, "contraction operand B"));
    }
    GFCC_TRY(check_extent(c.C, 0, kc, "contraction output C"));
  }
  if (t.kcluster > 1) {
    // whole K blocks per cluster block; every block of the cluster gets a (possibly empty) range
    cc.nsplit = t.kcluster;
    cc.kchunk = (((cc.K + t.kcluster - 1) / t.kcluster) + BK - 1) / BK * BK;
    cc.scz = 0;
  }
  if (t.bm == 32 && t.bn == 32) return launch_contract<16, 2, 2>(cc, t.kcluster, mt, nt, st);
  if (t.bm == 64) return launch_contract<64, 1, 1>(cc, t.kcluster, mt, nt, st);
  if (t.bm == 32) return launch_contract<32, 1, 1>(cc, t.kcluster, mt, nt, st);
  if (t.bm == 8) return launch_contract<8, 1, 1>(cc, t.kcluster, mt, nt, st);
  if (t.bm == 4) return launch_contract<4, 1, 1>(cc, t.kcluster, mt, nt, st);
  return launch_contract<16, 1, 1>(cc, t.kcluster, mt, nt, st);
}

int contract_listed(const Contract &c, const GuardList &list, cudaStream_t st) {
  Contract cc = c;
  cc.nsplit = 1;
  cc.kchunk = cc.K;
  const long long mt = (c.M + 31) / 32, tiles = mt * ((c.N + 31) / 32);
  const long long ka = imap_max(c.am, c.M) + imap_max(c.ak, c.K), kb = imap_max(c.bk, c.K) + imap_max(c.bn, c.N);
  GFCC_TRY(check_extent(c.A, 0, ka, "contraction operand A"));
  GFCC_TRY(check_extent(c.B, 0, kb, "contraction operand B"));
  GFCC_TRY(check_extent(c.C, 0, imap_max(c.cm, c.M) + imap_max(c.cn, c.N), "contraction output C"));
  contract_listed_kernel<<<(unsigned)std::min<long long>(tiles, LISTED_BLOCKS), NT, 0, st>>>(cc, list, mt, tiles);
  GFCC_LAUNCH_CHECK();
  return GFCC_OK;
}

namespace {
// C = alpha * sum_z part[z] + beta * C
__global__ void splitk_reduce_kernel(const double *part, int nsplit, long long M, long long N, double alpha, double beta,
                                     double *C, IMap cm, IMap cn) {
  const long long tot = M * N;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot; t += (long long)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int z = 0; z < nsplit; z++) s += part[z * tot + t];
    const long long m = t / N, n = t - m * N;
    const long long off = imap_apply(cm, m) + imap_apply(cn, n);
    C[off] = alpha * s + (beta != 0.0 ? beta * C[off] : 0.0);
  }
}

// split-K partial sums, one buffer per stream (work on a stream is ordered, so a buffer is never
// shared by concurrent contractions)
struct SplitBuf {
  double *p = nullptr;
  long long cap = 0;
};
std::mutex g_splitk_mu;
std::map<cudaStream_t, SplitBuf> g_splitk;
}  // namespace

thread_local bool g_emulate_big = false;
constexpr double EMULATE_MIN_FLOPS_DEFAULT = 4e12;
double g_emulate_min_flops = EMULATE_MIN_FLOPS_DEFAULT;
thread_local double g_emulate_min_flops_local = -1.0;

int gemm_f64(cudaStream_t st, long long M, long long N, long long K, double alpha,
             const double *A, IMap am, IMap ak, const double *B, IMap bk, IMap bn, double beta,
             double *C, IMap cm, IMap cn, long long batch, long long sab, long long sbb, long long scb) {
  Contract c;
  c.A = A; c.B = B; c.C = C;
  c.M = M; c.N = N; c.K = K;
  c.am = am; c.ak = ak; c.bk = bk; c.bn = bn; c.cm = cm; c.cn = cn;
  c.batch = batch; c.sab = sab; c.sbb = sbb; c.scb = scb;
  c.alpha = alpha; c.beta = beta;
  // Contractions whose owner allows it (mixed-precision set-up, emulated CCSD, closed-shell operator) run on
  // the tensor cores from digit planes: all of at least emu_min flops, and the smaller ones where the planes are faster
  // (unless the threshold was raised above its default), these with the outputs that 56 bits below the largest entries
  // do not serve summed in FP64.  Without room for the planes the FP64 units do it.
  const double emu_min = g_emulate_min_flops_local >= 0.0 ? g_emulate_min_flops_local : g_emulate_min_flops;
  const bool large = 2.0 * (double)M * (double)N * (double)K >= emu_min;
  if (batch == 1 && K > 0 && g_emulate_big &&
      (large || (g_emulate_min_flops <= EMULATE_MIN_FLOPS_DEFAULT && emulation_pays(M, N, K, false)))) {
    const int s = gemm_f64_emulated(st, M, N, K, alpha, A, am, ak, B, bk, bn, beta, C, cm, cn, !large);
    if (s != GFCC_ERR_OOM) return s;
  }
  // A few 16 x 16 output tiles and a long K: the K ranges of a cluster (8 at most) would not fill the
  // SMs, so K is split further into partial sums in global memory.
  const long long tiles = ((M + 15) / 16) * ((N + 15) / 16);
  if (batch == 1 && tiles * 8 < 2 * NUM_SM && K >= 8192) {
    long long nsplit = std::min<long long>(4 * NUM_SM / tiles, K / 512);
    nsplit = std::min<long long>(nsplit, 512);
    if (nsplit >= 2) {
      const long long need = nsplit * M * N;
      double *buf = nullptr;
      {
        std::lock_guard<std::mutex> lk(g_splitk_mu);
        SplitBuf &sb = g_splitk[st];
        if (need > sb.cap) {
          if (sb.p) dfree(sb.p);   // cudaFree synchronises: earlier work on the buffer is done
          sb.p = nullptr;
          sb.cap = 0;
          if (dmalloc((void **)&sb.p, sizeof(double) * need) != cudaSuccess) {
            cudaGetLastError();
            set_error("gemm_f64: cannot allocate %lld doubles of split-K workspace", need);
            return GFCC_ERR_OOM;
          }
          sb.cap = need;
        }
        buf = sb.p;
      }
      Contract p = c;
      p.C = buf;
      p.cm = imap1(N);
      p.cn = imap1(1);
      p.alpha = 1.0;
      p.beta = 0.0;
      p.nsplit = nsplit;
      p.kchunk = (K + nsplit - 1) / nsplit;
      p.scz = M * N;
      GFCC_TRY(contract_f64(p, st));
      splitk_reduce_kernel<<<grid1d(M * N), 256, 0, st>>>(buf, (int)nsplit, M, N, alpha, beta, C, cm, cn);
      GFCC_LAUNCH_CHECK();
      return GFCC_OK;
    }
  }
  return contract_f64(c, st);
}

}  // namespace gfcc
