// Tiled epilogues of the batched sigma product: antisymmetrise the contraction outputs, add the
// shift of eq. xplin and pack into y[s][mu].
//
// The contraction outputs are column-major in the systems (the planar column c = 2 s + re/im is
// the fastest index: T[(i,a)][(j,c)], Q[(i,j)][(a,c)], U[(i,a,j)][c] for IP; T[(i,b)][(a,c)],
// Qp[(a<b)][(i,c)], U[(i,b,a)][c] for EA), while y is row-major in the systems.  A block therefore
// handles a run of consecutive packed elements of one (i<j) pair (IP) or one i (EA): it reads the
// contraction outputs along c (coalesced), stages sigma in shared memory, and writes y along mu
// (coalesced).
//
// MODE_FULL: the outputs contain the whole operator (FP64 and FP64-accurate products):
//   IP y = z u + sigma(u), EA y = z u - sigma(u), u = x / D_s (right preconditioner) or x;
//   without omega y = sigma(x).
// MODE_OFFDIAG: the outputs contain the couplings only (BF16 products); the Fock-like diagonal d
//   is applied here in FP64: IP y = x + sigma_off(u) (preconditioned), (z + d) x + sigma_off(x);
//   EA y = x - sigma_off(u), (z - d) x - sigma_off(x); without omega y = d x + sigma_off(x).
#pragma once
#include <algorithm>

#include "sigma.cuh"

namespace gfcc {
namespace epi {

constexpr int MODE_FULL = 0, MODE_OFFDIAG = 1;
constexpr int THREADS = 256;

template <typename TIn>
constexpr int run_len() {
  return sizeof(TIn) == 4 ? 16 : 8;   // packed elements per block
}
// outputs a thread gathers at a time (four loads each in flight)
template <typename TIn>
constexpr int UNROLL = sizeof(TIn) == 4 ? 3 : 2;
// systems per launch: the shared tile run_len x (ns + 1) pairs stays below 33 KB
template <typename TIn>
constexpr int max_systems() {
  return 256;
}

__device__ __forceinline__ void load_x(const SysBatch &b, int s, long long mu, double &xr, double &xi) {
  s = sysv(b, s);
  if (b.xf != nullptr) {
    const float2 t = reinterpret_cast<const float2 *>(b.xf)[s * b.ldx + mu];
    xr = t.x;
    xi = t.y;
  } else {
    const double2 t = reinterpret_cast<const double2 *>(b.x)[s * b.ldx + mu];
    xr = t.x;
    xi = t.y;
  }
}

__device__ __forceinline__ void store_y(const SysBatch &b, int s, long long mu, double yr, double yi) {
  if (!sys_stores(b, s)) return;
  s = sysv(b, s);
  if (b.yf != nullptr)
    reinterpret_cast<float2 *>(b.yf)[s * b.ldy + mu] = make_float2((float)yr, (float)yi);
  else
    reinterpret_cast<double2 *>(b.y)[s * b.ldy + mu] = make_double2(yr, yi);
}

// sgn = +1 IP, -1 EA; diag = the operator's Fock-like diagonal (MODE_OFFDIAG)
template <int MODE, typename TIn>
__device__ __forceinline__ void combine(const SysBatch &b, int s, long long mu, TIn tr, TIn ti, const double *diag,
                                        double sgn) {
  if constexpr (MODE == MODE_OFFDIAG && sizeof(TIn) == 4) {
    // the preconditioned inner operator on FP32 vectors, y = x +/- sigma_off: one FP32 addition (eight
    // conversions and additions on the FP64 pipe instead held the epilogue to a third of the memory rate)
    if (b.xf != nullptr && b.diag != nullptr && b.omega != nullptr) {
      if (!sys_stores(b, s)) return;
      const long long v = sysv(b, s);
      const float2 x = reinterpret_cast<const float2 *>(b.xf)[v * b.ldx + mu];
      const float f = (float)sgn;
      reinterpret_cast<float2 *>(b.yf)[v * b.ldy + mu] = make_float2(fmaf(f, tr, x.x), fmaf(f, ti, x.y));
      return;
    }
  }
  const double sr = tr, si = ti;
  double xr, xi;
  load_x(b, s, mu, xr, xi);
  double yr, yi;
  if (MODE == MODE_FULL) {
    if (b.omega == nullptr) {
      yr = sr;
      yi = si;
    } else {
      double ur = xr, ui = xi;
      if (b.diag != nullptr) {
        const double dr = b.omega[sysv(b, s)] + b.dsign * b.diag[mu], di = b.zsign * b.eta;
        const double d2 = dr * dr + di * di;
        ur = (xr * dr + xi * di) / d2;
        ui = (xi * dr - xr * di) / d2;
      }
      const double zr = b.omega[sysv(b, s)], zi = b.zsign * b.eta;
      yr = zr * ur - zi * ui + sgn * sr;
      yi = zr * ui + zi * ur + sgn * si;
    }
  } else {
    const double d = diag[mu];
    if (b.omega == nullptr) {
      yr = d * xr + sr;
      yi = d * xi + si;
    } else if (b.diag != nullptr) {
      yr = xr + sgn * sr;
      yi = xi + sgn * si;
    } else {
      const double dr = b.omega[sysv(b, s)] + sgn * d, di = b.zsign * b.eta;
      yr = dr * xr - di * xi + sgn * sr;
      yi = dr * xi + di * xr + sgn * si;
    }
  }
  store_y(b, s, mu, yr, yi);
}

template <typename TIn>
struct Pair;
template <>
struct Pair<float> {
  using type = float2;
};
template <>
struct Pair<double> {
  using type = double2;
};

// the one-index block (IP 1h: n1 = o, sgn +1; EA 1p: n1 = v, sgn -1): S1[m][c], by the blocks past the first
// `first` of the grid's x dimension
template <typename TIn, int MODE>
__device__ __forceinline__ void one_index(const SysBatch &b, int n1, long long C2, const TIn *S1, const double *diag,
                                          double sgn, int s0, int ns, int first) {
  if (blockIdx.y != 0) return;
  const int tot = n1 * ns;
  for (int t = (blockIdx.x - first) * THREADS + threadIdx.x; t < tot; t += (gridDim.x - first) * THREADS) {
    const int s = t / n1, m = t - s * n1;
    const typename Pair<TIn>::type v = reinterpret_cast<const typename Pair<TIn>::type *>(S1 + m * C2)[s0 + s];
    combine<MODE, TIn>(b, s0 + s, m, v.x, v.y, diag, sgn);
  }
}

// IP 2h1p block: one block per (pair p = (i<j), run of a); grid (Po + blocks of the 1h part, cdiv(v, run)),
// dynamic shared memory run * (ns + 1) * 2 sizeof(TIn).  A thread handles both planes of a system.  Bound by the
// latency of its gathers: 19 us for 30 systems of o=27 v=133 in FP32 (31 us with one output at a time and the pair
// decoded by an FP64 square root in every thread).
template <typename TIn, int MODE>
__global__ __launch_bounds__(THREADS) void ip2_kernel(SysBatch b, int o, int v, long long C2, int s0, int ns, int Po,
                                                       const TIn *T, const TIn *Q, const TIn *U, const TIn *S1,
                                                       const double *diag) {
  chain_start();
  using P2 = typename Pair<TIn>::type;
  extern __shared__ __align__(16) unsigned char smem[];
  P2 *tile = reinterpret_cast<P2 *>(smem);
  constexpr int A = run_len<TIn>();
  if ((int)blockIdx.x >= Po) {
    one_index<TIn, MODE>(b, o, C2, S1, diag, 1.0, s0, ns, Po);
    return;
  }
  const long long p = blockIdx.x;
  const int a0 = blockIdx.y * A;
  long long i, j;
  pair_decode(p, o, i, j);
  const int ld = ns + 1, na = min(A, v - a0);
  // run a0 + al of the rows (i, a, j), (j, a, i), (i, j, a)
  const P2 *Tij = reinterpret_cast<const P2 *>(T + ((i * v + a0) * o + j) * C2) + s0;
  const P2 *Tji = reinterpret_cast<const P2 *>(T + ((j * v + a0) * o + i) * C2) + s0;
  const P2 *Qij = reinterpret_cast<const P2 *>(Q + ((i * o + j) * v + a0) * C2) + s0;
  const P2 *Uij = reinterpret_cast<const P2 *>(U + ((i * v + a0) * o + j) * C2) + s0;
  const long long row_o = o * (C2 / 2), row_1 = C2 / 2;
  for (int t0 = threadIdx.x; t0 < na * ns; t0 += UNROLL<TIn> * THREADS) {
    P2 tij[UNROLL<TIn>], tji[UNROLL<TIn>], q[UNROLL<TIn>], u[UNROLL<TIn>];
    int at[UNROLL<TIn>];
#pragma unroll
    for (int w = 0; w < UNROLL<TIn>; w++) {
      const int t = t0 + w * THREADS, al = t / ns, s = t - al * ns;
      at[w] = al * ld + s;
      if (t >= na * ns) break;
      tij[w] = Tij[al * row_o + s];
      tji[w] = Tji[al * row_o + s];
      q[w] = Qij[al * row_1 + s];
      u[w] = Uij[al * row_o + s];
    }
#pragma unroll
    for (int w = 0; w < UNROLL<TIn>; w++) {
      if (t0 + w * THREADS >= na * ns) break;
      P2 r;
      r.x = tij[w].x - tji[w].x + q[w].x + u[w].x;
      r.y = tij[w].y - tji[w].y + q[w].y + u[w].y;
      tile[at[w]] = r;
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < A * ns; t += THREADS) {
    const int s = t / A, al = t - s * A;
    if (al >= na) continue;
    const P2 r = tile[al * ld + s];
    combine<MODE, TIn>(b, s0 + s, o + p * v + a0 + al, r.x, r.y, diag, 1.0);
  }
}

// EA 2p1h block: one block per (i, run of pairs a<b); grid (o + blocks of the 1p part, cdiv(Pv, run))
template <typename TIn, int MODE>
__global__ __launch_bounds__(THREADS) void ea2_kernel(SysBatch b, int o, int v, long long Pv, long long C2, int s0,
                                                       int ns, const TIn *T, const TIn *Qp, const TIn *U, const TIn *S1,
                                                       const double *diag) {
  chain_start();
  using P2 = typename Pair<TIn>::type;
  extern __shared__ __align__(16) unsigned char smem[];
  P2 *tile = reinterpret_cast<P2 *>(smem);
  constexpr int A = run_len<TIn>();
  __shared__ int pa[A], pb[A];   // the block's pairs (a < b), decoded once
  if ((int)blockIdx.x >= o) {
    one_index<TIn, MODE>(b, v, C2, S1, diag, -1.0, s0, ns, o);
    return;
  }
  const long long i = blockIdx.x;
  const long long ab0 = (long long)blockIdx.y * A;
  if (threadIdx.x < A && ab0 + threadIdx.x < Pv) {
    long long a, bb;
    pair_decode(ab0 + threadIdx.x, v, a, bb);
    pa[threadIdx.x] = (int)a;
    pb[threadIdx.x] = (int)bb;
  }
  __syncthreads();
  const int ld = ns + 1, na = (int)min((long long)A, Pv - ab0);
  const long long row = C2 / 2;
  const P2 *Ti = reinterpret_cast<const P2 *>(T + i * v * v * C2) + s0;
  const P2 *Ui = reinterpret_cast<const P2 *>(U + i * v * v * C2) + s0;
  const P2 *Qi = reinterpret_cast<const P2 *>(Qp + (ab0 * o + i) * C2) + s0;
  for (int t0 = threadIdx.x; t0 < na * ns; t0 += UNROLL<TIn> * THREADS) {
    P2 tba[UNROLL<TIn>], tab[UNROLL<TIn>], q[UNROLL<TIn>], u[UNROLL<TIn>];
    int at[UNROLL<TIn>];
#pragma unroll
    for (int w = 0; w < UNROLL<TIn>; w++) {
      const int t = t0 + w * THREADS, al = t / ns, s = t - al * ns;
      if (t >= na * ns) break;
      const int a = pa[al], bb = pb[al];
      at[w] = al * ld + s;
      tba[w] = Ti[((long long)bb * v + a) * row + s];
      tab[w] = Ti[((long long)a * v + bb) * row + s];
      q[w] = Qi[(long long)al * o * row + s];
      u[w] = Ui[((long long)bb * v + a) * row + s];
    }
#pragma unroll
    for (int w = 0; w < UNROLL<TIn>; w++) {
      if (t0 + w * THREADS >= na * ns) break;
      P2 r;
      r.x = tba[w].x - tab[w].x + q[w].x + u[w].x;
      r.y = tba[w].y - tab[w].y + q[w].y + u[w].y;
      tile[at[w]] = r;
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < A * ns; t += THREADS) {
    const int s = t / A, al = t - s * A;
    if (al >= na) continue;
    const P2 r = tile[al * ld + s];
    combine<MODE, TIn>(b, s0 + s, v + i * Pv + ab0 + al, r.x, r.y, diag, -1.0);
  }
}

// blocks for the one-index block of n1 entries of ns systems
static inline int one_index_blocks(int n1, int ns) { return (int)cdiv((long long)n1 * ns, THREADS); }

template <typename TIn, int MODE>
int launch_ip(cudaStream_t st, const SysBatch &b, int o, int v, const TIn *S1, const TIn *T, const TIn *Q,
              const TIn *U, const double *diag) {
  const long long C2 = 2LL * b.nsys, Po = v > 0 ? (long long)o * (o - 1) / 2 : 0;
  constexpr int A = run_len<TIn>();
  for (int s0 = 0; s0 < b.nsys; s0 += max_systems<TIn>()) {
    const int ns = b.nsys - s0 < max_systems<TIn>() ? b.nsys - s0 : max_systems<TIn>();
    const size_t sm = (size_t)A * (ns + 1) * 2 * sizeof(TIn);
    GFCC_CUDA(launch_chained(ip2_kernel<TIn, MODE>, dim3((unsigned)Po + one_index_blocks(o, ns), std::max(1u, cdiv(v, A))), THREADS, sm, st, 
        b, o, v, C2, s0, ns, (int)Po, T, Q, U, S1, diag));
    GFCC_LAUNCH_CHECK();
  }
  return GFCC_OK;
}

template <typename TIn, int MODE>
int launch_ea(cudaStream_t st, const SysBatch &b, int o, int v, long long Pv, const TIn *S1, const TIn *T,
              const TIn *Qp, const TIn *U, const double *diag) {
  const long long C2 = 2LL * b.nsys;
  constexpr int A = run_len<TIn>();
  for (int s0 = 0; s0 < b.nsys; s0 += max_systems<TIn>()) {
    const int ns = b.nsys - s0 < max_systems<TIn>() ? b.nsys - s0 : max_systems<TIn>();
    const size_t sm = (size_t)A * (ns + 1) * 2 * sizeof(TIn);
    GFCC_CUDA(launch_chained(ea2_kernel<TIn, MODE>, dim3((unsigned)o + one_index_blocks(v, ns), std::max(1u, cdiv(Pv, A))), THREADS, sm, st, 
        b, o, v, Pv, C2, s0, ns, T, Qp, U, S1, diag));
    GFCC_LAUNCH_CHECK();
  }
  return GFCC_OK;
}

}  // namespace epi
}  // namespace gfcc
