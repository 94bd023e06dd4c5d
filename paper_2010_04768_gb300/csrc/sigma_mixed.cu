// Mixed-precision IP operator: the off-diagonal part of the sigma product on the BF16 tensor
// cores (FP32 accumulation), the Fock-like diagonal and the frequency shift in FP64.
//
//   sigma(u) = d * u + sigma_off(u),   d_i = -Fbar_ii,  d_ija = Fbar_aa - Fbar_ii - Fbar_jj
//   A u = (omega - i eta) u + sigma(u) = D u + sigma_off(u),   D = omega - i eta + d
//
// With right preconditioning by D (u = x / D) the operator is x + sigma_off(x / D).  The
// diagonal carries the orbital energies (order 1 Hartree); rounding it to BF16 would put an
// error of the size of eta on every resonant system, so it never leaves FP64.  The couplings
// (ring, oooo, ovoo, three-body, off-diagonal Fbar) are small and tolerate BF16 operands:
// the refinement loop recomputes the residual in FP64 and removes their rounding error.
//
// Contractions (all D[m][n] = A[m][k] B[n][k], BF16 K-major, FP32 out):
//   ring  T[(i,a)][(j,c)]  = Wr[(i,a)][(m,e)]   r2b[(j,c)][(m,e)],  r2b = r2[m,j,e]
//   oooo  Q[(i,j)][(a,c)]  = Wq[(i,j)][(m,n)]   r2o[(a,c)][(m,n)],  r2o = r2[m,n,a]
//   3-body, 1h
//         [Z[e]; S1[i]][c] = [V3 | 0; U1x][(m,e,n)|m]  rk[c][(m,e,n)|m]     (split K)
//   ovoo + 3-body
//         U[(i,a,j)][c]    = [W1 | T3][(i,a,j)][m | e]  rz[c][m | e],  rz = [r1 | Z]
#include <cuda_bf16.h>

#include "ctx.cuh"
#include "kernels.cuh"
#include "sigma.cuh"
#include "umma.cuh"
#include "epilogue.cuh"

namespace gfcc {

namespace {

// The BF16 operands only need FP32 accuracy: the vector (and the preconditioner division) is
// handled in FP32 on the FP32 pipe.
struct Cz {
  float r, i;
};

// x times the sign of d (+1 or -1), on the integer units
__device__ __forceinline__ float with_sign(double d, float x) {
  return __int_as_float(__float_as_int(x) ^ (__double2hiint(d) & 0x80000000));
}

__device__ __forceinline__ Cz load_u(const SysBatch &b, int s, long long mu) {
  s = sysv(b, s);
  Cz u;
  if (b.xf != nullptr) {
    const float2 t = reinterpret_cast<const float2 *>(b.xf)[s * b.ldx + mu];
    u = {t.x, t.y};
  } else {
    u = {d2f_trunc(b.x[2 * (s * b.ldx + mu)]), d2f_trunc(b.x[2 * (s * b.ldx + mu) + 1])};
  }
  if (b.diag != nullptr && b.omega != nullptr) {
    const float dr = d2f_trunc(b.omega[s]) + with_sign(b.dsign, d2f_trunc(b.diag[mu]));
    const float di = with_sign(b.zsign, d2f_trunc(b.eta));
    const float inv = 1.0f / (dr * dr + di * di);
    u = {(u.r * dr + u.i * di) * inv, (u.i * dr - u.r * di) * inv};
  }
  return u;
}

// r2[m, j, e] of system s as (re, im); zero on the diagonal m == j
__device__ __forceinline__ Cz r2_at(const SysBatch &b, int o, int v, int s, int m, int j, int e) {
  if (m == j) return {0.0f, 0.0f};
  const long long lo = m < j ? m : j, hi = m < j ? j : m;
  const long long mu = o + pair_index(lo, hi, o) * v + e;
  Cz u = load_u(b, s, mu);
  if (m > j) {
    u.r = -u.r;
    u.i = -u.i;
  }
  return u;
}

// element m of the one-index block of system s into row c = 2 s + re/im of rk (after o2v columns) and r1
__device__ __forceinline__ void put_r1(const SysBatch &b, int s, int m, long long off, long long ldk,
                                       __nv_bfloat16 *rk, long long ld1, __nv_bfloat16 *r1) {
  const Cz u = load_u(b, s, m);
  const __nv_bfloat16 hr = __float2bfloat16(u.r), hi = __float2bfloat16(u.i);
  rk[(long long)(2 * s) * ldk + off + m] = hr;
  rk[(long long)(2 * s + 1) * ldk + off + m] = hi;
  r1[(long long)(2 * s) * ld1 + m] = hr;
  r1[(long long)(2 * s + 1) * ld1 + m] = hi;
}

// r2b[(j, c)][(m, e)] = r2[m, j, e]
__global__ void unpack_ring_kernel(SysBatch b, int o, int v, long long ld, __nv_bfloat16 *out) {
  const int ns = b.nsys;
  const long long K = (long long)o * v;
  const long long tot = (long long)o * 2 * ns * K;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot; t += (long long)gridDim.x * blockDim.x) {
    const long long k = t % K, row = t / K;
    const int c = (int)(row % (2 * ns)), j = (int)(row / (2 * ns));
    const int m = (int)(k / v), e = (int)(k % v);
    const Cz u = r2_at(b, o, v, c >> 1, m, j, e);
    out[row * ld + k] = __float2bfloat16((c & 1) ? u.i : u.r);
  }
}

// r2o[(a, c)][(m, n)] = r2[m, n, a]: a 32 x 32 tile transpose through shared memory (reads
// coalesced along a, writes coalesced along (m, n)).  grid (K/32, v/32, C2), block (32, 8).
__global__ void unpack_oooo_kernel(SysBatch b, int o, int v, long long ld, __nv_bfloat16 *out) {
  __shared__ float tile[32][33];
  const int C2 = 2 * b.nsys;
  const long long K = (long long)o * o;
  const int c = blockIdx.z, s = c >> 1;
  const long long k0 = (long long)blockIdx.x * 32;
  const int a0 = blockIdx.y * 32;
  for (int r = threadIdx.y; r < 32; r += 8) {
    const long long k = k0 + r;
    const int a = a0 + threadIdx.x;
    float val = 0.f;
    if (k < K && a < v) {
      const Cz u = r2_at(b, o, v, s, (int)(k / o), (int)(k % o), a);
      val = (c & 1) ? u.i : u.r;
    }
    tile[r][threadIdx.x] = val;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int a = a0 + r;
    const long long k = k0 + threadIdx.x;
    if (a < v && k < K) out[((long long)a * C2 + c) * ld + k] = __float2bfloat16(tile[threadIdx.x][r]);
  }
}

// rk[c][(m, e, n)] = r2[m, n, e] (tile transpose over (e, n) for fixed m, c: reads coalesced along
// e, writes along n); grid (o/32, v/32, o * C2), block (32, 8)
__global__ void unpack_k_tiled_kernel(SysBatch b, int o, int v, long long ldk, __nv_bfloat16 *rk) {
  __shared__ float tile[32][33];
  const int C2 = 2 * b.nsys;
  const int c = blockIdx.z % C2, m = blockIdx.z / C2, s = c >> 1;
  const int n0 = blockIdx.x * 32, e0 = blockIdx.y * 32;
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int n = n0 + r, e = e0 + threadIdx.x;
    float val = 0.f;
    if (n < o && e < v) {
      const Cz u = r2_at(b, o, v, s, m, n, e);
      val = (c & 1) ? u.i : u.r;
    }
    tile[r][threadIdx.x] = val;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int e = e0 + r, n = n0 + threadIdx.x;
    if (e < v && n < o) rk[(long long)c * ldk + ((long long)m * v + e) * o + n] = __float2bfloat16(tile[threadIdx.x][r]);
  }
}

// A system's vector with the right preconditioner, the uniform parts read once
struct SysIn {
  const float2 *xf;
  const double2 *x;
  const double *diag;
  float om, di, di2, sgn;
  __device__ __forceinline__ SysIn(const SysBatch &b, int s) {
    const int t = sysv(b, s);
    xf = b.xf ? reinterpret_cast<const float2 *>(b.xf) + t * b.ldx : nullptr;
    x = b.xf ? nullptr : reinterpret_cast<const double2 *>(b.x) + t * b.ldx;
    diag = b.omega != nullptr ? b.diag : nullptr;
    om = diag != nullptr ? d2f_trunc(b.omega[t]) : 0.f;
    di = with_sign(b.zsign, d2f_trunc(b.eta));
    di2 = di * di;
    sgn = with_sign(b.dsign, 1.f);
  }
  // counting from element off
  __device__ __forceinline__ void shift(long long off) {
    if (xf != nullptr) xf += off;
    if (x != nullptr) x += off;
    if (diag != nullptr) diag += off;
  }
  __device__ __forceinline__ Cz operator()(int mu) const {
    Cz u;
    if (xf != nullptr) {
      const float2 t = xf[mu];
      u = {t.x, t.y};
    } else {
      const double2 t = x[mu];
      u = {d2f_trunc(t.x), d2f_trunc(t.y)};
    }
    if (diag != nullptr) {
      const float dr = om + sgn * d2f_trunc(diag[mu]);
      const float inv = 1.0f / (dr * dr + di2);
      u = {(u.r * dr + u.i * di) * inv, (u.i * dr - u.r * di) * inv};
    }
    return u;
  }
};

// BF16 pairs of a run of `len` (re, im) values, packed in 32 bits, to the rows re and re + ld (im): stores of
// two values wherever the address is a multiple of four bytes.  pack(i) is value i of the run, odd the parity of re's
// address in values; slot q holds values 2 q - odd and the next, q = 0 .. len / 2.
template <typename Pack>
__device__ __forceinline__ void put_pair(__nv_bfloat16 *re, long long ld, int odd, int len, int q, Pack pack) {
  const int i0 = 2 * q - odd, i1 = i0 + 1;
  const bool in0 = i0 >= 0 && i0 < len, in1 = i1 < len;
  const unsigned u0 = in0 ? pack(i0) : 0u, u1 = in1 ? pack(i1) : 0u;
  const unsigned r = __byte_perm(u0, u1, 0x5410), i = __byte_perm(u0, u1, 0x7632);
  __nv_bfloat16 *p = re + i0;
  if (in0 && in1) {
    *reinterpret_cast<unsigned *>(p) = r;
    *reinterpret_cast<unsigned *>(p + ld) = i;
  } else if (in0) {
    *reinterpret_cast<unsigned short *>(p) = (unsigned short)r;
    *reinterpret_cast<unsigned short *>(p + ld) = (unsigned short)i;
  } else if (in1) {
    *reinterpret_cast<unsigned short *>(p + 1) = (unsigned short)(r >> 16);
    *reinterpret_cast<unsigned short *>(p + ld + 1) = (unsigned short)(i >> 16);
  }
}

__device__ __forceinline__ unsigned pack_bf16(const Cz &u) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(u.r, u.i);
  return *reinterpret_cast<const unsigned *>(&h);
}

// All three 2h1p layouts in one pass.  One block per (e tile, m, system s): the tile r2[m, j, e]
// of system s for every j (each packed element is read by the blocks of its two occupied indices;
// the right preconditioner is applied once per read), rounded to BF16 in shared memory, then
//   ring   r2b[(j, c)][(m, e)]  rows of the tile's e range,
//   oooo   r2o[(e, c)][(m, j)]  rows of o consecutive columns,
//   long K rk[c][(m, e, j)]     one contiguous run of (e range) x o columns,
// for both planes c = 2 s + re/im, two columns a store.  Bound by instructions: 90 us for 40 systems of o=40 v=200 (154 MB
// written); one value a store, an index division for each and conversions on the FP64 pipe took 133 us.
constexpr int UNPACK_ET = 32;   // e values per block (a power of two)
constexpr int UNPACK_MAX_O = 180;   // tile o x (UNPACK_ET + 1) words within the default 48 KB

__global__ __launch_bounds__(256) void unpack_ip_kernel(SysBatch b, int o, int v, long long ld_ov, long long ld_o2,
                                                        long long ld_k1, __nv_bfloat16 *r2b, __nv_bfloat16 *r2o,
                                                        __nv_bfloat16 *rk, long long ld_ot, __nv_bfloat16 *rz) {
  chain_start();
  extern __shared__ unsigned tl[];   // [o][UNPACK_ET + 1] (re, im) in BF16
  constexpr int LD = UNPACK_ET + 1;
  const int e0 = blockIdx.x * UNPACK_ET, m = blockIdx.y, s = blockIdx.z;
  const int et = min(UNPACK_ET, v - e0);
  const int C2 = 2 * b.nsys, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  SysIn in(b, s);
  in.shift(o + e0 + lane);
#pragma unroll 4
  for (int j = warp; j < o; j += 8) {
    unsigned h = 0u;
    if (lane < et && j != m) {
      const int lo = min(m, j), hi = max(m, j);
      h = pack_bf16(in((lo * o - lo * (lo + 1) / 2 + hi - lo - 1) * v));
      if (m > j) h ^= 0x80008000u;
    }
    tl[j * LD + lane] = h;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) put_r1(b, s, m, (long long)o * o * v, ld_k1, rk, ld_ot, rz);
  __syncthreads();
  // ring: rows (j, 2 s + p), columns m v + e0 .. m v + e0 + et, 16 lanes a row (and one value more of an odd start);
  // row strides are even
  {
    const long long col = (long long)m * v + e0;
    const int q = lane & 15, odd = (int)(col & 1);
    __nv_bfloat16 *re = r2b + ((long long)(2 * warp + (lane >> 4)) * C2 + 2 * s) * ld_ov + col;
    for (int j = 2 * warp + (lane >> 4); j < o; j += 16, re += 16LL * C2 * ld_ov) {
      const unsigned *row = tl + j * LD;
      auto pack = [&](int i) { return row[i]; };
      put_pair(re, ld_ov, odd, et, q, pack);
      if (odd && q == 0) put_pair(re, ld_ov, odd, et, 16, pack);
    }
  }
  // oooo: rows (e, 2 s + p), columns m o + j; long K: row 2 s + p, columns (m v + e) o + j.  16 or 32 lanes a row
  const int half = o / 2 + 1 <= 16 ? 1 : 0, q0 = half ? lane & 15 : lane, step = half ? 16 : 32;
  const int el0 = half ? 2 * warp + (lane >> 4) : warp, stride = half ? 16 : 8;
  __nv_bfloat16 *re_k = rk + (long long)(2 * s) * ld_k1 + ((long long)m * v + e0 + el0) * o;
  __nv_bfloat16 *re_o = r2o + ((long long)(e0 + el0) * C2 + 2 * s) * ld_o2 + (long long)m * o;
  const int odd_o = (m * o) & 1;
  int odd_k = (int)((((long long)m * v + e0 + el0) * o) & 1);   // stays: the stride of el is even
  for (int el = el0; el < et; el += stride, re_k += stride * o, re_o += (long long)stride * C2 * ld_o2) {
    const unsigned *col = tl + el;
    auto pack = [&](int j) { return col[j * LD]; };
    for (int q = q0; q <= o / 2; q += step) {
      put_pair(re_o, ld_o2, odd_o, o, q, pack);
      put_pair(re_k, ld_k1, odd_k, o, q, pack);
    }
  }
}

// rk[c][o2v + m] = r1[m] and r1b[c][m] = r1[m] (the general unpacking; unpack_ip_kernel writes them itself)
__global__ void unpack_r1_kernel(SysBatch b, int o, int v, long long ldk, __nv_bfloat16 *rk, long long ld1,
                                 __nv_bfloat16 *r1b) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < b.nsys * o) put_r1(b, t / o, t % o, (long long)o * o * v, ldk, rk, ld1, r1b);
}

// Partial sums part[z][r][c] over the K splits: rows r < nz_rows (the three-body Z) go to zT[c][r] in BF16,
// rows r >= nz_rows (the one-index block) to S1[r - nz_rows][c].  A block adds 32 outputs, eight threads to
// each: with one thread for an output, which walks all splits, it took 14.7 us whatever the size.
__global__ __launch_bounds__(256) void reduce_splits_kernel(const float *part, int nsplit, int rows, int cols,
                                                            int nz_rows, __nv_bfloat16 *zT, long long ldT, float *S1) {
  chain_start();
  __shared__ float sh[8][33];
  const long long tot = (long long)rows * cols;
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  const long long t = (long long)blockIdx.x * 32 + x;
  float s = 0.f;
  if (t < tot) {
#pragma unroll 4
    for (int z = y; z < nsplit; z += 8) s += part[z * tot + t];
  }
  sh[y][x] = s;
  __syncthreads();
  if (y != 0 || t >= tot) return;
#pragma unroll
  for (int k = 1; k < 8; k++) s += sh[k][x];
  const int r = (int)(t / cols), c = (int)(t - (long long)r * cols);
  if (r < nz_rows)
    zT[c * ldT + r] = __float2bfloat16(s);
  else
    S1[(long long)(r - nz_rows) * cols + c] = s;
}

// ---------------------------------------------------------------------------------------- EA
// The ring and long-K layouts of the 2p1h block in one pass: block (e tile, a tile, (m, s)) holds the
// 32 x 32 tile Y[a][e] = y2[m, a, e] of system s (antisymmetric, zero for a == e: packed a < e, read along e above
// the diagonal and along a below it, so that reads stay coalesced), then writes, for both planes,
//   ring   r2e[(a, c)][(m, e)] =  Y[a][e]
//   long K rk[c][(m, a, e)]     = -Y[a][e]  (= y2[m, e, a])
// both along e.  grid (cdiv(v, 32), cdiv(v, 32), o * nsys), block (32, 8).
__global__ void unpack_ea_tile_kernel(SysBatch b, int o, int v, long long Pv, long long ld_ov, long long ldk,
                                      __nv_bfloat16 *r2e, __nv_bfloat16 *rk, long long ld_ot, __nv_bfloat16 *rz) {
  chain_start();
  __shared__ unsigned tile[32][33];   // (re, im) in BF16
  const int e0 = blockIdx.x * 32, a0 = blockIdx.y * 32;
  const int m = (int)(blockIdx.z % (unsigned)o), s = (int)(blockIdx.z / (unsigned)o);
  const int C2 = 2 * b.nsys, lane = threadIdx.x;
  // the 1p block, by the blocks of one (a tile, m)
  if (a0 == 0 && m == 0 && threadIdx.y == 0 && e0 + (int)threadIdx.x < v)
    put_r1(b, s, e0 + threadIdx.x, (long long)o * v * v, ldk, rk, ld_ot, rz);
  const bool below = e0 + 31 < a0;   // every a > e: packed pairs (e, a) run along a
  SysIn in(b, s);
  in.shift(v + (long long)m * Pv);
#pragma unroll
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int a = below ? a0 + lane : a0 + r, e = below ? e0 + r : e0 + lane;
    unsigned h = 0u;
    if (a < v && e < v && a != e) {
      const int lo = min(a, e), hi = max(a, e);
      h = pack_bf16(in((int)((unsigned)lo * (unsigned)(2 * v - lo - 1) / 2) + hi - lo - 1));   // pair_index in 32 bits
      if (a > e) h ^= 0x80008000u;
    }
    if (below)
      tile[lane][r] = h;
    else
      tile[r][lane] = h;
  }
  __syncthreads();
  // both along e, two columns a store: 16 lanes a row (and one value more of an odd start)
  const int et = min(32, v - e0), q = lane & 15;
  for (int r = 2 * threadIdx.y + (lane >> 4); r < 32 && a0 + r < v; r += 16) {
    const long long c1 = (long long)m * v + e0, c2 = ((long long)m * v + a0 + r) * v + e0;
    __nv_bfloat16 *re = r2e + ((long long)(a0 + r) * C2 + 2 * s) * ld_ov + c1, *re_k = rk + (long long)(2 * s) * ldk + c2;
    const int odd1 = (int)(c1 & 1), odd2 = (int)(c2 & 1);
    auto plus = [&](int i) { return tile[r][i]; };
    auto minus = [&](int i) { return tile[r][i] ^ 0x80008000u; };
    put_pair(re, ld_ov, odd1, et, q, plus);
    put_pair(re_k, ldk, odd2, et, q, minus);
    if (q == 0 && odd1) put_pair(re, ld_ov, odd1, et, 16, plus);
    if (q == 0 && odd2) put_pair(re_k, ldk, odd2, et, 16, minus);
  }
}

// r2p[(i, c)][ef] = y2[i, e < f] (row i of the packed 2p1h block), both planes; grid
// (cdiv(Pv, 512), o * nsys)
__global__ __launch_bounds__(256) void unpack_ea_pairs_kernel(SysBatch b, int o, int v, long long Pv, long long ld,
                                                              __nv_bfloat16 *out) {
  chain_start();
  const int i = (int)(blockIdx.y % (unsigned)o), s = (int)(blockIdx.y / (unsigned)o);
  const int ef = 2 * (int)(blockIdx.x * 256 + threadIdx.x);   // two values a thread; rows have room for an even count
  if (ef >= Pv) return;
  SysIn in(b, s);
  in.shift(v + (long long)i * Pv);
  const unsigned u0 = pack_bf16(in(ef)), u1 = ef + 1 < Pv ? pack_bf16(in(ef + 1)) : 0u;
  __nv_bfloat16 *re = out + ((long long)i * 2 * b.nsys + 2 * s) * ld + ef;
  *reinterpret_cast<unsigned *>(re) = __byte_perm(u0, u1, 0x5410);
  *reinterpret_cast<unsigned *>(re + ld) = __byte_perm(u0, u1, 0x7632);
}

constexpr int KSPLIT = 76;   // split of the long-K contraction (Z and the one-index row): two row tiles fill 152 SMs

struct MixedWork {
  __nv_bfloat16 *r2b, *r2o, *rk, *rz;
  float *T, *Q, *U, *Zp, *S1;
  long long bytes;
};

MixedWork layout(const gfcc_ctx *c, int nsys, void *base) {
  const long long o = c->o, v = c->v, C2 = 2LL * nsys;
  MixedWork w;
  unsigned char *p = static_cast<unsigned char *>(base);
  auto take = [&](long long bytes) {
    unsigned char *q = p;
    p += (bytes + 255) / 256 * 256;
    return q;
  };
  w.r2b = reinterpret_cast<__nv_bfloat16 *>(take(o * C2 * c->ld_ov * 2));
  w.r2o = reinterpret_cast<__nv_bfloat16 *>(take(v * C2 * c->ld_o2 * 2));
  w.rk = reinterpret_cast<__nv_bfloat16 *>(take(C2 * c->ld_k1 * 2));
  w.rz = reinterpret_cast<__nv_bfloat16 *>(take(C2 * c->ld_ot * 2));
  w.T = reinterpret_cast<float *>(take(o * v * o * C2 * 4));
  w.Q = reinterpret_cast<float *>(take(o * o * v * C2 * 4));
  w.U = reinterpret_cast<float *>(take(o * v * o * C2 * 4));
  w.Zp = reinterpret_cast<float *>(take(KSPLIT * (v + o) * C2 * 4));
  w.S1 = reinterpret_cast<float *>(take(o * C2 * 4));
  w.bytes = p - static_cast<unsigned char *>(base);
  return w;
}

}  // namespace

struct MixedWorkEA {
  __nv_bfloat16 *r2e, *r2p, *rk, *rz;
  float *T, *Qp, *U, *Zp, *S1;
  long long bytes;
};

MixedWorkEA layout_ea(const gfcc_ctx *c, int nsys, void *base) {
  const long long o = c->o, v = c->v, C2 = 2LL * nsys, Pv = c->Pv, ov2 = o * v * v;
  MixedWorkEA w;
  unsigned char *p = static_cast<unsigned char *>(base);
  auto take = [&](long long bytes) {
    unsigned char *q = p;
    p += (bytes + 255) / 256 * 256;
    return q;
  };
  w.r2e = reinterpret_cast<__nv_bfloat16 *>(take(v * C2 * c->ld_ov * 2));
  w.r2p = reinterpret_cast<__nv_bfloat16 *>(take(o * C2 * c->ld_pv * 2));
  w.rk = reinterpret_cast<__nv_bfloat16 *>(take(C2 * c->ld_k1e * 2));
  w.rz = reinterpret_cast<__nv_bfloat16 *>(take(C2 * c->ld_ot * 2));
  w.T = reinterpret_cast<float *>(take(o * v * v * C2 * 4));
  w.Qp = reinterpret_cast<float *>(take(std::max<long long>(Pv, 1) * o * C2 * 4));
  w.U = reinterpret_cast<float *>(take(ov2 * C2 * 4));
  w.Zp = reinterpret_cast<float *>(take(KSPLIT * (o + v) * C2 * 4));
  w.S1 = reinterpret_cast<float *>(take(v * C2 * 4));
  w.bytes = p - static_cast<unsigned char *>(base);
  return w;
}

long long sigma_mixed_work_doubles(const gfcc_ctx *c, int nsys) {
  long long b = 0;
  if (c->Wr_bf != nullptr) b = std::max(b, layout(c, nsys, nullptr).bytes);
  if (c->Wre_bf != nullptr) b = std::max(b, layout_ea(c, nsys, nullptr).bytes);
  return b / 8 + 64;
}

int apply_ip_mixed(gfcc_ctx *c, const SysBatch &b, double *work) {
  if (c->Wr_bf == nullptr) {
    set_error("mixed-precision sigma requested but the context was created in FP64");
    return GFCC_ERR_STATE;
  }
  cudaStream_t st = c->stream;
  const long long o = c->o, v = c->v, ov = o * v, oo = o * o, o2v = oo * v, C2 = 2LL * b.nsys;
  MixedWork w = layout(c, b.nsys, work);
  PhaseTimer tsig(c, PH_SIGMA, b.nsys * sigma_flops(c, GFCC_SECTOR_IP));
  {
  PhaseTimer tu(c, PH_UNPACK);
  if (v > 0 && o <= UNPACK_MAX_O) {
    const size_t sm = (size_t)o * (UNPACK_ET + 1) * sizeof(unsigned);
    GFCC_CUDA(launch_chained(unpack_ip_kernel, dim3(cdiv(v, UNPACK_ET), (unsigned)o, (unsigned)b.nsys), 256, sm, st, 
        b, (int)o, (int)v, c->ld_ov, c->ld_o2, c->ld_k1, w.r2b, w.r2o, w.rk, c->ld_ot, w.rz));
    GFCC_LAUNCH_CHECK();
  } else {
    unpack_ring_kernel<<<grid1d(o * C2 * ov), 256, 0, st>>>(b, (int)o, (int)v, c->ld_ov, w.r2b);
    GFCC_LAUNCH_CHECK();
    unpack_oooo_kernel<<<dim3(cdiv(oo, 32), cdiv(v, 32), C2), dim3(32, 8), 0, st>>>(b, (int)o, (int)v, c->ld_o2,
                                                                                     w.r2o);
    GFCC_LAUNCH_CHECK();
    unpack_k_tiled_kernel<<<dim3(cdiv(o, 32), cdiv(v, 32), o * C2), dim3(32, 8), 0, st>>>(b, (int)o, (int)v,
                                                                                          c->ld_k1, w.rk);
    GFCC_LAUNCH_CHECK();
    unpack_r1_kernel<<<cdiv(b.nsys * o, 128), 128, 0, st>>>(b, (int)o, (int)v, c->ld_k1, w.rk, c->ld_ot, w.rz);
    GFCC_LAUNCH_CHECK();
  }
  }
  {
    PhaseTimer tr(c, PH_RING_BF16, 2.0 * (double)ov * (double)ov * (double)(o * C2));
    GFCC_TRY(gemm_bf16_tn(st, c->Wr_bf, c->ld_ov, w.r2b, c->ld_ov, w.T, o * C2, (int)ov, (int)(o * C2), (int)ov, 1.0f,
                          0.0f));
  }
  {
    PhaseTimer tob(c, PH_BF16_OTHER, 2.0 * C2 * ((double)oo * oo * v + (double)v * o2v + (double)o2v * (o + v) +
                                                 (double)o * (o2v + o)));
    GFCC_TRY(gemm_bf16_tn(st, c->Wq_bf, c->ld_o2, w.r2o, c->ld_o2, w.Q, v * C2, (int)oo, (int)(v * C2), (int)oo, 1.0f,
                          0.0f));
    // three-body Z and the 1h row in one product (split K); Z -> BF16 transposed into rz[c][o + e]; then
    // U = [W1 | T3] [r1 | Z]
    const int zs = umma_splits((int)(o2v + o), KSPLIT);
    GFCC_TRY(gemm_bf16_tn(st, c->VU_bf, c->ld_k1, w.rk, c->ld_k1, w.Zp, C2, (int)(v + o), (int)C2, (int)(o2v + o), 1.0f,
                          0.0f, zs, (v + o) * C2));
    GFCC_CUDA(launch_chained(reduce_splits_kernel, cdiv((v + o) * C2, 32), 256, 0, st, w.Zp, zs, (int)(v + o), (int)C2, (int)v, w.rz + o,
                                                                 c->ld_ot, w.S1));
    GFCC_LAUNCH_CHECK();
    GFCC_TRY(gemm_bf16_tn(st, c->WT_bf, c->ld_ot, w.rz, c->ld_ot, w.U, C2, (int)o2v, (int)C2, (int)(o + v), 1.0f,
                          0.0f));
  }
  {
    PhaseTimer tp(c, PH_EPILOGUE, 4.0 * C2 * (3.0 * o2v + o) + (b.xf ? 16.0 : 32.0) * b.nsys * c->dim_ip);
    GFCC_TRY((epi::launch_ip<float, epi::MODE_OFFDIAG>(st, b, (int)o, (int)v, w.S1, w.T, w.Q, w.U, c->diag_ip)));
  }
  return GFCC_OK;
}


int apply_ea_mixed(gfcc_ctx *c, const SysBatch &b, double *work) {
  if (c->Wre_bf == nullptr) {
    set_error("mixed-precision EA sigma requested but its BF16 operands were not built");
    return GFCC_ERR_STATE;
  }
  cudaStream_t st = c->stream;
  const long long o = c->o, v = c->v, ov = o * v, ov2 = ov * v, C2 = 2LL * b.nsys, Pv = c->Pv;
  MixedWorkEA w = layout_ea(c, b.nsys, work);
  PhaseTimer tsig(c, PH_SIGMA, b.nsys * sigma_flops(c, GFCC_SECTOR_EA));
  {
    PhaseTimer tu(c, PH_UNPACK);
    GFCC_CUDA(launch_chained(unpack_ea_tile_kernel, dim3(cdiv(v, 32), cdiv(v, 32), (unsigned)(o * b.nsys)), dim3(32, 8), 0, st, 
        b, (int)o, (int)v, Pv, c->ld_ov, c->ld_k1e, w.r2e, w.rk, c->ld_ot, w.rz));
    GFCC_LAUNCH_CHECK();
    if (Pv > 0) {
      GFCC_CUDA(launch_chained(unpack_ea_pairs_kernel, dim3(cdiv(Pv, 512), (unsigned)(o * b.nsys)), 256, 0, st, b, (int)o, (int)v, Pv,
                                                                                        c->ld_pv, w.r2p));
      GFCC_LAUNCH_CHECK();
    }
  }
  // T[(i,b)][(a,c)] = Wr_ea[(i,b)][(m,e)] y2[m,a,e]
  {
    PhaseTimer tr(c, PH_RING_BF16, 2.0 * (double)ov * (double)ov * (double)(v * C2));
    GFCC_TRY(gemm_bf16_tn(st, c->Wre_bf, c->ld_ov, w.r2e, c->ld_ov, w.T, v * C2, (int)ov, (int)(v * C2), (int)ov, 1.0f,
                          0.0f));
  }
  // Qp[(a<b)][(i,c)] = Wp[(ab)][(ef)] y2[i,e,f]
  if (Pv > 0) {
    PhaseTimer tv(c, PH_VVVV, 2.0 * (double)Pv * (double)Pv * (double)(o * C2));
    GFCC_TRY(gemm_bf16_tn(st, c->Wp_bf, c->ld_pv, w.r2p, c->ld_pv, w.Qp, o * C2, (int)Pv, (int)(o * C2), (int)Pv,
                          1.0f, 0.0f));
  }
  {
    PhaseTimer tob(c, PH_BF16_OTHER, 2.0 * C2 * ((double)o * ov2 + (double)ov2 * (v + o) + (double)v * (ov2 + v)));
    // Z[m][c] = V3e[m][(n,f,e)] y2[n,e,f] (into rz[c][v + m]) and the 1p row [U1e | Fvv off-diagonal][a] . [y2 | y1](c)
    // in one product (split K); then U[(i,b,a)][c] = [W3 | T3e] [y1 | Z]
    const int zs = umma_splits((int)(ov2 + v), KSPLIT);
    GFCC_TRY(gemm_bf16_tn(st, c->VUe_bf, c->ld_k1e, w.rk, c->ld_k1e, w.Zp, C2, (int)(o + v), (int)C2, (int)(ov2 + v),
                          1.0f, 0.0f, zs, (o + v) * C2));
    GFCC_CUDA(launch_chained(reduce_splits_kernel, cdiv((o + v) * C2, 32), 256, 0, st, w.Zp, zs, (int)(o + v), (int)C2, (int)o, w.rz + v,
                                                                 c->ld_ot, w.S1));
    GFCC_LAUNCH_CHECK();
    GFCC_TRY(gemm_bf16_tn(st, c->WTe_bf, c->ld_ot, w.rz, c->ld_ot, w.U, C2, (int)ov2, (int)C2, (int)(v + o), 1.0f,
                          0.0f));
  }
  {
    PhaseTimer tp(c, PH_EPILOGUE, 4.0 * C2 * (2.0 * ov2 + (double)Pv * o + v) + (b.xf ? 16.0 : 32.0) * b.nsys * c->dim_ea);
    GFCC_TRY((epi::launch_ea<float, epi::MODE_OFFDIAG>(st, b, (int)o, (int)v, Pv, w.S1, w.T, w.Qp, w.U,
                                                       c->diag_ea)));
  }
  return GFCC_OK;
}

}  // namespace gfcc
