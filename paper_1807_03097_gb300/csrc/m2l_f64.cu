// M2L of the FP64 form with kept coupling matrices (a6, Sec. 4.2: acc_t(f, i) = sum_s sum_j
// G(x_ti, x_sj) u_s(f, j)), as exact integer products on the FP16 tensor cores.
//
// Why: GB300 issues one FP64 FMA warp instruction per 72 clocks and scheduler, so the 16 FMAs of an
// entry (4 complex fields) bound the product at 22 times the time that HBM needs to deliver the
// matrices.  Here every matrix entry and every folded source field is a fixed-point number of
// six 10-bit digits.  A digit is exact in FP16, a product of two digits has at most 18 bits, and
// the tensor core's FP32 accumulators hold the sums of 16 nodes (real and imaginary part)
// exactly; they go into 64-bit integers, which are rounded to FP64 once per target node.
//
// Fixed point.  w = rint(v 2^(58 - e)) with 2^e above the largest |Re|, |Im| (matrices: per target
// cluster, from the smallest node distance of its far list; sources: per tree level and field,
// found in every product); u = w + O, O = sum_k 512 1024^k, has the unsigned digits d_k, so that
// w = sum_k c_k 1024^k with c_k = d_k - 512 in [-512, 511] (the leading one in [-257, 256]).
// Digit products are summed by total weight: diagonal D holds c_k c'_l with (5 - k) + (5 - l) = D,
// D <= 5 (21 of 36 products; the rest is below 2^-57 of the largest product).  Sums over 16 nodes
// x 2 parts stay below 2^24 for D <= 3 (D = 3 in two accumulators), hence exact; a rounding of D = 4, 5
// is below 2^-58.  The product differs from the one with evaluated FP64 entries by 5.9e-16 (relative
// 2-norm, sphere of 1 536 elements, 81 nodes; the FP64 pipe's sums over kept matrices by 8.0e-16).
//
// Bound: HBM delivers the words (two FP64 a complex entry, rows padded to 16); beside it a
// scheduler spends about 64 clocks per 32 entries on products and digits.  Measured, M2L before (FP64 pipe,
// kept matrices) and after: 52.7 -> 3.5 ms at 125 760 pairs of 81 nodes (15.1 GB, 4.5 TB/s of 6.7), 163 -> 8.2 ms
// at 121 nodes, 6.95 -> 0.36 ms at 49, 1.55 -> 0.034 ms at 5 472 pairs of 25 (few targets: the K-steps
// of a target are split over blocks), 0.26 -> 0.041 ms at 4 nodes, where 12 of 16 rows are padding.
//
// Layout of the kept matrices: per target cluster, 16 source nodes (a K-step) x 16 target
// nodes (a row tile) at a time, the words of one A fragment of mma.m16n8k16 per lane.  A fragment
// register is a pair of entries (source nodes 2 q, 2 q + 1 of one row); its 2 x 6 digits take four
// 32-bit words: the low 10 bits of each half are the digits 5, 4, 3, 2, the high 6 bits hold digits
// 1 and 0 in pieces (6 + 4 bits).  So an entry keeps its 16 bytes, a warp reads 512 contiguous
// bytes per load, and a digit becomes FP16 by one mask-and-or (0x6400 | d is 1024 + d) and one
// packed subtraction (two more shifts for digits 1, 0).
#include <algorithm>
#include <cmath>
#include <cuda_fp16.h>

#include "efie_internal.h"

namespace efie {

namespace {

constexpr unsigned long long kOffset = 512ull * 0x0004010040100401ull;  // 512 sum_k 2^(10 k), k < 6
constexpr int kFixBits = 58;
constexpr int kF64Nodes = 64;  // source nodes staged at a time

struct LevOff {
  int off[12];
};

__device__ __forceinline__ int level_of(const LevOff &L, int m, int id) {
  int l = 0;
  while (l < m && id >= L.off[l + 1]) ++l;
  return l;
}

__device__ __forceinline__ unsigned long long fix(double v, int e) {
  return (unsigned long long)__double2ll_rn(scalbn(v, kFixBits - e)) + kOffset;
}

// four words of a pair of entries (x in the low halves)
__device__ __forceinline__ uint4 pack_pair(unsigned long long x, unsigned long long y) {
  auto half4 = [](unsigned long long u, unsigned *h) {
    const unsigned d0 = u & 1023, d1 = (u >> 10) & 1023;
    h[0] = (unsigned)((u >> 50) & 1023) | ((d1 >> 4) << 10);
    h[1] = (unsigned)((u >> 40) & 1023) | ((d1 & 15) << 12);
    h[2] = (unsigned)((u >> 30) & 1023) | ((d0 >> 4) << 10);
    h[3] = (unsigned)((u >> 20) & 1023) | ((d0 & 15) << 12);
  };
  unsigned a[4], b[4];
  half4(x, a);
  half4(y, b);
  return make_uint4(a[0] | (b[0] << 16), a[1] | (b[1] << 16), a[2] | (b[2] << 16), a[3] | (b[3] << 16));
}

// digit K (5 leading) of a pair as FP16 c_K
template <int K>
__device__ __forceinline__ unsigned digit(const uint4 &w) {
  unsigned d;
  if (K == 5) d = (w.x & 0x03ff03ffu) | 0x64006400u;
  if (K == 4) d = (w.y & 0x03ff03ffu) | 0x64006400u;
  if (K == 3) d = (w.z & 0x03ff03ffu) | 0x64006400u;
  if (K == 2) d = (w.w & 0x03ff03ffu) | 0x64006400u;
  if (K == 1) d = ((w.x >> 6) & 0x03f003f0u) | (((w.y >> 12) & 0x000f000fu) | 0x64006400u);
  if (K == 0) d = ((w.z >> 6) & 0x03f003f0u) | (((w.w >> 12) & 0x000f000fu) | 0x64006400u);
  const __half2 h = __hsub2(*reinterpret_cast<__half2 *>(&d), __float2half2_rn(1536.f));
  return *reinterpret_cast<const unsigned *>(&h);
}

__device__ __forceinline__ void mma_f16(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint4 ld_stream(const uint4 *p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// products of digit K of the entries with the digits of the sources, b[2 l], b[2 l + 1] = digit 5 - l
template <int K>
__device__ __forceinline__ void digit_products(float (&D)[7][4], const uint4 (&w)[4], const unsigned (&b)[12]) {
  const unsigned a[4] = {digit<K>(w[0]), digit<K>(w[1]), digit<K>(w[2]), digit<K>(w[3])};
#pragma unroll
  for (int l = 0; l <= K; ++l) {
    const int d = (5 - K) + l;
    // D = 3 in two accumulators (index 3: products with a leading digit, 6: the others)
    mma_f16(D[d == 3 && K != 5 && l != 0 ? 6 : d], a, b[2 * l], b[2 * l + 1]);
  }
}

}  // namespace

// Exponent e with 2^e >= 1.001 / (4 pi r) for every node distance r of a target's far list.  Distances are taken in
// FP32 from offsets to the cluster centres (81 nodes: 0.2 of the 29 ms of k_K_digits, which FP64 would take again)
// and once more in FP64 from the coordinates where FP32 may not resolve them: a centre distance whose square
// leaves its range, or nodes 1e3 times closer than the centres.  A list with a distance whose square FP64
// does not hold (or is 0) gets kBadExponent.
constexpr int kBadExponent = 1 << 20;
__global__ void k_K_exponent(const int *__restrict__ targets, const int *__restrict__ fptr, const int *__restrict__ fsrc,
                             int nI, const double *__restrict__ center, const float *__restrict__ nodeXf,
                             const double *__restrict__ nodeX, int *__restrict__ expo) {
  __shared__ double red[128];
  const int t = targets[blockIdx.x];
  double least = INFINITY;
  for (int k = fptr[t]; k < fptr[t + 1]; ++k) {
    const int s = fsrc[k];
    const double e0 = center[4 * t] - center[4 * s], e1 = center[4 * t + 1] - center[4 * s + 1],
                 e2 = center[4 * t + 2] - center[4 * s + 2];
    const float d0 = (float)e0, d1 = (float)e1, d2 = (float)e2, far = fmaxf(fabsf(d0), fmaxf(fabsf(d1), fabsf(d2)));
    const bool in_range = far > 0x1p-40f && far < 0x1p40f;
    float lo = 3e38f;
    if (in_range)
      for (int i = threadIdx.x; i < nI * nI; i += blockDim.x) {
        const float *a = nodeXf + ((size_t)t * nI + i / nI) * 3, *b = nodeXf + ((size_t)s * nI + i % nI) * 3;
        const float x = d0 + a[0] - b[0], y = d1 + a[1] - b[1], z = d2 + a[2] - b[2];
        lo = fminf(lo, x * x + y * y + z * z);
      }
    if (in_range && lo > 1e-6f * far * far) {
      least = fmin(least, (double)lo);
      continue;
    }
    for (int i = threadIdx.x; i < nI * nI; i += blockDim.x) {
      const double *a = nodeX + ((size_t)t * nI + i / nI) * 3, *b = nodeX + ((size_t)s * nI + i % nI) * 3;
      const double x = a[0] - b[0], y = a[1] - b[1], z = a[2] - b[2], r2 = x * x + y * y + z * z;
      least = r2 < INFINITY ? fmin(least, r2) : 0.0;  // an infinity or NaN: not representable
    }
  }
  red[threadIdx.x] = least;
  __syncthreads();
  for (int s = 64; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) red[threadIdx.x] = fmin(red[threadIdx.x], red[threadIdx.x + s]);
    __syncthreads();
  }
  if (threadIdx.x == 0)
    expo[t] = red[0] > 0.0 && red[0] < INFINITY ? ilogb(1.001 * 0.25 / (M_PI * sqrt(red[0]))) + 1 : kBadExponent;
}

constexpr int kCircle = 256;  // points e^{2 pi i n / kCircle} of the table

__global__ void k_circle(double2 *tab) {
  double sn, cs;
  sincospi(2.0 * threadIdx.x / kCircle, &sn, &cs);
  tab[threadIdx.x] = make_double2(cs, sn);
}

// v 2^(kFixBits - e) rounded to an integer (half away from zero), |v| < 2^e, by shifts of v's mantissa
__device__ __forceinline__ unsigned long long fix_shift(double v, int e) {
  const long long b = __double_as_longlong(v);
  const int ex = (int)((b >> 52) & 0x7ff), sh = ex - 1075 + kFixBits - e;
  const unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | (ex ? 1ull << 52 : 0ull);
  const unsigned long long u = sh >= 0 ? m << sh : (sh < -60 ? 0ull : (m + (1ull << (-sh - 1))) >> -sh);
  return (b < 0 ? 0ull - u : u) + kOffset;
}

// G = e^{i kappa r} / (4 pi r) from r^2 with 30 FP64 operations (the FP64 pipe takes 72 clocks an instruction and
// scheduler and bounds k_K_digits; with sqrt, division, sincos and conversions to integers the kernel took
// 55 ms for 62 880 unordered pairs of 81 nodes, now 29; assembly of the 1 536-element sphere 121.6 -> 95.3 ms).
// 1 / r: FP32 reciprocal root of the upper 23 mantissa bits, one step of the third-order iteration (relative error
// 2^-21 -> 2^-60); r = r^2 / r with one Newton correction.  e^{i x}: table lookup and Taylor polynomials of the
// remainder (Tang's table-driven method): x = n 2 pi / 256 + t, |t| <= 0.0123, two-constant reduction; sin t to
// t^5, cos t to t^6 (next terms 2^-57, 2^-66).
__device__ __forceinline__ double2 green(double r2, double kappa, const double2 *__restrict__ tab) {
  const long long b = __double_as_longlong(r2);
  const int ex = (int)(b >> 52);  // r2 = m 2^(ex - 1023); even power: f = m 2^odd in [1, 4), r2 = f 4^h
  if (ex < 200 || ex > 1800) {    // lengths beyond 1e-120 ... 1e120: the library's functions
    const double r = sqrt(r2), f = 0.25 / (M_PI * r);
    double sn, cs;
    sincos(kappa * r, &sn, &cs);
    return make_double2(f * cs, f * sn);
  }
  const int odd = (ex + 1) & 1, h = (ex - 1023 - odd) / 2;
  const float f = __int_as_float(((127 + odd) << 23) | (int)((b >> 29) & 0x7fffff));
  const int yb = __float_as_int(rsqrtf(f));  // in (1/2, 1]
  const double y0 = __longlong_as_double(((long long)((yb >> 23) - 127 + 1023 - h) << 52) | ((long long)(yb & 0x7fffff) << 29));
  const double t0 = r2 * y0, e = fma(-t0, y0, 1.0);
  const double y = fma(e * y0, fma(0.375, e, 0.5), y0);  // 1 / r
  const double ra = r2 * y, r = fma(0.5 * y, fma(-ra, ra, r2), ra);
  const double x = kappa * r, g = y * (0.25 / M_PI);
  if (!(x < 1e9)) {
    double sn, cs;
    sincos(x, &sn, &cs);
    return make_double2(g * cs, g * sn);
  }
  const double shifter = 6755399441055744.0;  // 1.5 2^52: the integer in the low bits
  const double ns = fma(x, kCircle / (2.0 * M_PI), shifter), n = ns - shifter;
  const double p1 = 2.0 * M_PI / kCircle, p2 = 2.4492935982947064e-16 / kCircle;  // 2 pi = fl(2 pi) + 2.449e-16
  const double t = fma(-n, p2, fma(-n, p1, x));
  const double2 cs = tab[(int)__double_as_longlong(ns) & (kCircle - 1)];
  const double t2 = t * t;
  const double st = fma(t * t2, fma(t2, 1.0 / 120, -1.0 / 6), t);                  // sin t
  const double ct = t2 * fma(t2, fma(t2, -1.0 / 720, 1.0 / 24), -0.5);             // cos t - 1
  return make_double2(g * (cs.x + fma(cs.x, ct, -cs.y * st)), g * (cs.y + fma(cs.y, ct, cs.x * st)));
}

// One block per unordered admissible pair {t, s}: G is symmetric, so every entry is evaluated once
// and written into both clusters' matrices.  A thread owns 2 x 2 entries (nodes 2 a, 2 a + 1 of t, 2 b,
// 2 b + 1 of s; the node count padded to an even nIe), i.e. two fragment words of either side.
__global__ void __launch_bounds__(128) k_K_digits(int ncl, const int *__restrict__ optr, const int *__restrict__ osrc,
                                                  const int *__restrict__ fptr, const int *__restrict__ fsrc,
                                                  const size_t *__restrict__ koff, const int *__restrict__ expo, int nI,
                                                  double kappa, const double *__restrict__ nodeX,
                                                  const double2 *__restrict__ circle, uint4 *__restrict__ K) {
  extern __shared__ double sx[];  // [2][nI][3]
  __shared__ double2 tab[kCircle];
  __shared__ int sh[4];
  const int u = blockIdx.x, tid = threadIdx.x;
  if (tid == 0) {
    int lo = 0, hi = ncl;  // the owner: optr[lo] <= u < optr[lo + 1]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (optr[mid] <= u) lo = mid; else hi = mid;
    }
    sh[0] = lo;
    sh[1] = osrc[u];
  }
  __syncthreads();
  const int cl[2] = {sh[0], sh[1]};
  for (int i = tid; i < kCircle; i += blockDim.x) tab[i] = circle[i];
  for (int side = 0; side < 2; ++side)
    for (int k = fptr[cl[side]] + tid; k < fptr[cl[side] + 1]; k += blockDim.x)
      if (fsrc[k] == cl[1 - side]) sh[2 + side] = k - fptr[cl[side]];
  for (int i = tid; i < 6 * nI; i += blockDim.x) sx[i] = nodeX[(size_t)cl[i / (3 * nI)] * 3 * nI + i % (3 * nI)];
  __syncthreads();
  const int nIe = (nI + 1) & ~1, nP = nIe >> 1, ntile = (nI + 15) >> 4;
  const int e0 = expo[cl[0]], e1 = expo[cl[1]];
  for (int idx = tid; idx < nP * nP; idx += blockDim.x) {
    const int a = idx / nP, b = idx % nP;
    double g[2][2][2];  // [node of t][node of s][re, im]
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const double *x = sx + 3 * min(2 * a + i, nI - 1), *y = sx + 3 * (nI + min(2 * b + j, nI - 1));
        const double dx = x[0] - y[0], dy = x[1] - y[1], dz = x[2] - y[2];
        const double2 v = green(dx * dx + dy * dy + dz * dz, kappa, tab);
        g[i][j][0] = v.x;
        g[i][j][1] = v.y;
      }
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const int e = side == 0 ? e0 : e1;
      const int J = sh[2 + side] * nIe + 2 * (side == 0 ? b : a), kk = J & 15;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int row = 2 * (side == 0 ? a : b) + i;
        if (row >= nI) continue;
        const int lane = 4 * (row & 7) + ((kk & 7) >> 1), reg = ((row >> 3) & 1) + 2 * (kk >> 3);
        uint4 *o = K + (((koff[cl[side]] + (J >> 4)) * ntile + (row >> 4)) * 8 + reg) * 32 + lane;
#pragma unroll
        for (int part = 0; part < 2; ++part) {
          const double x = side == 0 ? g[i][0][part] : g[0][i][part], y = side == 0 ? g[i][1][part] : g[1][i][part];
          __stcs(o + part * 128, pack_pair(fix_shift(x, e), fix_shift(y, e)));
        }
      }
    }
  }
}

// exponent e with 2^e above v (bit pattern); v = 0: any
__device__ __forceinline__ int max_exponent(unsigned long long v) { return (int)(v >> 52) - 1022; }

// fixed-point sources, node-major: fx[(cluster nI + node) 8 + 2 f + {re, im}]
__global__ void k_src_fix(long long tot, int nI, int m, LevOff L, const double2 *__restrict__ src,
                          const unsigned long long *__restrict__ smax, ulonglong2 *__restrict__ fx) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= tot) return;
  const int f = (int)(t & 3);
  const long long node = t >> 2;
  const int id = (int)(node / nI), i = (int)(node - (long long)id * nI);
  const int e = max_exponent(smax[4 * level_of(L, m, id) + f]);
  const double2 v = src[((size_t)id * 4 + f) * nI + i];
  fx[t] = make_ulonglong2(fix(v.x, e), fix(v.y, e));
}

// One block per (target cluster, split of its K-steps), one warp per row tile of 16 target nodes.
// 64 source nodes at a time are staged as B fragments (digits of (Re, Im) of the 4 fields on the 8
// columns, and of (-Im, Re) for the imaginary part of the entries); a warp streams its tile's
// words from HBM, the next four loads in flight during the 21 products of the present ones.
template <int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) k_m2l_f64_digits(
    const int *__restrict__ targets, const int *__restrict__ fptr, const int *__restrict__ fsrc,
    const size_t *__restrict__ koff, const int *__restrict__ expo, int nI, int m, LevOff L,
    const uint4 *__restrict__ K, const unsigned long long *__restrict__ fx,
    const unsigned long long *__restrict__ smax, double2 *__restrict__ acc, double2 *__restrict__ more, size_t slab) {
  __shared__ uint4 sB[kF64Nodes / 16][2][3][32];  // [step][part][digits 5 4, 3 2, 1 0][lane]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, ntile = blockDim.x >> 5;
  const int t = targets[blockIdx.x], k0 = fptr[t], nIe = (nI + 1) & ~1;
  const int total = (fptr[t + 1] - k0) * nIe, nch = (total + kF64Nodes - 1) / kF64Nodes, nst = (total + 15) >> 4;
  const int c0 = (int)((long long)nch * blockIdx.y / gridDim.y), c1 = (int)((long long)nch * (blockIdx.y + 1) / gridDim.y);
  const uint4 *Kt = K + ((koff[t] * ntile + warp) * 8) * 32 + lane;
  const size_t step = (size_t)ntile * 256;
  const int st1 = min(4 * c1, nst);
  long long hi[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0};
  uint4 nx[4];
  if (c0 < c1)
#pragma unroll
    for (int i = 0; i < 4; ++i) nx[i] = ld_stream(Kt + (size_t)(4 * c0) * step + 32 * i);
  for (int c = c0; c < c1; ++c) {
    __syncthreads();
    // four (node, column) a thread at a time, their loads in flight together
    for (int n0 = threadIdx.x; n0 < 8 * kF64Nodes; n0 += 4 * blockDim.x) {
      unsigned long long u4[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int n = n0 + v * blockDim.x, J = c * kF64Nodes + (n >> 3);
        u4[v] = kOffset;
        if (n < 8 * kF64Nodes && J < total) {
          const int k = J / nIe, i = J - k * nIe;
          if (i < nI) u4[v] = fx[((size_t)fsrc[k0 + k] * nI + i) * 8 + (n & 7)];
        }
      }
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int n = n0 + v * blockDim.x, node = n >> 3, col = n & 7;
        if (n >= 8 * kF64Nodes) continue;
        const unsigned long long u = u4[v];
        const int kk = node & 15, q = (kk & 7) >> 1, at = kk >> 3;
        __half *r = reinterpret_cast<__half *>(&sB[node >> 4][0][0][4 * col + q]) + 2 * at + (kk & 1);
        __half *s = reinterpret_cast<__half *>(&sB[node >> 4][1][0][4 * (col ^ 1) + q]) + 2 * at + (kk & 1);
#pragma unroll
        for (int d = 0; d < 6; ++d) {  // digit 5 - d: vector d / 2, words 2 (d % 2) + {0, 1}
          const float w = (float)((int)((u >> (50 - 10 * d)) & 1023) - 512);
          r[(d >> 1) * 256 + 4 * (d & 1)] = __float2half_rn(w);
          s[(d >> 1) * 256 + 4 * (d & 1)] = __float2half_rn((col & 1) ? -w : w);
        }
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int ks = 0; ks < 4; ++ks) {
      const int st = 4 * c + ks;
      if (st >= st1) break;
      float D[7][4];
#pragma unroll
      for (int d = 0; d < 7; ++d)
#pragma unroll
        for (int e = 0; e < 4; ++e) D[d][e] = 0.f;
#pragma unroll
      for (int part = 0; part < 2; ++part) {
        const uint4 w[4] = {nx[0], nx[1], nx[2], nx[3]};
        const size_t at = part == 0 ? (size_t)st * step + 128 : (size_t)min(st + 1, st1 - 1) * step;
#pragma unroll
        for (int i = 0; i < 4; ++i) nx[i] = ld_stream(Kt + at + 32 * i);
        unsigned b[12];
#pragma unroll
        for (int v = 0; v < 3; ++v) {
          const uint4 x = sB[ks][part][v][lane];
          b[4 * v] = x.x;
          b[4 * v + 1] = x.y;
          b[4 * v + 2] = x.z;
          b[4 * v + 3] = x.w;
        }
        digit_products<5>(D, w, b);
        digit_products<4>(D, w, b);
        digit_products<3>(D, w, b);
        digit_products<2>(D, w, b);
        digit_products<1>(D, w, b);
        digit_products<0>(D, w, b);
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        hi[e] += (long long)__float2int_rn(D[0][e]) * (1 << 20) + (long long)__float2int_rn(D[1][e]) * (1 << 10) +
                 __float2int_rn(D[2][e]);
        lo[e] += ((long long)__float2int_rn(D[3][e]) + __float2int_rn(D[6][e])) * (1 << 20) +
                 (long long)__float2int_rn(D[4][e]) * (1 << 10) + __float2int_rn(D[5][e]);
      }
    }
  }
  // accumulator registers: (row g, field q) Re, Im, then (row g + 8, field q)
  const int g = lane >> 2, f = lane & 3, row = 16 * warp + g;
  const unsigned long long big = smax[4 * level_of(L, m, t) + f];
  // an infinity or NaN among the sources of this level, or a distance without an FP64 square in the list
  const bool bad = (big >> 52) >= 2047 || expo[t] == kBadExponent;
  const int e = expo[t] + max_exponent(big) - 2 * kFixBits + 80;
  double v[4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
    v[i] = bad ? __longlong_as_double(0x7ff8000000000000ll) : scalbn((double)hi[i] + (double)lo[i] * 0x1p-30, e);
  double2 *o = (blockIdx.y == 0 ? acc : more + (blockIdx.y - 1) * slab) + ((size_t)t * 4 + f) * nI;
  if (row < nI) o[row] = make_double2(v[0], v[1]);
  if (row + 8 < nI) o[row + 8] = make_double2(v[2], v[3]);
}

static LevOff lev_off(const Ctx *c) {
  LevOff L;
  for (int l = 0; l < 12; ++l) L.off[l] = l < (int)c->lev_off.size() ? c->lev_off[l] : c->ncl;
  return L;
}

// K-steps before every cluster's matrices (and the total), 16 source nodes each
static std::vector<size_t> k_steps(const Ctx *c) {
  std::vector<int> cnt(c->ncl, 0);
  for (int f = 0; f < c->nfar; ++f) ++cnt[c->far[3 * f + 1]];
  std::vector<size_t> off(c->ncl + 1, 0);
  const size_t nIe = (c->nI + 1) & ~1;
  for (int t = 0; t < c->ncl; ++t) off[t + 1] = off[t] + (cnt[t] * nIe + 15) / 16;
  return off;
}

// splits of the K-steps: enough warps for the chip when there are few targets, two staged chunks each
static int k_splits(const Ctx *c, size_t steps) {
  const long long warps = 16ll * c->nsm, have = (long long)c->n_m2l_targets * ((c->nI + 15) / 16);
  const long long chunks = (long long)(steps / 4) / std::max(c->n_m2l_targets, 1);
  return (int)std::max(1ll, std::min({2 * warps / have, chunks / 2, 16ll}));
}

size_t m2l_f64_digits_bytes(const Ctx *c) {
  return k_steps(c).back() * (size_t)((c->nI + 15) / 16) * 4096;
}

size_t m2l_f64_digits_beside(const Ctx *c) {
  const size_t nodes = (size_t)c->ncl * c->nI;
  return 64 * nodes * k_splits(c, k_steps(c).back()) + 12 * (size_t)(c->ncl + 1) + 32 * (size_t)(c->m + 1) +
         sizeof(double2) * kCircle;
}

void m2l_f64_digits_free(Ctx *c) {
  dfree(c, c->d_K);
  dfree(c, c->d_koff);
  dfree(c, c->d_kexp);
  dfree(c, c->d_smax);
  dfree(c, c->d_fix);
  dfree(c, c->d_accmore);
}

// Evaluates and keeps the matrices in c->d_K (allocated by the caller, m2l_f64_digits_bytes).
efie_status m2l_f64_digits_build(Ctx *c) {
  const std::vector<size_t> off = k_steps(c);
  EFIE_TRY(dalloc(c, &c->d_koff, off.size()));
  EFIE_TRY(dalloc(c, &c->d_kexp, (size_t)c->ncl));
  EFIE_TRY(dalloc(c, &c->d_smax, 4 * (size_t)(c->m + 1)));
  EFIE_TRY(dalloc(c, &c->d_fix, (size_t)c->ncl * c->nI * 8));
  EFIE_CUDA(cudaMemcpyAsync(c->d_koff, off.data(), sizeof(size_t) * off.size(), cudaMemcpyHostToDevice, c->stream));
  k_K_exponent<<<c->n_m2l_targets, 128, 0, c->stream>>>(c->d_m2l_targets, c->d_far_ptr, c->d_far_src, c->nI, c->d_center,
                                                       c->d_nodeXf, c->d_nodeX, c->d_kexp); ++c->launches;
  DevTemp tmp;
  double2 *circle = nullptr;
  EFIE_TRY(tmp.get(c, &circle, kCircle));
  k_circle<<<1, kCircle, 0, c->stream>>>(circle); ++c->launches;
  k_K_digits<<<c->npairs, 128, sizeof(double) * 6 * c->nI, c->stream>>>(
      c->ncl, c->d_own_ptr, c->d_own_src, c->d_far_ptr, c->d_far_src, c->d_koff, c->d_kexp, c->nI, c->kappa, c->d_nodeX,
      circle, (uint4 *)c->d_K); ++c->launches;
  EFIE_CUDA(cudaGetLastError());
  c->f64_split = k_splits(c, off.back());
  if (c->f64_split > 1) {
    const size_t n = (size_t)(c->f64_split - 1) * c->ncl * 4 * c->nI;
    EFIE_TRY(dalloc(c, &c->d_accmore, n));
    EFIE_CUDA(cudaMemsetAsync(c->d_accmore, 0, sizeof(double2) * n, c->stream));
  }
  EFIE_CUDA(cudaStreamSynchronize(c->stream));
  return EFIE_OK;
}

// fixed-point sources from the folded ones and their largest values per level (d_smax)
efie_status m2l_f64_digits_fix(Ctx *c, cudaStream_t st, const double2 *src) {
  const long long tot = (long long)c->ncl * c->nI * 4;
  k_src_fix<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(tot, c->nI, c->m, lev_off(c), src, c->d_smax,
                                                           reinterpret_cast<ulonglong2 *>(c->d_fix)); ++c->launches;
  EFIE_CUDA(cudaGetLastError());
  return EFIE_OK;
}

efie_status m2l_f64_digits_apply(Ctx *c, cudaStream_t st) {
  const int ntile = (c->nI + 15) / 16;
  const dim3 grid(c->n_m2l_targets, c->f64_split);
  const size_t slab = (size_t)c->ncl * 4 * c->nI;
#define EFIE_DIGITS(T, B)                                                                                        \
  k_m2l_f64_digits<T, B><<<grid, 32 * ntile, 0, st>>>(c->d_m2l_targets, c->d_far_ptr, c->d_far_src, c->d_koff,    \
                                                      c->d_kexp, c->nI, c->m, lev_off(c), (const uint4 *)c->d_K,  \
                                                      c->d_fix, c->d_smax, c->d_acc, c->d_accmore, slab)
  if (ntile <= 8) EFIE_DIGITS(256, 2);
  else EFIE_DIGITS(640, 1);
#undef EFIE_DIGITS
  ++c->launches;
  EFIE_CUDA(cudaGetLastError());
  return EFIE_OK;
}

}  // namespace efie
