// Device steps of the restarted GMRES (a11) shared by the single-system solver, the lockstep
// batch of one context and the lockstep group of independent problems, so that all three take
// the same arithmetic in the same order.
#pragma once

#include <cuda_runtime.h>

namespace efie {

constexpr int kDotThreads = 256;
constexpr int kRowsPerThread = 2;
constexpr int kChunk = kDotThreads * kRowsPerThread;  // vector entries per partial dot product
constexpr int kVecPerBlock = 8;
static_assert(kVecPerBlock == kDotThreads / 32, "one warp sums one vector of a dot-product block");

// FP64 is GB300's scarcest pipe (one warp instruction per 72 clocks and scheduler), so what counts in
// all of these is the number of FP64 warp instructions and that every SM takes part, also for a
// few hundred unknowns.  Measured, an iteration beyond its product: 0.37 -> 0.15 ms on average over the
// 604 of 13 068 unknowns, 92 -> 28 us over the 129 of 768 (chunks of 2 048 entries, tiles of 32 and a
// single-thread Givens step before; a solve of six such systems in lockstep 178 -> 97 ms, whose
// steps were launched system by system).

// sums of x and y over the 32 lanes, x in lane 0 and y in lane 16 (5 additions a lane, fixed order)
__device__ __forceinline__ double warp_sum2(double x, double y) {
  const bool up = (threadIdx.x & 16) != 0;
  const double other = __shfl_xor_sync(0xffffffffu, up ? x : y, 16);
  double v = (up ? y : x) + other;
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Partial dot products of one chunk: part[i * nchunk + chunk] = sum_{t in chunk} conj(V_i[t]) w[t]
// for i = i0 .. i0 + 7 (i < nvec), one vector per warp: 64 FMAs and 5 additions a lane at 512 entries.
// Called by all kDotThreads threads of a block.
__device__ __forceinline__ void dot_partial_chunk(int N, int nvec, int i0, int chunk, const double2 *__restrict__ V,
                                                  size_t ldv, const double2 *__restrict__ w,
                                                  double2 *__restrict__ part, int nchunk) {
  const int lane = threadIdx.x & 31, i = i0 + (threadIdx.x >> 5);
  if (i >= nvec) return;
  const double2 *Vi = V + (size_t)i * ldv;
  double x = 0.0, y = 0.0;
  const int t0 = chunk * kChunk + lane, t1 = min(N, (chunk + 1) * kChunk);
#pragma unroll 4
  for (int t = t0; t < t1; t += 32) {
    // conj(a) w as four FMAs into the running sums
    const double2 a = Vi[t], wt = w[t];
    x = fma(a.x, wt.x, x);
    x = fma(a.y, wt.y, x);
    y = fma(a.x, wt.y, y);
    y = fma(-a.y, wt.x, y);
  }
  const double v = warp_sum2(x, y);
  double *o = reinterpret_cast<double *>(part + (size_t)i * nchunk + chunk);
  if ((lane & 15) == 0) o[lane >> 4] = v;
}

// h[i] = sum over the chunks of part[i][.], one warp, fixed order.
__device__ __forceinline__ void dot_final_warp(int i, int nchunk, const double2 *__restrict__ part,
                                               double2 *__restrict__ h) {
  const int lane = threadIdx.x & 31;
  double x = 0.0, y = 0.0;
  for (int k = lane; k < nchunk; k += 32) {
    const double2 v = part[(size_t)i * nchunk + k];
    x += v.x;
    y += v.y;
  }
  const double v = warp_sum2(x, y);
  if ((lane & 15) == 0) reinterpret_cast<double *>(h + i)[lane >> 4] = v;
}

// w[t] += sgn * sum_i c_i V_i[t] for the kCombRows entries t0 .. t0 + 7 of one block of kCombThreads
// threads: lane l of warp k sums the vectors i = 4 k + l / 8, + 32, ... for entry l % 8 (each load
// four 128-byte segments), so that a few hundred entries still make a block for every SM; the 32
// partial sums of an entry are added in a fixed order.  nrm (if not null): the new |w|^2 of the tile.
constexpr int kCombRows = 8;
constexpr int kCombThreads = 256;
__device__ __forceinline__ void combine_tile(int N, int t0, int nvec, const double2 *__restrict__ V, size_t ldv,
                                             const double2 *__restrict__ c, double sgn, double2 *__restrict__ w,
                                             double *nrm = nullptr) {
  __shared__ double2 part[kCombThreads / 8][kCombRows + 1];
  const int lane = threadIdx.x & 31, grp = threadIdx.x >> 3, t = t0 + (lane & 7);
  double x = 0.0, y = 0.0;
  if (t < N) {
#pragma unroll 4
    for (int i = grp; i < nvec; i += kCombThreads / 8) {
      const double2 a = V[(size_t)i * ldv + t], ci = c[i];
      x = fma(ci.x, a.x, x);
      x = fma(-ci.y, a.y, x);
      y = fma(ci.x, a.y, y);
      y = fma(ci.y, a.x, y);
    }
  }
  part[grp][lane & 7] = make_double2(x, y);
  __syncthreads();
  if (threadIdx.x < 32) {
    double sx = 0.0, sy = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const double2 v = part[8 * (lane >> 3) + k][lane & 7];
      sx += v.x;
      sy += v.y;
    }
#pragma unroll
    for (int o = 8; o < 32; o <<= 1) {
      sx += __shfl_xor_sync(0xffffffffu, sx, o);
      sy += __shfl_xor_sync(0xffffffffu, sy, o);
    }
    double q = 0.0;
    if (t < N && lane < 8) {
      const double2 v = w[t];
      const double2 n = make_double2(fma(sgn, sx, v.x), fma(sgn, sy, v.y));
      w[t] = n;
      q = fma(n.x, n.x, n.y * n.y);
    }
    if (nrm) {
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
      if (lane == 0) nrm[t0 / kCombRows] = q;
    }
  }
  __syncthreads();
}

__device__ __forceinline__ double2 scaled_entry(double2 w, double beta) {
  double f = beta > 0.0 ? 1.0 / beta : 0.0;
  return make_double2(w.x * f, w.y * f);
}

// Givens state layout in st: [0] beta of the new vector, [1] residual estimate,
// [2 .. 2+kr) cs, then sn (complex) [kr][2], then g (complex) [kr+1][2].
__device__ __forceinline__ void givens_init_dev(double *st, int kr, const double2 *h) {
  // g = (||r||, 0, ...); h[0] holds ||r||^2
  double beta = sqrt(h[0].x);
  double *g = st + 2 + kr + 2 * kr;
  for (int i = 0; i <= kr; ++i) {
    g[2 * i] = 0.0;
    g[2 * i + 1] = 0.0;
  }
  g[0] = beta;
  st[0] = beta;
  st[1] = beta;
}

// z <- -conj(s) z (+ v)
__device__ __forceinline__ double2 rot_pass(double sr, double si, double2 z, double2 v) {
  return make_double2(fma(-sr, z.x, fma(-si, z.y, v.x)), fma(-sr, z.y, fma(si, z.x, v.y)));
}
__device__ __forceinline__ double2 cmul_add(double2 a, double2 b, double2 v) {
  return make_double2(fma(a.x, b.x, fma(-a.y, b.y, v.x)), fma(a.x, b.y, fma(a.y, b.x, v.y)));
}

// hypot without its scaling where the squares are far inside the range
__device__ __forceinline__ double length2(double x, double y) {
  const double s = fma(x, x, y * y);
  return s > 1e-280 && s < 1e280 ? sqrt(s) : hypot(x, y);
}

// Column j of the Hessenberg matrix from the CGS2 coefficients h1 + h2 and the norm of the
// orthogonalised vector (nrm: |w|^2 of its tiles); previous rotations, new rotation, residual
// estimate |g_{j+1}|.  The entry that rotation i passes on, a_{i+1} = -conj(s_i) a_i + c_i b_{i+1},
// is an affine recurrence: the kGivThreads threads of the block compose their segments of it, scan
// the compositions and run their segments again from the right start (a single thread took
// 16 FP64 instructions of 72 clocks per rotation, 180 us at j = 300).
constexpr int kGivThreads = 128;
__device__ __forceinline__ void givens_step_block(int j, int kr, const double2 *h1, const double2 *h2,
                                                  const double *nrm, int ntile, double2 *H, double *st) {
  __shared__ double2 wP[kGivThreads / 32], wQ[kGivThreads / 32], last;
  __shared__ double wN[kGivThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double *cs = st + 2;
  double *sn = st + 2 + kr;     // complex [kr]
  double *g = st + 2 + 3 * kr;  // complex [kr+1]
  const double2 zero = make_double2(0.0, 0.0);
  double q = 0.0;
  for (int k = tid; k < ntile; k += kGivThreads) q += nrm[k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
  if (lane == 0) wN[warp] = q;
  const int L = (j + kGivThreads - 1) / kGivThreads, i0 = min(j, tid * L), i1 = min(j, i0 + L);
  const double2 a0 = make_double2(h1[0].x + h2[0].x, h1[0].y + h2[0].y);
  double2 P = make_double2(1.0, 0.0), Q = zero;
  for (int i = i0; i < i1; ++i) {
    const double2 b = make_double2(h1[i + 1].x + h2[i + 1].x, h1[i + 1].y + h2[i + 1].y);
    const double c = cs[i], sr = sn[2 * i], si = sn[2 * i + 1];
    P = rot_pass(sr, si, P, zero);
    Q = rot_pass(sr, si, Q, make_double2(c * b.x, c * b.y));
  }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {  // inclusive scan of the compositions, earlier segments first
    const double2 p = make_double2(__shfl_up_sync(0xffffffffu, P.x, o), __shfl_up_sync(0xffffffffu, P.y, o));
    const double2 r = make_double2(__shfl_up_sync(0xffffffffu, Q.x, o), __shfl_up_sync(0xffffffffu, Q.y, o));
    if (lane >= o) {
      Q = cmul_add(P, r, Q);
      P = cmul_add(P, p, zero);
    }
  }
  if (lane == 31) {
    wP[warp] = P;
    wQ[warp] = Q;
  }
  double2 eP = make_double2(__shfl_up_sync(0xffffffffu, P.x, 1), __shfl_up_sync(0xffffffffu, P.y, 1));
  double2 eQ = make_double2(__shfl_up_sync(0xffffffffu, Q.x, 1), __shfl_up_sync(0xffffffffu, Q.y, 1));
  if (lane == 0) {
    eP = make_double2(1.0, 0.0);
    eQ = zero;
  }
  __syncthreads();
  double2 a = a0;
  for (int k = 0; k < warp; ++k) a = cmul_add(wP[k], a, wQ[k]);
  a = cmul_add(eP, a, eQ);
  for (int i = i0; i < i1; ++i) {
    const double2 b = make_double2(h1[i + 1].x + h2[i + 1].x, h1[i + 1].y + h2[i + 1].y);
    const double c = cs[i], sr = sn[2 * i], si = sn[2 * i + 1];
    // [a; b] <- [c a + s b; -conj(s) a + c b]
    H[(size_t)i * kr + j] = cmul_add(make_double2(sr, si), b, make_double2(c * a.x, c * a.y));
    a = rot_pass(sr, si, a, make_double2(c * b.x, c * b.y));
  }
  if (i1 == j && (i0 < j || tid == 0)) last = a;  // the one thread whose segment ends the column (j = 0: thread 0)
  __syncthreads();
  if (tid > 0) return;
  a = last;
  double n2 = 0.0;
  for (int k = 0; k < kGivThreads / 32; ++k) n2 += wN[k];
  const double beta = sqrt(fmax(n2, 0.0));
  const double aa = length2(a.x, a.y), tt = length2(aa, beta);
  double c, sr, si;
  if (aa == 0.0) {
    c = 0.0; sr = 1.0; si = 0.0;
  } else {
    c = aa / tt;
    const double f = (beta / tt) / aa;
    sr = a.x * f;
    si = a.y * f;
  }
  cs[j] = c;
  sn[2 * j] = sr;
  sn[2 * j + 1] = si;
  H[(size_t)j * kr + j] = make_double2(c * a.x + sr * beta, c * a.y + si * beta);
  double gr = g[2 * j], gi = g[2 * j + 1];
  g[2 * (j + 1)] = -(sr * gr + si * gi);
  g[2 * (j + 1) + 1] = -(sr * gi - si * gr);
  g[2 * j] = c * gr;
  g[2 * j + 1] = c * gi;
  st[0] = beta;
  st[1] = length2(g[2 * (j + 1)], g[2 * (j + 1) + 1]);
}

// y = H(0:jd, 0:jd)^{-1} g(0:jd), one warp: row sums in parallel, rows in sequence.
__device__ __forceinline__ void backsolve_warp(int jd, int kr, const double2 *H, const double *st, double2 *y) {
  const double *g = st + 2 + 3 * kr;
  int lane = threadIdx.x & 31;
  for (int i = jd - 1; i >= 0; --i) {
    double x = 0.0, z = 0.0;
    for (int t = i + 1 + lane; t < jd; t += 32) {
      double2 hh = H[(size_t)i * kr + t], yy = y[t];
      x += hh.x * yy.x - hh.y * yy.y;
      z += hh.x * yy.y + hh.y * yy.x;
    }
    for (int o = 16; o > 0; o >>= 1) {
      x += __shfl_down_sync(0xffffffffu, x, o);
      z += __shfl_down_sync(0xffffffffu, z, o);
    }
    if (lane == 0) {
      double sr = g[2 * i] - x, si = g[2 * i + 1] - z;
      double2 d = H[(size_t)i * kr + i];
      double den = d.x * d.x + d.y * d.y;
      y[i] = make_double2((sr * d.x + si * d.y) / den, (si * d.x - sr * d.y) / den);
    }
    __syncwarp();
  }
}

}  // namespace efie
