// Near-field blocks of touching element pairs (a2: common vertex, common edge, identical elements)
// by the Sauter-Schwab substitutions [SS97], with sums factorised over the tensor structure that
// the substituted points still have.
//
// Every part of the three substitutions is a tensor rule in (a, x_i, x_j, x_m), a the singular
// coordinate, and for a fixed a one of the two directions of the canonical square depends on
// (i, j) only (the major direction), the other on m only (the minor one), on both elements.  So for
// a fixed a, with M = (i, j):
//   * the block sum over the g^2 x g points splits: first over M for every m (T = sum_M Q(M) X(M, m),
//     Q the products of the 1-D Bernstein functions of the two elements in the major direction), then
//     over m with the products of the minor direction.  For g = p + 4 = 6 that is about 150 FP64 FMAs
//     a point instead of 4 (2 (p + 1)^2)^2 = 1296;
//   * the geometry splits: the control nets are contracted along the minor direction once per m and
//     element, then along the major one per point, and only the coordinates that an element's points
//     depend on are run through (42 evaluations instead of 432 per a at a common vertex).
// The 1-D functions are the p + 1 Bernstein polynomials of degree p and the p of degree p - 1: the
// div-div term needs derivatives, and B_a' = p (B_{a-1}^{p-1} - B_a^{p-1}) is applied once per block.
//
// Bound: the FP64 pipe (one warp instruction per 72 clocks and scheduler; 92 % busy), as before, at
// a sixth of the instructions; loads from shared memory and index arithmetic are free beside it.  The
// 216 points of an a at g = 6 fill 6.75 warps, so 128 threads go twice and warps without work cost nothing.
// Measured, all touching pairs, direct kernel -> this one: sphere p = 2, 32 x 32 elements (30 708 pairs) 990 -> 168 ms;
// p = 1, 16 x 16: 65 -> 18 ms; torus p = 3, 16 x 16: 2 704 -> 276 ms; multi-cell surface p = 4: 703 -> 37 ms;
// blocks within 1e-14 of each other.  k_near_quad stays for what this rule leaves: geometry knots inside
// an element, and rules with more than 2 x 128 (p <= 2) or 2 x 256 points per a.
#include <algorithm>
#include <cmath>

#include "geom.cuh"

namespace efie {

namespace {

struct TouchArgs {
  const PatchDesc *patches;
  const double *knots;
  const double4 *cpw;
  const NearPair *pairs;
  const int *todo, *slot;
  int ntodo, n, g;
  const double *x, *w;  // Gauss rule on [0, 1]
  double kappa, h;
  double2 *blocks;  // [nnear][nb col][nb row]
};

template <int P>
struct TouchCfg {
  static constexpr int P1 = P + 1, NV = 2 * P + 1, NQ = NV * NV, NS = P1 * P1, NB = 2 * NS;
  static constexpr int kThreads = P <= 2 ? 128 : 256;
  static constexpr int kGeo = 4 * NS * NS, kDiv = P * P * NS;  // accumulators: geometry terms, one div variant
  static constexpr int kAcc = kGeo + 4 * kDiv;
  static constexpr int kT = 4 * NS + NQ;
  static constexpr int EPT = (kAcc + kThreads - 1) / kThreads;
};

// Shared memory (doubles): 1-D tables, product tables, contracted nets, T, then side geometry of the
// points (18 each), which the coefficients (10 each) and at the end the accumulators overwrite.
template <int P, int GD>
__host__ __device__ constexpr size_t touch_smem_doubles(int g) {
  using C = TouchCfg<P>;
  const size_t g2 = (size_t)g * g, g3 = g2 * g;
  const size_t pts = 18 * g3 > 2 * (size_t)C::kAcc ? 18 * g3 : 2 * (size_t)C::kAcc;
  return 2 * (g2 + g) * (2 * (GD + 1) + C::NV) + (g2 + g) * C::NQ + (size_t)2 * g * (GD + 1) * 8 + (size_t)2 * g * C::kT + 2 + pts;
}

// Part `part` of a substitution at a: which canonical direction is the major one, and for each element
// (0 target, 1 source) whether its points depend on i, j, m.
struct Part {
  int major;      // 0: direction 1, 1: direction 2
  int use[2][3];  // i, j, m
};

__device__ __forceinline__ Part part_of(int kind, int part) {
  if (kind == 3) return {part < 4 ? 1 : 0, {{1, 1, 1}, {1, 1, 1}}};
  if (kind == 2) {
    const int pyr = part >> 1;
    if (pyr == 0) return {1, {{1, 0, 1}, {0, 1, 1}}};
    if (pyr == 1) return {0, {{1, 1, 0}, {1, 1, 1}}};
    return {0, {{1, 1, 1}, {1, 1, 0}}};
  }
  if (part < 2) return {part == 0 ? 1 : 0, {{1, 0, 0}, {0, 1, 1}}};
  return {part == 2 ? 1 : 0, {{1, 0, 1}, {0, 1, 0}}};
}

// Canonical coordinates in the major direction at (xi, xj): s (target), t (source).
__device__ __forceinline__ void major_point(int kind, int part, double a, double xi, double xj, double &s, double &t) {
  if (kind == 3 || (kind == 2 && part >= 2)) {
    const bool neg = kind == 3 ? (part < 4 ? (part & 2) : (part & 1)) : (part & 1);
    const double z = a * xi;
    s = (neg ? z : 0.0) + (1.0 - z) * xj;
    t = s + (neg ? -z : z);
  } else {
    s = a * xi;
    t = a * xj;
  }
}

// Canonical coordinates in the minor direction at xm.
__device__ __forceinline__ void minor_point(int kind, int part, double a, double xm, double &s, double &t) {
  if (kind == 3 || (kind == 2 && part < 2)) {
    const bool neg = kind == 3 ? (part < 4 ? (part & 1) : (part & 2)) : (part & 1);
    s = (neg ? a : 0.0) + (1.0 - a) * xm;
    t = s + (neg ? -a : a);
  } else {
    const bool s_fixed = kind == 2 ? (part >> 1) == 1 : part < 2;
    s = s_fixed ? a : a * xm;
    t = s_fixed ? a * xm : a;
  }
}

// Jacobian of the substitution at (a, xi).
__device__ __forceinline__ double part_jacobian(int kind, int part, double a, double xi) {
  if (kind == 3) return a * (1.0 - a) * (1.0 - a * xi);
  if (kind == 2) return a * a * (1.0 - (part < 2 ? a : a * xi));
  return a * a * a;
}

// Accumulator e: products of the 1-D functions in directions 1 and 2 (index v_target NV + v_source;
// v < P1 degree p, else degree p - 1) and the coefficient (2 alpha + beta of the geometry term, 4).
template <int P>
__device__ __forceinline__ void decode(int e, int &q1, int &q2, int &k) {
  using C = TouchCfg<P>;
  if (e < C::kGeo) {
    k = e / (C::NS * C::NS);
    const int ac = (e / C::NS) % C::NS, bd = e % C::NS;
    q1 = (ac / C::P1) * C::NV + ac % C::P1;
    q2 = (bd / C::P1) * C::NV + bd % C::P1;
    return;
  }
  e -= C::kGeo;
  const int al = e / (2 * C::kDiv), be = (e / C::kDiv) & 1;
  e %= C::kDiv;
  const int nc = be == 0 ? P : C::P1, nb = al == 1 ? P : C::P1, nd = be == 1 ? P : C::P1;
  const int d = e % nd, b = (e / nd) % nb, c = (e / (nd * nb)) % nc, a = e / (nd * nb * nc);
  q1 = (a + (al == 0 ? C::P1 : 0)) * C::NV + c + (be == 0 ? C::P1 : 0);
  q2 = (b + (al == 1 ? C::P1 : 0)) * C::NV + d + (be == 1 ? C::P1 : 0);
  k = 4;
}

}  // namespace

// One block per element pair; see the head of the file.  Canonical direction d of an element is its
// patch direction d or, for a swapped pair of coordinates (bit 0 of the pair's symmetry code),
// 1 - d; reflections are applied to the coordinates, so functions and derivatives are the element's.
template <int P, int GD>
__global__ void __launch_bounds__(TouchCfg<P>::kThreads, P == 2 ? 3 : 1) k_near_touch(TouchArgs A) {
  using C = TouchCfg<P>;
  constexpr int NTH = C::kThreads, W1 = 2 * (GD + 1) + C::NV;
  extern __shared__ double sm[];
  const int g = A.g, g2 = g * g, g3 = g2 * g, tid = threadIdx.x;
  double *tab = sm;                                // [2 sides][g2 major, g minor][N, dN, V]
  double *Q = tab + 2 * (g2 + g) * W1;             // [g2 major, g minor][NQ]
  double *R = Q + (g2 + g) * C::NQ;                // [2][g][GD + 1][8]
  double2 *T = reinterpret_cast<double2 *>(R + 2 * g * (GD + 1) * 8 + (((g2 + g) * C::NQ) & 1));  // [g][kT]
  double *pts = reinterpret_cast<double *>(T + g * C::kT);
  __shared__ double sGx[16], sGw[16];
  __shared__ int sSpan[2][2];
  const NearPair pr = A.pairs[A.todo[blockIdx.x]];
  const int n = A.n, n2 = n * n, kind = pr.kind;
  const double h = A.h, h2 = h * h, h4 = h2 * h2, ik2 = 1.0 / (A.kappa * A.kappa);
  const int patch[2] = {pr.e / n2, pr.e2 / n2};
  int cell[2][2] = {{0, 0}, {0, 0}};  // [side][patch direction]
  for (int b = 0; b < 15; ++b) {
    cell[0][0] |= (((pr.e % n2) >> (2 * b)) & 1) << b;
    cell[0][1] |= (((pr.e % n2) >> (2 * b + 1)) & 1) << b;
    cell[1][0] |= (((pr.e2 % n2) >> (2 * b)) & 1) << b;
    cell[1][1] |= (((pr.e2 % n2) >> (2 * b + 1)) & 1) << b;
  }
  const int code[2] = {pr.r1, pr.r2};
  if (tid < g) {
    sGx[tid] = A.x[tid];
    sGw[tid] = A.w[tid];
  }
  if (tid < 4) {  // the element lies in one knot span of either direction
    const int side = tid >> 1, d = tid & 1;
    const PatchDesc &pd = A.patches[patch[side]];
    sSpan[side][d] = dev_span(A.knots + pd.kofs[d], pd.deg[d], pd.ncp[d], (cell[side][d] + 0.5) * h);
  }
  int q1[C::EPT], q2[C::EPT], kk[C::EPT];
  double2 acc[C::EPT];
#pragma unroll
  for (int t = 0; t < C::EPT; ++t) {
    acc[t] = make_double2(0.0, 0.0);
    q1[t] = q2[t] = kk[t] = 0;
    if (tid + t * NTH < C::kAcc) decode<P>(tid + t * NTH, q1[t], q2[t], kk[t]);
  }
  const int parts = kind == 3 ? 8 : (kind == 2 ? 6 : 4);
  for (int pa = 0; pa < parts * g; ++pa) {
    const int part = pa / g, ia = pa % g;
    const Part pt = part_of(kind, part);
    const int maj = pt.major, mnr = 1 - maj;
    __syncthreads();
    const double a = sGx[ia];
    // 1-D tables at the distinct coordinates of each element and direction
    for (int it = tid; it < 2 * (g2 + g); it += NTH) {
      const int side = it / (g2 + g), r = it % (g2 + g);
      const bool major = r < g2;
      const int i = r / g, j = r % g, m = r - g2;
      if (major ? ((!pt.use[side][0] && i) || (!pt.use[side][1] && j)) : (!pt.use[side][2] && m)) continue;
      double s, t;
      if (major) major_point(kind, part, a, sGx[i], sGx[j], s, t);
      else minor_point(kind, part, a, sGx[m], s, t);
      const int dir = major ? maj : mnr, pdir = (code[side] & 1) ? 1 - dir : dir;
      double u = side == 0 ? s : t;
      if (code[side] & (pdir == 0 ? 2 : 4)) u = 1.0 - u;
      const PatchDesc &pd = A.patches[patch[side]];
      double N[GD + 1], dN[GD + 1], B[kMaxP1], dB[kMaxP1];
      dev_bspline_at<GD>(A.knots + pd.kofs[pdir], A.knots + pd.iofs[pdir], pd.deg[pdir], pd.ncp[pdir],
                         sSpan[side][pdir], (cell[side][pdir] + u) * h, N, dN);
      double *o = tab + (side * (g2 + g) + r) * W1;
#pragma unroll
      for (int b = 0; b <= GD; ++b) {
        o[b] = N[b];
        o[GD + 1 + b] = dN[b];
      }
      dev_bernstein(P, u, B, dB);
#pragma unroll
      for (int b = 0; b < C::P1; ++b) o[2 * (GD + 1) + b] = B[b];
      if (P > 1) dev_bernstein(P - 1, u, B, dB);
#pragma unroll
      for (int b = 0; b < P; ++b) o[2 * (GD + 1) + C::P1 + b] = P > 1 ? B[b] : 1.0;
    }
    __syncthreads();
    // row of a side's table for the major index (i, j) / minor index m
    auto row = [&](int side, int i, int j) { return side * (g2 + g) + (pt.use[side][0] ? i : 0) * g + (pt.use[side][1] ? j : 0); };
    auto rowm = [&](int side, int m) { return side * (g2 + g) + g2 + (pt.use[side][2] ? m : 0); };
    // products of the 1-D functions of the two elements
    for (int it = tid; it < (g2 + g) * C::NQ; it += NTH) {
      const int r = it / C::NQ, v = it % C::NQ;
      const int rs = r < g2 ? row(0, r / g, r % g) : rowm(0, r - g2), rt = r < g2 ? row(1, r / g, r % g) : rowm(1, r - g2);
      Q[it] = tab[rs * W1 + 2 * (GD + 1) + v / C::NV] * tab[rt * W1 + 2 * (GD + 1) + v % C::NV];
    }
    // control nets contracted along the minor direction: values and derivatives (homogeneous)
    for (int it = tid; it < 2 * g * (GD + 1) * 2; it += NTH) {
      const int half = it & 1, b = (it >> 1) % (GD + 1), m = ((it >> 1) / (GD + 1)) % g, side = (it >> 1) / ((GD + 1) * g);
      const PatchDesc &pd = A.patches[patch[side]];
      const int pm = (code[side] & 1) ? 1 - mnr : mnr, pM = 1 - pm;  // patch directions: minor, major
      if (b > pd.deg[pM] || (!pt.use[side][2] && m)) continue;
      const double *N = tab + rowm(side, m) * W1 + (half ? GD + 1 : 0);
      const int k0 = sSpan[side][0] - pd.deg[0], k1 = sSpan[side][1] - pd.deg[1];
      double4 r = make_double4(0.0, 0.0, 0.0, 0.0);
      for (int c = 0; c <= pd.deg[pm]; ++c) {
        const double4 p = A.cpw[pd.cofs + (k1 + (pm == 1 ? c : b)) * pd.ncp[0] + k0 + (pm == 1 ? b : c)];
        const double v = N[c];
        r.x += v * p.x;
        r.y += v * p.y;
        r.z += v * p.z;
        r.w += v * p.w;
      }
      double *o = R + ((side * g + m) * (GD + 1) + b) * 8 + 4 * half;
      o[0] = r.x;
      o[1] = r.y;
      o[2] = r.z;
      o[3] = r.w;
    }
    __syncthreads();
    // F and its derivatives in directions 1, 2 at the distinct points of each element
    for (int it = tid; it < 2 * g3; it += NTH) {
      const int side = it / g3, r = it % g3, m = r % g, M = r / g, i = M / g, j = M % g;
      if ((!pt.use[side][0] && i) || (!pt.use[side][1] && j) || (!pt.use[side][2] && m)) continue;
      const PatchDesc &pd = A.patches[patch[side]];
      const int deg = pd.deg[(code[side] & 1) ? 1 - maj : maj];
      const double *N = tab + row(side, i, j) * W1, *Rm = R + (side * g + m) * (GD + 1) * 8;
      double f[4] = {0, 0, 0, 0}, fM[4] = {0, 0, 0, 0}, fm[4] = {0, 0, 0, 0};
#pragma unroll
      for (int b = 0; b <= GD; ++b)
        if (b <= deg) {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            f[c] = fma(N[b], Rm[8 * b + c], f[c]);
            fM[c] = fma(N[GD + 1 + b], Rm[8 * b + c], fM[c]);
            fm[c] = fma(N[b], Rm[8 * b + 4 + c], fm[c]);
          }
        }
      const double iw = 1.0 / f[3];
      double *o = pts + (side * g3 + r) * 9;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double X = f[c] * iw;
        o[c] = X;
        o[3 + 3 * maj + c] = (fM[c] - X * fM[3]) * iw;
        o[3 + 3 * mnr + c] = (fm[c] - X * fm[3]) * iw;
      }
    }
    __syncthreads();
    // kernel value and coefficients of every point; two points a thread at most (host rule)
    double co[2][10];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int r = tid + u * NTH;
      if (r < g3) {
        const int m = r % g, M = r / g, i = M / g, j = M % g;
        const double *S = pts + (((pt.use[0][0] ? i : 0) * g + (pt.use[0][1] ? j : 0)) * g + (pt.use[0][2] ? m : 0)) * 9;
        const double *Tt = pts + (g3 + ((pt.use[1][0] ? i : 0) * g + (pt.use[1][1] ? j : 0)) * g + (pt.use[1][2] ? m : 0)) * 9;
        const double dx = S[0] - Tt[0], dy = S[1] - Tt[1], dz = S[2] - Tt[2];
        const double rr = sqrt(dx * dx + dy * dy + dz * dz);
        double sn, cs;
        sincos(A.kappa * rr, &sn, &cs);
        const double W = sGw[ia] * sGw[i] * sGw[j] * sGw[m] * part_jacobian(kind, part, a, sGx[i]);
        const double f = W / (4.0 * M_PI * rr), gre = f * cs, gim = f * sn;
#pragma unroll
        for (int al = 0; al < 2; ++al)
#pragma unroll
          for (int be = 0; be < 2; ++be) {
            const double *Da = S + 3 + 3 * al, *Db = Tt + 3 + 3 * be;
            const double gg = h4 * (Da[0] * Db[0] + Da[1] * Db[1] + Da[2] * Db[2]);
            co[u][2 * (2 * al + be)] = gre * gg;
            co[u][2 * (2 * al + be) + 1] = gim * gg;
          }
        co[u][8] = -ik2 * h2 * gre;
        co[u][9] = -ik2 * h2 * gim;
      }
    }
    __syncthreads();
    double2 *X = reinterpret_cast<double2 *>(pts);  // [m][coefficient][M]
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int r = tid + u * NTH;
      if (r < g3)
#pragma unroll
        for (int c = 0; c < 5; ++c) X[((r % g) * 5 + c) * g2 + r / g] = make_double2(co[u][2 * c], co[u][2 * c + 1]);
    }
    __syncthreads();
    // T[m][t] = sum_M Q(M) X(M, m)
    for (int it = tid; it < g * C::kT; it += NTH) {
      const int m = it / C::kT, t = it % C::kT;
      const int c = t < 4 * C::NS ? t / C::NS : 4;
      const int v = t < 4 * C::NS ? ((t % C::NS) / C::P1) * C::NV + (t % C::NS) % C::P1 : t - 4 * C::NS;
      const double2 *Xm = X + (m * 5 + c) * g2;
      double re = 0.0, im = 0.0;
      for (int M = 0; M < g2; ++M) {
        const double q = Q[M * C::NQ + v];
        re = fma(q, Xm[M].x, re);
        im = fma(q, Xm[M].y, im);
      }
      T[it] = make_double2(re, im);
    }
    __syncthreads();
    // accumulators += sum_m Q(m) T[m]
#pragma unroll
    for (int t = 0; t < C::EPT; ++t) {
      const int qM = maj == 0 ? q1[t] : q2[t], qm = maj == 0 ? q2[t] : q1[t];
      const int ti = kk[t] < 4 ? kk[t] * C::NS + (qM / C::NV) * C::P1 + qM % C::NV : 4 * C::NS + qM;
      const double *qp = Q + g2 * C::NQ + qm;
      if (tid + t * NTH < C::kAcc)
        for (int m = 0; m < g; ++m) {
          const double q = qp[m * C::NQ];
          const double2 v = T[m * C::kT + ti];
          acc[t].x = fma(q, v.x, acc[t].x);
          acc[t].y = fma(q, v.y, acc[t].y);
        }
    }
  }
  __syncthreads();
  double2 *S = reinterpret_cast<double2 *>(pts);
#pragma unroll
  for (int t = 0; t < C::EPT; ++t)
    if (tid + t * NTH < C::kAcc) S[tid + t * NTH] = acc[t];
  __syncthreads();
  double2 *out = A.blocks + (size_t)A.slot[A.todo[blockIdx.x]] * C::NB * C::NB;
  for (int idx = tid; idx < C::NB * C::NB; idx += NTH) {
    const int cc = idx / C::NB, rr = idx % C::NB;
    // patch indices -> canonical: (direction, index in direction 1, index in direction 2)
    int al = rr / C::NS, b2 = (rr % C::NS) / C::P1, a1 = rr % C::P1;
    int be = cc / C::NS, d2 = (cc % C::NS) / C::P1, c1 = cc % C::P1;
    if (code[0] & 1) {
      const int x = a1;
      a1 = b2;
      b2 = x;
      al = 1 - al;
    }
    if (code[1] & 1) {
      const int x = c1;
      c1 = d2;
      d2 = x;
      be = 1 - be;
    }
    const double2 v = S[((2 * al + be) * C::NS + a1 * C::P1 + c1) * C::NS + b2 * C::P1 + d2];
    double re = 0.0, im = 0.0;
    const double2 *Dv = S + C::kGeo + (2 * al + be) * C::kDiv;
    const int nc = be == 0 ? P : C::P1, nb = al == 1 ? P : C::P1, nd = be == 1 ? P : C::P1;
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int w = 0; w < 2; ++w) {  // B' = p (L[index - 1] - L[index])
        const int a = al == 0 ? a1 - 1 + u : a1, b = al == 1 ? b2 - 1 + u : b2;
        const int c = be == 0 ? c1 - 1 + w : c1, d = be == 1 ? d2 - 1 + w : d2;
        const int ia = al == 0 ? a : b, ib = be == 0 ? c : d;
        if (ia < 0 || ia >= P || ib < 0 || ib >= P) continue;
        const double2 x = Dv[((a * nc + c) * nb + b) * nd + d];
        re += u == w ? x.x : -x.x;
        im += u == w ? x.y : -x.y;
      }
    out[idx] = make_double2(v.x + (double)(P * P) * re, v.y + (double)(P * P) * im);
  }
}

constexpr size_t kTouchSmem = 200 * 1024;  // rules that need more stay with k_near_quad

// Whether this geometry and rule can take the factorised kernel: at most two points a thread, shared
// memory for one block, and no knot inside an element (every element in one knot span).
template <int P>
static bool touch_fits(int g, int gdsel) {
  const size_t d = gdsel == 2 ? touch_smem_doubles<P, 2>(g) : (gdsel == 4 ? touch_smem_doubles<P, 4>(g) : touch_smem_doubles<P, 8>(g));
  return g <= 16 && g * g * g <= 2 * TouchCfg<P>::kThreads && d * sizeof(double) <= kTouchSmem;
}

bool near_touch_supported(const Ctx *c, int gdsel) {
  for (const PatchDesc &pd : c->patches)
    for (int d = 0; d < 2; ++d)
      for (int k = pd.deg[d] + 1; k < pd.ncp[d]; ++k) {
        const double v = c->knots[pd.kofs[d] + k] * c->n;
        if (std::fabs(v - std::round(v)) > 1e-12 * c->n) return false;
      }
  switch (c->p) {
    case 1: return touch_fits<1>(c->gs, gdsel);
    case 2: return touch_fits<2>(c->gs, gdsel);
    case 3: return touch_fits<3>(c->gs, gdsel);
    default: return touch_fits<4>(c->gs, gdsel);
  }
}

template <int P, int GD>
static efie_status launch_touch(Ctx *c, const TouchArgs &A) {
  const size_t smem = sizeof(double) * touch_smem_doubles<P, GD>(A.g);
  EFIE_TRY((allow_smem<kTouchSmem>(c, k_near_touch<P, GD>, smem)));
  k_near_touch<P, GD><<<A.ntodo, TouchCfg<P>::kThreads, smem, c->stream>>>(A);
  ++c->launches;
  EFIE_CUDA(cudaGetLastError());
  return EFIE_OK;
}

// Blocks of the touching pairs `todo` (device list), Gauss rule (x, w) of c->gs points.
efie_status dev_near_touch(Ctx *c, const NearPair *pairs, const int *todo, int ntodo, const int *slot, const double *x,
                           const double *w, int gdsel) {
  const TouchArgs A = {c->d_patches, c->d_knots, c->d_cpw, pairs, todo, slot, ntodo, c->n, c->gs, x, w,
                       c->kappa, 1.0 / c->n, c->d_nblk};
#define EFIE_TOUCH(PP)                                                  \
  if (c->p == PP)                                                       \
    return gdsel == 2 ? launch_touch<PP, 2>(c, A)                       \
                      : (gdsel == 4 ? launch_touch<PP, 4>(c, A) : launch_touch<PP, 8>(c, A));
  EFIE_TOUCH(1)
  EFIE_TOUCH(2)
  EFIE_TOUCH(3)
  EFIE_TOUCH(4)
#undef EFIE_TOUCH
  c->err = "device near-field quadrature supports 1 <= p <= 4";
  return EFIE_EINVAL;
}

}  // namespace efie
