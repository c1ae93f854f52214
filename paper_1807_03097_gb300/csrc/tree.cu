// The stages of a product around the M2L: leaf moments (a4), M2M (a5) and the fold of the vector moments
// into Cartesian sources on the way up; unfold, L2L (a7) and the evaluation at the test functions (a8) on
// the way down.
//   mu_beta(m) = h^2 sum_ab M[m1][a] M[m2][b] x*_{beta,b,a}
//   nu(m)      = h sum_ab (Md[m1][a] M[m2][b] x*_{0,b,a} + M[m1][a] Md[m2][b] x*_{1,b,a})
//   parent(f, m2, m1)   = sum_c sum_{m2'} E[c2][m2][m2'] sum_{m1'} E[c1][m1][m1'] child_c(f, m2', m1')
//   source: u_k = d_1 F_k mu_1 + d_2 F_k mu_2 (k = 1, 2, 3) and nu
//   local:  l_alpha = sum_k d_alpha F_k a_k, l_div = -kappa^-2 a_4 from the M2L result a, plus the parent's
//   child_c(f, m2', m1') += sum_{m2} E[c2][m2][m2'] sum_{m1} E[c1][m1][m1'] parent(f, m2, m1)
//   y*_{0,b,a} = h^2 sum_m M[m1][a] M[m2][b] l_0(m) + h sum_m Md[m1][a] M[m2][b] l_div(m), y*_1 alike
//
// One block per parent cluster and right-hand side.  The moments of its four children go to the parent from
// shared memory and a cluster's source is written where its moments are made; on the way down a
// child's M2L result is unfolded where the parent's expansion is added, and leaves are evaluated in
// place.  So a product takes 2 m launches here (2 m + 4 as separate stages; one more where source lists are split), and the moments and
// expansions of the leaves, three quarters of all, never touch memory.  Measured, whole
// mixed product before and after (with the T and T^T launches of all vectors as one): 96 elements 110 -> 92 us, 13 068
// unknowns 4.34 -> 4.24 ms, leaf-level variant 0.511 -> 0.434 ms, 64 right-hand sides on 1 024 elements 37.7 -> 35.8 ms.
#include <algorithm>

#include "efie_internal.h"

namespace efie {

namespace {

template <class R> struct Cx;
template <> struct Cx<double> { using T = double2; };
template <> struct Cx<float> { using T = float2; };
template <class R> using C2 = typename Cx<R>::T;
template <class R> __device__ __forceinline__ C2<R> mk(R a, R b) {
  C2<R> v;
  v.x = a;
  v.y = b;
  return v;
}
template <class R> __device__ __forceinline__ void fma2(C2<R> &s, R a, C2<R> b) {
  s.x += a * b.x;
  s.y += a * b.y;
}

constexpr int kTreeThreads = 256;

// What all stages share.  Fields of the M2L: FP32 [cluster nI + node] ld + 4 r + f, FP64 [cluster][f][node].
template <class R>
struct TreeArgs {
  int q1, p1, nI;
  const R *M, *Md, *E;  // [q1][p1], [q1][p1], [2][q1][q1]
  const R *D;           // [cluster][node][6]: d_1 F, d_2 F
  R h, ik2;
  int ld;
};

template <class R>
__device__ __forceinline__ size_t field(const TreeArgs<R> &A, int id, int m, int r, int f, int ld) {
  return sizeof(R) == 8 ? ((size_t)id * 4 + f) * A.nI + m : ((size_t)id * A.nI + m) * ld + 4 * r + f;
}

// Largest |Re|, |Im| of the folded sources of a block's clusters, for the fixed point of the FP64 M2L
// (bit patterns of non-negative doubles order as integers; infinities and NaN come out above all).
struct FieldMax {
  unsigned long long v[4] = {0, 0, 0, 0};
  __device__ __forceinline__ void note(int f, double2 z) {
    const unsigned long long a = __double_as_longlong(fabs(z.x)), b = __double_as_longlong(fabs(z.y));
    v[f] = max(v[f], max(a, b));
  }
  __device__ __forceinline__ void note(int, float2) {}
  __device__ __forceinline__ void flush(unsigned long long *out) {  // all threads of the block
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      unsigned long long m = v[f];
      for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
      if ((threadIdx.x & 31) == 0 && m > *reinterpret_cast<volatile unsigned long long *>(out + f)) atomicMax(out + f, m);
    }
  }
};

// source of node m of cluster id from its moments in shared memory [3][nI]
template <class R>
__device__ __forceinline__ void fold_node(const TreeArgs<R> &A, int id, int m, int r, const C2<R> *mom,
                                          C2<R> *__restrict__ src, FieldMax &fm) {
  const R *D = A.D + ((size_t)id * A.nI + m) * 6;
  const C2<R> m0 = mom[m], m1 = mom[A.nI + m], nu = mom[2 * A.nI + m];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const C2<R> u = mk<R>(D[k] * m0.x + D[3 + k] * m1.x, D[k] * m0.y + D[3 + k] * m1.y);
    src[field(A, id, m, r, k, A.ld)] = u;
    fm.note(k, u);
  }
  src[field(A, id, m, r, 3, A.ld)] = nu;
  fm.note(3, nu);
}

// parent moments par[3][nI] from ch[4][3][nI] through T[4][3][nI] (all shared memory, par may be ch)
template <class R>
__device__ __forceinline__ void m2m_block(const TreeArgs<R> &A, const R *sE, const C2<R> *ch, C2<R> *T, C2<R> *par) {
  const int q1 = A.q1, nI = A.nI;
  for (int i = threadIdx.x; i < 12 * nI; i += blockDim.x) {
    const int cf = i / nI, rem = i % nI, m2p = rem / q1, m1 = rem % q1, c1 = (cf / 3) & 1;
    C2<R> s = mk<R>(0, 0);
    const C2<R> *p = ch + cf * nI + m2p * q1;
    const R *e = sE + (c1 * q1 + m1) * q1;
    for (int k = 0; k < q1; ++k) fma2<R>(s, e[k], p[k]);
    T[i] = s;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 3 * nI; i += blockDim.x) {
    const int f = i / nI, rem = i % nI, m2 = rem / q1, m1 = rem % q1;
    C2<R> s = mk<R>(0, 0);
    for (int c = 0; c < 4; ++c) {
      const C2<R> *t = T + (c * 3 + f) * nI + m1;
      const R *e = sE + ((c >> 1) * q1 + m2) * q1;
      for (int k = 0; k < q1; ++k) fma2<R>(s, e[k], t[k * q1]);
    }
    par[i] = s;
  }
  __syncthreads();
}

// unfolded local expansion, component f (0, 1 vector, 2 div)
template <class R>
__device__ __forceinline__ C2<R> unfold_value(const TreeArgs<R> &A, const C2<R> *__restrict__ acc, int id, int m, int r, int f) {
  if (f == 2) {
    const C2<R> v = acc[field(A, id, m, r, 3, A.ld)];
    return mk<R>(-A.ik2 * v.x, -A.ik2 * v.y);
  }
  const R *D = A.D + ((size_t)id * A.nI + m) * 6 + 3 * f;
  C2<R> s = mk<R>(0, 0);
#pragma unroll
  for (int k = 0; k < 3; ++k) fma2<R>(s, D[k], acc[field(A, id, m, r, k, A.ld)]);
  return s;
}

template <class R>
__host__ __device__ constexpr size_t up_leaf_smem(int q1, int p1, int nc) {
  const size_t nI = (size_t)q1 * q1, c = sizeof(C2<R>);
  return c * (nc * 2 * p1 * p1 + nc * 3 * p1 * q1 + nc * 3 * nI + (nc == 4 ? 12 * nI : 0)) +
         sizeof(R) * (2 * q1 * p1 + 2 * q1 * q1);
}

}  // namespace

// Leaf moments and sources of the NC leaves of a block, and (NC = 4) the moments and source of their parent.
template <class R, int NC>
__global__ void __launch_bounds__(kTreeThreads) k_up_leaf(TreeArgs<R> A, int leaf_off, int par_off,
                                                          const double2 *__restrict__ xs, size_t xstride,
                                                          C2<R> *__restrict__ mom, size_t mstride, C2<R> *__restrict__ src,
                                                          unsigned long long *smax_leaf, unsigned long long *smax_par) {
  const int q1 = A.q1, p1 = A.p1, nI = A.nI, r = blockIdx.y, p2 = p1 * p1;
  extern __shared__ double2 smt[];
  C2<R> *sx = reinterpret_cast<C2<R> *>(smt);  // [NC][2 p2]
  C2<R> *T0 = sx + NC * 2 * p2;                // [NC][3][p1][q1]: x_0, x_1 by M; x_0 by Md
  C2<R> *ch = T0 + NC * 3 * p1 * q1;           // [NC][3][nI]
  C2<R> *T = ch + NC * 3 * nI;                 // [12][nI] (NC = 4)
  R *sM = reinterpret_cast<R *>(T + (NC == 4 ? 12 * nI : 0)), *sMd = sM + q1 * p1, *sE = sMd + q1 * p1;
  const int e0 = blockIdx.x * NC;
  for (int i = threadIdx.x; i < q1 * p1; i += blockDim.x) {
    sM[i] = A.M[i];
    sMd[i] = A.Md[i];
  }
  if (NC == 4)
    for (int i = threadIdx.x; i < 2 * nI; i += blockDim.x) sE[i] = A.E[i];
  for (int i = threadIdx.x; i < NC * 2 * p2; i += blockDim.x) {
    const double2 v = xs[r * xstride + (size_t)e0 * 2 * p2 + i];
    sx[i] = mk<R>((R)v.x, (R)v.y);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < NC * p1 * q1; i += blockDim.x) {
    const int c = i / (p1 * q1), b = (i / q1) % p1, m1 = i % q1;
    C2<R> a0 = mk<R>(0, 0), a1 = a0, ad = a0;
    for (int a = 0; a < p1; ++a) {
      const R M = sM[m1 * p1 + a], Md = sMd[m1 * p1 + a];
      const C2<R> x0 = sx[c * 2 * p2 + b * p1 + a], x1 = sx[c * 2 * p2 + p2 + b * p1 + a];
      fma2<R>(a0, M, x0);
      fma2<R>(a1, M, x1);
      fma2<R>(ad, Md, x0);
    }
    C2<R> *o = T0 + (c * 3 * p1 + b) * q1 + m1;
    o[0] = a0;
    o[p1 * q1] = a1;
    o[2 * p1 * q1] = ad;
  }
  __syncthreads();
  const R h = A.h, h2 = h * h;
  for (int i = threadIdx.x; i < NC * nI; i += blockDim.x) {
    const int c = i / nI, mi = i % nI, m1 = mi % q1, m2 = mi / q1;
    C2<R> u0 = mk<R>(0, 0), u1 = u0, v = u0;
    for (int b = 0; b < p1; ++b) {
      const R M = sM[m2 * p1 + b], Md = sMd[m2 * p1 + b];
      const C2<R> *t = T0 + (c * 3 * p1 + b) * q1 + m1;
      const C2<R> t0 = t[0], t1 = t[p1 * q1], td = t[2 * p1 * q1];
      fma2<R>(u0, M, t0);
      fma2<R>(u1, M, t1);
      v.x += M * td.x + Md * t1.x;
      v.y += M * td.y + Md * t1.y;
    }
    C2<R> *o = ch + c * 3 * nI + mi;
    o[0] = mk<R>(h2 * u0.x, h2 * u0.y);
    o[nI] = mk<R>(h2 * u1.x, h2 * u1.y);
    o[2 * nI] = mk<R>(h * v.x, h * v.y);
  }
  __syncthreads();
  FieldMax fl;
  for (int i = threadIdx.x; i < NC * nI; i += blockDim.x)
    fold_node<R>(A, leaf_off + e0 + i / nI, i % nI, r, ch + (i / nI) * 3 * nI, src, fl);
  if (sizeof(R) == 8 && smax_leaf) fl.flush(smax_leaf);
  if (NC == 1) {
    C2<R> *out = mom + r * mstride + (size_t)(leaf_off + e0) * 3 * nI;
    for (int i = threadIdx.x; i < 3 * nI; i += blockDim.x) out[i] = ch[i];
    return;
  }
  m2m_block<R>(A, sE, ch, T, ch);  // (every thread has folded its leaves before the parent overwrites them)
  const int id = par_off + blockIdx.x;
  C2<R> *out = mom + r * mstride + (size_t)id * 3 * nI;
  for (int i = threadIdx.x; i < 3 * nI; i += blockDim.x) out[i] = ch[i];
  FieldMax fp;
  for (int i = threadIdx.x; i < nI; i += blockDim.x) fold_node<R>(A, id, i, r, ch, src, fp);
  if (sizeof(R) == 8 && smax_par) fp.flush(smax_par);
}

// Moments and source of a cluster from its children's moments.
template <class R>
__global__ void __launch_bounds__(kTreeThreads) k_up(TreeArgs<R> A, int par_off, int ch_off, C2<R> *__restrict__ mom,
                                                     size_t mstride, C2<R> *__restrict__ src, unsigned long long *smax) {
  const int nI = A.nI, r = blockIdx.y, id = par_off + blockIdx.x;
  extern __shared__ double2 smt[];
  C2<R> *ch = reinterpret_cast<C2<R> *>(smt), *T = ch + 12 * nI;
  R *sE = reinterpret_cast<R *>(T + 12 * nI);
  mom += r * mstride;
  for (int i = threadIdx.x; i < 2 * nI; i += blockDim.x) sE[i] = A.E[i];
  const C2<R> *cm = mom + (size_t)(ch_off + 4 * blockIdx.x) * 3 * nI;
  for (int i = threadIdx.x; i < 12 * nI; i += blockDim.x) ch[i] = cm[i];
  __syncthreads();
  m2m_block<R>(A, sE, ch, T, ch);
  C2<R> *out = mom + (size_t)id * 3 * nI;
  for (int i = threadIdx.x; i < 3 * nI; i += blockDim.x) out[i] = ch[i];
  FieldMax fm;
  for (int i = threadIdx.x; i < nI; i += blockDim.x) fold_node<R>(A, id, i, r, ch, src, fm);
  if (sizeof(R) == 8 && smax) fm.flush(smax);
}

// acc += the further partial results of an M2L whose source lists were split, in order.  A pass of its own:
// the stages below read a result three times, and with 9 to 16 splits (small problems) that
// took 20 us a level instead of 4 once.
template <class R>
__global__ void k_add_splits(size_t rows, int cols, int ld, int ldm, int nslab, size_t slab, const C2<R> *__restrict__ more,
                             C2<R> *__restrict__ acc) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= rows * cols) return;
  const size_t row = t / cols, col = t % cols;
  C2<R> v = acc[row * ld + col];
#pragma unroll 4
  for (int j = 0; j < nslab - 1; ++j) {
    const C2<R> b = more[j * slab + row * ldm + col];
    v.x += b.x;
    v.y += b.y;
  }
  acc[row * ld + col] = v;
}

// Local expansions of the children of a cluster; LEAF: the children are leaves, evaluated into ys.  The
// cluster's own expansion is in loc, or (root) unfolded here.  NC = 1: a root that is a leaf.
template <class R, bool LEAF, int NC>
__global__ void __launch_bounds__(kTreeThreads) k_down(TreeArgs<R> A, const C2<R> *__restrict__ acc, int par_off, int ch_off, int root,
                                                       C2<R> *__restrict__ loc, size_t lstride, double2 *__restrict__ ys,
                                                       size_t ystride) {
  const int q1 = A.q1, p1 = A.p1, nI = A.nI, r = blockIdx.y;
  extern __shared__ double2 smt[];
  C2<R> *par = reinterpret_cast<C2<R> *>(smt);  // [3][nI]
  C2<R> *T = par + 3 * nI;                      // [2][3][nI]
  C2<R> *lc = T + 6 * nI;                       // [NC][3][nI] (LEAF)
  C2<R> *Q = lc + (LEAF ? NC * 3 * nI : 0);     // [NC][4][q1][p1] (LEAF): l_0, l_1, l_2 by M; l_2 by Md
  R *sE = reinterpret_cast<R *>(Q + (LEAF ? NC * 4 * q1 * p1 : 0)), *sM = sE + 2 * nI, *sMd = sM + q1 * p1;
  loc += r * lstride;
  for (int i = threadIdx.x; i < 2 * nI; i += blockDim.x) sE[i] = A.E[i];
  if (LEAF)
    for (int i = threadIdx.x; i < q1 * p1; i += blockDim.x) {
      sM[i] = A.M[i];
      sMd[i] = A.Md[i];
    }
  const int id = par_off + blockIdx.x;
  for (int i = threadIdx.x; i < 3 * nI; i += blockDim.x)
    (NC == 1 ? lc : par)[i] = root ? unfold_value<R>(A, acc, id, i % nI, r, i / nI) : loc[(size_t)id * 3 * nI + i];
  __syncthreads();
  if (NC == 4) {
    for (int i = threadIdx.x; i < 6 * nI; i += blockDim.x) {
      const int c1 = i / (3 * nI), rem = i % (3 * nI), f = rem / nI, m2 = (rem % nI) / q1, m1p = rem % nI % q1;
      C2<R> s = mk<R>(0, 0);
      const C2<R> *pp = par + f * nI + m2 * q1;
      const R *e = sE + c1 * nI + m1p;
      for (int k = 0; k < q1; ++k) fma2<R>(s, e[k * q1], pp[k]);
      T[i] = s;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 12 * nI; i += blockDim.x) {
      const int c = i / (3 * nI), rem = i % (3 * nI), f = rem / nI, m = rem % nI, m2p = m / q1, m1p = m % q1;
      const C2<R> *tt = T + ((c & 1) * 3 + f) * nI + m1p;
      const R *e = sE + (c >> 1) * nI + m2p;
      C2<R> s = mk<R>(0, 0);
      for (int k = 0; k < q1; ++k) fma2<R>(s, e[k * q1], tt[k * q1]);
      const int cid = ch_off + 4 * blockIdx.x + c;
      const C2<R> o = unfold_value<R>(A, acc, cid, m, r, f);
      const C2<R> v = mk<R>(o.x + s.x, o.y + s.y);
      if (LEAF) lc[i] = v;
      else loc[(size_t)cid * 3 * nI + rem] = v;
    }
    if (LEAF) __syncthreads();
  }
  if (!LEAF) return;
  for (int i = threadIdx.x; i < NC * q1 * p1; i += blockDim.x) {
    const int c = i / (q1 * p1), m2 = (i / p1) % q1, a = i % p1;
    const C2<R> *l = lc + c * 3 * nI + m2 * q1;
    C2<R> s0 = mk<R>(0, 0), s1 = s0, s2 = s0, sd = s0;
    for (int k = 0; k < q1; ++k) {
      const R M = sM[k * p1 + a], Md = sMd[k * p1 + a];
      fma2<R>(s0, M, l[k]);
      fma2<R>(s1, M, l[nI + k]);
      fma2<R>(s2, M, l[2 * nI + k]);
      fma2<R>(sd, Md, l[2 * nI + k]);
    }
    C2<R> *o = Q + c * 4 * q1 * p1 + m2 * p1 + a;
    o[0] = s0;
    o[q1 * p1] = s1;
    o[2 * q1 * p1] = s2;
    o[3 * q1 * p1] = sd;
  }
  __syncthreads();
  const R h = A.h, h2 = h * h;
  const int p2 = p1 * p1;
  for (int i = threadIdx.x; i < NC * 2 * p2; i += blockDim.x) {
    const int c = i / (2 * p2), al = (i / p2) & 1, b = (i / p1) % p1, a = i % p1;
    const C2<R> *q = Q + c * 4 * q1 * p1 + a;
    R ax = 0, ay = 0;
    for (int m2 = 0; m2 < q1; ++m2) {
      const R M = sM[m2 * p1 + b], W = al == 0 ? M : sMd[m2 * p1 + b];
      const C2<R> u = q[(al * q1 + m2) * p1], d = q[((al == 0 ? 3 : 2) * q1 + m2) * p1];
      ax += h2 * M * u.x + h * W * d.x;
      ay += h2 * M * u.y + h * W * d.y;
    }
    ys[r * ystride + (size_t)blockIdx.x * NC * 2 * p2 + i] = make_double2((double)ax, (double)ay);
  }
}

namespace {

TreeArgs<float> tree_args(const Ctx *c, const float *D, int ld) {
  return {c->q1, c->p1, c->nI, c->d_Mf, c->d_Mdf, c->d_Ef, D, (float)(1.0 / c->n), (float)(1.0 / (c->kappa * c->kappa)), ld};
}
TreeArgs<double> tree_args(const Ctx *c, const double *D, int ld) {
  return {c->q1, c->p1, c->nI, c->d_M, c->d_Md, c->d_E, D, 1.0 / c->n, 1.0 / (c->kappa * c->kappa), ld};
}

// dynamic shared memory of k_up and k_down (leaves: of NC children evaluated in the block); their largest
// sizes at kMaxQ1, kMaxP1 are the functions' limits
template <class R>
constexpr size_t up_smem(int q1) {
  return sizeof(C2<R>) * 24 * q1 * q1 + sizeof(R) * 2 * q1 * q1;
}
template <class R>
constexpr size_t down_smem(int q1, int p1, int leaves) {
  const size_t nI = (size_t)q1 * q1;
  return sizeof(C2<R>) * 9 * nI + sizeof(R) * (2 * nI + 2 * q1 * p1) + leaves * sizeof(C2<R>) * (3 * nI + 4 * q1 * p1);
}

// Leaves with their parents in one block; not in FP64 while the parents are fewer than the SMs: the FP64
// pipe of an SM is slow enough that four times the blocks gain more than a launch costs.
template <class R>
bool leaves_fused(const Ctx *c) {
  return c->m > 0 && (sizeof(R) == 4 || c->nE / 4 >= c->nsm);
}

template <class R>
efie_status up(Ctx *c, cudaStream_t st, int nrhs, const R *D, const double2 *xs, size_t xstride, C2<R> *mom, size_t mstride,
               C2<R> *src, int ld, unsigned long long *smax) {
  const TreeArgs<R> A = tree_args(c, D, ld);
  const int m = c->m;
  auto mx = [&](int l) { return smax ? smax + 4 * l : nullptr; };
  const bool fused = leaves_fused<R>(c);
  if (!fused) {
    const size_t sm = up_leaf_smem<R>(c->q1, c->p1, 1);
    EFIE_TRY((allow_smem<up_leaf_smem<R>(kMaxQ1, kMaxP1, 1)>(c, k_up_leaf<R, 1>, sm)));
    k_up_leaf<R, 1><<<dim3(c->nE, nrhs), kTreeThreads, sm, st>>>(A, c->lev_off[m], 0, xs, xstride, mom, mstride, src, mx(m),
                                                              nullptr);
    ++c->launches;
  } else {
    const size_t sm = up_leaf_smem<R>(c->q1, c->p1, 4);
    EFIE_TRY((allow_smem<up_leaf_smem<R>(kMaxQ1, kMaxP1, 4)>(c, k_up_leaf<R, 4>, sm)));
    k_up_leaf<R, 4><<<dim3(c->nE / 4, nrhs), kTreeThreads, sm, st>>>(A, c->lev_off[m], c->lev_off[m - 1], xs, xstride, mom,
                                                                  mstride, src, mx(m), mx(m - 1));
    ++c->launches;
  }
  const size_t sm = up_smem<R>(c->q1);
  EFIE_TRY((allow_smem<up_smem<R>(kMaxQ1)>(c, k_up<R>, sm)));
  for (int l = m - (fused ? 2 : 1); l >= 0; --l) {
    k_up<R><<<dim3(c->np << (2 * l), nrhs), kTreeThreads, sm, st>>>(A, c->lev_off[l], c->lev_off[l + 1], mom, mstride, src, mx(l));
    ++c->launches;
  }
  EFIE_CUDA(cudaGetLastError());
  return EFIE_OK;
}

template <class R>
efie_status down(Ctx *c, cudaStream_t st, int nrhs, const R *D, int ld, const C2<R> *acc, C2<R> *loc, size_t lstride,
                 double2 *ys, size_t ystride) {
  const TreeArgs<R> A = tree_args(c, D, ld);
  const int m = c->m;
  const size_t base = down_smem<R>(c->q1, c->p1, 0);
  const bool fused = leaves_fused<R>(c);
  EFIE_TRY((allow_smem<down_smem<R>(kMaxQ1, kMaxP1, 0)>(c, k_down<R, false, 4>, base)));
  for (int l = 0; l < m - (fused ? 1 : 0); ++l) {
    k_down<R, false, 4><<<dim3(c->np << (2 * l), nrhs), kTreeThreads, base, st>>>(A, acc, c->lev_off[l], c->lev_off[l + 1],
                                                                                  l == 0, loc, lstride, ys, ystride);
    ++c->launches;
  }
  if (fused) {
    const size_t sm = down_smem<R>(c->q1, c->p1, 4);
    EFIE_TRY((allow_smem<down_smem<R>(kMaxQ1, kMaxP1, 4)>(c, k_down<R, true, 4>, sm)));
    k_down<R, true, 4><<<dim3(c->nE / 4, nrhs), kTreeThreads, sm, st>>>(A, acc, c->lev_off[m - 1], c->lev_off[m], m == 1,
                                                                     loc, lstride, ys, ystride);
  } else {
    const size_t sm = down_smem<R>(c->q1, c->p1, 1);
    EFIE_TRY((allow_smem<down_smem<R>(kMaxQ1, kMaxP1, 1)>(c, k_down<R, true, 1>, sm)));
    k_down<R, true, 1><<<dim3(c->nE, nrhs), kTreeThreads, sm, st>>>(A, acc, c->lev_off[m], 0, m == 0, loc, lstride, ys,
                                                                 ystride);
  }
  ++c->launches;
  EFIE_CUDA(cudaGetLastError());
  return EFIE_OK;
}

}  // namespace

efie_status tree_up_f32(Ctx *c, cudaStream_t st, int nrhs, const double2 *xs, float2 *mom, float2 *src, int ld) {
  return up<float>(c, st, nrhs, c->d_nodeDf, xs, (size_t)c->nsup, mom, (size_t)c->ncl * 3 * c->nI, src, ld, nullptr);
}
efie_status tree_up_f64(Ctx *c, cudaStream_t st, const double2 *xs, double2 *mom, double2 *src, unsigned long long *smax) {
  return up<double>(c, st, 1, c->d_nodeD, xs, 0, mom, 0, src, 0, smax);
}
efie_status tree_down_f32(Ctx *c, cudaStream_t st, int nrhs, float2 *acc, int ld, const float2 *more, int ldm, int nslab,
                          size_t slab, float2 *loc, double2 *ys) {
  if (nslab > 1) {
    const size_t rows = (size_t)c->ncl * c->nI, tot = rows * 4 * nrhs;
    k_add_splits<float><<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(rows, 4 * nrhs, ld, ldm, nslab, slab, more, acc);
    ++c->launches;
  }
  return down<float>(c, st, nrhs, c->d_nodeDf, ld, acc, loc, (size_t)c->ncl * 3 * c->nI, ys, (size_t)c->nsup);
}
efie_status tree_down_f64(Ctx *c, cudaStream_t st, double2 *acc, const double2 *more, int nslab, size_t slab, double2 *loc,
                          double2 *ys) {
  if (nslab > 1) {
    k_add_splits<double><<<(unsigned)((slab + 255) / 256), 256, 0, st>>>(slab, 1, 1, 1, nslab, slab, more, acc);
    ++c->launches;
  }
  return down<double>(c, st, 1, c->d_nodeD, 0, acc, loc, 0, ys, 0);
}

}  // namespace efie
