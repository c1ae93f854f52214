// M2L of one or a few right-hand sides in the mixed form (a6, Sec. 4.2): for every target
// cluster t and target node i, acc(i, f) = sum_s sum_j G(x_ti, x_sj) w_s(j, f) over the admissible
// sources s, G = e^{i kappa r} / (4 pi r) and 4 complex fields f per right-hand side.
//
// A warp holds 16-row tiles of target nodes and sweeps the flattened list of source nodes (source
// cluster, node) of its target, 8 nodes at a time.  The kernel entries are evaluated by the lane
// that holds them in the A operand of mma.sync.m16n8k8 (TF32), so that they go from the
// special-function unit into the tensor core without passing through memory; the 4 complex
// fields of a right-hand side are the 8 columns of B (Re, Im in turn), and a complex product is two
// real ones, Re G x (Re w, Im w) + Im G x (-Im w, Re w).  tcgen05 would want the entries in shared
// or tensor memory and at least 16 columns: with one right-hand side the tile would be written
// and read once for half the columns in use.
//
// Precision.  Both operands are split x = hi + lo with hi in TF32 (11 bits): the fields rounded
// (|lo| <= 2^-12 |x|), the entries truncated, because the tensor core reads the upper 19 bits of a
// register as it is: hi costs no instruction then, lo = x - (x & mask) two.  Of lo's 13 bits the tensor
// core in turn drops up to two, 0.875 units of 2^-23 on average over evenly distributed lo, which is
// 7.5e-8 of x over evenly distributed logarithms; that mean is given back when the sums are
// written.  hi hi + hi lo + lo hi leaves out about 2^-23.  The tensor core truncates when it accumulates, so
// every 8 source nodes get a fresh accumulator (the four small products first), which is added
// to FP32 sums on the CUDA cores; these enter the running sums by two-sum (compensated) addition
// once per 64 source nodes.  The two large products of a step still shorten its accumulator by half a unit of
// 2^-23 each on average, 6.4e-8 of the sum: at kappa <= 1, where the phases' errors are small, the far part is
// 9e-8 to 13e-8 too small (FP32 sums on the CUDA cores: up to 6e-8) and the whole product up to 1.23 times as far
// from 64 bits, at kappa >= 3 0.3 to 0.7 times.  kCut = 1.39e-7 would give that mean back too (1.13 times); it was
// taken back because it moves residuals at the tolerance of a solve by some percent, and so the step at which
// some stop (a cube of 24 elements in a group: errors of 1e-6 instead of 1e-7 to 6e-7 at a tolerance of 1e-6).
//
// Kernel entry.  Per source node and target, y = x_s - d with d = c_t - c_s is the node seen from
// the target's centre and a = |y|; the fields carry e^{i kappa a} / (4 pi), from the FP64 phase of
// the centres times e^{i kappa (a - r0)} with a - r0 = (|x_s|^2 - 2 d.x_s) / (a + r0).  Per entry,
// num = r^2 - a^2 = |x_t|^2 - 2 x_t.y has no cancellation against a^2, and delta = r - a solves
// delta (delta + 2 a) = num: one Newton step from r^2 rsqrt(r^2) - a takes the place of a
// reciprocal (three FP32 operations against 8 cycles of the special-function unit) and leaves
// delta with an error of a few 2^-24 of |x_t|, not of r.
//
// Bound: the issue slots and register ports of a scheduler, about 36 clocks per 32 entries: 13 packed
// FP32 instructions per two entries at 2 to 3 clocks, 6 mma per 4 entries at 7 (an mma.sync holds
// the ports that long), the special-function unit at 24.  Measured, M2L of one right-hand side: 4.38 ->
// 4.01 ms at 519 480 pairs of 81 nodes, 1.34 -> 1.05 ms at 125 760, 92 -> 18 us at 5 472 pairs of 25 nodes
// (split lists), 15.7 -> 0.82 ms for two right-hand sides with 144 nodes; error of the product against
// 64 bits 4.2e-7 -> 1.6e-7 (sphere, kappa = 10).  More warps with fewer tiles (2 or 1 a warp), fewer registers,
// separate accumulators for Re G and Im G, and 128 nodes a stage were measured and slower by 1 to 20 %.  Entries
// rounded instead of truncated to hi: 7 % slower at 81 nodes, 3 % at 49, products 1 to 7 % closer to 64 bits.
#include <algorithm>

#include "efie_internal.h"
#include "fastmath.cuh"

namespace efie {

namespace {

constexpr int kMmaNodes = 64;   // source nodes staged at a time
constexpr int kMmaSteps = kMmaNodes / 8;
constexpr float kCut = 7.5e-8f; // mean share of an entry lost to the truncation of its lo part
constexpr int kMmaMaxWarps = 7; // ceil(17^2 / 16) = 19 row tiles, 3 per warp

// Shared memory of one block (float4 units): B fragments [step][rhs][re, im][lane] (steps 64 bytes
// apart more than their size, against bank conflicts of the staging stores), constants of the
// source nodes [node][3], running sums and compensation [warp][rhs][tile][2][lane].
template <int MT, int NR>
struct MmaLayout {
  static constexpr int kStep = NR * 2 * 32 + 4;
  static constexpr int kB = kMmaSteps * kStep;
  static constexpr int kC = 3 * kMmaNodes;
  static constexpr int kH = NR * MT * 2 * 32;  // per warp
  static constexpr size_t bytes(int warps) { return sizeof(float4) * (kB + kC + (size_t)warps * kH); }
};

__device__ __forceinline__ float tf32_hi(float x) {
  return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xffffe000u);
}

// the part of x that the tensor core reads
__device__ __forceinline__ float tf32_cut(float x) { return __uint_as_float(__float_as_uint(x) & 0xffffe000u); }

__device__ __forceinline__ void mma_tf32(float (&c)[4], const float (&a)[4], float b0, float b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(__float_as_uint(a[0])), "r"(__float_as_uint(a[1])), "r"(__float_as_uint(a[2])), "r"(__float_as_uint(a[3])),
        "r"(__float_as_uint(b0)), "r"(__float_as_uint(b1)));
}

__device__ __forceinline__ void two_sum2(float2 &h, float2 &l, float2 b) {
  const float2 s = make_float2(h.x + b.x, h.y + b.y), p = make_float2(s.x - h.x, s.y - h.y);
  l.x += (h.x - (s.x - p.x)) + (b.x - p.x);
  l.y += (h.y - (s.y - p.y)) + (b.y - p.y);
  h = s;
}

// Row constants of one tile (rows g and g + 8 packed): 2 x_t and -|x_t|^2.
struct RowConst {
  float2 ux, uy, uz, un;
};

// NT row tiles x the staged source nodes: part += G w (packed accumulator registers 0-1, 2-3).
// The stages of the evaluation run over all tiles in turn, and the accumulators of a step are added
// to the sums in the next step, so that a warp has 2 NT independent chains under way while its
// MMAs run.
template <int NT, int MT, int NR, bool FAST>
__device__ __forceinline__ void sweep(const RowConst (&u)[MT], const float4 *__restrict__ sB,
                                      const float4 *__restrict__ sC, int steps, int lane, float kappa,
                                      float2 (&part)[NR][MT][2]) {
  const float2 m1 = make_float2(-1.f, -1.f), mh = make_float2(-0.5f, -0.5f), kap = make_float2(kappa, kappa);
  const int q = lane & 3;
  float s[NR][NT][4];
#pragma unroll
  for (int r = 0; r < NR; ++r)
#pragma unroll
    for (int i = 0; i < NT; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) s[r][i][e] = 0.f;
#pragma unroll 1
  for (int ks = 0; ks < steps; ++ks) {
    // entries (rows g, g + 8) x (nodes q, q + 4 for h = 0, 1), the order of the A fragment
    float2 ri[NT][2], p[NT][2], v[NT][2];
    const float4 *cs = sC + 3 * (8 * ks + q);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float4 c0 = cs[12 * h], c1 = cs[12 * h + 1];
#pragma unroll
      for (int i = 0; i < NT; ++i) {
        float2 x = __ffma2_rn(u[i].ux, make_float2(c0.x, c0.y), u[i].un);  // -num
        x = __ffma2_rn(u[i].uy, make_float2(c0.z, c0.w), x);
        x = __ffma2_rn(u[i].uz, make_float2(c1.x, c1.y), x);
        v[i][h] = x;
        p[i][h] = __ffma2_rn(x, m1, make_float2(c1.z, c1.w));  // r^2
        ri[i][h] = make_float2(rsqrt_ftz(p[i][h].x), rsqrt_ftz(p[i][h].y));
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float4 c2 = cs[12 * h + 2];
#pragma unroll
      for (int i = 0; i < NT; ++i) {
        const float2 dl = __ffma2_rn(p[i][h], ri[i][h], make_float2(c2.x, c2.y));
        const float2 e = __ffma2_rn(dl, __fadd2_rn(dl, make_float2(c2.z, c2.w)), v[i][h]);
        float2 x = __ffma2_rn(__fmul2_rn(ri[i][h], e), mh, dl);
        if (!FAST) {
          const float inv2pi = 0.15915494309189535f, p1 = 6.28318548202514648f, p2 = -1.7484555e-7f;
          x = __fmul2_rn(x, kap);
          const float2 n = make_float2(-rintf(x.x * inv2pi), -rintf(x.y * inv2pi));
          x = __ffma2_rn(n, make_float2(p1, p1), x);
          x = __ffma2_rn(n, make_float2(p2, p2), x);
        }
        p[i][h] = __fmul2_rn(make_float2(cos_ftz(x.x), cos_ftz(x.y)), ri[i][h]);   // Re G
        v[i][h] = __fmul2_rn(make_float2(sin_ftz(x.x), sin_ftz(x.y)), ri[i][h]);   // Im G
      }
    }
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
      for (int i = 0; i < NT; ++i) {
        part[r][i][0] = __fadd2_rn(part[r][i][0], make_float2(s[r][i][0], s[r][i][1]));
        part[r][i][1] = __fadd2_rn(part[r][i][1], make_float2(s[r][i][2], s[r][i][3]));
      }
    const float4 *bs = sB + ks * MmaLayout<MT, NR>::kStep + lane;
#pragma unroll
    for (int i = 0; i < NT; ++i) {
      float ar[4], ai[4], br[4], bi[4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float2 hr = make_float2(tf32_cut(p[i][h].x), tf32_cut(p[i][h].y));
        const float2 hi = make_float2(tf32_cut(v[i][h].x), tf32_cut(v[i][h].y));
        const float2 lr = __ffma2_rn(hr, m1, p[i][h]), li = __ffma2_rn(hi, m1, v[i][h]);
        ar[2 * h] = p[i][h].x;
        ar[2 * h + 1] = p[i][h].y;
        ai[2 * h] = v[i][h].x;
        ai[2 * h + 1] = v[i][h].y;
        br[2 * h] = lr.x;
        br[2 * h + 1] = lr.y;
        bi[2 * h] = li.x;
        bi[2 * h + 1] = li.y;
      }
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const float4 wr = bs[r * 64], wi = bs[r * 64 + 32];  // (hi 0, hi 1, lo 0, lo 1)
#pragma unroll
        for (int e = 0; e < 4; ++e) s[r][i][e] = 0.f;
        mma_tf32(s[r][i], br, wr.x, wr.y);
        mma_tf32(s[r][i], bi, wi.x, wi.y);
        mma_tf32(s[r][i], ar, wr.z, wr.w);
        mma_tf32(s[r][i], ai, wi.z, wi.w);
        mma_tf32(s[r][i], ar, wr.x, wr.y);
        mma_tf32(s[r][i], ai, wi.x, wi.y);
      }
    }
  }
#pragma unroll
  for (int r = 0; r < NR; ++r)
#pragma unroll
    for (int i = 0; i < NT; ++i) {
      part[r][i][0] = __fadd2_rn(part[r][i][0], make_float2(s[r][i][0], s[r][i][1]));
      part[r][i][1] = __fadd2_rn(part[r][i][1], make_float2(s[r][i][2], s[r][i][3]));
    }
}

}  // namespace

// One block per (target cluster, split of its source list, group of NR right-hand sides).
//   src[(cluster nI + node) ld + 4 r + f], acc likewise for the first split; the others go to
//   more[(split - 1) slab + (cluster nI + node) ldm + 4 r + f] and are added, in order, by k_add_splits.
// FAST: lengths are scaled by kappa while they are staged, so that delta is the phase; else (kappa so
// small or large that squares of scaled lengths could leave the FP32 range, or phases beyond
// +-100 pi) lengths stay as they are, and the phase is reduced to [-pi, pi] (two-constant
// Cody-Waite) before the hardware sine and cosine.
template <int MT, int NR, bool FAST>
__global__ void __launch_bounds__(32 * kMmaMaxWarps, 2) k_m2l_mma(
    const int *__restrict__ targets, const int *__restrict__ fptr, const int *__restrict__ fsrc,
    const float4 *__restrict__ pgeo, const float2 *__restrict__ pph, int nI, int R, int ld, float kappa,
    const float4 *__restrict__ nodeX4, const float2 *__restrict__ src, float2 *__restrict__ acc, float2 *__restrict__ more,
    int ldm, size_t slab) {
  using L = MmaLayout<MT, NR>;
  extern __shared__ float4 sm4[];
  float4 *sB = sm4, *sC = sB + L::kB;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  float4 *sH = sC + L::kC + warp * L::kH;
  const int g = lane >> 2, q = lane & 3;
  const int t = targets[blockIdx.x], r0 = blockIdx.z * NR, nr = min(NR, R - r0);
  const int k0 = fptr[t], total = (fptr[t + 1] - k0) * nI;
  const int nch = (total + kMmaNodes - 1) / kMmaNodes;
  const int c0 = (int)((long long)nch * blockIdx.y / gridDim.y), c1 = (int)((long long)nch * (blockIdx.y + 1) / gridDim.y);
  const int ntile = (nI + 15) / 16;
  src += 4 * r0;
  float2 *out = 4 * r0 + (blockIdx.y == 0 ? acc : more + (blockIdx.y - 1) * slab);
  const int ldo = blockIdx.y == 0 ? ld : ldm;

  // this warp's row tiles are warp, warp + nw, ...; rows beyond nI repeat the last node
  const float sc = FAST ? kappa : 1.f;
  RowConst u[MT];
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    const int row = 16 * (warp + i * nw) + g;
    float4 x = nodeX4[(size_t)t * nI + min(row, nI - 1)], z = nodeX4[(size_t)t * nI + min(row + 8, nI - 1)];
    x = make_float4(sc * x.x, sc * x.y, sc * x.z, 0.f);
    z = make_float4(sc * z.x, sc * z.y, sc * z.z, 0.f);
    u[i].ux = make_float2(2.f * x.x, 2.f * z.x);
    u[i].uy = make_float2(2.f * x.y, 2.f * z.y);
    u[i].uz = make_float2(2.f * x.z, 2.f * z.z);
    u[i].un = make_float2(-(x.x * x.x + x.y * x.y + x.z * x.z), -(z.x * z.x + z.y * z.y + z.z * z.z));
  }
#pragma unroll
  for (int i = 0; i < NR * MT * 2; ++i) sH[i * 32 + lane] = make_float4(0.f, 0.f, 0.f, 0.f);

  for (int c = c0; c < c1; ++c) {
    const int base = c * kMmaNodes, nn = min(kMmaNodes, total - base);
    const int steps = (nn + 7) / 8;
    __syncthreads();
    for (int n = threadIdx.x; n < 8 * steps; n += blockDim.x) {
      const int J = base + min(n, nn - 1);  // nodes past the end of the list: the last one, without fields
      const int k = J / nI, m = J - k * nI;
      const int s = fsrc[k0 + k];
      float4 d = pgeo[k0 + k], x = nodeX4[(size_t)s * nI + m];
      const float2 ph = pph[k0 + k];
      float2 w[NR][4];
#pragma unroll
      for (int r = 0; r < NR; ++r)
#pragma unroll
        for (int f = 0; f < 4; f += 2) {
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          if (n < nn && r < nr) v = *reinterpret_cast<const float4 *>(src + ((size_t)s * nI + m) * ld + 4 * r + f);
          w[r][f] = make_float2(v.x, v.y);
          w[r][f + 1] = make_float2(v.z, v.w);
        }
      d = make_float4(sc * d.x, sc * d.y, sc * d.z, sc * d.w);
      x = make_float4(sc * x.x, sc * x.y, sc * x.z, 0.f);
      const float yx = x.x - d.x, yy = x.y - d.y, yz = x.z - d.z;
      const float aa = yx * yx + yy * yy + yz * yz;
      const float a = aa * rsqrt_ftz(aa);
      const float bb = x.x * x.x + x.y * x.y + x.z * x.z - 2.f * (d.x * x.x + d.y * x.y + d.z * x.z);
      float sn, cs;
      const float da = bb * rcp_ftz(a + d.w);
      sincosf(FAST ? da : kappa * da, &sn, &cs);
      const float pr = sc * (ph.x * cs - ph.y * sn), pi = sc * (ph.x * sn + ph.y * cs);
      sC[3 * n] = make_float4(yx, yx, yy, yy);
      sC[3 * n + 1] = make_float4(yz, yz, aa, aa);
      sC[3 * n + 2] = make_float4(-a, -a, 2.f * a, 2.f * a);
      // node n of its step is row n % 8 of B: lane 4 column + n % 4, register (n % 8) / 4
      float *o = reinterpret_cast<float *>(sB + (n >> 3) * L::kStep) + 4 * (n & 3) + ((n >> 2) & 1);
#pragma unroll
      for (int r = 0; r < NR; ++r)
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          const float re = pr * w[r][f].x - pi * w[r][f].y, im = pr * w[r][f].y + pi * w[r][f].x;
          const float rh = tf32_hi(re), ih = tf32_hi(im), rl = re - rh, il = im - ih;
          float *b = o + r * 256 + 32 * f;  // columns 2 f (Re) and 2 f + 1 (Im), 16 floats each
          b[0] = rh;
          b[2] = rl;
          b[16] = ih;
          b[18] = il;
          b[128] = -ih;
          b[130] = -il;
          b[144] = rh;
          b[146] = rl;
        }
    }
    __syncthreads();
    float2 part[NR][MT][2];
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
      for (int i = 0; i < MT; ++i) part[r][i][0] = part[r][i][1] = make_float2(0.f, 0.f);
    if (MT == 1 || warp + (MT - 1) * nw < ntile)
      sweep<MT, MT, NR, FAST>(u, sB, sC, steps, lane, kappa, part);
    else
      sweep<(MT > 1 ? MT - 1 : 1), MT, NR, FAST>(u, sB, sC, steps, lane, kappa, part);
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
      for (int i = 0; i < MT; ++i) {
        float4 *hp = sH + (r * MT + i) * 64 + lane;
        const float4 hi = hp[0], lo = hp[32];
        float2 h0 = make_float2(hi.x, hi.y), h1 = make_float2(hi.z, hi.w);
        float2 l0 = make_float2(lo.x, lo.y), l1 = make_float2(lo.z, lo.w);
        two_sum2(h0, l0, part[r][i][0]);
        two_sum2(h1, l1, part[r][i][1]);
        hp[0] = make_float4(h0.x, h0.y, h1.x, h1.y);
        hp[32] = make_float4(l0.x, l0.y, l1.x, l1.y);
      }
  }
  // accumulator registers: (row g, field q) Re, Im, then (row g + 8, field q)
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    const int row = 16 * (warp + i * nw) + g;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      if (r >= nr) break;
      const float4 hi = sH[(r * MT + i) * 64 + lane], lo = sH[(r * MT + i) * 64 + 32 + lane];
      float2 *o = out + ((size_t)t * nI + row) * ldo + 4 * r + q;
      if (row < nI) o[0] = make_float2(hi.x + fmaf(hi.x, kCut, lo.x), hi.y + fmaf(hi.y, kCut, lo.y));
      if (row + 8 < nI) o[(size_t)8 * ldo] = make_float2(hi.z + fmaf(hi.z, kCut, lo.z), hi.w + fmaf(hi.w, kCut, lo.w));
    }
  }
}

// Row tiles over warps: at most 3 tiles a warp, evenly.
static int mma_warps(int nI) { return ((nI + 15) / 16 + 2) / 3; }

template <int MT, int NR, bool FAST>
static efie_status launch_mma_t(Ctx *c, cudaStream_t st, const MmaArgs &A) {
  const int nw = mma_warps(c->nI);
  const size_t sm = MmaLayout<MT, NR>::bytes(nw);
  const dim3 grid(c->n_m2l_targets, A.split, (A.R + NR - 1) / NR);
  EFIE_CUDA(cudaFuncSetAttribute(k_m2l_mma<MT, NR, FAST>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)MmaLayout<MT, NR>::bytes(kMmaMaxWarps)));
  k_m2l_mma<MT, NR, FAST><<<grid, 32 * nw, sm, st>>>(c->d_m2l_targets, c->d_far_ptr, c->d_far_src, c->d_pgeo, c->d_pph,
                                                   c->nI, A.R, A.ld, (float)c->kappa, c->d_nodeX4, A.src, A.acc,
                                                   A.more, A.ldm, A.slab);
  ++c->launches;
  EFIE_CUDA(cudaGetLastError());
  return EFIE_OK;
}

template <int MT, int NR>
static efie_status launch_mma_m(Ctx *c, cudaStream_t st, const MmaArgs &A) {
  const bool fast = m2l_scaled_lengths(c);
  return fast ? launch_mma_t<MT, NR, true>(c, st, A) : launch_mma_t<MT, NR, false>(c, st, A);
}

template <int MT>
static efie_status launch_mma_r(Ctx *c, cudaStream_t st, const MmaArgs &A) {
  // right-hand sides in even groups of at most 3, which share the evaluation of the kernel
  const int groups = (A.R + 2) / 3;
  switch ((A.R + groups - 1) / groups) {
    case 1: return launch_mma_m<MT, 1>(c, st, A);
    case 2: return launch_mma_m<MT, 2>(c, st, A);
    default: return launch_mma_m<MT, 3>(c, st, A);
  }
}

// Splits of the source lists: enough blocks for the chip when there are few targets, at least two
// staged chunks each.
int m2l_mma_splits(const Ctx *c) {
  if (c->n_m2l_targets == 0) return 1;
  const long long blocks = 2ll * c->nsm * 8;
  const long long chunks = (long long)c->nfar * c->nI / kMmaNodes / c->n_m2l_targets;
  return (int)std::max(1ll, std::min({blocks / c->n_m2l_targets, chunks / 2, 16ll}));
}

// A batch takes this kernel while it is faster than k_m2l_tc, whose cost does not change up to 16
// right-hand sides, while this one's grows with them.  Measured (ms, this kernel / k_m2l_tc, sphere of
// 1 536 elements): 16 nodes, 6 right-hand sides 0.31 / 0.38; 25 nodes 6: 0.64 / 0.67; 49 nodes 3: 0.85 / 1.06,
// 4: 1.23 / 1.06; 81 nodes 2: 1.47 / 1.96, 3: 2.27 / 1.96; 121 nodes 2: 3.02 / 3.42, 3: 4.37 / 3.42.  Per pair
// k_m2l_tc takes (rows + 94) x source nodes (rows padded to 64, 96 or 128, nodes to 8), this kernel a
// right-hand side's (rows + 8) x nodes / 1.36 (rows padded to its tiles).  From 24 to 6 144 elements and 9 to
// 121 nodes a batch of this kernel is at most 3 % behind k_m2l_tc, but for 7 right-hand sides at 16 nodes and 1 024
// elements or more (2.19 against 1.77 ms at 4 096); for a few dozen targets, where only this kernel splits
// lists, it could take more than 7 (24 elements, 9 nodes: 8 us for 7, 22 us for 8).
int m2l_mma_rhs(const Ctx *c) {
  if (!m2l_tc_supported(c)) return 1 << 30;
  const int nI = c->nI, nw = mma_warps(nI), mt = ((nI + 15) / 16 + nw - 1) / nw;
  const double here = (16.0 * nw * mt + 8) * nI, tc = ((nI <= 64 ? 64 : (nI <= 96 ? 96 : 128)) + 94.0) * 8 * ((nI + 7) / 8);
  return std::max(1, std::min(kMmaMaxRhs, (int)(1.36 * tc / here)));
}

efie_status launch_m2l_mma(Ctx *c, cudaStream_t st, const MmaArgs &A) {
  if (c->n_m2l_targets == 0) return EFIE_OK;
  const int tiles = (c->nI + 15) / 16, nw = mma_warps(c->nI);
  switch ((tiles + nw - 1) / nw) {
    case 1: return launch_mma_r<1>(c, st, A);
    case 2: return launch_mma_r<2>(c, st, A);
    default: return launch_mma_r<3>(c, st, A);
  }
}

}  // namespace efie
