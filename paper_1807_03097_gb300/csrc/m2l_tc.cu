// M2L of several right-hand sides on the tensor cores (a6, Sec. 4.2: the coupling of an
// admissible block is the kernel sampled at the tensor Chebyshev points of both clusters).
//
// For a target cluster t, a group of 64 fields (16 right-hand sides x {x, y, z, div}) and the
// far list of t, the contribution is C(i, f) = sum_s sum_j G_ts(i, j) S_s(j, f) with complex G
// and S.  On the tensor cores it runs transposed, with the fields on the 128 MMA rows:
//   A_s = [Re S_s^T; Im S_s^T]        (128 x nI, per source cluster),
//   D1  = A_s (Re G_ts)^T,  D2 = A_s (Im G_ts)^T      (128 x nI each, FP32 in tensor memory),
//   Re C^T = D1[0:64] - D2[64:128],  Im C^T = D1[64:128] + D2[0:64].
// Each FP32 operand is scaled by a power of two and split as hi + lo in FP16 (2 x 11 bits); the three
// products hi*hi, hi*lo and lo*hi carry 21 to 22 bits.  Scales: one per target cluster for G (its
// smallest node distance), one per field for the sources (the field's largest entry); both are
// taken back in the epilogue.  FP16 keeps hi and lo of a source whole down to 2^-16 of the field's largest
// (below that with an absolute error of 2^-39 of it); an entry G, whose bound 2^9 / (4 pi) leaves room for nodes
// closer than their clusters' balls, down to 2^-7 of that bound, which the distances of a far list reach.
// The tensor core rounds its accumulator more coarsely than an FP32 add, so every group of 4 block pairs
// gets a fresh accumulator D = [D1 D2] (one MMA of N = 2 NP against B = [Re G; Im G]), and the group's
// result is added to running sums S in tensor memory with FP32 adds on the CUDA cores.
//
// Kernel entry: as in k_m2l_mma (y = x_s - d is the source node seen from the target's centre, a = |y|;
// delta = r - a from num = r^2 - a^2 without cancellation, by one Newton step), but the factor
// e^{i kappa a} / (4 pi) belongs to the pair and goes onto the entry: A is the same for all targets.
//
// A block has 19 warps.  Warp 18 prepares the constants of the source nodes of a stage, one node a lane.
// Warps 0-15 evaluate the entries of B, fold D into S and write the result; warp 0 also allocates
// tensor memory.  The A operands are split once per product (k_tc_split, in the order of the
// shared-memory tiles) and fetched by lane 0 of warp 17 with bulk copies of 4 KB.  Lane 0 of warp 16
// issues the MMAs of a stage once its operands are there: the issuing thread stalls while the
// tensor pipe is busy, which an evaluating warp cannot afford.  Shared memory holds four stages of 4
// groups of 8 source nodes; the groups of all sources follow one another without padding to whole
// stages.  Stages are handed over with mbarriers; every wait is bounded and a wait that runs out
// sets an error flag for the host.  The copy lane and the MMA lane then issue nothing more and wait, with a
// fresh bound, for what they have in flight, so that the block neither reuses nor leaves its memory under
// a copy or an MMA.
//
// Bound: shared memory (a stage of 32 nodes at 121 target nodes: 1 740 clocks, of which the MMAs read 580, their
// pipe is busy 770, the A copies take 130 and the loads and stores of the evaluation 650) and the latency of
// four evaluating warps a scheduler (FMA pipe 42 %).  Measured, M2L of 64 right-hand sides at about 181 000 pairs of
// 121 nodes: operands in split TF32, sources split for every pair, target and source node constants per thread,
// 31.5 ms; FP16 and the sources split once 25.4 ms; the entry of k_m2l_mma from prepared constants, two
// target nodes at a time 18.2 ms; the targets' constants in registers 17.2 ms.  Error of the product against
// 64 bits 2.3e-6 -> 1.3e-6.
#include "efie_internal.h"
#include "tc.cuh"
#include "tc_pipeline.h"
#include "fastmath.cuh"
#include <cuda_fp16.h>
#include <type_traits>

namespace efie {

namespace {

constexpr int kTcFields = 64;      // fields per block (MMA rows = 2 x 64)
constexpr int kTcWarps = 16;                    // evaluating warps
constexpr int kTcProducers = 32 * kTcWarps;
constexpr int kTcThreads = kTcProducers + 96;   // + the MMA-issue, bulk-copy and node-constant warps
constexpr long long kTcWaitCycles = 1ll << 31;  // about a second
constexpr int kTcGroup = 4;   // block pairs accumulated in D before it is folded into S
constexpr int kTcStages = 4;  // shared-memory stages of 4 groups of 8 source nodes
static_assert(kTcGroup == 4, "a group of pairs is one stage per group of 8 source nodes");

// Tiles are K-major grids of core matrices (8 rows x 16 bytes = 8 source nodes), rows first: row r
// of node group g at g (group bytes) + 16 r.  A group of A is the 4 KB chunk of k_tc_split.
template <int NP>
struct TcLayout {
  static constexpr uint32_t kA = 128 * 16;             // 8 source nodes of A, hi or lo
  static constexpr uint32_t kB = 2 * NP * 16;          // 8 source nodes of B (Re rows, Im rows), hi or lo
  static constexpr uint32_t kOffB = 4 * 2 * kA;        // a stage: 4 groups of A [hi, lo], 4 of B [hi, lo]
  static constexpr uint32_t kStage = kOffB + 4 * 2 * kB;
  static constexpr uint32_t kConst = kTcStages * kStage;  // source node constants, per stage float4 [4][16 pairs]
  static constexpr uint32_t kBars = kConst + kTcStages * 1024;
  static constexpr uint32_t kBytes = kBars + 160;
  static constexpr uint32_t kCols = 4 * NP <= 256 ? 256 : 512;  // D1, D2, S1, S2
  static_assert(2 * 128 * (NP + 1) * 4 <= kTcStages * kStage, "epilogue staging must fit in the stages");
};

// 2^e as a float from its biased exponent
__device__ __forceinline__ float pow2_biased(int b) { return __uint_as_float((unsigned)b << 23); }
// Biased exponent of a field's scale, from the bits of its largest |entry|: the largest entry goes to
// [2^14, 2^15), half of the FP16 range.  254 minus it is that of the inverse.  A field with an
// infinity or a NaN keeps the scale 1.
__device__ __forceinline__ int field_scale(unsigned mx) {
  const int e = (int)(mx >> 23);
  return e == 255 ? 127 : min(268 - e, 253);
}

// x0, x1 = hi + lo (packed pairs), both rounded to nearest
__device__ __forceinline__ void split_f16(float x0, float x1, uint32_t &hi, uint32_t &lo) {
  const __half2 h = __floats2half2_rn(x0, x1);
  const float2 hf = __half22float2(h);
  const __half2 l = __floats2half2_rn(x0 - hf.x, x1 - hf.y);
  hi = *reinterpret_cast<const uint32_t *>(&h);
  lo = *reinterpret_cast<const uint32_t *>(&l);
}

// Largest |Re|, |Im| of every field over the source clusters (the list is symmetric: the targets), as
// float bits.  One block per cluster and 64 fields.
__global__ void __launch_bounds__(256) k_tc_max(const int *__restrict__ targets, int nI, int F, int ld,
                                                const float2 *__restrict__ src, unsigned *__restrict__ mx) {
  __shared__ unsigned part[64];
  const int fl = threadIdx.x & 63, f = blockIdx.y * kTcFields + fl;
  if (threadIdx.x < 64) part[threadIdx.x] = 0u;
  __syncthreads();
  if (f < F) {
    const float2 *s = src + (size_t)targets[blockIdx.x] * nI * ld + f;
    unsigned m = 0;
#pragma unroll 4
    for (int j = threadIdx.x >> 6; j < nI; j += 4) {
      const float2 v = s[(size_t)j * ld];
      m = max(m, max(__float_as_uint(v.x) & 0x7fffffffu, __float_as_uint(v.y) & 0x7fffffffu));
    }
    atomicMax(&part[fl], m);
  }
  __syncthreads();
  if (threadIdx.x < 64 && f < F && part[fl]) atomicMax(&mx[f], part[fl]);
}

// A operands: out[((cluster KG + g) NFB + block of 64 fields)][hi, lo][128 rows][8 nodes] in FP16, rows f (Re)
// and 64 + f (Im), node j = 8 g + k; zero beyond the nodes and fields.  One block per cluster and 64
// fields; bounded by HBM (8 bytes read and written an entry).
__global__ void __launch_bounds__(256) k_tc_split(const int *__restrict__ targets, int nI, int F, int ld,
                                                  const float2 *__restrict__ src, const unsigned *__restrict__ mx,
                                                  uint4 *__restrict__ out) {
  const int t = targets[blockIdx.x], fl = threadIdx.x & 63, f = blockIdx.y * kTcFields + fl;
  const int KG = (nI + 7) / 8;
  const float sc = f < F ? pow2_biased(field_scale(mx[f])) : 1.f;
  for (int g = threadIdx.x >> 6; g < KG; g += 4) {
    float2 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int j = 8 * g + k;
      v[k] = (f < F && j < nI) ? src[((size_t)t * nI + j) * ld + f] : make_float2(0.f, 0.f);
    }
    uint4 *o = out + (((size_t)t * KG + g) * gridDim.y + blockIdx.y) * 256;
    uint32_t h[4], l[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) split_f16(v[2 * k].x * sc, v[2 * k + 1].x * sc, h[k], l[k]);
    o[fl] = make_uint4(h[0], h[1], h[2], h[3]);
    o[128 + fl] = make_uint4(l[0], l[1], l[2], l[3]);
#pragma unroll
    for (int k = 0; k < 4; ++k) split_f16(v[2 * k].y * sc, v[2 * k + 1].y * sc, h[k], l[k]);
    o[64 + fl] = make_uint4(h[0], h[1], h[2], h[3]);
    o[192 + fl] = make_uint4(l[0], l[1], l[2], l[3]);
  }
}

// Kernel entries of N target nodes (constants u: 2 x, -|x|^2) and two source nodes (constants c), times
// their factors: (Re G0, Re G1), (Im G0, Im G1) of each.  num in scalar FMA: two cost what a packed one
// does with three distinct operands, and the target's constants need not be held twice.
template <int N, bool FAST>
__device__ __forceinline__ void kernel_entries(const float4 *u, const float4 (&c)[4], float kappa,
                                               float2 (&re)[N], float2 (&im)[N]) {
  const float2 m1 = make_float2(-1.f, -1.f), mh = make_float2(-0.5f, -0.5f);
  const float2 na = make_float2(c[2].x, c[2].y), a2 = make_float2(c[2].z, c[2].w);
  const float2 fr = make_float2(c[3].x, c[3].y), fi = make_float2(c[3].z, c[3].w);
  const float2 nfi = make_float2(-fi.x, -fi.y);
  float2 v[N], p[N], ri[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float2 x = make_float2(fmaf(u[i].z, c[1].x, fmaf(u[i].y, c[0].z, fmaf(u[i].x, c[0].x, u[i].w))),
                                 fmaf(u[i].z, c[1].y, fmaf(u[i].y, c[0].w, fmaf(u[i].x, c[0].y, u[i].w))));  // -num
    v[i] = x;
    p[i] = __ffma2_rn(x, m1, make_float2(c[1].z, c[1].w));  // r^2
    ri[i] = make_float2(rsqrt_ftz(p[i].x), rsqrt_ftz(p[i].y));
  }
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float2 dl = __ffma2_rn(p[i], ri[i], na);
    const float2 e = __ffma2_rn(dl, __fadd2_rn(dl, a2), v[i]);
    float2 x = __ffma2_rn(__fmul2_rn(ri[i], e), mh, dl);
    if (!FAST) {
      const float inv2pi = 0.15915494309189535f, p1 = 6.28318548202514648f, p2 = -1.7484555e-7f;
      x = __fmul2_rn(x, make_float2(kappa, kappa));
      const float2 n = make_float2(-rintf(x.x * inv2pi), -rintf(x.y * inv2pi));
      x = __ffma2_rn(n, make_float2(p1, p1), x);
      x = __ffma2_rn(n, make_float2(p2, p2), x);
    }
    const float2 cs = __fmul2_rn(make_float2(cos_ftz(x.x), cos_ftz(x.y)), ri[i]);
    const float2 sn = __fmul2_rn(make_float2(sin_ftz(x.x), sin_ftz(x.y)), ri[i]);
    re[i] = __ffma2_rn(fr, cs, __fmul2_rn(nfi, sn));
    im[i] = __ffma2_rn(fr, sn, __fmul2_rn(fi, cs));
  }
}

// Read-only loads issued where they stand (volatile: the scheduler does not sink them towards
// their use), so that the loads of the next stage overlap the evaluation of this one.
__device__ __forceinline__ float4 ldg_pin(const float4 *p) {
  float4 v;
  asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ float2 ldg_pin(const float2 *p) {
  float2 v;
  asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ int ldg_pin(const int *p) {
  int v;
  asm volatile("ld.global.nc.b32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

}  // namespace

// Staging map of a stage: warp w covers the node group w % 4 (its own pair and first node: groups of
// all pairs in a row), lane l the nodes 2 (l / 8) + e (e < 2) of it and the target nodes
// n = l % 8 + 8 (w / 4) + 32 i (B rows n and NP + n), so that a warp store fills one core matrix (128
// contiguous bytes).  Tensor memory: D1 [0, NP), D2 [NP, 2 NP) hold the group of block pairs in
// flight, S1 [2 NP, 3 NP), S2 [3 NP, 4 NP) the running sums over the far list.  rfrac: the smallest
// node distance of an admissible pair relative to its centre distance, 1 / (1 + eta).  FAST: lengths scaled
// by kappa or not, as in k_m2l_mma.
template <int NP, bool FAST>
__global__ void __launch_bounds__(kTcThreads, 1) k_m2l_tc(
    const int *__restrict__ targets, const int *__restrict__ fptr, const int *__restrict__ fsrc,
    const float4 *__restrict__ pgeo, const float2 *__restrict__ pph, int nI, float kappa, float rfrac,
    const float4 *__restrict__ nodeX4, int F, int ld, const uint4 *__restrict__ opA, const unsigned *__restrict__ mx,
    float2 *__restrict__ acc, int *__restrict__ err) {
  using L = TcLayout<NP>;
  extern __shared__ __align__(1024) uint8_t smem[];
  float4 *sC = reinterpret_cast<float4 *>(smem + L::kConst);
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L::kBars);
  uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + 3 * kTcStages + 3);
  int *sRmin = reinterpret_cast<int *>(tslot + 1);
  const uint32_t b_full = tc::smem_u32(&bars[0]), b_empty = tc::smem_u32(&bars[kTcStages]);
  const uint32_t b_const = tc::smem_u32(&bars[2 * kTcStages + 2]), b_done = tc::smem_u32(&bars[3 * kTcStages + 2]);
  const uint32_t b_tfull = tc::smem_u32(&bars[2 * kTcStages]), b_tempty = tc::smem_u32(&bars[2 * kTcStages + 1]);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int t = targets[blockIdx.x];
  const int f0 = blockIdx.y * kTcFields;
  const int k0 = fptr[t], nsrc = fptr[t + 1] - k0;
  const int KG = (nI + 7) / 8;                       // groups of 8 source nodes of a pair
  const int ngrp = nsrc * KG, T = (ngrp + 3) / 4;    // groups and stages of the block

  if (tid == 0) {
    for (int i = 0; i < kTcStages; ++i) {
      tc::mbar_init(b_full + 8 * i, kTcProducers + 1);
      tc::mbar_init(b_empty + 8 * i, 1);
      tc::mbar_init(b_const + 8 * i, 32);
    }
    tc::mbar_init(b_tfull, 1);
    tc::mbar_init(b_tempty, kTcProducers);
    tc::mbar_init(b_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *sRmin = 0x7f7fffff;
  }
  const float sc = FAST ? kappa : 1.f;
  // B rows of target nodes n >= nI (padding up to NP, in the Re and the Im half): finite from the start
  for (int i = tid; i < kTcStages * 16 * (NP - nI); i += kTcThreads) {
    const int n = nI + i % (NP - nI), tl = i / (NP - nI);  // tl: stage (bits 4-5), group and hi/lo, Re/Im half (bit 0)
    *reinterpret_cast<float4 *>(smem + (tl >> 4) * L::kStage + L::kOffB + ((tl >> 1) & 7) * L::kB +
                                16 * ((tl & 1) * NP + n)) = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  tc::fence_proxy_async();
  if (warp == 0) tc::tmem_alloc(tc::smem_u32(tslot), L::kCols);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  for (int i = tid; i < nsrc; i += kTcThreads) atomicMin(sRmin, __float_as_int(pgeo[k0 + i].w));
  __syncthreads();
  // G <= 1 / (rfrac r0) goes to 2^9 at most: the bounding balls are sampled, and nodes 128 times closer than
  // their bound still fit in FP16
  const int gexp = min(max((int)(__float_as_uint(__int_as_float(*sRmin) * rfrac) >> 23) + 9, 1), 253);
  const uint32_t tbase = *tslot;
  const uint32_t idesc = tc::idesc_f16(128, 2 * NP);
  const int q = warp & 3, r4 = warp >> 2;  // lane quadrant and column quarter of the drain
  const uint32_t tq = tbase + ((uint32_t)(32 * q) << 16);
  long long patience = kTcWaitCycles;  // of this thread's waits; none after one has run out
  auto wait = [&](uint32_t bar, uint32_t parity, int code) {
    if (tc::mbar_wait(bar, parity, patience)) return true;
    atomicOr(err, code);
    patience = 0;
    return false;
  };

  if (warp < kTcWarps) {
  // S += D for group g of block pairs (S = D for the first), then release D to the MMAs.
  // This thread covers lane 32 q + lane and the column blocks b = r4 + 4 i of D1/S1, D2/S2.
  auto drain = [&](int g) {
    constexpr int NB = NP / 32;
    const int p = g;
    wait(b_tfull, g & 1, 1);
    tc::fence_after_sync();
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      uint32_t d[NB][8], sv[NB][8];
#pragma unroll
      for (int i = 0; i < NB; ++i) {
        const uint32_t cd = tq + half * NP + 8 * (r4 + 4 * i);
        tc::tmem_ld8_async(cd, d[i]);
        if (p > 0) tc::tmem_ld8_async(cd + 2 * NP, sv[i]);
      }
      tc::tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < NB; ++i) {
        tc::touch8(d[i]);
        if (p > 0) {
          tc::touch8(sv[i]);
#pragma unroll
          for (int k = 0; k < 8; ++k) d[i][k] = __float_as_uint(__uint_as_float(d[i][k]) + __uint_as_float(sv[i][k]));
        }
        tc::tmem_st8_async(tq + half * NP + 8 * (r4 + 4 * i) + 2 * NP, d[i]);
      }
    }
    tc::tmem_wait_st();
    tc::fence_before_sync();
    tc::mbar_arrive(b_tempty);
  };

  const int kg = warp & 3, kp = lane >> 3;         // node group of a stage, pair of nodes in it
  const int rbase = (lane & 7) + 8 * (warp >> 2);  // target nodes rbase + 32 i
  const int rows = (nI - 8 * (warp >> 2) + 31) / 32;  // i below this (the same for the warp)
  float4 u[NP / 32];  // rows past nI: the last node
#pragma unroll
  for (int i = 0; i < NP / 32; ++i) {
    const float4 v = nodeX4[(size_t)t * nI + min(rbase + 32 * i, nI - 1)];
    const float x = sc * v.x, y = sc * v.y, z = sc * v.z;
    u[i] = make_float4(2.f * x, 2.f * y, 2.f * z, -(x * x + y * y + z * z));
  }
  for (int it = 0, c = 0, g = 0; it < T; ++it) {
    const int st = it % kTcStages;
    wait(b_const + 8 * st, (it / kTcStages) & 1, 2);
    float4 cn[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) cn[v] = sC[64 * st + 16 * v + 4 * kg + kp];
    if (it >= kTcStages) wait(b_empty + 8 * st, ((it / kTcStages) & 1) ^ 1, 2);
    uint8_t *sB = smem + st * L::kStage + L::kOffB + kg * 2 * L::kB + 16 * rbase + 4 * kp;
    // target nodes k and (N = 2) k + 1: two chains at a time
    auto put = [&](auto count, int k) {
      constexpr int N = decltype(count)::value;
      float2 re[N], im[N];
      kernel_entries<N, FAST>(u + k, cn, kappa, re, im);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        uint32_t rh, rl, ih, il;
        split_f16(re[i].x, re[i].y, rh, rl);
        split_f16(im[i].x, im[i].y, ih, il);
        uint32_t *o = reinterpret_cast<uint32_t *>(sB + 512 * (k + i));
        o[0] = rh;
        o[4 * NP] = ih;
        o[L::kB / 4] = rl;
        o[L::kB / 4 + 4 * NP] = il;
      }
    };
    if (rows > 0) put(std::integral_constant<int, 2>(), 0);
    if (NP > 64 && rows > 2) put(std::integral_constant<int, NP == 96 ? 1 : 2>(), 2);
    tc::fence_proxy_async();
    tc::mbar_arrive(b_full + 8 * st);
    // the previous group's MMAs are done by now: fold it into the running sums
    if (c == 0 && it > 0) drain(g++);
    if (++c == KG) c = 0;
  }
  if (nsrc >= 1) drain((nsrc - 1) / kTcGroup);
  } else if (warp == kTcWarps && lane == 0) {
    // ------------------------------------------------------------------- MMA issue
    // One thread, so that its waits on the tensor pipe stall no evaluating warp.  Descriptors are
    // built once; the start address sits in the low bits, so stage st and K-step ks are reached by
    // adding their bytes / 16 (shared addresses stay below 2^18 bytes).  A group of 4 pairs is KG stages.
    const uint32_t a0 = tc::smem_u32(smem);
    const uint64_t dah0 = tc::smem_desc(a0, 2 * L::kA, 128), dal0 = tc::smem_desc(a0 + L::kA, 2 * L::kA, 128);
    const uint64_t dbh0 = tc::smem_desc(a0 + L::kOffB, 2 * L::kB, 128);
    const uint64_t dbl0 = tc::smem_desc(a0 + L::kOffB + L::kB, 2 * L::kB, 128);
    int c = 0, g = 0;  // stage of the group, group
    const int issued = issue_stages(
        T,
        [&](int it) {
          if (c == 0 && it > 0 && !wait(b_tempty, g++ & 1, 4)) return false;
          return wait(b_full + 8 * (it % kTcStages), (it / kTcStages) & 1, 8);
        },
        [&](int it) {
          // [D1 D2] (+)= A [Re B; Im B]^T, three split products per K-step
          const int st = it % kTcStages;
          tc::fence_after_sync();
#pragma unroll
          for (int ks = 0; ks < 2; ++ks) {
            if (4 * it + 2 * ks >= ngrp) break;
            const uint64_t oa = (uint64_t)(st * (L::kStage >> 4) + ks * (4 * L::kA >> 4));
            const uint64_t ob = (uint64_t)(st * (L::kStage >> 4) + ks * (4 * L::kB >> 4));
            tc::mma_f16(tbase, dah0 + oa, dbh0 + ob, idesc, (c == 0 && ks == 0) ? 0u : 1u);
            tc::mma_f16(tbase, dah0 + oa, dbl0 + ob, idesc, 1u);
            tc::mma_f16(tbase, dal0 + oa, dbh0 + ob, idesc, 1u);
          }
          tc::mma_commit(b_empty + 8 * st);
          if (++c == KG) c = 0;
          if (c == 0 || it == T - 1) tc::mma_commit(b_tfull);
        });
    // no MMA is in flight when the block goes on: the last group's completion, or after an early end that of
    // what was issued
    if (issued < T) tc::mma_commit(b_done);
    if (T > 0 && !(issued < T ? tc::mbar_wait(b_done, 0, kTcWaitCycles)
                              : tc::mbar_wait(b_tfull, ((T - 1) / KG) & 1, kTcWaitCycles)))
      atomicOr(err, 128);
  } else if (warp == kTcWarps + 1 && lane == 0) {
    // -------------------------------------------------------------- bulk copies of A
    // A stage past the last group repeats it: its B is zero.
    int lp = 0, lc = 0;
    int s = nsrc > 0 ? ldg_pin(fsrc + k0) : 0;
    const int issued = issue_stages(
        T, [&](int it) { return it < kTcStages || wait(b_empty + 8 * (it % kTcStages), ((it / kTcStages) & 1) ^ 1, 32); },
        [&](int it) {
          const int st = it % kTcStages;
          tc::mbar_arrive_expect(b_full + 8 * st, 4 * 2 * L::kA);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            tc::bulk_load(tc::smem_u32(smem) + st * L::kStage + i * 2 * L::kA,
                          opA + (((size_t)s * KG + lc) * gridDim.y + blockIdx.y) * 256, 2 * L::kA, b_full + 8 * st);
            if (4 * it + i + 1 >= ngrp) continue;
            if (++lc == KG) {
              lc = 0;
              s = ldg_pin(fsrc + k0 + ++lp);
            }
          }
        });
    // a phase completes only with its copies (it was armed after the one before had completed), and the
    // evaluating warps arrive in every phase
    drain_stages(issued, kTcStages, [&](int it) {
      if (!tc::mbar_wait(b_full + 8 * (it % kTcStages), (it / kTcStages) & 1, kTcWaitCycles)) atomicOr(err, 32);
    });
  } else if (warp == kTcWarps + 2) {
    // -------------------------------------------------------- source node constants
    // Lane l: node l % 8 of the stage's group l / 8.  Nodes past the pair's or the list's end repeat the
    // last one with factor 0.  A stage's slot is free once its previous entries are evaluated.
    const float sg = sc * pow2_biased(gexp);
    int lp = (lane >> 3) / KG, lc = (lane >> 3) % KG;  // pair and group of the next load
    float4 nx = make_float4(0, 0, 0, 0), ng = make_float4(0, 0, 0, 1);
    float2 nph = make_float2(0, 0);
    auto load = [&]() {
      const int k = min(lp, nsrc - 1), j = 8 * lc + (lane & 7);
      nx = ldg_pin(nodeX4 + (size_t)ldg_pin(fsrc + k0 + k) * nI + min(j, nI - 1));
      ng = ldg_pin(pgeo + k0 + k);
      nph = lp < nsrc && j < nI ? ldg_pin(pph + k0 + k) : make_float2(0.f, 0.f);
      lc += 4;
      while (lc >= KG) {
        lc -= KG;
        ++lp;
      }
    };
    if (T > 0) load();
    for (int it = 0; it < T; ++it) {
      const int st = it % kTcStages;
      const float4 x = make_float4(sc * nx.x, sc * nx.y, sc * nx.z, 0.f);
      const float4 d = make_float4(sc * ng.x, sc * ng.y, sc * ng.z, sc * ng.w);
      const float2 ph = make_float2(sg * nph.x, sg * nph.y);
      load();
      const float yx = x.x - d.x, yy = x.y - d.y, yz = x.z - d.z;
      const float aa = yx * yx + yy * yy + yz * yz;
      const float a = aa * rsqrt_ftz(aa);
      const float bb = x.x * x.x + x.y * x.y + x.z * x.z - 2.f * (d.x * x.x + d.y * x.y + d.z * x.z);
      const float da = bb * rcp_ftz(a + d.w);
      float sn, cs;
      sincosf(FAST ? da : kappa * da, &sn, &cs);
      const float fr = ph.x * cs - ph.y * sn, fi = ph.x * sn + ph.y * cs;
      if (it >= kTcStages) wait(b_full + 8 * st, ((it / kTcStages) & 1) ^ 1, 64);
      float *o = reinterpret_cast<float *>(sC + 64 * st + (lane >> 1)) + (lane & 1);
      o[0] = yx;
      o[2] = yy;
      o[64] = yz;
      o[66] = aa;
      o[128] = -a;
      o[130] = 2.f * a;
      o[192] = fr;
      o[194] = fi;
      tc::mbar_arrive(b_const + 8 * st);
    }
  }
  __syncwarp();
  // ------------------------------------------------------------------------- epilogue
  // every MMA is complete and drained: stage the sums as [128][NP + 1] in the stage memory
  __syncthreads();
  float *sS1 = reinterpret_cast<float *>(smem), *sS2 = sS1 + 128 * (NP + 1);
  const int m = 32 * q + lane;
  if (warp >= kTcWarps) {
    // the MMA, copy and constants warps take no part in staging the sums
  } else if (nsrc >= 1) {
    tc::fence_after_sync();
#pragma unroll 1
    for (int b = r4; b < NP / 8; b += 4) {
      float v[8];
      tc::tmem_ld8(tq + 2 * NP + 8 * b, v);
#pragma unroll
      for (int i = 0; i < 8; ++i) sS1[m * (NP + 1) + 8 * b + i] = v[i];
      tc::tmem_ld8(tq + 3 * NP + 8 * b, v);
#pragma unroll
      for (int i = 0; i < 8; ++i) sS2[m * (NP + 1) + 8 * b + i] = v[i];
    }
  } else {
    for (int b = r4; b < NP / 8; b += 4)
      for (int i = 0; i < 8; ++i) sS1[m * (NP + 1) + 8 * b + i] = sS2[m * (NP + 1) + 8 * b + i] = 0.f;
  }
  __syncthreads();
  for (int idx = tid; idx < nI * kTcFields; idx += kTcThreads) {
    const int f = idx & (kTcFields - 1), i = idx >> 6;
    if (f0 + f >= F) continue;
    const float re = sS1[f * (NP + 1) + i] - sS2[(64 + f) * (NP + 1) + i];
    const float im = sS1[(64 + f) * (NP + 1) + i] + sS2[f * (NP + 1) + i];
    const float ug = pow2_biased(254 - gexp), uf = pow2_biased(254 - field_scale(mx[f0 + f]));
    acc[((size_t)t * nI + i) * ld + f0 + f] = make_float2(re * ug * uf, im * ug * uf);
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 0) tc::tmem_dealloc(tbase, L::kCols);
}

template <int NP, bool FAST>
static efie_status tc_attr() {
  cudaError_t e = cudaFuncSetAttribute(k_m2l_tc<NP, FAST>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)TcLayout<NP>::kBytes);
  return e == cudaSuccess ? EFIE_OK : EFIE_ECUDA;
}

template <int NP>
static efie_status tc_attrs() {
  const efie_status e = tc_attr<NP, true>();
  return e == EFIE_OK ? tc_attr<NP, false>() : e;
}

bool m2l_tc_supported(const Ctx *c) { return c->nI <= 128; }

// bytes of the split A operands of `nrhs` right-hand sides (16 right-hand sides at a time)
size_t m2l_tc_bytes(const Ctx *c, int nrhs) {
  return (size_t)c->ncl * ((c->nI + 7) / 8) * ((nrhs + 15) / 16) * 4096;
}

// for batches of up to nrhs right-hand sides (0: the error flag only)
efie_status m2l_tc_prepare(Ctx *c, int nrhs) {
  EFIE_TRY(tc_attrs<64>());
  EFIE_TRY(tc_attrs<96>());
  EFIE_TRY(tc_attrs<128>());
  if (!c->d_tc_err) {
    EFIE_TRY(dalloc(c, &c->d_tc_err, 1));
    EFIE_CUDA(cudaMemsetAsync(c->d_tc_err, 0, sizeof(int), c->stream));
  }
  if (nrhs > 0) {
    EFIE_TRY(dalloc(c, &c->d_tcA, m2l_tc_bytes(c, nrhs) / sizeof(uint4)));
    EFIE_TRY(dalloc(c, &c->d_tcmax, 4 * (size_t)nrhs));
  }
  return EFIE_OK;
}

template <int NP>
static void launch_np(Ctx *c, cudaStream_t st, dim3 grid, int F, int ld, float2 *acc) {
  const float kf = (float)c->kappa, rfrac = (float)(1.0 / (1.0 + c->eta));
#define EFIE_TC(MV)                                                                                      \
  k_m2l_tc<NP, MV><<<grid, kTcThreads, TcLayout<NP>::kBytes, st>>>(c->d_m2l_targets, c->d_far_ptr,          \
                                                                   c->d_far_src, c->d_pgeo, c->d_pph, c->nI, \
                                                                   kf, rfrac, c->d_nodeX4, F, ld, c->d_tcA,   \
                                                                   c->d_tcmax, acc, c->d_tc_err)
  if (m2l_scaled_lengths(c)) EFIE_TC(true);
  else EFIE_TC(false);
#undef EFIE_TC
}

// acc[t][i][f] for the targets of the M2L, f < F = 4 R, row stride ld (float2 entries)
efie_status launch_m2l_tc(Ctx *c, cudaStream_t st, int F, int ld, const float2 *src, float2 *acc) {
  if (c->n_m2l_targets == 0) return EFIE_OK;
  const int nI = c->nI;
  dim3 grid(c->n_m2l_targets, (F + kTcFields - 1) / kTcFields);
  EFIE_CUDA(cudaMemsetAsync(c->d_tcmax, 0, sizeof(unsigned) * F, st));
  k_tc_max<<<grid, 256, 0, st>>>(c->d_m2l_targets, nI, F, ld, src, c->d_tcmax);
  k_tc_split<<<grid, 256, 0, st>>>(c->d_m2l_targets, nI, F, ld, src, c->d_tcmax, c->d_tcA);
  c->launches += 2;
  if (nI <= 64) launch_np<64>(c, st, grid, F, ld, acc);
  else if (nI <= 96) launch_np<96>(c, st, grid, F, ld, acc);
  else if (nI <= 128) launch_np<128>(c, st, grid, F, ld, acc);
  else return EFIE_EINVAL;
  ++c->launches;
  EFIE_CUDA(cudaGetLastError());
  return EFIE_OK;
}

// One bounded wait on an mbarrier that nothing ever completes (the situation of a stalled
// pipeline stage): the wait gives up after `cycles` clocks and sets the same error flag as the
// tensor-core M2L.  The barrier lives in shared memory and is abandoned when the block exits.
__global__ void k_wait_selftest(long long cycles, int *err) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    tc::mbar_init(tc::smem_u32(&bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (!tc::mbar_wait(tc::smem_u32(&bar), 0, cycles)) atomicOr(err, 16);
  }
}

efie_status dev_wait_selftest(Ctx *c, long long cycles) {
  EFIE_TRY(m2l_tc_prepare(c, 0));
  k_wait_selftest<<<1, 32, 0, c->stream>>>(cycles, c->d_tc_err);
  ++c->launches;
  EFIE_CUDA(cudaGetLastError());
  return m2l_tc_check(c);
}

efie_status m2l_tc_check(Ctx *c) {
  if (!c->d_tc_err) return EFIE_OK;
  int e = 0;
  EFIE_CUDA(cudaMemcpyAsync(&e, c->d_tc_err, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  EFIE_CUDA(cudaStreamSynchronize(c->stream));
  if (e) {
    c->err = "tensor-core M2L: a pipeline wait ran out (code " + std::to_string(e) + ")";
    cudaMemsetAsync(c->d_tc_err, 0, sizeof(int), c->stream);
    return EFIE_ETIMEOUT;
  }
  return EFIE_OK;
}

}  // namespace efie
