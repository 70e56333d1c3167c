// FP64-class Gram matrix G = Y^H Y of an FP32 thin quaternion sketch on the tcgen05 tensor cores
// (the Gram product of CholeskyQR, Def. 1 eq. QQR and every QR of Algorithms 1-4).
//
// G's components are sums of the real Gram W = Yh^T Yh of the plane-stacked Yh = [Y0 Y1 Y2 Y3]
// (m x 4l).  W is formed exactly enough for FP64-class use by an error-free splitting:
//  - every column c of Yh gets the exponent e_c with max_r |Yh(r, c)| < 2^e_c, and each entry is
//    written in balanced base 128, y = 2^(e_c - 6) (q_1 + q_2 2^-7 + ... + q_7 2^-42) + rest with
//    integers |q_i| <= 64, each the nearest to what is left (the rest is at most 2^-49 of 2^e_c; an
//    entry of at least 2^-25 of it is represented exactly);
//  - the q_i are exact in BF16, their products exact in FP32, and the tensor core's FP32 sums of
//    such integer products stay exact while they stay below 2^24: the slice pairs (i, j) of equal
//    weight s = i + j - 2 share one TMEM accumulator, at most 7 pairs x 512 rows x 64^2 < 2^24,
//    so every CTA reduces a chunk of at most 512 rows;
//  - pairs with i + j > 8 (weight 2^-49 and below) are left out: 28 BF16 products per entry and row
//    (digits rounded toward zero hold one bit less: 8 of 6 bits and 36 products for 48 bits);
//  - the 7 exact integer sums of a chunk are scaled by 2^-7s (exact) and added in double-FP32,
//    the chunks are added in double-FP32, and the result is scaled by 2^(e_a + e_b - 12).
// The error of W(a, b) is about 2^-45 of max|y_a| max|y_b| m: FP64-class, as the Gram of the
// double-FP32 SIMT path (orth.cu), at tensor-core throughput.
//
// Kernels: gram_slice_kernel (one CTA per column: exponent, then the 7 slices, BF16, column-major
// per slice with rows padded to a multiple of 8), gram_tc_kernel (persistent CTAs over the (128 x 64
// tile of W's upper part, 512-row chunk) items: TMA of the 7 slices of both operands into a ring of two 32-row
// stages, 10 MMAs of 128 x (64..256) x 16 per 16 rows into 7 x 64 TMEM columns, epilogue to
// double-FP32 partial tiles), gram_tc_combine_kernel (chunk sums, scaling, the quaternion
// components of G).
// Bound: a stage row is 64 bytes of one column and slice, and the TMA's row rate, then the MMAs, set
// the pace: 16-row stages (32-byte rows) and 8 slices took 391 us at 20000 x 180 and 76 us at
// 20000 x 60, this form 251 and 43 (error over max|y_a| max|y_b| m: 2^-48.1, before 2^-45.9).
#include <algorithm>
#include <cstring>

#include "qlr_internal.h"
#include "tc_common.cuh"

namespace {

using namespace qlr_tc;

// The two splittings.  Slices7 (single problems): balanced base 128, as above.  Slices8 (batch
// plans): 8 digits of 6 bits rounded toward zero, 36 products, 2^-48 of the column maximum; the
// plans' results hang on every bit of their factors (the phase of each singular vector pair is set
// by rounding errors), so they keep the digits they were released with.
template <int N>
struct Slices {
  static constexpr int GS = N;                    // slices per entry
  static constexpr int GBITS = (N == 7) ? 7 : 6;  // weight step of the slices
  static constexpr bool NEAREST = (N == 7);
  static constexpr int NGRP = N;                  // weight groups s = i + j - 2 = 0 .. N - 1
};
constexpr int GTOP = 6;          // bits of the first slice
constexpr int GTMEM = 512;       // TMEM columns allocated for the weight groups' accumulators (a power of two)
constexpr int GA = 128;          // W rows per tile (MMA M)
constexpr int GB = 64;           // W columns per tile (MMA N)
constexpr int GK = 32;           // rows of Y per pipeline stage (64-byte swizzled BF16 rows, two MMA K)
constexpr int GCHUNK = 512;      // rows of Y per item at most (exactness of the TMEM sums)
constexpr int GSTAGES = 2;
constexpr int GEPI = 8;                // epilogue warps: a lane quarter and half the columns each
constexpr int GTHREADS = 64 + 32 * GEPI;
constexpr int GSW = GK * 2;           // bytes per K-major row = swizzle span
constexpr int GMODE = 4;              // descriptor swizzle mode: 64 bytes
constexpr int A_TILE = GA * GK * 2;   // bytes of one slice's A tile
constexpr int B_TILE = GB * GK * 2;
constexpr size_t gsmem(int gs) { return (size_t)GSTAGES * gs * (A_TILE + B_TILE) + 1024 + 256; }

struct GramTcParams {
  CUtensorMap tmA;      // slices as (mp rows inner) x (GS L4p columns outer), box {GK, GA}
  CUtensorMap tmB;      // the same array, box {GK, GB}
  float2* part;         // [chunk] L4 x L4 column-major: W(a, b) at b L4 + a, double-FP32 (h, l)
  int L4, nA, nB;       // W order, a-blocks of GA, b-blocks of GB
  int L4p;              // columns per slice (L4 rounded up to GB; an A tile may run into the
                        // next slice: those W rows a >= L4 are never stored)
  int kiters;           // GK-row stages over all m rows
  int cstages;          // stages per chunk
  int* err;
};

// A problem of a batch plan: the MMA parameters (tensor maps first, 64-byte aligned) and what the
// slicing and the combine need.
struct GramTcProb {
  GramTcParams tc;
  const float* y[4];
  int64_t m, ld, mp;
  int l, nchunks;
  __nv_bfloat16* S;
  int* ex;
  float* G;             // double-FP32 upper triangle, 8 floats per entry at G + 8 (j l + i)
};

// Columns of Yh (L4p columns, the padding zero) by CTAs of 8 warps, WPC warps per column (8 for
// one tall problem, 1 for the many short ones of a batch): the column exponent, then the
// slices (two rows a lane and 4-byte stores took 60 us at 20000 x 180, now 51).
template <int N, int WPC>
__device__ __forceinline__ void gram_slice_cols(const float* __restrict__ y0, const float* __restrict__ y1,
                                                const float* __restrict__ y2, const float* __restrict__ y3, int64_t m,
                                                int l, int64_t ld, int L4p, int64_t mp, __nv_bfloat16* __restrict__ S,
                                                int* __restrict__ ex, const int g) {
  __shared__ float red[8];
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int c = g * (8 / WPC) + warp / WPC, sub = warp % WPC;
  const bool valid = c < L4p;
  const float* y = nullptr;
  if (valid && c < 4 * l) {
    const int pl = c / l, j = c % l;
    y = (pl == 0 ? y0 : pl == 1 ? y1 : pl == 2 ? y2 : y3) + (int64_t)j * ld;
  }
  // eight rows a lane and turn: two 16-byte loads where the column allows, one 16-byte store a slice
  const bool vec = (reinterpret_cast<uintptr_t>(y) & 15u) == 0;
  auto load8 = [&](int64_t r, float (&v)[8]) {
    if (vec && r + 8 <= m) {
      const float4 a = *reinterpret_cast<const float4*>(y + r), b = *reinterpret_cast<const float4*>(y + r + 4);
      v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else {
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = (r + u < m) ? y[r + u] : 0.f;
    }
  };
  float mx = 0.f;
  if (y)
#pragma unroll 2
    for (int64_t r = 8 * (sub * 32 + lane); r < m; r += 256 * WPC) {
      float v[8];
      load8(r, v);
#pragma unroll
      for (int u = 0; u < 8; ++u) mx = fmaxf(mx, fabsf(v[u]));
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (WPC > 1) {
    if (lane == 0) red[warp] = mx;
    __syncthreads();
    const int w0 = warp - sub;
    for (int w = 0; w < WPC; ++w) mx = fmaxf(mx, red[w0 + w]);
  }
  if (!valid) return;
  int e = 0;
  if (mx > 0.f) frexpf(mx, &e);   // max < 2^e
  if (sub == 0 && lane == 0) ex[c] = e;
  // 2^(GTOP - e) as two factors (its exponent may exceed FP32's)
  const int k = GTOP - e, k1 = k / 2;
  const float f1 = __int_as_float((127 + k1) << 23), f2 = __int_as_float((127 + k - k1) << 23);
  for (int64_t r = 8 * (sub * 32 + lane); r < mp; r += 256 * WPC) {   // mp is a multiple of 8
    float v[8] = {};
    if (y && r < m) load8(r, v);
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = (v[u] * f1) * f2;               // |v| < 64, exact
#pragma unroll
    for (int i = 0; i < N; ++i) {
      __nv_bfloat162 p[4];
#pragma unroll
      for (int u = 0; u < 8; u += 2) {
        const float q0 = Slices<N>::NEAREST ? rintf(v[u]) : truncf(v[u]);   // |q| <= 64, or 63
        const float q1 = Slices<N>::NEAREST ? rintf(v[u + 1]) : truncf(v[u + 1]);
        p[u / 2] = __floats2bfloat162_rn(q0, q1);
        v[u] = (v[u] - q0) * (float)(1 << Slices<N>::GBITS);                // exact
        v[u + 1] = (v[u + 1] - q1) * (float)(1 << Slices<N>::GBITS);
      }
      *reinterpret_cast<uint4*>(S + ((size_t)i * L4p + c) * mp + r) = *reinterpret_cast<const uint4*>(p);
    }
  }
}

__global__ void __launch_bounds__(256) gram_slice_kernel(const float* __restrict__ y0, const float* __restrict__ y1,
                                                         const float* __restrict__ y2, const float* __restrict__ y3,
                                                         int64_t m, int l, int64_t ld, int L4p, int64_t mp,
                                                         __nv_bfloat16* __restrict__ S, int* __restrict__ ex) {
  gram_slice_cols<7, 8>(y0, y1, y2, y3, m, l, ld, L4p, mp, S, ex, blockIdx.x);
}

// (s, e) += x exactly into a two-float sum (Knuth's two-sum, the rounding error kept in e).
__device__ __forceinline__ void two_sum_acc(float& s, float& e, float x) {
  const float t = __fadd_rn(s, x);
  const float v = __fsub_rn(t, s);
  const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, v)), __fsub_rn(x, v));
  s = t;
  e = __fadd_rn(e, err);
}

// A tile of W for one chunk of rows: tile index tl enumerates (ab, bb) with bb >= 2 ab (the upper part
// of W).
struct GramTile {
  int a0, b0, it0, nit, chunk;
};
__device__ __forceinline__ GramTile gram_tile(const GramTcParams& p, int tl, int chunk) {
  int ab = 0;
  while (ab < p.nA && tl >= max(0, p.nB - 2 * ab)) { tl -= max(0, p.nB - 2 * ab); ++ab; }
  const int it0 = chunk * p.cstages;
  return {ab * GA, (2 * ab + tl) * GB, it0, min(p.kiters, it0 + p.cstages) - it0, chunk};
}

// Persistent CTAs: CTA b takes items b, b + gridDim.x, ...  `item(i)` gives the parameters and the tile.
// The accumulators fill the TMEM, so an item's MMAs wait for the one before to be read out; its
// first stages are loaded meanwhile, and eight warps read (one CTA per item with four epilogue
// warps spent 21 of 50 thousand cycles outside the MMAs).
template <int N, class Item>
__device__ __forceinline__ void gram_tc_items(const int nitems, Item item, int* err) {
  constexpr int GS = Slices<N>::GS, GBITS = Slices<N>::GBITS, NGRP = Slices<N>::NGRP, GPAIR_MAX = NGRP + 1;
  constexpr int STAGE_BYTES = GS * (A_TILE + B_TILE);
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + GSTAGES * STAGE_BYTES);
  uint64_t* full = bars;
  uint64_t* empty = bars + GSTAGES;
  uint64_t* tmem_full = bars + 2 * GSTAGES;
  uint64_t* tmem_empty = tmem_full + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tmem_empty + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  auto a_tile = [&](int s, int i) { return smem + s * STAGE_BYTES + i * A_TILE; };
  auto b_tile = [&](int s, int j) { return smem + s * STAGE_BYTES + GS * A_TILE + j * B_TILE; };

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x / 32, 0), lane = threadIdx.x % 32;
  if (threadIdx.x == 0) {
    for (int s = 0; s < GSTAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(tmem_full, 1);
    mbar_init(tmem_empty, GEPI);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == GEPI + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(GTMEM)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == GEPI) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      int issued = 0, s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int x = blockIdx.x; x < nitems && ok; x += gridDim.x) {
        const GramTcParams* pp;
        const GramTile g = item(x, pp, true);
        for (int i = 0; i < g.nit; ++i) {
          ok = mbar_wait(&empty[s], ph ^ 1u, abort_flag, err);
          if (!ok) break;
          mbar_expect_tx(&full[s], (uint32_t)STAGE_BYTES);
          const int k0 = (g.it0 + i) * GK;
          for (int q = 0; q < GS; ++q) {
            tma_load_2d(smem_u32(a_tile(s, q)), &pp->tmA, k0, q * pp->L4p + g.a0, &full[s]);
            tma_load_2d(smem_u32(b_tile(s, q)), &pp->tmB, k0, q * pp->L4p + g.b0, &full[s]);
          }
          ++issued;
          if (++s == GSTAGES) { s = 0; ph ^= 1u; }
        }
      }
      // drain: every issued stage must have landed before the CTA may exit
      for (int i = max(0, issued - GSTAGES); i < issued; ++i) {
        const uint64_t t0 = now_ns();
        while (!mbar_try_wait(&full[i % GSTAGES], (uint32_t)(i / GSTAGES) & 1u) && now_ns() - t0 < WAIT_NS) __nanosleep(64);
      }
    }
  } else if (warp == GEPI + 1) {
    // ---------------- MMA issuer ----------------
    {   // the whole warp, MMAs by one elected lane
      const uint32_t lead = elect_one();
      // BF16 A and B, FP32 D, both K-major, M = GA; N = t GB for t consecutive B slices: the B
      // slice tiles are adjacent in shared memory, and one MMA of A_i against slices j .. j+t-1
      // writes pair (i, j + u) to TMEM columns (i + j + u) GB, the accumulator of its weight group
      const uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(GA >> 4) << 24);
      // stage 0's descriptors; a stage, slice or K step moves the 16-byte address field
      const uint64_t ad0 = make_desc(smem_u32(a_tile(0, 0)), 16, 8 * GSW, GMODE);
      const uint64_t bd0 = make_desc(smem_u32(b_tile(0, 0)), 16, 8 * GSW, GMODE);
      bool ok = true;
      int s = 0;
      uint32_t ph = 0, done = 0;                 // done: items handed to the epilogue
      for (int x = blockIdx.x; x < nitems && ok; x += gridDim.x, ++done) {
        const GramTcParams* pp;
        const GramTile g = item(x, pp, false);
        if (done > 0) {
          ok = mbar_wait_warp(tmem_empty, (done - 1) & 1u, abort_flag, err);
          if (!ok) break;
        }
        tc_fence_after();
        for (int i = 0; i < g.nit; ++i) {
          ok = mbar_wait_warp(&full[s], ph, abort_flag, err);
          if (!ok) break;
          tc_fence_after();
          const uint64_t so = (uint64_t)(s * (STAGE_BYTES >> 4));
#pragma unroll
          for (int ks = 0; ks < GK / 16; ++ks) {
#pragma unroll
            for (int qi = 0; qi < GS; ++qi) {
              const uint64_t ad = ad0 + so + (uint64_t)((qi * A_TILE + ks * 32) >> 4);
#pragma unroll
              for (int qj = 0; qj <= GPAIR_MAX - 2 - qi; qj += 4) {
                const int t = min(4, GPAIR_MAX - 1 - qi - qj);   // slices qj .. qj + t - 1
                const uint64_t bd = bd0 + so + (uint64_t)((qj * B_TILE + ks * 32) >> 4);
                const uint32_t idesc = idesc0 | ((uint32_t)((t * GB) >> 3) << 17);
                // first products of the weight groups in this chunk: qi == 0, first stage and k-step
                const uint32_t acc = (i > 0 || ks > 0 || qi > 0) ? 1u : 0u;
                umma_bf16(lead, tmem + (uint32_t)((qi + qj) * GB), ad, bd, idesc, acc);
              }
            }
          }
          umma_commit(lead, &empty[s]);   // frees the stage once these MMAs have read it
          if (++s == GSTAGES) { s = 0; ph ^= 1u; }
        }
        umma_commit(lead, tmem_full);     // accumulators complete (also fires after an abort)
      }
    }
  } else {
    // ---------------- epilogue: the exact integer sums -> double-FP32 ----------------
    const int q = warp & 3, c0 = (warp >> 2) * (GB / 2);
    uint32_t done = 0;
    for (int x = blockIdx.x; x < nitems; x += gridDim.x, ++done) {
      const GramTcParams* pp;
      const GramTile g = item(x, pp, false);
      if (!mbar_wait(tmem_full, done & 1u, abort_flag, err) || *abort_flag) break;
      tc_fence_after();
      float h[GB / 2], e[GB / 2];
#pragma unroll
      for (int jj = 0; jj < GB / 2; ++jj) h[jj] = e[jj] = 0.f;
#pragma unroll
      for (int gr = NGRP - 1; gr >= 0; --gr) {
        const float w = __int_as_float((127 - GBITS * gr) << 23);   // 2^(-GBITS gr)
        uint32_t r[32];
        tmem_ld32_issue(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(gr * GB + c0), r);
        tmem_wait_ld();
#pragma unroll
        for (int jj = 0; jj < GB / 2; ++jj) two_sum_acc(h[jj], e[jj], __uint_as_float(r[jj]) * w);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tmem_empty);
      const int a = g.a0 + q * 32 + lane, L4 = pp->L4;
      if (a < L4) {
        float2* P = pp->part + (size_t)g.chunk * L4 * L4;
#pragma unroll
        for (int jj = 0; jj < GB / 2; ++jj) {
          const int b = g.b0 + c0 + jj;
          if (b < L4) P[(size_t)b * L4 + a] = make_float2(h[jj], e[jj]);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == GEPI + 1) {
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(GTMEM) : "memory");
  }
}

__global__ void __launch_bounds__(GTHREADS, 1) gram_tc_kernel(const __grid_constant__ GramTcParams p, int ntiles, int nitems) {
  gram_tc_items<7>(
      nitems,
      [&](int x, const GramTcParams*& pp, bool) {
        pp = &p;
        return gram_tile(p, x % ntiles, x / ntiles);
      },
      p.err);
}

// Batch plans: item (problem, tile, chunk) with that problem's parameters in global memory
// (tensor maps 64-byte aligned, written before the launch).
__global__ void __launch_bounds__(GTHREADS, 1) gram_tc_grouped_kernel(const GramTcProb* __restrict__ probs,
                                                                      const int4* __restrict__ items, int nitems, int* err) {
  gram_tc_items<8>(
      nitems,
      [&](int x, const GramTcParams*& pp, bool tma) {
        const int4 it = items[x];
        pp = &probs[it.x].tc;
        if (tma) {   // the TMA-issuing thread
          asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(&pp->tmA) : "memory");
          asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(&pp->tmB) : "memory");
        }
        return gram_tile(*pp, it.y, it.z);
      },
      err);
}

// W(I, J) for I <= J: the chunk partials added in double-FP32, scaled by 2^(e_I + e_J - 12).
__device__ __forceinline__ double w_tc(const float2* __restrict__ part, int nchunks, const int* __restrict__ ex, int L4,
                                       int I, int J) {
  if (I > J) { const int t = I; I = J; J = t; }
  const size_t o = (size_t)J * L4 + I, step = (size_t)L4 * L4;
  float s = 0.f, e = 0.f;
  for (int c = 0; c < nchunks; ++c) {
    const float2 v = part[c * step + o];
    two_sum_acc(s, e, v.x);
    e = __fadd_rn(e, v.y);
  }
  return ldexp((double)s + (double)e, ex[I] + ex[J] - 2 * GTOP);
}

// W(I, J), I <= J, as a scaled double-FP32 pair (s, e).
__device__ __forceinline__ float2 w_tc_d32(const float2* __restrict__ part, int nchunks, const int* __restrict__ ex,
                                           int L4, int I, int J) {
  if (I > J) { const int t = I; I = J; J = t; }
  const size_t o = (size_t)J * L4 + I, step = (size_t)L4 * L4;
  float s = 0.f, e = 0.f;
  for (int c = 0; c < nchunks; ++c) {
    const float2 v = part[c * step + o];
    two_sum_acc(s, e, v.x);
    e = __fadd_rn(e, v.y);
  }
  const int k = ex[I] + ex[J] - 2 * GTOP;
  return make_float2(ldexpf(s, k), ldexpf(e, k));
}

// Batch plans: item (problem, block of 128 entries); G's upper triangle in double-FP32.
__global__ void __launch_bounds__(128) gram_tc_combine_grouped_kernel(const GramTcProb* __restrict__ probs,
                                                                      const int4* __restrict__ items) {
  const int4 it = items[blockIdx.x];
  const GramTcProb& a = probs[it.x];
  const int l = a.l, L4 = 4 * l;
  const int idx = it.y * 128 + (int)threadIdx.x;
  if (idx >= l * l) return;
  const int i = idx % l, j = idx / l;
  if (i > j) return;
  // component signs of conj(y_i) y_j from the 16 plane products W(c l + i, d l + j)
  const float sg[4][4][4] = {{{1, 0, 0, 0}, {0, 1, 0, 0}, {0, 0, 1, 0}, {0, 0, 0, 1}},
                             {{0, -1, 0, 0}, {1, 0, 0, 0}, {0, 0, 0, -1}, {0, 0, 1, 0}},
                             {{0, 0, -1, 0}, {0, 0, 0, 1}, {1, 0, 0, 0}, {0, -1, 0, 0}},
                             {{0, 0, 0, -1}, {0, 0, -1, 0}, {0, 1, 0, 0}, {1, 0, 0, 0}}};
  float gs[4] = {0.f, 0.f, 0.f, 0.f}, ge[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int d = 0; d < 4; ++d) {
      const float2 w = w_tc_d32(a.tc.part, a.nchunks, a.ex, L4, c * l + i, d * l + j);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (sg[c][d][q] != 0.f) {
          two_sum_acc(gs[q], ge[q], sg[c][d][q] * w.x);
          ge[q] = __fadd_rn(ge[q], sg[c][d][q] * w.y);
        }
    }
  float h[4], lo[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    h[q] = __fadd_rn(gs[q], ge[q]);
    lo[q] = __fsub_rn(ge[q], __fsub_rn(h[q], gs[q]));
    if (i == j && q > 0) h[q] = lo[q] = 0.f;
  }
  float4* o = reinterpret_cast<float4*>(a.G + 8 * ((size_t)j * l + i));
  o[0] = make_float4(h[0], h[1], h[2], h[3]);
  o[1] = make_float4(lo[0], lo[1], lo[2], lo[3]);
}

__global__ void __launch_bounds__(256) gram_slice_grouped_kernel(const GramTcProb* __restrict__ probs,
                                                                 const int4* __restrict__ items) {
  const int4 it = items[blockIdx.x];
  const GramTcProb& a = probs[it.x];
  gram_slice_cols<8, 1>(a.y[0], a.y[1], a.y[2], a.y[3], a.m, a.l, a.ld, a.tc.L4p, a.mp, a.S, a.ex, it.y);
}

// The quaternion Gram from W, FP64 planes: 16 threads per entry (i <= j), thread (c, d) forms
// W(c l + i, d l + j); component q = c xor d of conj(y_i) y_j takes it with the sign of the
// Hamilton table (negative for (c, d) in {(1,0),(2,0),(3,0),(1,2),(2,3),(3,1)}), and the four
// threads of each component add their terms by two shuffles.
__global__ void __launch_bounds__(128) gram_tc_combine_kernel(const float2* __restrict__ part, int nchunks,
                                                              const int* __restrict__ ex, int l, double* __restrict__ G) {
  const int e = blockIdx.x * 8 + (int)(threadIdx.x >> 4);
  const int lane16 = threadIdx.x & 15, c = lane16 >> 2, d = lane16 & 3;
  const int ntri = l * (l + 1) / 2;
  // entry e of the column-by-column listing of the upper triangle: j the largest with j (j + 1) / 2 <= e
  int j = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
  while (j > 0 && j * (j + 1) / 2 > e) --j;
  while ((j + 1) * (j + 2) / 2 <= e) ++j;
  const int i = e - j * (j + 1) / 2;
  double v = 0.0;
  if (e < ntri) {
    v = w_tc(part, nchunks, ex, 4 * l, c * l + i, d * l + j);
    if ((0x3950u >> (c * 4 + d)) & 1u) v = -v;
  }
  v += __shfl_xor_sync(0xffffffffu, v, 5);
  v += __shfl_xor_sync(0xffffffffu, v, 10);
  if (e < ntri && c == 0) {   // thread (0, q) holds component q
    const int q = d;
    const size_t ll = (size_t)l * l;
    const double gq = (i == j && q > 0) ? 0.0 : v;
    G[q * ll + (size_t)j * l + i] = gq;
    if (i != j) G[q * ll + (size_t)i * l + j] = (q == 0) ? gq : -gq;
  }
}

struct GramTcDims {
  int L4, L4p, nA, nB, ntiles, nchunks, kiters, chunk;
  int64_t mp;
};
// `single`: rows per chunk such that the items fill whole waves of the SMs, an item's time outside its
// MMAs counted as 100 rows (4096 x 40: 32 items of 512 rows took 25 us, 128 of 128 rows 12; 20000 x 60: 49 and
// 43 us); from four waves on, and in batch plans, 512.
GramTcDims gram_tc_dims(int64_t m, int l, bool single) {
  GramTcDims d{};
  d.L4 = 4 * l;
  d.L4p = (d.L4 + GB - 1) / GB * GB;
  d.nA = (d.L4 + GA - 1) / GA;
  d.nB = (d.L4 + GB - 1) / GB;
  d.ntiles = 0;
  for (int ab = 0; ab < d.nA; ++ab) d.ntiles += std::max(0, d.nB - 2 * ab);
  d.mp = std::max<int64_t>(GK, (m + 7) / 8 * 8);   // at least one TMA box of rows
  d.kiters = (int)((m + GK - 1) / GK);
  d.chunk = GCHUNK;
  constexpr int64_t SMS = 152;
  if (single && d.ntiles * ((m + GCHUNK - 1) / GCHUNK) < 4 * SMS) {
    int64_t best = INT64_MAX;
    for (int c = GCHUNK; c >= 128; c -= GK) {
      const int64_t items = d.ntiles * ((m + c - 1) / c), cost = (items + SMS - 1) / SMS * (std::min<int64_t>(c, m) + 100);
      if (cost < best) { best = cost; d.chunk = c; }
    }
  }
  d.nchunks = (int)((m + d.chunk - 1) / d.chunk);
  return d;
}

struct GramTcBufs {
  __nv_bfloat16* S;
  int* ex;
  float2* part;
};
size_t rup256(size_t b) { return (b + 255) / 256 * 256; }
GramTcBufs gram_tc_carve(char* base, const GramTcDims& d, int gs) {
  GramTcBufs b;
  b.S = reinterpret_cast<__nv_bfloat16*>(base);
  base += rup256((size_t)gs * d.L4p * d.mp * 2);
  b.ex = reinterpret_cast<int*>(base);
  base += rup256((size_t)d.L4p * 4);
  b.part = reinterpret_cast<float2*>(base);
  return b;
}

// Tensor maps and dimensions of one problem (host side).
bool gram_tc_params(GramTcParams& prm, const GramTcDims& d, const GramTcBufs& bufs, int gs, int* err) {
  memset(&prm, 0, sizeof(prm));
  const uint64_t cols = (uint64_t)gs * d.L4p;
  if (!encode_2d(&prm.tmA, bufs.S, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (uint64_t)d.mp, cols, (uint64_t)d.mp * 2, GK, GA,
                 CU_TENSOR_MAP_SWIZZLE_64B) ||
      !encode_2d(&prm.tmB, bufs.S, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (uint64_t)d.mp, cols, (uint64_t)d.mp * 2, GK, GB,
                 CU_TENSOR_MAP_SWIZZLE_64B))
    return false;
  prm.part = bufs.part;
  prm.L4 = d.L4;
  prm.nA = d.nA;
  prm.nB = d.nB;
  prm.L4p = d.L4p;
  prm.kiters = d.kiters;
  prm.cstages = d.chunk / GK;
  prm.err = err;
  return true;
}

}  // namespace

namespace qlr {

size_t gram_tc_ws(int64_t m, int l, bool single) {
  const GramTcDims d = gram_tc_dims(m, l, single);
  return rup256((size_t)8 * d.L4p * d.mp * 2) + rup256((size_t)d.L4p * 4) + rup256((size_t)d.nchunks * d.L4 * d.L4 * 8);
}

bool gram_tc_supported(const qlr_qmat& Y) {
  if (Y.dtype != QLR_F32 || Y.layout != QLR_COL_MAJOR || Y.rows <= 0 || Y.cols <= 0) return false;
  for (int c = 0; c < 4; ++c)
    if (Y.plane[c] == nullptr) return false;
  const GramTcDims d = gram_tc_dims(Y.rows, (int)Y.cols, false);
  return Y.cols <= 1024 && (int64_t)8 * d.L4p < (1 << 30) && d.nchunks < 65536 && get_encode() != nullptr;
}

int gram_tc(qlr_ctx* ctx, const qlr_qmat& Y, double* G, WsArena& ws) {
  const int64_t m = Y.rows;
  const int l = (int)Y.cols;
  const GramTcDims d = gram_tc_dims(m, l, true);
  const size_t mark = ws.off;
  char* base = ws.take<char>(gram_tc_ws(m, l, true));
  if (!ws.ok) { ws.off = mark; ws.ok = true; return QLR_ENOMEM; }
  const GramTcBufs bufs = gram_tc_carve(base, d, 7);
  __nv_bfloat16* S = bufs.S;
  int* ex = bufs.ex;
  float2* part = bufs.part;
  GramTcParams prm;
  if (!gram_tc_params(prm, d, bufs, 7, ctx->d_err)) {
    ws.off = mark;
    return QLR_ECUDA;
  }
  KTimer kt(ctx, QLR_KID_GRAM);
  gram_slice_kernel<<<d.L4p, 256, 0, ctx->stream>>>(
      static_cast<const float*>(Y.plane[0]), static_cast<const float*>(Y.plane[1]), static_cast<const float*>(Y.plane[2]),
      static_cast<const float*>(Y.plane[3]), m, l, Y.ld, d.L4p, d.mp, S, ex);
  qlr_count_launch();
  QLR_CUDA_TRY(cudaGetLastError());
  QLR_TRY(qlr_allow_smem(gram_tc_kernel));
  const int nitems = d.ntiles * d.nchunks, sms = ctx->num_sms > 0 ? ctx->num_sms : 148;
  gram_tc_kernel<<<(unsigned)std::min(nitems, sms), GTHREADS, gsmem(7), ctx->stream>>>(prm, d.ntiles, nitems);
  qlr_count_launch();
  QLR_CUDA_TRY(cudaGetLastError());
  const int64_t ntri = (int64_t)l * (l + 1) / 2;
  gram_tc_combine_kernel<<<(unsigned)((ntri + 7) / 8), 128, 0, ctx->stream>>>(part, d.nchunks, ex, l, G);
  qlr_count_launch();
  QLR_CUDA_TRY(cudaGetLastError());
  ws.off = mark;   // the buffers are dead once the combine is enqueued (stream order)
  return QLR_OK;
}

size_t gram_tc_record_bytes() { return sizeof(GramTcProb); }

int gram_tc_record(void* dst, const qlr_qmat& Y, char* scratch, float* G, int* err) {
  const int l = (int)Y.cols;
  const GramTcDims d = gram_tc_dims(Y.rows, l, false);
  const GramTcBufs bufs = gram_tc_carve(scratch, d, 8);
  GramTcProb r;
  memset(&r, 0, sizeof(r));
  if (!gram_tc_params(r.tc, d, bufs, 8, err)) return QLR_ECUDA;
  for (int c = 0; c < 4; ++c) r.y[c] = static_cast<const float*>(Y.plane[c]);
  r.m = Y.rows;
  r.ld = Y.ld;
  r.mp = d.mp;
  r.l = l;
  r.nchunks = d.nchunks;
  r.S = bufs.S;
  r.ex = bufs.ex;
  r.G = G;
  memcpy(dst, &r, sizeof(r));
  return QLR_OK;
}

void gram_tc_grouped_items(int64_t m, int l, int prob, std::vector<int4>& slice, std::vector<int4>& mma,
                           std::vector<int4>& comb) {
  const GramTcDims d = gram_tc_dims(m, l, false);
  for (int g = 0; g < (d.L4p + 7) / 8; ++g) slice.push_back(make_int4(prob, g, 0, 0));
  for (int ch = 0; ch < d.nchunks; ++ch)
    for (int t = 0; t < d.ntiles; ++t) mma.push_back(make_int4(prob, t, ch, 0));
  for (int b = 0; b < (l * l + 127) / 128; ++b) comb.push_back(make_int4(prob, b, 0, 0));
}

int gram_tc_grouped(qlr_ctx* ctx, const void* d_probs, const int4* slice, int n_slice, const int4* mma, int n_mma,
                    const int4* comb, int n_comb) {
  if (n_slice <= 0) return QLR_OK;
  const GramTcProb* probs = static_cast<const GramTcProb*>(d_probs);
  KTimer kt(ctx, QLR_KID_GRAM);
  gram_slice_grouped_kernel<<<n_slice, 256, 0, ctx->stream>>>(probs, slice);
  qlr_count_launch();
  QLR_CUDA_TRY(cudaGetLastError());
  QLR_TRY(qlr_allow_smem(gram_tc_grouped_kernel));
  gram_tc_grouped_kernel<<<std::min(n_mma, ctx->num_sms > 0 ? ctx->num_sms : 148), GTHREADS, gsmem(8), ctx->stream>>>(
      probs, mma, n_mma, ctx->d_err);
  qlr_count_launch();
  QLR_CUDA_TRY(cudaGetLastError());
  gram_tc_combine_grouped_kernel<<<n_comb, 128, 0, ctx->stream>>>(probs, comb);
  qlr_count_launch();
  QLR_CUDA_TRY(cudaGetLastError());
  return QLR_OK;
}

}  // namespace qlr
