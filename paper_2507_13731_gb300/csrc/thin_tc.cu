// FP32-accurate products of a tall thin quaternion matrix with a small or wide factor, on the
// tensor cores (tcgen05 kind::f16 with BF16 operands):
//   C = alpha T S + beta C    Q = Y R^{-1}, the lifts, the deflation Y - B (B^H Y)   (thin x small)
//   C = mask .* M + (1 - mask) .* U diag(S) V^H                    (matrix completion, eq. Step2)
//
// Arithmetic.  An FP32 value is the sum of three BF16 values, x = x0 + x1 + x2 (each the rounding
// to nearest of what the earlier ones leave: 8 bits each, 24 in all), so a product of two FP32
// values is the sum of the six products x_i y_j with i + j <= 2 up to ~2^-26 relative.  From
// TINY = 2^-100 on all three are normal BF16 numbers.  A tile whose operands hold smaller entries that
// count, or entries that are not finite (a split's 0 times an infinity is a NaN that FP32 does not
// give), or whose sums may come near FP32's largest number (x0 may lie 2^-9 above x), is formed by FP32
// multiply-adds in the epilogue instead: the split kernels note what they see.  The tensor cores' FP32 accumulation truncates (each MMA that adds into an
// accumulator loses half an ulp of it on average, always toward zero), so the reduction is cut into
// chunks of 32 elements (16 where it is at most 64 long), each in a fresh accumulator: the
// corrections first, 2^-8 of the sum or less, then the one or two MMAs of x0 y0.  The epilogue
// adds the chunks in registers, rounding to nearest.
//
// The Hamilton product (eq. 1) is a real product: row i of the tall operand holds its 4 l plane
// entries (reduction index 4 r + c), and output plane d of column j is its product with the row
// sign(c, d) X_{c xor d}(r, j) of the small factor, which the expansion kernel writes out (4 rows
// per output column).  The tall operand is split once, elementwise, in its own column-major layout
// and read by the MMA as an MN-major tile, so nothing is transposed.
//
// A CTA takes 128 rows of the tall operand by 32 output columns of all four planes (one MMA of
// M = 128, N = 128 per product) and walks a contiguous range of tiles, column tiles fastest: the
// rows' operand stays in shared memory while that leaves a ring of four stages (k <= 40) and only
// the factor streams.  Four chunk accumulators go round (all 512 TMEM columns), so the MMAs run
// ahead of the epilogue, into the next tile too.  A stage's 12 MMAs take about 770 cycles, and its
// issuer spends 500 more on barriers and commits, with the pipe idle: two issuing warps take the
// stages in turn.
//
// Bound and measurements (CUDA events, GB300, whole calls): the masked update writes 16 bytes per entry
// for 6 * 32 k flops.  At 20000 x 10000, k = 50 the six products are 0.83 ms of tensor time and the
// writes 0.5 ms; it takes 1.83 ms against 9.03 ms on the FP32 pipe (4096 x 4096, k = 30: 123 against
// 457 us).  No unit is at its limit (k = 30: tensor pipe active 39 % of the time, DRAM 52 %, L2 37 %); MMAs
// and stores take turns within a CTA.  Q = Y R^{-1} at 20000 x 180: 115 us with the splits against 255.
// Error against 64 bits, random operands: 8.5e-8 (4096 x 4096, k = 30) and 8.9e-8 (20000 x 10000, k = 50)
// relative, FP32 fused multiply-adds 1.5e-7 and more.  About 5e-8 of it is truncation, always toward zero: a
// product that follows another truncating one adds to its error rather than averaging out.  (Chunks of 16
// elements at any length: 4e-8, but up to 24 % more error in all from k = 100 on, and 4 to 9 % more time.)
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "qlr_internal.h"
#include "tc_common.cuh"

namespace {

using namespace qlr_tc;

constexpr int TL_M = 128, TL_J = 32, TL_N = 4 * TL_J;   // tile: rows, output columns, MMA N
constexpr int TL_BK = 32;                               // reduction elements per stage
constexpr int TL_SPLIT = TL_M * TL_BK * 2;              // one split of one operand tile: 8 KB
constexpr int TL_OP = 3 * TL_SPLIT;                     // one operand's three splits
constexpr int TL_EPI = 8;                               // epilogue warps
constexpr int TL_ISSUERS = 2;                           // MMA-issuing warps
constexpr int TL_THREADS = 32 * (TL_EPI + 1 + TL_ISSUERS);   // epilogue, TMA producer, issuers
constexpr int TL_RES_CHUNKS = 5;                        // chunks of the resident operand (K <= 160)
constexpr int TL_MAX_STAGES = 4;
constexpr int TL_ACC = 4;                               // chunk accumulators
constexpr int TALL_MAX_L = 256;

struct TallArgs {
  CUtensorMap tmA, tmB;
  int64_t M, N;                 // rows of the tall operand, output columns
  int K, Kq;                    // reduction length (4 per column of the tall operand), padded to TL_BK
  int mtiles, ntiles;
  int upper;                    // column tile nt reduces only indices below 4 (32 nt + 32)
  int resident, stages, per;    // per: MMA steps (of 16 reduction elements) per chunk, 1 or 2
  float* c[4];
  int64_t ldc;
  float alpha, beta;            // thin x small
  const float* m[4];            // masked update: M (m[0] null: zero real part), mask
  int64_t ldm;
  const uint8_t* mask;
  int64_t ldk;
  // the operands as given, for tiles formed in FP32, and what the split kernels found in them
  const float* t[4];            // tall operand, column-major
  int64_t ldt;
  const double* s[4];           // small FP64 factor, column-major; masked update: U and S
  int64_t lds;
  const float* u[4];
  int64_t ldu;
  const double* sigma;
  const uint8_t* aflags;        // [512-row block][column of the tall operand]: largest biased exponent, 255 also
                                // for entries below TINY
  const uint4* bflags;          // [column tile][32-column block of the reduction]: columns with entries below
                                // TINY, columns with entries that dwarf such, largest biased exponent
  int* err;
};
constexpr float TINY = 7.888609e-31f, DWARF = 1.3234890e-23f;   // 2^-100, 2^-76
// Operands below 2^(ea - 126) and 2^(eb - 126): a sum of 4 l <= 2^10 products stays below 2^126.
constexpr unsigned EXP_SUM_MAX = 126 + 252 - 10;
constexpr int TL_MAX_RB = TALL_MAX_L / 32;                      // 32-column blocks of the reduction
constexpr int SPLIT_ROWS = 512;                                 // rows per CTA of the split kernel
__device__ __forceinline__ bool is_tiny(float x) { return x != 0.f && fabsf(x) < TINY; }

// Signs of the real product, bit 4 c + d: T_c X_{c xor d} enters output plane d negatively.
constexpr uint32_t neg_bits(std::initializer_list<std::pair<int, int>> cd) {
  uint32_t m = 0;
  for (const auto& e : cd) m |= 1u << (4 * e.first + e.second);
  return m;
}
constexpr uint32_t NEG_THIN = neg_bits({{1, 0}, {2, 0}, {3, 0}, {3, 1}, {1, 2}, {2, 3}});   // T S, eq. 1
constexpr uint32_t NEG_MASKED = neg_bits({{1, 1}, {3, 1}, {1, 2}, {2, 2}, {2, 3}, {3, 3}});  // u conj(v), T = V, X = U S

// x = s0 + s1 + s2.  A value that rounds beyond BF16's range is truncated instead; a non-finite
// value is kept whole in s0.
__device__ __forceinline__ void split3(float x, __nv_bfloat16 (&s)[3]) {
  s[0] = __float2bfloat16_rn(x);
  if (__hisinf(s[0]) && isfinite(x)) s[0] = __float2bfloat16_rz(x);
  const float r1 = isfinite(x) ? x - __bfloat162float(s[0]) : 0.f;
  s[1] = __float2bfloat16_rn(r1);
  s[2] = __float2bfloat16_rn(r1 - __bfloat162float(s[1]));
}

// Tall operand T (rows x l, column-major planes): out[s][4 r + c][row], rows padded to Kq with
// zero reduction rows.  A thread takes two matrix rows of one column's four planes.
struct SplitArgs {
  const float* t[4];
  int64_t ld, rows, ldo;
  int l, Kq;
  __nv_bfloat16* out;
  uint8_t* flags;
};
__global__ void __launch_bounds__(SPLIT_ROWS / 2) tall_split_kernel(const SplitArgs a) {
  __shared__ unsigned wmax[SPLIT_ROWS / 64];
  const int r = blockIdx.y;
  const int64_t i = (int64_t)blockIdx.x * SPLIT_ROWS + 2 * threadIdx.x;
  float x[4][2] = {};
  if (r < a.l) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float* src = a.t[c] + (int64_t)r * a.ld;
      if (i < a.rows) x[c][0] = src[i];
      if (i + 1 < a.rows) x[c][1] = src[i + 1];
    }
  }
  float mx = 0.f;
  bool odd = false;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const float v = x[e / 2][e % 2];
    mx = fmaxf(mx, fabsf(v));
    odd = odd || is_tiny(v) || isnan(v);
  }
  const unsigned m = __reduce_max_sync(0xffffffffu, odd ? 0x7f800000u : __float_as_uint(mx));
  if (threadIdx.x % 32 == 0) wmax[threadIdx.x / 32] = m;
  if (i < a.ldo) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      __nv_bfloat16 s0[3], s1[3];
      split3(x[c][0], s0);
      split3(x[c][1], s1);
#pragma unroll
      for (int s = 0; s < 3; ++s)
        *reinterpret_cast<__nv_bfloat162*>(a.out + ((size_t)s * a.Kq + 4 * r + c) * a.ldo + i) = __nv_bfloat162(s0[s], s1[s]);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned b = 0;
    for (int w = 0; w < SPLIT_ROWS / 64; ++w) b = max(b, wmax[w]);
    a.flags[(size_t)blockIdx.x * (a.Kq / 4) + r] = (uint8_t)(b >> 23);
  }
}

// Expanded factor: out[s][128 nt + 64 h + 16 d + jj][4 r + c] = sign(c, d) X_{c xor d}(r, 32 nt + 16 h + jj):
// the 64 accumulator columns of an epilogue warp (16 output columns, four planes) lie together.
// X is the small FP64 factor (column-major, rounded to FP32), or, for the masked update, U diag(S)
// with the matrix row as the column index.  A CTA stages 32 r x 32 columns of the four planes.
struct ExpandArgs {
  const double* s[4];           // small factor planes (null: masked update)
  int64_t lds;
  const float* u[4];            // U, column-major; S
  int64_t ldu;
  const double* sigma;
  int l;
  int64_t N;                    // valid output columns
  int Kq;
  int64_t rows;                 // rows of one split
  uint32_t neg;                 // NEG_THIN or NEG_MASKED
  __nv_bfloat16* out;
  uint4* flags;
};
__global__ void __launch_bounds__(256) tall_expand_kernel(const ExpandArgs a) {
  __shared__ float X[4][32][33];   // plane, r, column
  __shared__ unsigned tiny_cols[8], big_cols[8], wmax[8];
  const int t = threadIdx.x;
  const int64_t j0 = (int64_t)blockIdx.x * TL_J;
  const int r0 = blockIdx.y * 32;
  for (int e = t; e < 4096; e += 256) {
    const int q = e / 1024, f = e % 1024;
    const int jj = a.u[1] ? f % 32 : f / 32, rr = a.u[1] ? f / 32 : f % 32;   // coalesced either way
    const int64_t j = j0 + jj;
    const int r = r0 + rr;
    float v = 0.f;
    if (j < a.N && r < a.l)
      v = a.u[1] ? a.u[q][(int64_t)r * a.ldu + j] * (float)a.sigma[r] : (float)a.s[q][j * a.lds + r];
    X[q][rr][jj] = v;
  }
  __syncthreads();
  {   // a lane per column, four r a warp
    bool tiny = false, odd = false;
    float mx = 0.f;
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const float v = X[e / 4][4 * (t / 32) + e % 4][t % 32];
      tiny = tiny || is_tiny(v);
      odd = odd || isnan(v);
      mx = fmaxf(mx, fabsf(v));
    }
    const unsigned tb = __ballot_sync(0xffffffffu, tiny), bb = __ballot_sync(0xffffffffu, mx >= DWARF);
    const unsigned mb = __reduce_max_sync(0xffffffffu, odd ? 0x7f800000u : __float_as_uint(mx));
    if (t % 32 == 0) { tiny_cols[t / 32] = tb; big_cols[t / 32] = bb; wmax[t / 32] = mb; }
    __syncthreads();
    if (t == 0) {
      uint4 f = make_uint4(0u, 0u, 0u, 0u);
      for (int w = 0; w < 8; ++w) { f.x |= tiny_cols[w]; f.y |= big_cols[w]; f.z = max(f.z, wmax[w] >> 23); }
      a.flags[(size_t)blockIdx.x * TL_MAX_RB + blockIdx.y] = f;
    }
  }
  const int rr = t % 32;
  if (4 * (r0 + rr) >= a.Kq) return;
  for (int w = t / 32; w < TL_N; w += 8) {
    const int d = (w / 16) % 4, jj = (w / 64) * 16 + w % 16;
    __nv_bfloat16 h[4][3];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float v = X[c ^ d][rr][jj];
      split3(((a.neg >> (4 * c + d)) & 1u) ? -v : v, h[c]);
    }
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      __nv_bfloat162 p[2] = {__nv_bfloat162(h[0][s], h[1][s]), __nv_bfloat162(h[2][s], h[3][s])};
      *reinterpret_cast<uint2*>(a.out + ((size_t)s * a.rows + (size_t)blockIdx.x * TL_N + w) * a.Kq + 4 * (r0 + rr)) =
          *reinterpret_cast<uint2*>(p);
    }
  }
}

template <bool MASKED>
__global__ void __launch_bounds__(TL_THREADS, 1) tall_gemm_kernel(const __grid_constant__ TallArgs p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int nchunks = p.Kq / TL_BK, stages = p.stages, per = p.per;
  const bool res = p.resident != 0;
  const int a_res = res ? nchunks * TL_OP : 0;                   // resident operand, then the ring
  const int stage_bytes = res ? TL_OP : 2 * TL_OP;
  unsigned char* ring = smem + a_res;
  uint64_t* bars = reinterpret_cast<uint64_t*>(ring + stages * stage_bytes);
  uint64_t* full = bars;                         // [TL_MAX_STAGES]
  uint64_t* empty = bars + TL_MAX_STAGES;        // [TL_MAX_STAGES]
  uint64_t* afull = bars + 2 * TL_MAX_STAGES;    // [TL_RES_CHUNKS]
  uint64_t* adone = afull + TL_RES_CHUNKS;       // [1]
  uint64_t* acc_full = adone + 1;                // [TL_ACC]
  uint64_t* acc_empty = acc_full + TL_ACC;       // [TL_ACC]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + TL_ACC);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  unsigned* seen = tmem_slot + 2;                // [3] over the whole operands: largest exponents, tiny entries
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x / 32, 0), lane = threadIdx.x % 32;
  const int64_t tiles = (int64_t)p.mtiles * p.ntiles;
  const int64_t t0 = tiles * blockIdx.x / gridDim.x, t1 = tiles * (blockIdx.x + 1) / gridDim.x;
  auto ksteps_of = [&](int nt) {
    const int k = p.upper ? min(p.K, 4 * TL_J * (nt + 1)) : p.K;
    return (k + 15) / 16;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < TL_MAX_STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int s = 0; s < TL_RES_CHUNKS; ++s) mbar_init(&afull[s], 1);
    mbar_init(adone, TL_ISSUERS);
    for (int b = 0; b < TL_ACC; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], TL_EPI); }
    *abort_flag = 0;
    seen[0] = seen[1] = seen[2] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == TL_EPI + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == TL_EPI) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      auto load_a = [&](unsigned char* dst, int mt, int ch, uint64_t* bar) {
        for (int s = 0; s < 3; ++s)
          for (int h = 0; h < 2; ++h)
            tma_load_2d(smem_u32(dst + s * TL_SPLIT + h * (TL_SPLIT / 2)), &p.tmA, mt * TL_M + 64 * h,
                        s * p.Kq + ch * TL_BK, bar);
      };
      int it = 0, cur = -1, nm = 0, s = 0;
      uint32_t sph = 0;
      bool ok = true;
      int mt = (int)(t0 / p.ntiles), nt = (int)(t0 % p.ntiles);
      for (int left = (int)(t1 - t0); left > 0 && ok; --left) {
        if (res && mt != cur) {
          if (nm > 0) ok = mbar_wait(adone, (uint32_t)(nm - 1) & 1u, abort_flag, p.err);   // the previous rows are done with
          if (!ok) break;
          for (int ch = 0; ch < nchunks; ++ch) {
            mbar_expect_tx(&afull[ch], TL_OP);
            load_a(smem + ch * TL_OP, mt, ch, &afull[ch]);
          }
          ++nm;
        }
        cur = mt;
        const int nch = (ksteps_of(nt) + 1) / 2;
        for (int ch = 0; ch < nch; ++ch, ++it) {
          ok = mbar_wait(&empty[s], sph ^ 1u, abort_flag, p.err);
          if (!ok) break;
          mbar_expect_tx(&full[s], (uint32_t)stage_bytes);
          unsigned char* st = ring + s * stage_bytes;
          if (!res) load_a(st, mt, ch, &full[s]);
          unsigned char* bt = res ? st : st + TL_OP;
          for (int q = 0; q < 3; ++q)
            tma_load_2d(smem_u32(bt + q * TL_SPLIT), &p.tmB, ch * TL_BK, q * p.ntiles * TL_N + nt * TL_N, &full[s]);
          if (++s == stages) { s = 0; sph ^= 1u; }
        }
        if (++nt == p.ntiles) { nt = 0; ++mt; }
      }
      // drain: every issued copy must have landed before the CTA may exit
      const uint64_t w0 = now_ns();
      for (int i = max(0, it - stages); i < it; ++i)
        while (!mbar_try_wait(&full[i % stages], (uint32_t)(i / stages) & 1u) && now_ns() - w0 < WAIT_NS) __nanosleep(64);
      if (nm > 0)
        for (int ch = 0; ch < nchunks; ++ch)
          while (!mbar_try_wait(&afull[ch], (uint32_t)(nm - 1) & 1u) && now_ns() - w0 < WAIT_NS) __nanosleep(64);
    }
  } else if (warp > TL_EPI) {
    // ---------------- MMA issuers: stages in turn ----------------
    {   // the whole warp, MMAs by one elected lane
      const uint32_t lead = elect_one();
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | ((uint32_t)(TL_N >> 3) << 17) |
                             ((uint32_t)(TL_M >> 4) << 24);
      // descriptors of the first stage (later ones move the 16-byte address field): the tall operand
      // MN-major, 64-row atoms of 128 bytes (stride TL_SPLIT / 2) in 8-step groups of 1024 bytes; the
      // factor K-major, 64-byte rows
      const uint64_t adesc0 = make_desc(smem_u32(res ? smem : ring), TL_SPLIT / 2, 1024, 2);
      const uint64_t bdesc0 = make_desc(smem_u32(res ? ring : ring + TL_OP), 16, 512, 4);
      int cur = -1, nm = 0, s = 0, b = 0, turn = warp - TL_EPI - 1;
      // Phases of the ring and of the accumulators.  An issuer skips the other's stages without waiting, and
      // yet none of its waits by parity is two phases behind: the ring holds an even number of stages
      // (TL_MAX_STAGES), so a slot is always the same issuer's; of the accumulators between two uses of one,
      // at most two belong to a stage of the other issuer, so this one has waited for the drain of a
      // later one than the use before the last, and they are drained in order.
      uint32_t sph = 0, bph = 0;
      bool ok = true;
      int mt = (int)(t0 / p.ntiles), nt = (int)(t0 % p.ntiles);
      for (int left = (int)(t1 - t0); left > 0 && ok; --left) {
        if (res && mt != cur) {   // new rows: their resident operand is on its way
          if (cur >= 0) umma_commit(lead, adone);   // the old one may be overwritten once these MMAs have read it
          // Both issuers wait for every phase of afull, also one whose rows have no stage for them (a range
          // that begins on the last column tile of its rows): a wait by parity would take a phase not yet
          // begun for one that is over.
          for (int c2 = 0; c2 < nchunks && ok; ++c2) ok = mbar_wait_warp(&afull[c2], (uint32_t)nm & 1u, abort_flag, p.err);
          if (!ok) break;
          ++nm;
        }
        cur = mt;
        const int ks_n = ksteps_of(nt);
        for (int ch = 0; 2 * ch < ks_n; ++ch) {
          const int nacc = (per == 2 || 2 * ch + 1 == ks_n) ? 1 : 2;   // chunks of this stage
          if (turn != 0) {                           // another issuer's
            --turn;
            b += nacc;
            if (b >= TL_ACC) { b -= TL_ACC; bph ^= 1u; }
            if (++s == stages) { s = 0; sph ^= 1u; }
            continue;
          }
          turn = TL_ISSUERS - 1;
          ok = mbar_wait_warp(&full[s], sph, abort_flag, p.err);
          if (!ok) break;
          const uint64_t ad = adesc0 + (uint64_t)(uint32_t)((res ? ch * TL_OP : s * stage_bytes) >> 4);
          const uint64_t bd = bdesc0 + (uint64_t)(uint32_t)((s * stage_bytes) >> 4);
          constexpr uint64_t SP = TL_SPLIT >> 4, KA = (16 * 128) >> 4, KB = 32 >> 4;
          // one accumulation chunk: the corrections of its steps [h0, h1), then x0 y0
          auto chunk = [&](auto H0, auto H1) {
            constexpr int h0 = decltype(H0)::value, h1 = decltype(H1)::value;
            ok = mbar_wait_warp(&acc_empty[b], bph ^ 1u, abort_flag, p.err);
            if (!ok) return;
            tc_fence_after();
            const uint32_t acc = tmem + (uint32_t)(b * TL_N);
#pragma unroll
            for (int h = h0; h < h1; ++h) {
              const uint64_t x = ad + h * KA, y = bd + h * KB;
              umma_bf16(lead, acc, x, y + 2 * SP, idesc, h > h0);
              umma_bf16(lead, acc, x + 2 * SP, y, idesc, 1u);
              umma_bf16(lead, acc, x + SP, y + SP, idesc, 1u);
              umma_bf16(lead, acc, x, y + SP, idesc, 1u);
              umma_bf16(lead, acc, x + SP, y, idesc, 1u);
            }
#pragma unroll
            for (int h = h0; h < h1; ++h) umma_bf16(lead, acc, ad + h * KA, bd + h * KB, idesc, 1u);
            umma_commit(lead, &acc_full[b]);
            if (++b == TL_ACC) { b = 0; bph ^= 1u; }
          };
          using I0 = std::integral_constant<int, 0>;
          using I1 = std::integral_constant<int, 1>;
          using I2 = std::integral_constant<int, 2>;
          if (per == 2 && 2 * ch + 1 < ks_n) {
            chunk(I0{}, I2{});
          } else {
            chunk(I0{}, I1{});
            if (ok && 2 * ch + 1 < ks_n) chunk(I1{}, I2{});
          }
          if (!ok) break;
          umma_commit(lead, &empty[s]);
          if (++s == stages) { s = 0; sph ^= 1u; }
        }
        if (++nt == p.ntiles) { nt = 0; ++mt; }
      }
    }
  } else {
    // ---------------- epilogue: 8 warps, a lane quarter and half the columns each ----------------
    const int q = warp & 3, half = warp >> 2;
    int mt = (int)(t0 / p.ntiles), nt = (int)(t0 % p.ntiles), b = 0, cur = -1;
    uint32_t bph = 0;
    unsigned ea = 0;                                   // largest biased exponent of these rows
    bool ok = true;
    // What the split kernels found, over the whole operands, while the first tile is on its way: tiles are
    // looked at one by one only if there is something to find (their 16 bytes a tile cost 6 % of an update of
    // rank 8).
    const int rblocks = (p.Kq + 4 * 32 - 1) / (4 * 32);
    bool look;
    {
      unsigned a4 = 0, be = 0, tiny = 0;
      const unsigned* af = reinterpret_cast<const unsigned*>(p.aflags);
      const int64_t words = (p.M + SPLIT_ROWS - 1) / SPLIT_ROWS * (p.Kq / 16);
      for (int64_t i = threadIdx.x; i < words; i += 32 * TL_EPI) a4 = __vmaxu4(a4, af[i]);
      for (int i = threadIdx.x; i < p.ntiles * rblocks; i += 32 * TL_EPI) {
        const uint4 f = p.bflags[(size_t)(i / rblocks) * TL_MAX_RB + i % rblocks];
        tiny |= f.x;
        be = max(be, f.z);
      }
      a4 = __vmaxu4(a4, a4 >> 16);
      a4 = __reduce_max_sync(0xffffffffu, __vmaxu4(a4, a4 >> 8) & 255u);
      be = __reduce_max_sync(0xffffffffu, be);
      tiny = __reduce_or_sync(0xffffffffu, tiny);
      if (lane == 0) { atomicMax(&seen[0], a4); atomicMax(&seen[1], be); atomicOr(&seen[2], tiny); }
      asm volatile("bar.sync 1, %0;" ::"n"(32 * TL_EPI) : "memory");
      look = seen[0] == 255u || seen[1] == 255u || seen[2] != 0 || seen[0] + seen[1] > EXP_SUM_MAX;
    }
    for (int left = (int)(t1 - t0); left > 0 && ok; --left) {
      const int64_t row = (int64_t)mt * TL_M + q * 32 + lane, j0 = (int64_t)nt * TL_J + half * 16;
      const int nch = (ksteps_of(nt) + per - 1) / per;
      const int tmt = mt;
      if (++nt == p.ntiles) { nt = 0; ++mt; }
      const bool row_ok = row < p.M;
      const int nj = (int)max((int64_t)0, min((int64_t)16, p.N - j0));   // valid columns of this warp's 16
      uint8_t mk[16];   // the mask, in flight while the MMAs run
      if (MASKED && row_ok) {
        const uint8_t* mp = p.mask + j0 * p.ldk + row;
#pragma unroll
        for (int jj = 0; jj < 16; ++jj, mp += p.ldk) mk[jj] = jj < nj ? *mp : 0;
      }
      float v[4][16];
#pragma unroll
      for (int e = 0; e < 64; ++e) v[e / 16][e % 16] = 0.f;
      for (int ch = 0; ch < nch; ++ch) {
        ok = mbar_wait(&acc_full[b], bph, abort_flag, p.err) && !*abort_flag;
        if (!ok) break;
        tc_fence_after();
        const uint32_t base = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * TL_N + half * 64);
#pragma unroll
        for (int d = 0; d < 4; d += 2) {
          uint32_t r[32];
          tmem_ld32_issue(base + d * 16, r);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 32; ++e) v[d + e / 16][e % 16] += __uint_as_float(r[e]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[b]);   // one arrival a warp: 32 lanes' would serialise
        if (++b == TL_ACC) { b = 0; bph ^= 1u; }
      }
      if (!ok) break;
      bool again = false;
      if (look) {
        if (tmt != cur) {
          unsigned a4 = 0;
          const unsigned* af = reinterpret_cast<const unsigned*>(p.aflags + (size_t)(tmt / (SPLIT_ROWS / TL_M)) * (p.Kq / 4));
          for (int w = lane; w < p.Kq / 16; w += 32) a4 = __vmaxu4(a4, af[w]);
          a4 = __vmaxu4(a4, a4 >> 16);
          ea = __reduce_max_sync(0xffffffffu, __vmaxu4(a4, a4 >> 8) & 255u);
          cur = tmt;
        }
        const uint4 f = lane < rblocks ? p.bflags[(size_t)(j0 / TL_J) * TL_MAX_RB + lane] : make_uint4(0u, 0u, 0u, 0u);
        const unsigned eb = __reduce_max_sync(0xffffffffu, f.z);
        const unsigned tc = __reduce_or_sync(0xffffffffu, f.x) & ~__reduce_or_sync(0xffffffffu, f.y);
        again = tc != 0 || ea == 255u || eb == 255u || ea + eb > EXP_SUM_MAX;
      }
      if (!row_ok) continue;
      if (again) {   // FP32 multiply-adds on the operands as given (the sums' values are not used)
        constexpr uint32_t neg = MASKED ? NEG_MASKED : NEG_THIN;
#pragma unroll
        for (int e = 0; e < 64; ++e) v[e / 16][e % 16] = 0.f;
        const int rend = p.upper ? (int)min((int64_t)p.K / 4, j0 + 16) : p.K / 4;
#pragma unroll 1
        for (int r = 0; r < rend; ++r) {
          float t[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) t[c] = p.t[c][(int64_t)r * p.ldt + row];
          const float sg = MASKED ? (float)p.sigma[r] : 0.f;
#pragma unroll
          for (int jj = 0; jj < 16; ++jj) {
            if (jj >= nj) continue;
            float x[4];
#pragma unroll
            for (int c = 0; c < 4; ++c)
              x[c] = MASKED ? p.u[c][(int64_t)r * p.ldu + j0 + jj] * sg : (float)p.s[c][(j0 + jj) * p.lds + r];
#pragma unroll
            for (int d = 0; d < 4; ++d)
#pragma unroll
              for (int c = 0; c < 4; ++c)
                v[d][jj] = fmaf(((neg >> (4 * c + d)) & 1u) ? -t[c] : t[c], x[c ^ d], v[d][jj]);
          }
        }
      }
      // pointers are stepped by the pitch: 64-bit index products for every entry made this
      // epilogue the bound (50 instructions an entry: 211 us at 4096 x 4096, k = 30)
      if (MASKED) {   // C(i, j): i = output column, j = row of the tall operand
        uint32_t seen = 0;
#pragma unroll
        for (int jj = 0; jj < 16; ++jj) seen |= (mk[jj] != 0 ? 1u : 0u) << jj;
        if (seen) {
#pragma unroll
          for (int d = 0; d < 4; ++d) {
            if (!p.m[d]) {
#pragma unroll
              for (int jj = 0; jj < 16; ++jj)
                if ((seen >> jj) & 1u) v[d][jj] = 0.f;
              continue;
            }
            const float* m = p.m[d] + j0 * p.ldm + row;
            float mv[16];
#pragma unroll
            for (int jj = 0; jj < 16; ++jj, m += p.ldm) mv[jj] = ((seen >> jj) & 1u) ? *m : 0.f;
#pragma unroll
            for (int jj = 0; jj < 16; ++jj)
              if ((seen >> jj) & 1u) v[d][jj] = mv[jj];
          }
        }
#pragma unroll
        for (int d = 0; d < 4; ++d) {
          float* c = p.c[d] + j0 * p.ldc + row;
          if (nj == 16) {
#pragma unroll
            for (int jj = 0; jj < 16; ++jj, c += p.ldc) __stcs(c, v[d][jj]);
          } else {
#pragma unroll
            for (int jj = 0; jj < 16; ++jj, c += p.ldc)
              if (jj < nj) __stcs(c, v[d][jj]);
          }
        }
      } else {
#pragma unroll
        for (int d = 0; d < 4; ++d) {
          float* c = p.c[d] + j0 * p.ldc + row;
          if (p.beta != 0.f) {
            float old[16];
            const float* o = c;
#pragma unroll
            for (int jj = 0; jj < 16; ++jj, o += p.ldc) old[jj] = jj < nj ? *o : 0.f;
#pragma unroll
            for (int jj = 0; jj < 16; ++jj) v[d][jj] = p.alpha * v[d][jj] + p.beta * old[jj];
          } else {
#pragma unroll
            for (int jj = 0; jj < 16; ++jj) v[d][jj] *= p.alpha;
          }
#pragma unroll
          for (int jj = 0; jj < 16; ++jj, c += p.ldc)
            if (jj < nj) *c = v[d][jj];
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == TL_EPI + 1) {
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
}

int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }
// The operands' splits, and with what was found in them behind (multiples of 16 bytes).
size_t a_split(int64_t rows, int64_t l) { return (size_t)3 * round_up(4 * l, TL_BK) * round_up(rows, 8) * 2; }
size_t b_split(int64_t N, int64_t l) { return (size_t)3 * round_up(N, TL_J) * 4 * round_up(4 * l, TL_BK) * 2; }
size_t a_bytes(int64_t rows, int64_t l) {
  return a_split(rows, l) + (size_t)(round_up(rows, SPLIT_ROWS) / SPLIT_ROWS) * (round_up(4 * l, TL_BK) / 4);
}
size_t b_bytes(int64_t N, int64_t l) { return b_split(N, l) + (size_t)(round_up(N, TL_J) / TL_J) * TL_MAX_RB * sizeof(uint4); }

// Split the tall operand (rows [0, rows) of its planes) into `out`.
void run_split(cudaStream_t st, const void* const t[4], int64_t ld, int64_t rows, int l, char* out, TallArgs& p) {
  SplitArgs a{};
  for (int c = 0; c < 4; ++c) a.t[c] = static_cast<const float*>(t[c]);
  a.ld = ld; a.rows = rows; a.ldo = round_up(rows, 8); a.l = l; a.Kq = (int)round_up(4 * l, TL_BK);
  a.out = reinterpret_cast<__nv_bfloat16*>(out);
  a.flags = reinterpret_cast<uint8_t*>(out + a_split(rows, l));
  for (int c = 0; c < 4; ++c) p.t[c] = a.t[c];
  p.ldt = ld;
  p.aflags = a.flags;
  tall_split_kernel<<<dim3((unsigned)((rows + SPLIT_ROWS - 1) / SPLIT_ROWS), (unsigned)(a.Kq / 4)), SPLIT_ROWS / 2, 0, st>>>(a);
  qlr_count_launch();
}

// Fill in the tile plan and the tensor maps and launch.
template <bool MASKED>
int run_gemm(qlr_ctx* ctx, TallArgs& p, const char* A, const char* B, int l) {
  p.K = 4 * l;
  p.Kq = (int)round_up(p.K, TL_BK);
  p.mtiles = (int)((p.M + TL_M - 1) / TL_M);
  p.ntiles = (int)((p.N + TL_J - 1) / TL_J);
  p.resident = (p.Kq <= TL_RES_CHUNKS * TL_BK && p.ntiles > 1) ? 1 : 0;
  const size_t budget = (size_t)227 * 1024 - 1024 - 256;
  const size_t ares = p.resident ? (size_t)(p.Kq / TL_BK) * TL_OP : 0, stage = p.resident ? TL_OP : 2 * TL_OP;
  p.stages = (int)std::min<size_t>(TL_MAX_STAGES, (budget - ares) / stage / 2 * 2);   // even: see the issuers
  p.per = (p.K <= 64) ? 1 : 2;
  const int64_t ldo = round_up(p.M, 8);
  if (!encode_2d(&p.tmA, A, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (uint64_t)p.M, (uint64_t)3 * p.Kq, (uint64_t)ldo * 2, 64,
                 TL_BK, CU_TENSOR_MAP_SWIZZLE_128B) ||
      !encode_2d(&p.tmB, B, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (uint64_t)p.Kq, (uint64_t)3 * p.ntiles * TL_N,
                 (uint64_t)p.Kq * 2, TL_BK, TL_N, CU_TENSOR_MAP_SWIZZLE_64B))
    return QLR_ECUDA;
  const size_t smem = ares + p.stages * stage + 1024 + 256;
  auto kern = tall_gemm_kernel<MASKED>;
  QLR_TRY(qlr_allow_smem(kern));
  const int64_t tiles = (int64_t)p.mtiles * p.ntiles;
  const unsigned grid = (unsigned)std::min<int64_t>(tiles, ctx->num_sms > 0 ? ctx->num_sms : 148);
  kern<<<grid, TL_THREADS, smem, ctx->stream>>>(p);
  qlr_count_launch();
  QLR_CUDA_TRY(cudaGetLastError());
  return QLR_OK;
}

int run_expand(cudaStream_t st, ExpandArgs& e, int l, int64_t N, char* out, TallArgs& p) {
  e.l = l;
  e.N = N;
  e.Kq = (int)round_up(4 * l, TL_BK);
  e.rows = round_up(N, TL_J) * 4;
  e.out = reinterpret_cast<__nv_bfloat16*>(out);
  e.flags = reinterpret_cast<uint4*>(out + b_split(N, l));
  for (int c = 0; c < 4; ++c) { p.s[c] = e.s[c]; p.u[c] = e.u[c]; }
  p.lds = e.lds; p.ldu = e.ldu; p.sigma = e.sigma; p.bflags = e.flags;
  tall_expand_kernel<<<dim3((unsigned)((N + TL_J - 1) / TL_J), (unsigned)((e.Kq + 127) / 128)), 256, 0, st>>>(e);
  qlr_count_launch();
  QLR_CUDA_TRY(cudaGetLastError());
  return QLR_OK;
}

// Panels of the masked update: the expanded factor of a panel of rows of C stays in L2 while the
// panel's entries stream out.
constexpr size_t PANEL_BYTES = (size_t)48 << 20;
constexpr int64_t PANEL_COLS = 65536;
int64_t panel_rows(int64_t m, int k) {
  const int64_t per = (int64_t)b_bytes(TL_J, k);
  return std::min<int64_t>(round_up(m, TL_J), std::max<int64_t>(1, (int64_t)PANEL_BYTES / per) * TL_J);
}

}  // namespace

namespace qlr {

// The line lies where three launches on the tensor cores and one on the FP32 pipe take the same
// time: 410 against 418 us for a CholeskyQR2 at rows N l = 24e6 (l = 110), 323 / 322 at 36e6 (l = 60),
// 434 / 445 at 36e6 (l = 110), 405 / 423 at 72e6 (l = 60), 1465 / 1753 at 20000 x 180.
bool tall_gemm_wanted(int64_t rows, int64_t N, int l) {
  return l >= 1 && l <= TALL_MAX_L && N >= 1 && rows < (1LL << 31) - TL_M && N < (1LL << 28) && rows * N * l >= (int64_t)24000000 && get_encode() != nullptr;
}
size_t tall_gemm_ws(int64_t rows, int64_t N, int l) { return a_bytes(rows, l) + b_bytes(N, l) + 1024; }

int tall_gemm(qlr_ctx* ctx, const qlr_qmat& T, const double* const S[4], int64_t lds, int64_t N, float alpha, float beta,
              bool upper, qlr_qmat& C, WsArena& ws) {
  const int l = (int)T.cols;
  const size_t mark = ws.off;
  char* A = ws.take<char>(a_bytes(T.rows, l));
  char* B = ws.take<char>(b_bytes(N, l));
  if (!ws.ok) { ws.ok = true; ws.off = mark; return QLR_ENOMEM; }
  KTimer kt(ctx, QLR_KID_APPLY);
  TallArgs p;
  memset(&p, 0, sizeof(p));
  run_split(ctx->stream, T.plane, T.ld, T.rows, l, A, p);
  ExpandArgs e{};
  for (int c = 0; c < 4; ++c) e.s[c] = S[c];
  e.lds = lds;
  e.neg = NEG_THIN;
  int rc = run_expand(ctx->stream, e, l, N, B, p);
  if (rc == QLR_OK) {
    p.M = T.rows; p.N = N; p.upper = upper ? 1 : 0;
    for (int c = 0; c < 4; ++c) p.c[c] = static_cast<float*>(C.plane[c]);
    p.ldc = C.ld; p.alpha = alpha; p.beta = beta; p.err = ctx->d_err;
    rc = run_gemm<false>(ctx, p, A, B, l);
  }
  ws.off = mark;
  return rc;
}

// On warm operands 24.4 against 21.8 us at m n k = 1e7 and 27.8 / 35.1 at 3e7; with L2 flushed and 30 % observed
// 37.5 / 54.4 at 1.6e7, 47.8 / 97.4 at 3e7, 131 / 415 at 4096 x 4096, k = 8.  No more rows than the other forms take, so that what is refused does not depend on the form.
bool masked_update_tc_wanted(int64_t m, int64_t n, int k) {
  return k >= 1 && k <= TALL_MAX_L && m <= COMPLETE_MAX_ROWS && n < (1LL << 31) && m * n * k >= (int64_t)15000000 &&
         get_encode() != nullptr;
}
size_t masked_update_tc_ws(int64_t m, int64_t n, int k) {
  return a_bytes(std::min<int64_t>(n, PANEL_COLS), k) + b_bytes(panel_rows(m, k), k) + 1024;
}

int masked_update_tc(qlr_ctx* ctx, const CompleteArgs& a, WsArena& ws) {
  const size_t mark = ws.off;
  const int64_t pr = panel_rows(a.m, a.k), pc = std::min<int64_t>(a.n, PANEL_COLS);
  char* A = ws.take<char>(a_bytes(pc, a.k));
  char* B = ws.take<char>(b_bytes(pr, a.k));
  if (!ws.ok) { ws.ok = true; ws.off = mark; return QLR_ENOMEM; }
  KTimer kt(ctx, QLR_KID_COMPLETE);
  int rc = QLR_OK;
  for (int64_t j0 = 0; j0 < a.n && rc == QLR_OK; j0 += pc) {
    const int64_t nc = std::min(pc, a.n - j0);
    const void* v[4];
    for (int c = 0; c < 4; ++c) v[c] = static_cast<const float*>(a.V[c]) + j0;
    TallArgs tall;
    memset(&tall, 0, sizeof(tall));
    run_split(ctx->stream, v, a.ldv, nc, a.k, A, tall);
    for (int64_t i0 = 0; i0 < a.m && rc == QLR_OK; i0 += pr) {
      const int64_t nr = std::min(pr, a.m - i0);
      ExpandArgs e{};
      for (int c = 0; c < 4; ++c) e.u[c] = static_cast<const float*>(a.U[c]) + i0;
      e.ldu = a.ldu; e.sigma = a.S;
      e.neg = NEG_MASKED;
      TallArgs p = tall;
      rc = run_expand(ctx->stream, e, a.k, nr, B, p);
      if (rc != QLR_OK) break;
      p.M = nc; p.N = nr;
      for (int c = 0; c < 4; ++c) {
        p.c[c] = static_cast<float*>(a.C[c]) + i0 * a.ldc + j0;
        p.m[c] = a.M[c] ? static_cast<const float*>(a.M[c]) + i0 * a.ldm + j0 : nullptr;
      }
      p.ldc = a.ldc; p.ldm = a.ldm; p.mask = a.mask + i0 * a.ldk + j0; p.ldk = a.ldk; p.err = ctx->d_err;
      rc = run_gemm<true>(ctx, p, A, B, a.k);
    }
  }
  ws.off = mark;
  return rc;
}

}  // namespace qlr
