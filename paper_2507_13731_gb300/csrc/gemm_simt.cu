// SIMT (CUDA-core) quaternion GEMM:  C = alpha * op(A) * B + beta * C.
//
// Used for (i) the plain FP32 / FP64 sketch passes Y = A X and Z = A^H Y (the comparator path
// and the FP64 mode), and (ii) thin-times-small products Q = Y R^{-1}, U = Q1 U_hat, V = Q2 V_hat.
// Each output entry is a sum of Hamilton products (Section 2, eq. 1); op(A) = A or conj(A)
// elementwise, with A's (i, k) addressing given by two strides so that A, A^T-views and
// column-major thin matrices all use the same kernels: a register-tiled one for FP32 and one cut
// for the FP64 pipe's rate (gemm_f64_kernel), which also forms the FP64 Gram's partial sums.
#include <algorithm>

#include "qlr_internal.h"

namespace {

constexpr int BM = 64, BN = 32, BK = 16, NT = 256;

template <class TAcc>
__device__ __forceinline__ TAcc load_elem(const void* p, int64_t idx, int dt) {
  if (dt == QLR_F64) return (TAcc)static_cast<const double*>(p)[idx];
  if (dt == QLR_F32) return (TAcc)static_cast<const float*>(p)[idx];
  return (TAcc)__bfloat162float(static_cast<const __nv_bfloat16*>(p)[idx]);
}

// One BM x BN output tile (row tile bx, column tile by) of C.
template <class TAcc, bool I_CONTIG, bool CONJ>
__device__ __forceinline__ void gemm_simt_tile(const qlr::GemmArgs& g, int64_t bx, int64_t by) {
  // one element of padding for 4-byte types (bank conflicts); none for doubles (48 KB static limit)
  constexpr int PAD = sizeof(TAcc) == 4 ? 1 : 0;
  __shared__ TAcc As[4][BK][BM + PAD];
  __shared__ TAcc Bs[4][BK][BN + PAD];
  const int t = threadIdx.x;
  const int tx = t % 16, ty = t / 16;
  const int64_t i0 = bx * BM, j0 = by * BN;

  Quat<TAcc> acc[4][2];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int s = 0; s < 2; ++s) acc[r][s] = {0, 0, 0, 0};

  TAcc ra[4][4], rb[4][2];
  auto load_tile = [&](int64_t k0) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        int ii, kk;
        if (I_CONTIG) { ii = t % BM; kk = t / BM + 4 * r; }
        else { kk = t % BK; ii = t / BK + 16 * r; }
        int64_t gi = i0 + ii, gk = k0 + kk;
        TAcc v = 0;
        if (g.a[c] != nullptr && gi < g.M && gk < g.K) v = load_elem<TAcc>(g.a[c], gi * g.sa_i + gk * g.sa_k, g.a_dtype);
        ra[c][r] = v;
      }
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        int kk = t % BK, jj = t / BK + 16 * r;
        int64_t gk = k0 + kk, gj = j0 + jj;
        TAcc v = 0;
        if (gk < g.K && gj < g.N) v = load_elem<TAcc>(g.b[c], gk + gj * g.ldb, g.b_dtype);
        rb[c][r] = v;
      }
    }
  };
  auto store_tile = [&]() {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        int ii, kk;
        if (I_CONTIG) { ii = t % BM; kk = t / BM + 4 * r; }
        else { kk = t % BK; ii = t / BK + 16 * r; }
        As[c][kk][ii] = ra[c][r];
      }
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        int kk = t % BK, jj = t / BK + 16 * r;
        Bs[c][kk][jj] = rb[c][r];
      }
    }
  };

  // rows of an upper-triangular B below the column tile's last column are zero
  const int64_t kend = g.b_upper ? min(g.K, j0 + BN) : g.K;
  load_tile(0);
  for (int64_t k0 = 0; k0 < kend; k0 += BK) {
    store_tile();
    __syncthreads();
    if (k0 + BK < kend) load_tile(k0 + BK);   // prefetch next tile into registers
#pragma unroll 4
    for (int kk = 0; kk < BK; ++kk) {
      Quat<TAcc> a[4], b[2];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        int ii = tx + 16 * r;
        a[r] = {As[0][kk][ii], As[1][kk][ii], As[2][kk][ii], As[3][kk][ii]};
      }
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        int jj = 2 * ty + s;
        b[s] = {Bs[0][kk][jj], Bs[1][kk][jj], Bs[2][kk][jj], Bs[3][kk][jj]};
      }
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          Quat<TAcc> p = CONJ ? qcmul(a[r], b[s]) : qmul(a[r], b[s]);
          acc[r][s].w += p.w; acc[r][s].x += p.x; acc[r][s].y += p.y; acc[r][s].z += p.z;
        }
    }
    __syncthreads();
  }

  const TAcc alpha = (TAcc)g.alpha, beta = (TAcc)g.beta;
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      int64_t gi = i0 + tx + 16 * r, gj = j0 + 2 * ty + s;
      if (gi >= g.M || gj >= g.N) continue;
      TAcc v[4] = {acc[r][s].w, acc[r][s].x, acc[r][s].y, acc[r][s].z};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        int64_t o = gi + gj * g.ldc;
        TAcc out = alpha * v[c];
        if (g.c_dtype == QLR_F64) {
          double* C = static_cast<double*>(g.c[c]);
          C[o] = (g.beta != 0.0) ? (double)out + g.beta * C[o] : (double)out;
        } else {
          float* C = static_cast<float*>(g.c[c]);
          C[o] = (g.beta != 0.0) ? (float)out + (float)beta * C[o] : (float)out;
        }
      }
    }
}

template <class TAcc, bool I_CONTIG, bool CONJ>
__global__ void __launch_bounds__(NT) gemm_simt_kernel(qlr::GemmArgs g) {
  gemm_simt_tile<TAcc, I_CONTIG, CONJ>(g, blockIdx.x, blockIdx.y);
}

// acc += a b (or conj(a) b) as 16 fused multiply-adds.
template <bool CONJ>
__device__ __forceinline__ void fma_q(Quat<double>& acc, const Quat<double>& a, const Quat<double>& b) {
  const double x = CONJ ? -a.x : a.x, y = CONJ ? -a.y : a.y, z = CONJ ? -a.z : a.z;
  acc.w = fma(-z, b.z, fma(-y, b.y, fma(-x, b.x, fma(a.w, b.w, acc.w))));
  acc.x = fma(-z, b.y, fma(y, b.z, fma(x, b.w, fma(a.w, b.x, acc.x))));
  acc.y = fma(z, b.x, fma(y, b.w, fma(-x, b.z, fma(a.w, b.y, acc.y))));
  acc.z = fma(z, b.w, fma(-y, b.x, fma(x, b.y, fma(a.w, b.z, acc.z))));
}

// FP64 product.  The FP64 pipe does under two multiply-adds per SM and cycle, so what bounds a
// product is how evenly its multiply-adds are spread over the SMs; operand reuse hardly matters
// (one output quaternion per thread reads 8 shared-memory values per 16 multiply-adds).  A CTA
// of 256 threads therefore takes only TM x TN outputs, with 256 / (TM TN) threads per output that
// share the reduction and are summed in a fixed order at the end: at 256 x 192 x 15 the 64 x 32
// tiles of the FP32 kernel put the whole product on 4 SMs (2.1 ms op N, 2.8 ms op H); 8 x 4
// tiles put it on 128.  blockIdx.z takes chunks of `kchunk` reduction steps into separate outputs
// `zstride` elements apart (the Gram's partial sums); `upper` skips tiles below the diagonal.
constexpr int FBK = 32;
template <int TM, int TN, bool I_CONTIG, bool CONJ>
__global__ void __launch_bounds__(NT) gemm_f64_kernel(const qlr::GemmArgs g, int64_t kchunk, int64_t zstride, int upper) {
  constexpr int OUT = TM * TN, KS = NT / OUT;
  constexpr int NA = 4 * FBK * TM / NT, NB = 4 * FBK * TN / NT;
  constexpr int ASZ = 4 * FBK * (TM + 1), BSZ = 4 * FBK * (TN + 1);
  __shared__ double smem[ASZ + BSZ > KS * OUT * 4 ? ASZ + BSZ : KS * OUT * 4];
  double* As = smem;
  double* Bs = smem + ASZ;
  const int64_t i0 = (int64_t)blockIdx.x * TM, j0 = (int64_t)blockIdx.y * TN;
  if (upper && i0 > j0 + TN - 1) return;
  const int t = threadIdx.x, oi = t % TM, oj = (t / TM) % TN, sl = t / OUT;
  const int64_t kbeg = (int64_t)blockIdx.z * kchunk;
  int64_t kend = min(g.K, kbeg + kchunk);
  if (g.b_upper) kend = min(kend, j0 + TN);   // an upper-triangular B is zero below its diagonal
  double ra[NA], rb[NB];
  auto load_tile = [&](int64_t k0) {
#pragma unroll
    for (int r = 0; r < NA; ++r) {
      const int e = t + NT * r, c = e / (FBK * TM), q = e % (FBK * TM);
      const int ii = I_CONTIG ? q % TM : q / FBK, kk = I_CONTIG ? q / TM : q % FBK;
      const int64_t gi = i0 + ii, gk = k0 + kk;
      ra[r] = (g.a[c] != nullptr && gi < g.M && gk < kend)
                  ? load_elem<double>(g.a[c], gi * g.sa_i + gk * g.sa_k, g.a_dtype) : 0.0;
    }
#pragma unroll
    for (int r = 0; r < NB; ++r) {
      const int e = t + NT * r, c = e / (FBK * TN), q = e % (FBK * TN), kk = q % FBK, jj = q / FBK;
      const int64_t gj = j0 + jj, gk = k0 + kk;
      rb[r] = (gj < g.N && gk < kend) ? load_elem<double>(g.b[c], gk + gj * g.ldb, g.b_dtype) : 0.0;
    }
  };
  auto store_tile = [&]() {
#pragma unroll
    for (int r = 0; r < NA; ++r) {
      const int e = t + NT * r, c = e / (FBK * TM), q = e % (FBK * TM);
      const int ii = I_CONTIG ? q % TM : q / FBK, kk = I_CONTIG ? q / TM : q % FBK;
      As[(c * FBK + kk) * (TM + 1) + ii] = ra[r];
    }
#pragma unroll
    for (int r = 0; r < NB; ++r) {
      const int e = t + NT * r, c = e / (FBK * TN), q = e % (FBK * TN), kk = q % FBK, jj = q / FBK;
      Bs[(c * FBK + kk) * (TN + 1) + jj] = rb[r];
    }
  };
  Quat<double> acc = {0, 0, 0, 0};
  if (kbeg < kend) load_tile(kbeg);
  for (int64_t k0 = kbeg; k0 < kend; k0 += FBK) {
    store_tile();
    __syncthreads();
    if (k0 + FBK < kend) load_tile(k0 + FBK);
#pragma unroll
    for (int kk = sl; kk < FBK; kk += KS) {
      const double* ap = As + kk * (TM + 1) + oi;
      const double* bp = Bs + kk * (TN + 1) + oj;
      constexpr int AP = FBK * (TM + 1), BP = FBK * (TN + 1);
      fma_q<CONJ>(acc, {ap[0], ap[AP], ap[2 * AP], ap[3 * AP]}, {bp[0], bp[BP], bp[2 * BP], bp[3 * BP]});
    }
    __syncthreads();
  }
  if (KS > 1) {   // the threads of one output, in slice order
    Quat<double>* red = reinterpret_cast<Quat<double>*>(smem);
    red[t] = acc;
    __syncthreads();
    if (sl != 0) return;
    for (int s = 1; s < KS; ++s) {
      const Quat<double> q = red[t + s * OUT];
      acc.w += q.w; acc.x += q.x; acc.y += q.y; acc.z += q.z;
    }
  }
  const int64_t gi = i0 + oi, gj = j0 + oj;
  if (gi >= g.M || gj >= g.N) return;
  const double v[4] = {acc.w, acc.x, acc.y, acc.z};
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int64_t o = gi + gj * g.ldc + (int64_t)blockIdx.z * zstride;
    const double out = g.alpha * v[c];
    if (g.c_dtype == QLR_F64) {
      double* C = static_cast<double*>(g.c[c]);
      C[o] = (g.beta != 0.0) ? out + g.beta * C[o] : out;
    } else {
      float* C = static_cast<float*>(g.c[c]);
      C[o] = (g.beta != 0.0) ? (float)out + (float)g.beta * C[o] : (float)out;
    }
  }
}

template <int TM, int TN>
void launch_f64(const qlr::GemmArgs& g, int64_t kchunk, int nz, int64_t zstride, int upper, cudaStream_t s) {
  const dim3 grid((unsigned)((g.M + TM - 1) / TM), (unsigned)((g.N + TN - 1) / TN), (unsigned)nz);
  if (g.i_contig) {
    if (g.conj_a) gemm_f64_kernel<TM, TN, true, true><<<grid, NT, 0, s>>>(g, kchunk, zstride, upper);
    else gemm_f64_kernel<TM, TN, true, false><<<grid, NT, 0, s>>>(g, kchunk, zstride, upper);
  } else {
    if (g.conj_a) gemm_f64_kernel<TM, TN, false, true><<<grid, NT, 0, s>>>(g, kchunk, zstride, upper);
    else gemm_f64_kernel<TM, TN, false, false><<<grid, NT, 0, s>>>(g, kchunk, zstride, upper);
  }
  qlr_count_launch();
}

void launch_f32(const qlr::GemmArgs& g, cudaStream_t s) {
  dim3 grid((unsigned)((g.M + BM - 1) / BM), (unsigned)((g.N + BN - 1) / BN));
  if (g.i_contig) {
    if (g.conj_a) gemm_simt_kernel<float, true, true><<<grid, NT, 0, s>>>(g);
    else gemm_simt_kernel<float, true, false><<<grid, NT, 0, s>>>(g);
  } else {
    if (g.conj_a) gemm_simt_kernel<float, false, true><<<grid, NT, 0, s>>>(g);
    else gemm_simt_kernel<float, false, false><<<grid, NT, 0, s>>>(g);
  }
  qlr_count_launch();
}

}  // namespace

namespace qlr {
// Partial sums of G = Y^H Y over `chunks` chunks of `rpc` rows in FP64 (FP32 or FP64 Y): chunk z's
// upper-triangle tiles at part + z 4 l^2 (entries below the tiles that meet the diagonal unset).
int gram_f64_partials(qlr_ctx* ctx, const qlr_qmat& Y, int64_t chunks, int64_t rpc, double* part) {
  GemmArgs g{};
  const int64_t l = Y.cols;
  for (int c = 0; c < 4; ++c) { g.a[c] = Y.plane[c]; g.b[c] = Y.plane[c]; g.c[c] = part + c * l * l; }
  g.sa_i = Y.ld; g.sa_k = 1; g.i_contig = false; g.conj_a = true; g.a_dtype = Y.dtype;
  g.ldb = Y.ld; g.b_dtype = Y.dtype; g.ldc = l; g.c_dtype = QLR_F64;
  g.M = l; g.N = l; g.K = Y.rows; g.alpha = 1.0; g.beta = 0.0; g.acc64 = true;
  // the larger tile halves the shared-memory traffic; it is taken when there are tiles enough
  if (l > 64) launch_f64<16, 8>(g, rpc, (int)chunks, 4 * l * l, 1, ctx->stream);
  else launch_f64<8, 4>(g, rpc, (int)chunks, 4 * l * l, 1, ctx->stream);
  QLR_CUDA_TRY(cudaGetLastError());
  return QLR_OK;
}

int gemm_simt(qlr_ctx* ctx, const GemmArgs& g) {
  if (g.M == 0 || g.N == 0) return QLR_OK;
  if (g.N > 65535LL * BN || g.M > (int64_t)INT32_MAX * BM) return QLR_EUNSUPPORTED;
  KTimer kt(ctx, g.kid);
  if (!g.acc64) {
    launch_f32(g, ctx->stream);
  } else {
    // 16 x 8 tiles once they give every SM two CTAs (half the shared-memory reads), 8 x 4 tiles for
    // anything smaller: 2048 x 2048 x 60 takes 7.1 ms and 20000 x 300 x 110 18 ms, the FP64 pipe's time (22 and 30
    // to 216 ms in the FP32 kernel's tiles), 517 x 389 x 23 0.17 ms (4.4); 8 x 32 tiles where the column tiles would exceed the grid's y limit
    const int64_t big = ((g.M + 15) / 16) * ((g.N + 7) / 8), K = std::max<int64_t>(g.K, 1);
    if (g.N > 65535LL * 8) launch_f64<8, 32>(g, K, 1, 0, 0, ctx->stream);
    else if (big >= 2 * (int64_t)(ctx->num_sms > 0 ? ctx->num_sms : 148)) launch_f64<16, 8>(g, K, 1, 0, 0, ctx->stream);
    else launch_f64<8, 4>(g, K, 1, 0, 0, ctx->stream);
  }
  QLR_CUDA_TRY(cudaGetLastError());
  return QLR_OK;
}
}  // namespace qlr
