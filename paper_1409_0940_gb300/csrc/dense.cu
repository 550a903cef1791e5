// Batched dense linear algebra on the SIMT pipes: the Gram matrices
// I + Z_ij^T Z_ij of eq. (cache), their FP64 Cholesky factorisation, the cached
// inverse Q_ij = (I + Z_ij^T Z_ij)^-1 (the paper's "Q_ij can be cached"), and the
// per-iteration products with Q_ij and H_ij.
#include "common.cuh"
#include "internal.h"
#include "simt.cuh"

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <vector>

namespace rff {

namespace {

// ------------------------------------------------------------------ generic GEMM
// D = alpha * op(A) op(B) + beta * Cm for a batch of row-major matrices.
// Tile 64 x 64, 256 threads, 4 x 4 outputs per thread.  Loads are bounds-checked
// so any M, N, K works.  lower_only skips tiles strictly above the diagonal.
template <typename T, int BK>
__global__ void __launch_bounds__(256) k_gemm(const GemmDesc* __restrict__ descs, int transA, int transB, T alpha,
                                              T beta, int lower_only) {
  const GemmDesc g = descs[blockIdx.z];
  const int tm = blockIdx.x, tn = blockIdx.y;
  if (tm * 64 >= g.M || tn * 64 >= g.N) return;
  if (lower_only && tn > tm) return;
  const T* __restrict__ A = static_cast<const T*>(g.A);
  const T* __restrict__ B = static_cast<const T*>(g.B);
  __shared__ T As[BK][64 + 1];
  __shared__ T Bs[BK][64 + 1];
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  T acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = T(0);
  const int m0 = tm * 64, n0 = tn * 64;
  for (int k0 = 0; k0 < g.K; k0 += BK) {
    for (int t = tid; t < 64 * BK; t += 256) {
      int mm, kk;
      if (transA) { mm = t % 64; kk = t / 64; } else { kk = t % BK; mm = t / BK; }
      const int gm = m0 + mm, gk = k0 + kk;
      T v = T(0);
      if (gm < g.M && gk < g.K) v = transA ? A[(int64_t)gk * g.lda + gm] : A[(int64_t)gm * g.lda + gk];
      As[kk][mm] = v;
      int nn, kb;
      if (transB) { kb = t % BK; nn = t / BK; } else { nn = t % 64; kb = t / 64; }
      const int gn = n0 + nn, gkb = k0 + kb;
      T w = T(0);
      if (gn < g.N && gkb < g.K) w = transB ? B[(int64_t)gn * g.ldb + gkb] : B[(int64_t)gkb * g.ldb + gn];
      Bs[kb][nn] = w;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      T a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[k][ty * 4 + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[k][tx * 4 + j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  const T* __restrict__ Cm = static_cast<const T*>(g.Cm);
  T* __restrict__ D = static_cast<T*>(g.D);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int gm = m0 + ty * 4 + i;
    if (gm >= g.M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int gn = n0 + tx * 4 + j;
      if (gn >= g.N) continue;
      T v = alpha * acc[i][j];
      if (beta != T(0)) v = fma(beta, Cm[(int64_t)gm * g.ldc + gn], v);
      D[(int64_t)gm * g.ldd + gn] = v;
    }
  }
}

// ------------------------------------------------------------------ FP32 NN GEMM
// The per-iteration products with the cached factors, W' += Q r and y = -P e, and the scores of
// sketched rows: D = alpha A B + beta C, A (M x K) row-major with 16-byte aligned rows, B (K x N)
// with N = 16 MQ = ldb columns.  One CTA per 128 rows and all N columns, so A is read once; 8 x MQ
// outputs per thread (rows ty + 16 i, columns tx + 16 q); 32 K elements per stage of a four-stage
// ring of asynchronous copies.
//
// FP32 products are summed 32 at a time, each chunk's sum folded into a float-float accumulator
// (TwoSum): the error of a K-term dot product is that of one 32-term FP32 sum instead of a K-term
// one (K = s_j = 4096 for the cached projection).  For N > 64 the float-float accumulators wait
// in tensor memory.
//
// cl = GEMM_CL: the K chunks of a product are shared by a cluster of GEMM_CL CTAs, whose
// float-float sums are added in order through distributed shared memory.
// Measured against 64 x 64 tiles without a pipeline: four 4096 x 4096 by 160, 1.92 -> 0.71 ms (30
// TFLOP/s); 256 of 625 x 625 by 16, 856 -> 180 us (2.2 TB/s of factors); and, split over clusters,
// 512 x 512 by 16, 68 -> 5.6 us, 2048 x 8192 by 16, 1265 -> 61 us.
constexpr int GEMM_NS = 4, GEMM_CL = 8, GEMM_M = 128, GEMM_K = 32, GEMM_LDK = simt::row_stride(GEMM_K);
constexpr int GEMM_CL_MAX_N = 144;   // the float-float sums of 128 rows fit the ring's memory
__host__ __device__ constexpr int gemm_stage(int n) { return GEMM_M * GEMM_LDK + GEMM_K * n; }   // floats
__host__ __device__ constexpr size_t gemm_smem(int n) { return (size_t)GEMM_NS * gemm_stage(n) * 4; }
static_assert((size_t)2 * GEMM_M * GEMM_CL_MAX_N * 4 <= gemm_smem(GEMM_CL_MAX_N), "");
static_assert(gemm_smem(256) <= 232448 - 256, "the ring fits a CTA's shared memory at N = 256");
// tensor-memory columns of the parked accumulators (16 MQ words a thread, two threads a lane)
__host__ __device__ constexpr uint32_t gemm_tmem_cols(int mq) { return mq <= 8 ? 256u : 512u; }

template <int MQ>
__global__ void __launch_bounds__(256) k_gemm_f32_nn(const GemmDesc* __restrict__ descs,
                                                     const __grid_constant__ GemmDesc one, float alpha, float beta,
                                                     const uint8_t* __restrict__ bmask, int cl) {
  using namespace simt;
  constexpr int N = 16 * MQ, STG = gemm_stage(N);
  constexpr bool PARK = MQ > 4;
  if (bmask && !bmask[blockIdx.y]) return;
  const GemmDesc g = descs ? descs[blockIdx.y] : one;
  const int rank = cl > 1 ? (int)tc5::cluster_rank() : 0;
  const int m0 = (int)(blockIdx.x / cl) * GEMM_M;
  if (m0 >= g.M) return;   // (a cluster's CTAs share m0)
  extern __shared__ __align__(16) float gm_smem[];
  __shared__ uint32_t tmem_word;
  const int tid = threadIdx.x, tx = thread_tx(), ty = thread_ty();
  if (PARK && tid < 32) tc5::tmem_alloc<1>(tc5::smem_u32(&tmem_word), gemm_tmem_cols(MQ));
  const float* __restrict__ A = static_cast<const float*>(g.A);
  const float* __restrict__ B = static_cast<const float*>(g.B);
  const int nch = (g.K + GEMM_K - 1) / GEMM_K;
  const int c0 = (int)((int64_t)rank * nch / cl), c1 = (int)((int64_t)(rank + 1) * nch / cl);
  auto issue = [&](int c) {
    if (c < c1) {
      float* As = gm_smem + ((c - c0) % GEMM_NS) * STG;
      float* Bs = As + GEMM_M * GEMM_LDK;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int e = tid + 256 * q, r = e / 8, k = c * GEMM_K + 4 * (e % 8);
        const int bytes = m0 + r < g.M ? max(0, min(16, 4 * (g.K - k))) : 0;
        cp_async16_fill(As + r * GEMM_LDK + 4 * (e % 8), bytes ? A + (int64_t)(m0 + r) * g.lda + k : A, bytes);
      }
      for (int e = tid; e < GEMM_K * N / 4; e += 256) {
        const int k = c * GEMM_K + e / (N / 4);
        const int bytes = k < g.K ? 16 : 0;
        cp_async16_fill(Bs + 4 * e, bytes ? B + (int64_t)k * N + 4 * (e % (N / 4)) : B, bytes);
      }
    }
    cp_commit();
  };
#pragma unroll
  for (int c = 0; c < GEMM_NS - 1; ++c) issue(c0 + c);
  uint32_t park = 0;
  float hi[PARK ? 1 : MQ][8], lo[PARK ? 1 : MQ][8];
#pragma unroll
  for (int q = 0; q < (PARK ? 1 : MQ); ++q)
#pragma unroll
    for (int i = 0; i < 8; ++i) hi[q][i] = lo[q][i] = 0.f;
  if (PARK) {
    tc5::fence_before();
    __syncthreads();
    tc5::fence_after();
    park = park_base(tmem_word, gemm_tmem_cols(MQ));
    for (int q = 0; q < 2 * MQ; ++q) park8(park + 8 * q, hi[0]);
    tc5::tmem_wait_st();
  }
  for (int c = c0; c < c1; ++c) {
    cp_wait<GEMM_NS - 2>();
    __syncthreads();   // chunk c has landed; everyone is done with chunk c - 1
    issue(c + GEMM_NS - 1);
    const float* ap = gm_smem + ((c - c0) % GEMM_NS) * STG + ty * GEMM_LDK;
    const float* bp = gm_smem + ((c - c0) % GEMM_NS) * STG + GEMM_M * GEMM_LDK + tx;
    float acc[MQ][8];
#pragma unroll
    for (int q = 0; q < MQ; ++q)
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[q][i] = 0.f;
#pragma unroll 2
    for (int k4 = 0; k4 < GEMM_K / 4; ++k4) {
      float a[8][4];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(ap + 16 * i * GEMM_LDK + 4 * k4);
        a[i][0] = v.x; a[i][1] = v.y; a[i][2] = v.z; a[i][3] = v.w;
      }
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
#pragma unroll
        for (int q = 0; q < MQ; ++q) {
          const float b = bp[(4 * k4 + kk) * N + 16 * q];
#pragma unroll
          for (int i = 0; i < 8; ++i) acc[q][i] = fmaf(a[i][kk], b, acc[q][i]);
        }
    }
#pragma unroll
    for (int q = 0; q < MQ; ++q) {
      if (PARK) {
        float h[8], l[8];
        unpark8(park + 8 * q, h);
        unpark8(park + 8 * (MQ + q), l);
#pragma unroll
        for (int i = 0; i < 8; ++i) two_sum_into(h[i], l[i], acc[q][i]);
        park8(park + 8 * q, h);
        park8(park + 8 * (MQ + q), l);
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) two_sum_into(hi[PARK ? 0 : q][i], lo[PARK ? 0 : q][i], acc[q][i]);
      }
    }
    if (PARK) tc5::tmem_wait_st();
  }
  cp_wait<0>();   // (only empty groups are left)
  const float* __restrict__ Cm = static_cast<const float*>(g.Cm);
  float* __restrict__ D = static_cast<float*>(g.D);
  if (cl == 1) {
#pragma unroll
    for (int q = 0; q < MQ; ++q) {
      float h[8], l[8];
      if (PARK) {
        unpark8(park + 8 * q, h);
        unpark8(park + 8 * (MQ + q), l);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int gm = m0 + ty + 16 * i;
        if (gm >= g.M) continue;
        float v = alpha * (PARK ? h[i] + l[i] : hi[PARK ? 0 : q][i] + lo[PARK ? 0 : q][i]);
        if (beta != 0.f) v = fmaf(beta, Cm[(int64_t)gm * g.ldc + tx + 16 * q], v);
        D[(int64_t)gm * g.ldd + tx + 16 * q] = v;
      }
    }
    if (PARK) tmem_return(tmem_word, gemm_tmem_cols(MQ));
  } else {
    __syncthreads();   // everyone is done reading the ring
#pragma unroll
    for (int q = 0; q < MQ; ++q) {
      float h[8], l[8];
      if (PARK) {
        unpark8(park + 8 * q, h);
        unpark8(park + 8 * (MQ + q), l);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        gm_smem[(ty + 16 * i) * N + tx + 16 * q] = PARK ? h[i] : hi[PARK ? 0 : q][i];
        gm_smem[(GEMM_M + ty + 16 * i) * N + tx + 16 * q] = PARK ? l[i] : lo[PARK ? 0 : q][i];
      }
    }
    if (PARK) tmem_return_and_meet(tmem_word, gemm_tmem_cols(MQ));
    else tc5::cluster_sync_all();
    constexpr int SHARE = GEMM_M * N / GEMM_CL;
    const uint32_t base = tc5::smem_u32(gm_smem);
    for (int e = rank * SHARE + tid; e < (rank + 1) * SHARE; e += 256) {
      float h[GEMM_CL], l[GEMM_CL];
#pragma unroll
      for (int r = 0; r < GEMM_CL; ++r) {
        h[r] = ld_cluster(base + 4 * e, r);
        l[r] = ld_cluster(base + 4 * (GEMM_M * N + e), r);
      }
      float th = h[0], tl = l[0];
#pragma unroll
      for (int r = 1; r < GEMM_CL; ++r) {
        two_sum_into(th, tl, h[r]);
        tl = __fadd_rn(tl, l[r]);
      }
      const int gm = m0 + e / N, col = e % N;
      if (gm < g.M) {
        float v = alpha * (th + tl);
        if (beta != 0.f) v = fmaf(beta, Cm[(int64_t)gm * g.ldc + col], v);
        D[(int64_t)gm * g.ldd + col] = v;
      }
    }
    tc5::cluster_sync_all();   // nobody leaves while others read its shared memory
  }
}

// ------------------------------------------------------------------ Gram
// H (s x s, f64, lower tiles) += Z^T Z for Z (n x s) float32.  Products and
// 32-row partial sums in FP32; the partial sums are accumulated in a
// float-float pair (Knuth's TwoSum), so the sum over all n rows carries about
// the error of one 32-term FP32 sum.  (An FP32 accumulator over all rows, or
// over chunks of a few hundred rows, perturbs H enough to move the ADMM fixed
// point by ~kappa(H) * 1e-7.)
// ------------------------------------------------------------------ double-float GEMM
// The FP64 GEMM of the set-up factorisation in double-float arithmetic on the FP32 pipes
// (this part issues FP32 FMAs at 64 times its FP64 rate).  Each FP64 input is held as a
// float pair x = hi + lo (48 significant bits); a product a b is formed exactly as
// p + e by p = a_hi b_hi, e = fma(a_hi, b_hi, -p), plus the cross terms a_hi b_lo and
// a_lo b_hi (a_lo b_lo, 2^-48 relative, is dropped); the accumulator is a float pair
// updated by TwoSum (Knuth), the error terms gathered in its low part.  The result is
// hi + lo in FP64: about 2^-44 relative per K = 64 dot product, enough for a factor whose
// inverse feeds FP32 and three-term BF16 iterations.  Same tiling and interface as k_gemm.
// An operand given as float pairs (PA / PB) is read as such; one given in FP64 is split on
// load (that takes FP64-pipe work, so operands that many CTAs read are split once
// beforehand by k_to_pairs).
constexpr int DF_BK = 16;

__device__ __forceinline__ void load_pair(const void* base, int64_t idx, bool paired, float& h, float& l) {
  if (paired) {
    const float2 v = static_cast<const float2*>(base)[idx];
    h = v.x;
    l = v.y;
  } else {
    const double v = static_cast<const double*>(base)[idx];
    h = __double2float_rn(v);
    l = __double2float_rn(v - (double)h);
  }
}

template <bool PA, bool PB>
__global__ void __launch_bounds__(256) k_gemm_df(const GemmDesc* __restrict__ descs, int transA, int transB,
                                                 double alpha, double beta, int lower_only) {
  const GemmDesc g = descs[blockIdx.z];
  const int tm = blockIdx.x, tn = blockIdx.y;
  if (tm * 64 >= g.M || tn * 64 >= g.N) return;
  if (lower_only && tn > tm) return;
  __shared__ float Ah[DF_BK][64 + 1], Al[DF_BK][64 + 1];
  __shared__ float Bh[DF_BK][64 + 1], Bl[DF_BK][64 + 1];
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  float hi[4][4], lo[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) hi[i][j] = lo[i][j] = 0.f;
  const int m0 = tm * 64, n0 = tn * 64;
  for (int k0 = 0; k0 < g.K; k0 += DF_BK) {
    for (int t = tid; t < 64 * DF_BK; t += 256) {
      int mm, kk;
      if (transA) { mm = t % 64; kk = t / 64; } else { kk = t % DF_BK; mm = t / DF_BK; }
      const int gm = m0 + mm, gk = k0 + kk;
      float vh = 0.f, vl = 0.f;
      if (gm < g.M && gk < g.K)
        load_pair(g.A, transA ? (int64_t)gk * g.lda + gm : (int64_t)gm * g.lda + gk, PA, vh, vl);
      Ah[kk][mm] = vh;
      Al[kk][mm] = vl;
      int nn, kb;
      if (transB) { kb = t % DF_BK; nn = t / DF_BK; } else { nn = t % 64; kb = t / 64; }
      const int gn = n0 + nn, gkb = k0 + kb;
      float wh = 0.f, wl = 0.f;
      if (gn < g.N && gkb < g.K)
        load_pair(g.B, transB ? (int64_t)gn * g.ldb + gkb : (int64_t)gkb * g.ldb + gn, PB, wh, wl);
      Bh[kb][nn] = wh;
      Bl[kb][nn] = wl;
    }
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < DF_BK; ++k) {
      float ah[4], al[4], bh[4], bl[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        ah[i] = Ah[k][ty * 4 + i];
        al[i] = Al[k][ty * 4 + i];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        bh[j] = Bh[k][tx * 4 + j];
        bl[j] = Bl[k][tx * 4 + j];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          // the rounded product and the TwoSum steps must not be contracted into FMAs:
          // the exact-error identities hold only for separately rounded operations
          const float p = __fmul_rn(ah[i], bh[j]);
          float e = fmaf(ah[i], bh[j], -p);
          e = fmaf(ah[i], bl[j], e);
          e = fmaf(al[i], bh[j], e);
          const float s = __fadd_rn(hi[i][j], p);
          const float bb = __fsub_rn(s, hi[i][j]);
          const float err = __fadd_rn(__fsub_rn(hi[i][j], __fsub_rn(s, bb)), __fsub_rn(p, bb));
          lo[i][j] += err + e;
          hi[i][j] = s;
        }
    }
    __syncthreads();
  }
  const double* __restrict__ Cm = static_cast<const double*>(g.Cm);
  double* __restrict__ D = static_cast<double*>(g.D);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int gm = m0 + ty * 4 + i;
    if (gm >= g.M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int gn = n0 + tx * 4 + j;
      if (gn >= g.N) continue;
      double v = alpha * ((double)hi[i][j] + (double)lo[i][j]);
      if (beta != 0.0) v = fma(beta, Cm[(int64_t)gm * g.ldc + gn], v);
      D[(int64_t)gm * g.ldd + gn] = v;
    }
  }
}

// dst (float pairs, ld ldd) = src (FP64, ld lda), M x N per job (desc.A = src, desc.D = dst)
__global__ void k_to_pairs(const GemmDesc* __restrict__ descs) {
  const GemmDesc g = descs[blockIdx.z];
  const int64_t r = (int64_t)blockIdx.x * 8 + threadIdx.y, c = (int64_t)blockIdx.y * 32 + threadIdx.x;
  if (r >= g.M || c >= g.N) return;
  const double v = static_cast<const double*>(g.A)[r * g.lda + c];
  const float h = __double2float_rn(v);
  static_cast<float2*>(g.D)[r * g.ldd + c] = make_float2(h, __double2float_rn(v - (double)h));
}

// Gram accumulation H (FP64) += Z^T Z over the n rows of Z (row-major, ld ldz): one CTA per
// 128 x 128 tile of H on or below the diagonal, 8 x 8 outputs per thread (rows ty*4 + {0..3} and
// 64 + ty*4 + {0..3}, columns the same of tx), 32 rows of both operands per stage of a
// four-stage ring of asynchronous copies.  Bound: the FP32 pipe (64 multiply-adds for four
// 16-byte shared-memory loads).  Products and 64-row partial sums in FP32 (round to nearest,
// unbiased), folded into a float-float accumulator (TwoSum) after every 64 rows, added to H in
// FP64 at the end: about 2^-44 relative per entry.  The 128 words of the float-float accumulator
// wait in tensor memory between folds.  Against 128 x 64 tiles of 8 x 4 outputs with the
// accumulator in registers (238 of them, one CTA of eight warps): the 256 blocks of
// 625 rows x 4096 features of a 32 x 8 grid 86 ms in 512 launches -> 15.3 ms in 16 (34 TFLOP/s).
// cl = GR_CL: the rows are shared by a cluster of GR_CL CTAs, whole runs of 64 each, whose float-float
// sums are added in order through distributed shared memory.  Few tiles leave most SMs idle for as
// long as a CTA takes for all rows: the set-up of 60,000 rows in 2 blocks at D = 300 (6 tiles) 7.3 ->
// 1.7 ms (5.8 with 128 x 64 tiles), at D = 1000 9.2 -> 5.2 (8.5), four blocks of 1024 30.0 -> 14.0 (24.4)
constexpr int GR_T = 128, GR_K = 32, GR_NS = 4, GR_CL = 8;
constexpr size_t GR_SMEM = (size_t)GR_NS * 2 * GR_K * GR_T * 4;
static_assert((size_t)2 * GR_T * GR_T * 4 <= GR_SMEM, "a tile's float-float sums fit the ring's memory");

__global__ void __launch_bounds__(256, 1) k_gram_tile(const float* __restrict__ Zall, int64_t ldz, int64_t n,
                                                      const int64_t* __restrict__ slot,
                                                      const int64_t* __restrict__ size, int64_t s_one,
                                                      double* __restrict__ Hall, int64_t h_stride, int cl) {
  using namespace simt;
  const int rank = cl > 1 ? (int)tc5::cluster_rank() : 0, tile = (int)blockIdx.x / cl;
  // tile (ta, tb), tb <= ta, of the lower triangle
  int ta = (int)((sqrtf(8.f * (float)tile + 1.f) - 1.f) * 0.5f);
  while (ta * (ta + 1) / 2 > tile) --ta;
  while ((ta + 1) * (ta + 2) / 2 <= tile) ++ta;
  const int64_t a0 = (int64_t)ta * GR_T, b0 = ((int64_t)tile - (int64_t)ta * (ta + 1) / 2) * GR_T;
  const int64_t s = size ? size[blockIdx.y] : s_one;
  if (a0 >= s) return;   // past this matrix
  const float* Z = Zall + (slot ? slot[blockIdx.y] - slot[0] : 0);
  double* H = Hall + blockIdx.y * h_stride;
  extern __shared__ __align__(16) float gr_smem[];
  __shared__ uint32_t tmem_word;
  const int tid = threadIdx.x, tx = thread_tx(), ty = thread_ty();
  if (tid < 32) tc5::tmem_alloc<1>(tc5::smem_u32(&tmem_word), 512);
  // stages st0 .. st1 of 32 rows, st0 even (sums are folded after every second one)
  const int64_t runs = ceil_div(n, 2 * GR_K);
  const int64_t st0 = 2 * (rank * runs / cl), st1 = min(ceil_div(n, GR_K), 2 * ((rank + 1) * runs / cl));
  // this thread's four columns of either operand: zeros past the matrix (rows are padded to 16 bytes)
  const int c4 = 4 * (tid % 32);
  const bool a_in = a0 + c4 < s, b_in = b0 + c4 < s;
  const int64_t a_col = a_in ? a0 + c4 : 0, b_col = b_in ? b0 + c4 : 0;
  auto issue = [&](int64_t st) {
    if (st < st1) {
      float* As = gr_smem + (st % GR_NS) * (2 * GR_K * GR_T);
      float* Bs = As + GR_K * GR_T;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = tid / 32 + 8 * q;
        const int64_t gr = st * GR_K + r;
        const float* row = Z + (gr < n ? gr : n - 1) * ldz;   // rows past n: zeros
        cp_async16_fill(As + r * GR_T + c4, row + a_col, gr < n && a_in ? 16 : 0);
        cp_async16_fill(Bs + r * GR_T + c4, row + b_col, gr < n && b_in ? 16 : 0);
      }
    }
    cp_commit();
  };
#pragma unroll
  for (int st = 0; st < GR_NS - 1; ++st) issue(st0 + st);
  tc5::fence_before();
  __syncthreads();
  tc5::fence_after();
  const uint32_t park = park_base(tmem_word, 512);
  float acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
#pragma unroll
  for (int i = 0; i < 16; ++i) park8(park + 8 * i, acc[0]);
  tc5::tmem_wait_st();
  for (int64_t st = st0; st < st1; ++st) {
    cp_wait<GR_NS - 2>();
    __syncthreads();   // stage st has landed; everyone is done with stage st - 1
    issue(st + GR_NS - 1);
    const float* As = gr_smem + (st % GR_NS) * (2 * GR_K * GR_T);
    const float* Bs = As + GR_K * GR_T;
#pragma unroll 4
    for (int k = 0; k < GR_K; ++k) {
      const float4 al = *reinterpret_cast<const float4*>(As + k * GR_T + ty * 4);
      const float4 ah = *reinterpret_cast<const float4*>(As + k * GR_T + 64 + ty * 4);
      const float4 bl = *reinterpret_cast<const float4*>(Bs + k * GR_T + tx * 4);
      const float4 bh = *reinterpret_cast<const float4*>(Bs + k * GR_T + 64 + tx * 4);
      const float a[8] = {al.x, al.y, al.z, al.w, ah.x, ah.y, ah.z, ah.w};
      const float b[8] = {bl.x, bl.y, bl.z, bl.w, bh.x, bh.y, bh.z, bh.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if ((st & 1) || st + 1 == st1) {   // every 64 rows: fold the partial sums into hi + lo
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float hi[8], lo[8];
        unpark8(park + 16 * i, hi);
        unpark8(park + 16 * i + 8, lo);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          two_sum_into(hi[j], lo[j], acc[i][j]);
          acc[i][j] = 0.f;
        }
        park8(park + 16 * i, hi);
        park8(park + 16 * i + 8, lo);
      }
      tc5::tmem_wait_st();
    }
  }
  if (cl == 1) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float hi[8], lo[8];
      unpark8(park + 16 * i, hi);
      unpark8(park + 16 * i + 8, lo);
      const int64_t gm = a0 + (i < 4 ? ty * 4 + i : 64 + ty * 4 + i - 4);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int64_t gn = b0 + (j < 4 ? tx * 4 + j : 64 + tx * 4 + j - 4);
        if (gm < s && gn < s) H[gm * s + gn] += (double)hi[j] + (double)lo[j];
      }
    }
    tmem_return(tmem_word, 512);
  } else {
    cp_wait<0>();      // (only empty groups are left)
    __syncthreads();   // everyone is done reading the ring
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float v[8];
      float* row = gr_smem + (i < 4 ? ty * 4 + i : 64 + ty * 4 + i - 4) * GR_T;
#pragma unroll
      for (int part = 0; part < 2; ++part) {   // the sums, then their low parts
        unpark8(park + 16 * i + 8 * part, v);
        *reinterpret_cast<float4*>(row + part * GR_T * GR_T + tx * 4) = make_float4(v[0], v[1], v[2], v[3]);
        *reinterpret_cast<float4*>(row + part * GR_T * GR_T + 64 + tx * 4) = make_float4(v[4], v[5], v[6], v[7]);
      }
    }
    tmem_return_and_meet(tmem_word, 512);
    constexpr int SHARE = GR_T * GR_T / GR_CL;
    const uint32_t base = tc5::smem_u32(gr_smem);
    for (int e = rank * SHARE + tid; e < (rank + 1) * SHARE; e += 256) {
      float th = ld_cluster(base + 4 * e, 0), tl = ld_cluster(base + 4 * (GR_T * GR_T + e), 0);
#pragma unroll
      for (int r = 1; r < GR_CL; ++r) {
        two_sum_into(th, tl, ld_cluster(base + 4 * e, r));
        tl = __fadd_rn(tl, ld_cluster(base + 4 * (GR_T * GR_T + e), r));
      }
      const int64_t gm = a0 + e / GR_T, gn = b0 + e % GR_T;
      if (gm < s && gn < s) H[gm * s + gn] += (double)th + (double)tl;
    }
    tc5::cluster_sync_all();   // nobody leaves while others read its shared memory
  }
}

// ------------------------------------------------------------------ diagonal potrf
// Blocks whose diagonal lies far from 1 (a subnormal pivot's reciprocal would be infinite, though its
// square root is an ordinary number) are factored as S A S, S = diag(2^sexp) bringing the diagonal into
// [1, 4); L of S A S is S L, and its inverse L^-1 S^-1.  Called, not inlined: they are rare, and the
// kernel's code is fetched anew for every one of its short launches.
__device__ __noinline__ void scale_block(double (*M)[65], int* sexp) {
  const int tid = threadIdx.x;
  if (tid < 64) {
    int e = 1;
    const double d = M[tid][tid];
    if (d > 0.0 && isfinite(d)) frexp(d, &e);   // in [2^(e-1), 2^e)
    sexp[tid] = -((e - 1) >> 1);
  }
  __syncthreads();
  for (int t = tid; t < 64 * 64; t += 256)
    M[t / 64][t % 64] = ldexp(ldexp(M[t / 64][t % 64], sexp[t / 64]), sexp[t % 64]);
  __syncthreads();
}
__device__ __noinline__ void unscale_block(double* A, int64_t ld, double* inv, int bs, const int* sexp) {
  for (int t = threadIdx.x; t < 64 * 64; t += 256) {   // (the elements this thread wrote)
    const int r = t / 64, c = t % 64;
    if (r < bs && c < bs) A[r * ld + c] = ldexp(A[r * ld + c], -sexp[r]);
    inv[t] = ldexp(inv[t], sexp[c]);
  }
}

// One CTA per matrix: factor the bs x bs diagonal block starting at column kcol
// (bs = min(64, s - kcol)) in shared memory, write L back (upper part zeroed) and
// the inverse of L into inv (64 x 64, zero padded).  info = column+1 of the first
// non-positive pivot (the pivot is replaced by 1 so the factorisation finishes).
//
// The factorisation runs as L D L^T with unit lower L: step c needs the reciprocal of pivot d_c
// only, and one multiplication per element of the column, t_r = A_rc / d_c, before the updates
//   A_rq -= t_r A_qc   (c < q <= r)      and, the forward substitution L X = I in place of the
//   X_rq -= t_r X_cq   (r > c, q <= c)   identity, so that the inverse needs no sweep of its own;
// the square roots of all pivots are taken together at the end (L_rc sqrt(d_c), X_rq / sqrt(d_r)).
// X_rq takes the place of A_rq in M once column q has been eliminated, so that step c updates the
// elements (r, q), q <= r, of every row r > c by the same rule, with u_q = A_qc for q > c and X_cq
// for q <= c: a prefix of one table of the lower triangle's elements, last row first, in which
// no lane of a warp idles.  Warp 0 updates the next pivot first and inverts it while the other
// warps run the updates: on this part's 1/64-rate FP64 pipe a square root and a division in front
// of every step's updates, by one thread, took as long as the updates.
// Bound: that pipe (2 multiply-adds per clock and SM: 89k of them, 23 us).  measured 61 us
// per 64 columns, 92 us with square root, division and column scaling in front of every step.
__global__ void __launch_bounds__(256) k_potrf_diag(const DiagJob* __restrict__ jobs, int kcol) {
  __shared__ double M[64][65];
  __shared__ double L[64][65];  // eliminated columns: A_rc at step c
  __shared__ double col[64];    // t of the current step
  __shared__ double u[64];
  __shared__ double piv[64];    // the pivots d_c, then their square roots
  __shared__ double rinv[64];   // 1 / d_c, then 1 / sqrt(d_c)
  __shared__ uint16_t elem[64 * 65 / 2];   // (r << 8) | q, r = 63 first
  __shared__ int bad, sexp[64];   // S = diag(2^sexp)
  const int tid = threadIdx.x;
  for (int t = tid; t < 64 * 64; t += 256) {
    const int r = t / 64, c = t % 64;
    if (c <= r) elem[64 * 65 / 2 - (r + 1) * (r + 2) / 2 + c] = (uint16_t)((r << 8) | c);
  }
  if (tid == 0) bad = 0;
  const DiagJob jb = jobs[blockIdx.x];
  if (kcol >= jb.s) return;
  const int bs = min(64, jb.s - kcol);
  // pivot c: positive, or recorded and replaced by 1
  auto pivot = [&](int c, double d) {
    if (!(d > 0.0)) {
      if (bad == 0) bad = kcol + c + 1;
      d = 1.0;
    }
    piv[c] = d;
    // 1 / d by Newton's iteration from the FP32 reciprocal, shorter than a division: everything
    // waits for it.  The second step's error is 2^-92 before its rounding (0.5000 ulp at most in
    // 20,000 random pivots)
    const float f = (float)d;
    double r;
    if (f > 1e-30f && f < 1e30f) {
      r = (double)(1.f / f);
      r = fma(r, fma(-d, r, 1.0), r);
      r = fma(r, fma(-d, r, 1.0), r);
    } else {
      r = 1.0 / d;
    }
    rinv[c] = r;
  };
  int far = 0;
  for (int t = tid; t < 64 * 64; t += 256) {
    const int r = t / 64, c = t % 64;
    const double v = (r < bs && c < bs) ? jb.A[(int64_t)(kcol + r) * jb.ld + kcol + c] : (r == c ? 1.0 : 0.0);
    M[r][c] = v;
    if (r == c) far |= (unsigned)((__double2hiint(v) >> 20) - (1023 - 96)) > 2u * 96u;   // sign and exponent
  }
  const bool scaled = __syncthreads_or(far) != 0;
  if (scaled) scale_block(M, sexp);
  if (tid == 0) pivot(0, M[0][0]);
  __syncthreads();
  for (int c = 0; c < bs; ++c) {
    if (tid < 64) {
      double v;
      if (tid > c) {
        v = M[tid][c];
        col[tid] = v * rinv[c];
        L[tid][c] = v;
        M[tid][c] = 0.0;   // X_rc starts from the identity's zero
      } else {
        v = tid == c ? 1.0 : M[c][tid];
      }
      u[tid] = tid == c ? 1.0 : v;
    }
    __syncthreads();
    if (tid == 0 && c + 1 < bs) pivot(c + 1, M[c + 1][c + 1] - col[c + 1] * u[c + 1]);
    if (tid >= 32) {
      const int len = 64 * 65 / 2 - (c + 1) * (c + 2) / 2 - 1;   // (the last element is the next pivot)
#pragma unroll 2
      for (int p = tid - 32; p < len; p += 224) {
        const uint32_t v = elem[p];
        const int r = (int)(v >> 8), q = (int)(v & 0xffu);
        M[r][q] -= col[r] * u[q];
      }
    }
    __syncthreads();
  }
  if (tid < bs) {
    const double s = sqrt(piv[tid]);
    piv[tid] = s;
    rinv[tid] = 1.0 / s;
  }
  __syncthreads();
  for (int t = tid; t < 64 * 64; t += 256) {
    const int r = t / 64, c = t % 64;
    const bool in = r < bs && c < bs;
    if (in) jb.A[(int64_t)(kcol + r) * jb.ld + kcol + c] = c < r ? L[r][c] * rinv[c] : c == r ? piv[r] : 0.0;
    jb.inv[t] = in && c <= r ? (c < r ? M[r][c] : 1.0) * rinv[r] : 0.0;
  }
  if (scaled) unscale_block(jb.A + (int64_t)kcol * jb.ld + kcol, jb.ld, jb.inv, bs, sexp);
  if (tid == 0 && bad && jb.info && *jb.info == 0) *jb.info = bad;
}

__global__ void k_zero_strict_upper(double* A, int64_t s) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= s * s) return;
  if (t % s > t / s) A[t] = 0.0;
}

}  // namespace

namespace {
template <int MQ>
cudaError_t launch_gemm_mq(const GemmDesc* descs, const GemmDesc& one, int nbatch, int maxM, int maxK, float alpha,
                           float beta, const uint8_t* bmask, cudaStream_t st) {
  constexpr size_t smem = gemm_smem(16 * MQ);
  cudaError_t e = cudaFuncSetAttribute(k_gemm_f32_nn<MQ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // One CTA per 128 rows, or a cluster sharing its K chunks where that ends sooner: waves times
  // chunks per CTA, four chunks for filling the ring and, in a cluster, the exchange (clusters of
  // eight leave about an eighth of the SMs unused)
  const int64_t ctas = ceil_div(maxM, GEMM_M) * nbatch, nch = ceil_div(maxK, GEMM_K), nsm = device_sms();
  const int64_t whole = ceil_div(ctas, nsm) * (nch + 2);
  const int64_t shared = ceil_div(ctas * GEMM_CL, nsm * 7 / 8) * (ceil_div(nch, GEMM_CL) + 4);
  const int cl = 16 * MQ <= GEMM_CL_MAX_N && shared < whole ? GEMM_CL : 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(ceil_div(maxM, GEMM_M) * cl), (unsigned)nbatch);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cl;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_gemm_f32_nn<MQ>, descs, one, alpha, beta, bmask, cl);
}

cudaError_t launch_gemm(const GemmDesc* descs, const GemmDesc& one, int nbatch, int maxM, int maxK, int N, float alpha,
                        float beta, const uint8_t* bmask, cudaStream_t st) {
  if (nbatch <= 0 || maxM <= 0) return cudaSuccess;
  if (N % 16) return cudaErrorInvalidValue;
  switch (N / 16) {
#define RFF_MQ(q) \
  case q:         \
    return launch_gemm_mq<q>(descs, one, nbatch, maxM, maxK, alpha, beta, bmask, st);
    RFF_MQ(1) RFF_MQ(2) RFF_MQ(3) RFF_MQ(4) RFF_MQ(5) RFF_MQ(6) RFF_MQ(7) RFF_MQ(8)
    RFF_MQ(9) RFF_MQ(10) RFF_MQ(11) RFF_MQ(12) RFF_MQ(13) RFF_MQ(14) RFF_MQ(15) RFF_MQ(16)
#undef RFF_MQ
    default:
      return cudaErrorInvalidValue;
  }
}
}  // namespace

cudaError_t launch_gemm_f32_nn(const GemmDesc* descs_dev, int nbatch, int maxM, int maxK, int N, float alpha,
                               float beta, cudaStream_t st, const uint8_t* bmask) {
  return launch_gemm(descs_dev, GemmDesc{}, nbatch, maxM, maxK, N, alpha, beta, bmask, st);
}

cudaError_t launch_gemm_f32_nn_one(const GemmDesc& g, float alpha, float beta, cudaStream_t st) {
  if (g.lda % 4 || g.ldb != g.N || (reinterpret_cast<uintptr_t>(g.A) | reinterpret_cast<uintptr_t>(g.B)) % 16)
    return cudaErrorInvalidValue;
  return launch_gemm(nullptr, g, 1, g.M, g.K, g.N, alpha, beta, nullptr, st);
}

cudaError_t launch_gemm_f64(const GemmDesc* descs_dev, int nbatch, int maxM, int maxN, int transA, int transB,
                            double alpha, double beta, int lower_only, cudaStream_t st, bool double_float) {
  if (nbatch <= 0 || maxM <= 0 || maxN <= 0) return cudaSuccess;
  dim3 grid((unsigned)ceil_div(maxM, 64), (unsigned)ceil_div(maxN, 64), (unsigned)nbatch);
  if (double_float)
    k_gemm_df<false, false><<<grid, 256, 0, st>>>(descs_dev, transA, transB, alpha, beta, lower_only);
  else
    k_gemm<double, 16><<<grid, 256, 0, st>>>(descs_dev, transA, transB, alpha, beta, lower_only);
  return cudaGetLastError();
}

// double-float GEMM with both operands given as float pairs
cudaError_t launch_gemm_df_pairs(const GemmDesc* descs_dev, int nbatch, int maxM, int maxN, int transA, int transB,
                                 double alpha, double beta, int lower_only, cudaStream_t st) {
  if (nbatch <= 0 || maxM <= 0 || maxN <= 0) return cudaSuccess;
  dim3 grid((unsigned)ceil_div(maxM, 64), (unsigned)ceil_div(maxN, 64), (unsigned)nbatch);
  k_gemm_df<true, true><<<grid, 256, 0, st>>>(descs_dev, transA, transB, alpha, beta, lower_only);
  return cudaGetLastError();
}

cudaError_t launch_to_pairs(const GemmDesc* descs_dev, int nbatch, int maxM, int maxN, cudaStream_t st) {
  if (nbatch <= 0 || maxM <= 0 || maxN <= 0) return cudaSuccess;
  dim3 grid((unsigned)ceil_div(maxM, 8), (unsigned)ceil_div(maxN, 32), (unsigned)nbatch);
  k_to_pairs<<<grid, dim3(32, 8), 0, st>>>(descs_dev);
  return cudaGetLastError();
}

cudaError_t launch_gram_f32_to_f64(const float* Z, int64_t ldz, int64_t n, const int64_t* slot, const int64_t* size,
                                   int64_t s_max, int nb, double* H, int64_t h_stride, cudaStream_t st) {
  if (n <= 0 || s_max <= 0 || nb <= 0) return cudaSuccess;
  const int64_t nt = ceil_div(s_max, GR_T);
  const cudaError_t e = cudaFuncSetAttribute(k_gram_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GR_SMEM);
  if (e != cudaSuccess) return e;
  // One CTA per tile, or a cluster sharing its rows where that ends sooner (waves times stages per CTA, four
  // for filling the ring and, in a cluster, six more for the exchange; clusters of eight leave about an
  // eighth of the SMs unused).  One matrix only: how many are launched together may depend on the
  // memory there is, which must not show in the sums.
  const int64_t tiles = nt * (nt + 1) / 2, nst = ceil_div(n, GR_K), nsm = device_sms();
  const int64_t whole = ceil_div(tiles, nsm) * (nst + 4);
  const int64_t shared = ceil_div(tiles * GR_CL, nsm * 7 / 8) * (ceil_div(nst, GR_CL) + 10);
  const int cl = !size && nb == 1 && shared < whole ? GR_CL : 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(tiles * cl), (unsigned)nb);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = GR_SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cl;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_gram_tile, Z, ldz, n, slot, size, s_max, H, h_stride, cl);
}

cudaError_t launch_zero_strict_upper(double* A, int64_t s, int nbatch, cudaStream_t st) {
  for (int b = 0; b < nbatch; ++b) {
    k_zero_strict_upper<<<(unsigned)ceil_div(s * s, 256), 256, 0, st>>>(A + (size_t)b * s * s, s);
  }
  return cudaGetLastError();
}

cudaError_t launch_potrf_diag(const DiagJob* jobs_dev, int njobs, int kcol, cudaStream_t st) {
  if (njobs <= 0) return cudaSuccess;
  k_potrf_diag<<<njobs, 256, 0, st>>>(jobs_dev, kcol);
  return cudaGetLastError();
}

// Blocked right-looking Cholesky (64-column panels) of every A_b in place, then
// optionally Q_b = A_b^-1 by forward and backward substitution against the
// identity, using the inverted 64 x 64 diagonal factors:
//   potrf step k:  L_kk = chol(A_kk);  A_ik <- A_ik L_kk^-T;  A_il -= A_ik A_lk^T
//   L Y = I:       Y_k = L_kk^-1 B_k;  B_i -= L_ik Y_k   (i > k)
//   L^T Q = Y:     Q_k = L_kk^-T Y_k;  Y_i -= L_ki^T Q_k (i < k)
// Descriptors live in `dev_scratch` (>= factor_scratch_bytes bytes).
// Kernels over the matrices of a batch take up to MAT_BATCH jobs by value (one launch instead of
// one per matrix: 256 blocks of order 625 took 1280 launches of ~3 us for what these do in 24).
constexpr int MAT_BATCH = 64;
struct MatBatch {
  double* A[MAT_BATCH];   // the matrix, or the source
  void* D[MAT_BATCH];     // the second matrix, or the destination
  int64_t ld[MAT_BATCH];
  int s[MAT_BATCH];
};

template <typename Fill, typename Launch>
static cudaError_t over_batches(const std::vector<MatJob>& jobs, Fill&& fill, Launch&& launch) {
  for (size_t b0 = 0; b0 < jobs.size(); b0 += MAT_BATCH) {
    const int nb = (int)std::min<size_t>(MAT_BATCH, jobs.size() - b0);
    MatBatch mb;
    int smax = 0;
    for (int b = 0; b < nb; ++b) {
      fill(mb, b, b0 + b);
      smax = std::max(smax, mb.s[b]);
    }
    if (smax <= 0) continue;
    launch(mb, nb, smax);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// 32 x 32 tiles of the strict lower triangle and the diagonal, through shared memory so that both
// the reads and the writes run along rows
__global__ void __launch_bounds__(256) k_mirror_lower(const __grid_constant__ MatBatch mb) {
  const int s = mb.s[blockIdx.z], r0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
  if (r0 >= s || c0 > r0) return;
  double* Q = mb.A[blockIdx.z];
  const int64_t ld = mb.ld[blockIdx.z];
  __shared__ double t[32][33];
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  for (int y = ty; y < 32; y += 8)
    if (r0 + y < s && c0 + tx < s) t[y][tx] = Q[(int64_t)(r0 + y) * ld + c0 + tx];
  __syncthreads();
  for (int y = ty; y < 32; y += 8)   // element (c0 + y, r0 + tx) from (r0 + tx, c0 + y)
    if (c0 + y < s && r0 + tx < s && r0 + tx > c0 + y) Q[(int64_t)(c0 + y) * ld + r0 + tx] = t[tx][y];
}

cudaError_t launch_mirror_lower(const std::vector<MatJob>& jobs, cudaStream_t st) {
  return over_batches(
      jobs,
      [&](MatBatch& mb, int b, size_t k) {
        mb.A[b] = jobs[k].Q;
        mb.D[b] = nullptr;
        mb.ld[b] = jobs[k].ldq;
        mb.s[b] = jobs[k].Q ? jobs[k].s : 0;
      },
      [&](const MatBatch& mb, int nb, int smax) {
        const unsigned g = (unsigned)ceil_div(smax, 32);
        k_mirror_lower<<<dim3(g, g, (unsigned)nb), 256, 0, st>>>(mb);
      });
}

__global__ void k_factor_init(const __grid_constant__ MatBatch mb) {
  const int64_t s = mb.s[blockIdx.y], t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= s * s) return;
  const int64_t r = t / s, c = t % s;
  static_cast<double*>(mb.D[blockIdx.y])[t] = r == c ? 1.0 : 0.0;
  if (r == c) mb.A[blockIdx.y][r * mb.ld[blockIdx.y] + r] += 1.0;
}

cudaError_t launch_factor_init(const std::vector<MatJob>& jobs, cudaStream_t st) {
  return over_batches(
      jobs,
      [&](MatBatch& mb, int b, size_t k) {
        mb.A[b] = jobs[k].A;
        mb.D[b] = jobs[k].Q;   // ldq = s
        mb.ld[b] = jobs[k].ld;
        mb.s[b] = jobs[k].s;
      },
      [&](const MatBatch& mb, int nb, int smax) {
        k_factor_init<<<dim3((unsigned)ceil_div((int64_t)smax * smax, 256), (unsigned)nb), 256, 0, st>>>(mb);
      });
}

__global__ void k_convert_factors(const __grid_constant__ MatBatch mb) {
  const int64_t s = mb.s[blockIdx.y], t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t < s * s) static_cast<float*>(mb.D[blockIdx.y])[t / s * round_up(s, 4) + t % s] = (float)mb.A[blockIdx.y][t];
}

cudaError_t launch_convert_factors(const std::vector<MatJob>& jobs, float* const* dst, cudaStream_t st) {
  return over_batches(
      jobs,
      [&](MatBatch& mb, int b, size_t k) {
        mb.A[b] = jobs[k].Q;
        mb.D[b] = dst[k];
        mb.ld[b] = jobs[k].ldq;
        mb.s[b] = jobs[k].s;
      },
      [&](const MatBatch& mb, int nb, int smax) {
        k_convert_factors<<<dim3((unsigned)ceil_div((int64_t)smax * smax, 256), (unsigned)nb), 256, 0, st>>>(mb);
      });
}

// descriptor phases of the blocked factorisation: 0 panel, 1 trailing update, 2-3 forward
// sweep, 4-5 backward sweep, 6-9 conversions to float pairs (double-float mode)
constexpr int FACTOR_PHASES = 10;

// RFF_FACTOR=df selects the double-float block updates below instead of the tensor-core ones
// of ozaki.cu (read once)
static bool use_double_float_updates() {
  static const bool df = [] {
    const char* e = getenv("RFF_FACTOR");
    return e && strcmp(e, "df") == 0;
  }();
  return df;
}

size_t factor_scratch_bytes(int njobs, int smax) {
  const int nb = (int)ceil_div(smax, 64);
  // per job: the diagonal inverses, and two 64 x (nb * 64) float-pair staging buffers
  const size_t df = (size_t)njobs * nb * 64 * 64 * sizeof(double) +
                    (size_t)njobs * 2 * 64 * nb * 64 * sizeof(float2) + (size_t)njobs * sizeof(DiagJob) * nb +
                    (size_t)njobs * nb * FACTOR_PHASES * sizeof(GemmDesc) + 1024;
  return std::max(df, oz_factor_scratch_bytes(njobs, smax));
}

cudaError_t factor_and_invert_f64(const std::vector<MatJob>& jobs, bool invert, void* dev_scratch, cudaStream_t st,
                                  bool double_float, int oz_bits, bool overlap) {
  const int nj = (int)jobs.size();
  if (nj == 0) return cudaSuccess;
  if (!use_double_float_updates()) return factor_and_invert_oz(jobs, invert, dev_scratch, st, oz_bits, overlap);
  int smax = 0;
  for (const auto& j : jobs) smax = std::max(smax, j.s);
  const int nb = (int)ceil_div(smax, 64);
  char* p = static_cast<char*>(dev_scratch);
  double* inv = reinterpret_cast<double*>(p);
  p += (size_t)nj * nb * 64 * 64 * sizeof(double);
  // float-pair copies of the operands that many CTAs of one double-float GEMM read: P2 holds
  // the L panel below the diagonal block (rest x 64, ld 64) or the L block row (64 x c0,
  // ld ldp); B2 the block row of Q (64 x ncol, ld ldp)
  const int64_t ldp = (int64_t)nb * 64;
  float2* pairs = reinterpret_cast<float2*>(p);
  p += (size_t)nj * 2 * 64 * ldp * sizeof(float2);
  DiagJob* djobs = reinterpret_cast<DiagJob*>(p);
  p += (size_t)nj * nb * sizeof(DiagJob);
  GemmDesc* gd = reinterpret_cast<GemmDesc*>(p);

  std::vector<DiagJob> hd((size_t)nj * nb);
  for (int k = 0; k < nb; ++k)
    for (int b = 0; b < nj; ++b)
      hd[(size_t)k * nj + b] = DiagJob{jobs[b].A, jobs[b].ld, jobs[b].s, inv + ((size_t)b * nb + k) * 4096,
                                       jobs[b].info};
  cudaError_t e = cudaMemcpyAsync(djobs, hd.data(), hd.size() * sizeof(DiagJob), cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return e;

  // descriptor table: [phase][k][b]
  std::vector<GemmDesc> g((size_t)FACTOR_PHASES * nb * nj);
  auto at = [&](int ph, int k, int b) -> GemmDesc& { return g[((size_t)ph * nb + k) * nj + b]; };
  for (int k = 0; k < nb; ++k)
    for (int b = 0; b < nj; ++b) {
      const MatJob& J = jobs[b];
      const int64_t c0 = (int64_t)k * 64;
      const int bs = (int)std::max<int64_t>(0, std::min<int64_t>(64, J.s - c0));
      const int rest = (int)std::max<int64_t>(0, J.s - c0 - 64);
      double* Ikk = inv + ((size_t)b * nb + k) * 4096;
      float2* P2 = pairs + (size_t)b * 2 * 64 * ldp;
      float2* B2 = P2 + 64 * ldp;
      double* Lp = J.A + (c0 + 64) * J.ld + c0;   // L panel below the diagonal block
      GemmDesc z{};
      // panel: A_ik <- A_ik * inv^T (in place)
      GemmDesc pn = z;
      if (bs > 0 && rest > 0) pn = GemmDesc{J.A + (c0 + 64) * J.ld + c0, Ikk, nullptr, J.A + (c0 + 64) * J.ld + c0,
                                            rest, bs, bs, J.ld, 64, 0, J.ld};
      at(0, k, b) = pn;
      GemmDesc tr = z, cp = z;
      if (bs > 0 && rest > 0) {
        if (double_float) {
          cp = GemmDesc{Lp, nullptr, nullptr, P2, rest, bs, 0, J.ld, 0, 0, 64};
          tr = GemmDesc{P2, P2, Lp + 64, Lp + 64, rest, rest, bs, 64, 64, J.ld, J.ld};
        } else {
          tr = GemmDesc{Lp, Lp, Lp + 64, Lp + 64, rest, rest, bs, J.ld, J.ld, J.ld, J.ld};
        }
      }
      at(1, k, b) = tr;
      at(6, k, b) = cp;
      // Inverse Q = L^-T L^-1 from Q = I: the forward sweep (L Y = I) touches only the
      // columns up to the diagonal block of block row k (Y is lower triangular); the
      // backward sweep (L^T Q = Y) computes the block lower triangle of the symmetric Q,
      // which needs the same columns; the strict upper triangle is mirrored afterwards.
      // s^3/3 flops per sweep instead of s^3.
      GemmDesc fa = z, fb = z, ba = z, bb = z, cq = z, cl = z, cqb = z;
      const int ncol = (int)(c0 + bs);
      double* Qk = J.Q + c0 * J.ldq;   // block row k of Q
      if (invert && bs > 0) {
        fa = GemmDesc{Ikk, Qk, nullptr, Qk, bs, ncol, bs, 64, J.ldq, 0, J.ldq};
        ba = fa;
        if (double_float) {
          // the forward update reads the panel pairs of phase 6 and Q_k converted after fa
          cq = GemmDesc{Qk, nullptr, nullptr, B2, bs, ncol, 0, J.ldq, 0, 0, ldp};
          if (rest > 0) fb = GemmDesc{P2, B2, Qk + 64 * J.ldq, Qk + 64 * J.ldq, rest, ncol, bs, 64, ldp, J.ldq,
                                      J.ldq};
          if (c0 > 0) {
            cl = GemmDesc{J.A + c0 * J.ld, nullptr, nullptr, P2, bs, (int)c0, 0, J.ld, 0, 0, ldp};
            cqb = GemmDesc{Qk, nullptr, nullptr, B2, bs, (int)c0, 0, J.ldq, 0, 0, ldp};
            bb = GemmDesc{P2, B2, J.Q, J.Q, (int)c0, (int)c0, bs, ldp, ldp, J.ldq, J.ldq};
          }
        } else {
          if (rest > 0) fb = GemmDesc{Lp, Qk, Qk + 64 * J.ldq, Qk + 64 * J.ldq, rest, ncol, bs, J.ld, J.ldq, J.ldq,
                                      J.ldq};
          if (c0 > 0) bb = GemmDesc{J.A + c0 * J.ld, Qk, J.Q, J.Q, (int)c0, (int)c0, bs, J.ld, J.ldq, J.ldq, J.ldq};
        }
      }
      at(2, k, b) = fa;
      at(3, k, b) = fb;
      at(4, k, b) = ba;
      at(5, k, b) = bb;
      at(7, k, b) = cq;
      at(8, k, b) = cl;
      at(9, k, b) = cqb;
    }
  e = cudaMemcpyAsync(gd, g.data(), g.size() * sizeof(GemmDesc), cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return e;
  auto dev = [&](int ph, int k) { return gd + ((size_t)ph * nb + k) * nj; };

  // the GEMMs that many CTAs feed from one panel or block row (trailing update, forward and
  // backward updates) read float pairs converted once per step in double-float mode; the
  // 64-row products (panel solve, diagonal-block products) split their FP64 operands on load
  const bool df = double_float;
  auto upd = [&](int ph, int k, int M, int N, int tA, int tB, int lower) {
    return df ? launch_gemm_df_pairs(dev(ph, k), nj, M, N, tA, tB, -1.0, 1.0, lower, st)
              : launch_gemm_f64(dev(ph, k), nj, M, N, tA, tB, -1.0, 1.0, lower, st);
  };
  for (int k = 0; k < nb; ++k) {
    const int c0 = k * 64, rest = std::max(0, smax - c0 - 64);
    if ((e = launch_potrf_diag(djobs + (size_t)k * nj, nj, c0, st)) != cudaSuccess) return e;
    if (rest > 0) {
      if ((e = launch_gemm_f64(dev(0, k), nj, rest, 64, 0, 1, 1.0, 0.0, 0, st, df)) != cudaSuccess) return e;
      if (df && (e = launch_to_pairs(dev(6, k), nj, rest, 64, st)) != cudaSuccess) return e;
      if ((e = upd(1, k, rest, rest, 0, 1, 1)) != cudaSuccess) return e;
    }
  }
  if (!invert) return cudaSuccess;
  for (int k = 0; k < nb; ++k) {
    const int c0 = k * 64, rest = std::max(0, smax - c0 - 64), ncol = std::min(smax, c0 + 64);
    if ((e = launch_gemm_f64(dev(2, k), nj, 64, ncol, 0, 0, 1.0, 0.0, 0, st, df)) != cudaSuccess) return e;
    if (rest > 0) {
      if (df && ((e = launch_to_pairs(dev(6, k), nj, rest, 64, st)) != cudaSuccess ||
                 (e = launch_to_pairs(dev(7, k), nj, 64, ncol, st)) != cudaSuccess))
        return e;
      if ((e = upd(3, k, rest, ncol, 0, 0, 0)) != cudaSuccess) return e;
    }
  }
  for (int k = nb - 1; k >= 0; --k) {
    const int c0 = k * 64, ncol = std::min(smax, c0 + 64);
    if ((e = launch_gemm_f64(dev(4, k), nj, 64, ncol, 1, 0, 1.0, 0.0, 0, st, df)) != cudaSuccess) return e;
    if (c0 > 0) {
      if (df && ((e = launch_to_pairs(dev(8, k), nj, 64, c0, st)) != cudaSuccess ||
                 (e = launch_to_pairs(dev(9, k), nj, 64, c0, st)) != cudaSuccess))
        return e;
      if ((e = upd(5, k, c0, c0, 1, 0, 0)) != cudaSuccess) return e;
    }
  }
  return launch_mirror_lower(jobs, st);
}

}  // namespace rff
