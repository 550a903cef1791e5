// Split-BF16 streaming GEMM on tensor cores, driven by a job table.
//
// Every job multiplies one 128-row tile of operand A (rows a_row.., K from a_k0)
// by the m_pad-row operand B (rows b_row.., K from b_k0) over nk chunks of 32:
//
//   acc (TMEM, 128 x m_pad fp32) = sum over the split products A_s . B_t^T
//
// with A = A1 + A2 (+ A3) and B = B1 + B2 (+ B3) split into 16-bit terms.  Three
// BF16 terms each (NA = NB = 3) take the six products whose exponents sum to at
// most 2^-16 (11, 12, 21, 13, 22, 31): the accuracy of an FP32 product.  Two
// terms each (scaled FP16 hi/lo, 22 significant bits) take 11, 12, 21.  The
// accumulator times out_scale (and the inverse FP16 scale of B, from the device
// maximum b_amax) is written row-major to out + job.out (ld m_pad); amax, when
// given, collects max |result| for the FP16 split of the result that follows.
//
// Users: the cached projection of eq. (gpWij) (A = Q_ij split three ways, B = the
// right-hand side), and the two chained products of the cached-Z precision
// (pass 1: A = Z^T, B = V^T; pass 2: A = Z, B = W'^T; eq. (gpWij), (gpOij)).
//
// A TMA ring of 32-element K chunks (64-byte swizzle), or 64-element ones (128-byte
// swizzle), feeds the tiles of each chunk.  Warp 0 issues the copies, one thread of warp 1
// the MMAs, warps 2..9 write the result.  Waits are bounded as in the regeneration kernel: on a timeout
// the CTA records an error code, waits (bounded) for its copies and products in
// flight, frees TMEM and returns.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "common.cuh"
#include "tc.h"
#include "tcgen05.cuh"

namespace rff {

namespace {

using namespace tc5;

constexpr int QKC = 32;                      // K elements of a job's chunk count (SgJob::nk)
constexpr int QMAXS = 8;
constexpr int QEPI = 8;                      // writing warps: two per TMEM lane quarter, half the columns each
constexpr int QNT = 64 + 32 * QEPI;
constexpr int ERR_Q = 8;

struct QArgs {
  CUtensorMap tA[3], tB[3];
  int mpad, ns;
  uint32_t stage_bytes, tmem_cols;
  uint32_t acc_b;            // column of the second accumulator (the small products), 0 = one accumulator
  uint32_t nbuf;             // accumulator sets in TMEM (2: the next job's products overlap the epilogue)
  uint32_t buf_cols;         // TMEM columns of one set
  int njobs;
  const SgJob* jobs;
  float* out;
  int64_t out_elems;
  float out_scale;
  const unsigned* b_amax;
  unsigned* amax;
  const uint8_t* bmask;      // active blocks of a stochastic iteration, or null
  int accumulate;            // 1: out += result (amax of the sum)
  int cl;                    // CTAs (a cluster) that share a job's K stages
  const __nv_bfloat16 *c_a, *c_b;   // leading terms of A and B where the chains are centred, or null
  int64_t c_lda, c_ldb;
  int* err;
  long long timeout_cycles;
};

struct QShared {
  uint64_t full[QMAXS], empty[QMAXS];
  uint64_t acc_full[2], acc_empty[2], mma_done;
  uint32_t tmem;
  int abort_flag;
};

__device__ __forceinline__ bool qwait(uint32_t bar, uint32_t parity, QShared& sh, const QArgs& a) {
  if (mbar_try(bar, parity)) return true;
  const long long t0 = clock64();
  while (true) {
    if (mbar_try(bar, parity)) return true;
    if (*(volatile int*)&sh.abort_flag) return false;
    if (clock64() - t0 > a.timeout_cycles) {
      *(volatile int*)&sh.abort_flag = 1;
      atomicOr(a.err, ERR_Q);
      return false;
    }
  }
}

__device__ __forceinline__ float4 ld_cluster4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}

// Where a chain of accumulations starts.  The tensor cores' accumulator rounds toward zero, a bias in
// proportion to the running sum.  A factor's product Q r is mostly cancellation (Q = (I + Z^T Z)^-1 takes
// r's part along Z's large singular vectors down by their squares): row k's sum runs from 0 down to some
// -Q_kk r_k times k's place, jumps by Q_kk r_k at k and falls back to about 0, and over the rows, whose
// jumps lie anywhere, the bias cancels.  Cut into chains that start at 0, the one with the jump stays at
// Q_kk r_k and the others run from 0 to a fraction of -Q_kk r_k: these biases differ by a tenth, a share of
// r that Q should have taken out and that Z brings back enlarged.  So each chain starts at minus half of
// what it will add (its share of -Q_kk r_k, and Q_kk r_k where it holds the jump), and over the rows
// it lies on one side of 0 as much as on the other; what it started from is subtracted at the end.
// Scores after two iterations (TensorSketch, degree 3, n = 2002, D = 4096, l1 loss, largest eigenvalue
// 6e4), error against float64: one chain 2.6e-4, eight from 0 9.7e-4, eight from here 3.2e-4; where
// little cancels the error is that of the short chains (binary fit of 20k rows 4.5e-6, 3.8e-6, 3.8e-6).
struct ChainStart {   // of the 32 output rows of a writing warp, a row per lane
  const __nv_bfloat16* r;   // B's leading term at the first row's own feature, column 0
  int64_t ldr;
  float w;                  // A's leading term at this lane's own feature, times the weight
  __device__ __forceinline__ ChainStart() : r(nullptr), ldr(0), w(0.f) {}
  // row0: the warp's first row; the chain takes K elements k0 .. k1 of k_all
  __device__ __forceinline__ ChainStart(const SgJob& job, const QArgs& a, int row0, int k0, int k1, int k_all)
      : ldr(a.c_ldb), w(0.f) {
    // the A column, and K element, of a row's own feature: out's row, counted from the job's first feature
    // (m_pad is a multiple of 16, and a 16th of out's elements a 32-bit number)
    const uint32_t out_row = (uint32_t)(job.out >> 4) / (uint32_t)(a.mpad >> 4);
    const int first = (int)(out_row - (uint32_t)(job.b_row / a.mpad) * (uint32_t)a.c_ldb - (uint32_t)job.b_k0) + row0;
    const int row = row0 + (int)(threadIdx.x & 31), k = first + (int)(threadIdx.x & 31);
    r = a.c_b + job.b_row * a.c_ldb + job.b_k0 + first;
    if (k < a.c_lda)   // (past it a padding row)
      w = __bfloat162float(a.c_a[(job.a_row + row) * a.c_lda + job.a_k0 + k]) *
          (0.5f * (float)(k1 - k0) / (float)k_all - (k >= k0 && k < k1 ? 0.5f : 0.f));
  }
  // columns c .. c + 31, those below c_end (a multiple of 8): 8 columns of 32 rows at a time as one
  // 16-byte load per lane, all in flight together, turned through the warp's 512 bytes of buf (a
  // 2-byte load per row and column took 14 us of a product of 128 columns, these 4)
  __device__ __forceinline__ void load(int c, int c_end, uint4* buf, float (&o)[32]) const {
    const int lane = threadIdx.x & 31;
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      v[u] = c + 8 * u < c_end ? *reinterpret_cast<const uint4*>(r + (c + 8 * u + lane / 4) * ldr + 8 * (lane % 4))
                               : make_uint4(0, 0, 0, 0);
    const __nv_bfloat16* mine = reinterpret_cast<const __nv_bfloat16*>(buf) + lane;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      __syncwarp();
      buf[lane] = v[u];
      __syncwarp();
#pragma unroll
      for (int t = 0; t < 8; ++t) o[8 * u + t] = w * __bfloat162float(mine[32 * t]);
    }
  }
};

// split-product order (A term, B term): exponents summing to at most 2^-16
__host__ __device__ constexpr int prod_a(int p) { return p == 2 || p == 4 ? 1 : p == 5 ? 2 : 0; }
__host__ __device__ constexpr int prod_b(int p) { return p == 1 || p == 4 ? 1 : p == 3 ? 2 : 0; }

// A job is skipped by every role alike when it has no K chunks or its block is inactive.
__device__ __forceinline__ bool q_skip(const SgJob& j, const QArgs& a) {
  return j.nk <= 0 || (a.bmask && !a.bmask[j.blk]);
}

// Each CTA takes the jobs blockIdx.x, blockIdx.x + gridDim.x, ... (one job per CTA when the
// grid covers the table).  The copies run ahead through the ring across jobs; a job's products
// go to accumulator set (its count) mod nbuf, which the writing warps free after reading it.
// KC: K elements per ring stage, 32 (64-byte rows, 64-byte swizzle) or 64 (128-byte rows and
// swizzle: fewer shared-memory wavefronts per product, half as many stages); a job's nk counts
// chunks of 32, so with KC = 64 an odd count reads 32 more K columns, which the caller keeps
// zero in A (or beyond the tensor, where the copy fills zeros).
//
// cl > 1: a cluster of cl CTAs takes one job, each a run of its K stages; the partial results meet
// in distributed shared memory and are added in rank order, each CTA finishing 128 / cl rows.
template <int NA, int NB, int F16, int KC>
__global__ void __launch_bounds__(QNT) k_split_gemm(const __grid_constant__ QArgs a) {
  constexpr int NPROD = (NA == 3 && NB == 3) ? 6 : 3;
  constexpr uint32_t ATILE = 128 * KC * 2;                  // one 128-row A term
  constexpr uint32_t SBO = 8 * KC * 2, LAYOUT = KC == 64 ? 2 : 4;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  QShared& sh = *reinterpret_cast<QShared*>(base + a.ns * a.stage_bytes);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const uint32_t bar_full = smem_u32(&sh.full[0]), bar_empty = smem_u32(&sh.empty[0]);
  const uint32_t bar_accf = smem_u32(&sh.acc_full[0]), bar_acce = smem_u32(&sh.acc_empty[0]);
  const uint32_t bar_done = smem_u32(&sh.mma_done);
  const uint32_t mb = (uint32_t)a.mpad * (KC * 2);   // one B term: m_pad rows
  const int rank = a.cl > 1 ? (int)cluster_rank() : 0;
  const int job0 = blockIdx.x / a.cl, job_step = gridDim.x / a.cl;
  // this CTA's stages of KC elements of a job of nk chunks
  auto stages_of = [&](int nk, int& s0, int& s1) {
    const int n = (nk * QKC + KC - 1) / KC;
    s0 = rank * n / a.cl;
    s1 = (rank + 1) * n / a.cl;
  };
  if (threadIdx.x == 0) {
    sh.abort_flag = 0;
    for (int i = 0; i < a.ns; ++i) {
      mbar_init(bar_full + 8 * i, 1);
      mbar_init(bar_empty + 8 * i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar_accf + 8 * i, 1);
      mbar_init(bar_acce + 8 * i, QEPI);   // one arrival per writing warp
    }
    mbar_init(bar_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem)),
                 "r"(a.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = sh.tmem;

  if (warp == 0) {
    if (lane == 0) {
      uint32_t issued = 0;   // ring stages filled, over all of this CTA's jobs
      bool ok = true;
      for (int jx = job0; ok && jx < a.njobs; jx += job_step) {
        const SgJob job = a.jobs[jx];
        if (q_skip(job, a)) continue;
        int s0, s1;
        stages_of(job.nk, s0, s1);
        for (int kc = s0; kc < s1; ++kc) {
          const int st = issued % a.ns;
          const uint32_t use = issued / a.ns;
          if (use > 0 && !qwait(bar_empty + 8 * st, (use - 1) & 1, sh, a)) {
            ok = false;
            break;
          }
          const uint32_t fb = bar_full + 8 * st;
          mbar_expect_tx(fb, a.stage_bytes);
          const uint32_t dst = smem_u32(base + st * a.stage_bytes);
#pragma unroll
          for (int s = 0; s < NA; ++s) tma_load_2d(dst + s * ATILE, &a.tA[s], job.a_k0 + kc * KC, job.a_row, fb);
#pragma unroll
          for (int s = 0; s < NB; ++s)
            tma_load_2d(dst + NA * ATILE + s * mb, &a.tB[s], job.b_k0 + kc * KC, job.b_row, fb);
          ++issued;
        }
      }
      // copies in flight finish before the CTA may exit (bounded)
      for (uint32_t u = issued > (uint32_t)a.ns ? issued - a.ns : 0; u < issued; ++u) {
        const int st = u % a.ns;
        const long long t0 = clock64();
        while (!mbar_try(bar_full + 8 * st, (u / a.ns) & 1) && clock64() - t0 < a.timeout_cycles) {
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = F16 ? idesc_f16(128, a.mpad) : idesc_bf16(128, a.mpad);
      bool ok = true;
      uint32_t used = 0, done_jobs = 0;   // ring stages consumed, jobs multiplied
      for (int jx = job0; ok && jx < a.njobs; jx += job_step) {
        const SgJob job = a.jobs[jx];
        if (q_skip(job, a)) continue;
        const uint32_t buf = done_jobs % a.nbuf, round = done_jobs / a.nbuf;
        if (round > 0 && !qwait(bar_acce + 8 * buf, (round - 1) & 1, sh, a)) {
          ok = false;
          break;
        }
        // (one accumulator set: the second's barrier says that the chains' starts are in place)
        if (NA == 3 && a.c_a && !qwait(bar_acce + 8, 0, sh, a)) {
          ok = false;
          break;
        }
        fence_after();
        const uint32_t acc = tmem + buf * a.buf_cols;
        int s0, s1;
        stages_of(job.nk, s0, s1);
        for (int kc = s0; kc < s1; ++kc, ++used) {
          const int st = used % a.ns;
          if (!qwait(bar_full + 8 * st, (used / a.ns) & 1, sh, a)) {
            ok = false;
            break;
          }
          fence_after();
          const uint32_t sa = smem_u32(base + st * a.stage_bytes);
          const uint32_t sb = sa + NA * ATILE;
#pragma unroll
          for (int kk = 0; kk < KC / 16; ++kk) {
#pragma unroll
            for (int p = 0; p < NPROD; ++p) {
              const uint64_t da = smem_desc(sa + prod_a(p) * ATILE + kk * 32, SBO, LAYOUT);
              const uint64_t db = smem_desc(sb + prod_b(p) * mb + kk * 32, SBO, LAYOUT);
              if (a.acc_b) {
                // hi.hi alone in the first accumulator, the smaller products in the second
                const uint32_t d = p == 0 ? acc : acc + a.acc_b;
                mma_bf16(d, da, db, idesc, (kc > s0 || kk > 0 || p > 1 || (NA == 3 && p == 0 && a.c_a)) ? 1u : 0u);
              } else {
                mma_bf16(acc, da, db, idesc, (kc > s0 || kk > 0 || p > 0) ? 1u : 0u);
              }
            }
          }
          mma_commit(bar_empty + 8 * st);
        }
        if (!ok) break;
        mma_commit(bar_accf + 8 * buf);
        ++done_jobs;
      }
      mma_commit(bar_done);
      qwait(bar_done, 0, sh, a);
    }
  } else {
    // epilogue: lanes = rows of the A tile; warps 2..5 take the first m_pad/2 columns, warps
    // 6..9 the rest, 8 per TMEM read
    const int quarter = warp & 3;
    const int c_begin = ((warp - 2) >> 2) * (a.mpad / 2), c_end = c_begin + a.mpad / 2;
    const int row = quarter * 32 + lane;
    uint32_t done_jobs = 0;
    float mx = 0.f;
    __shared__ uint4 turn[QEPI][32];   // (see ChainStart::load)
    ChainStart start;
    float o[32];   // the chains' starts of 32 columns
    if (NA == 3 && a.c_a) {
      const SgJob job = a.jobs[job0];
      if (!q_skip(job, a)) {
        int s0, s1;
        stages_of(job.nk, s0, s1);
        start = ChainStart(job, a, quarter * 32, s0 * KC, s1 * KC, job.nk * QKC);
        for (int c = c_begin; c < c_end; c += 32) {
          start.load(c, c_end, turn[warp - 2], o);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float v[8] = {o[8 * u], o[8 * u + 1], o[8 * u + 2], o[8 * u + 3], o[8 * u + 4], o[8 * u + 5], o[8 * u + 6], o[8 * u + 7]};
            if (c + 8 * u < c_end) tmem_st8(tmem + ((uint32_t)(quarter * 32) << 16) + c + 8 * u, v);
          }
        }
        tmem_wait_st();
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_acce + 8);
        if (c_end - c_begin > 32) start.load(c_begin, c_end, turn[warp - 2], o);   // again the first 32, before the products end
      }
    }
    for (int jx = job0; jx < a.njobs; jx += job_step) {
      const SgJob job = a.jobs[jx];
      if (q_skip(job, a)) continue;
      const uint32_t buf = done_jobs % a.nbuf, round = done_jobs / a.nbuf;
      int ok = 0;
      if (lane == 0) ok = qwait(bar_accf + 8 * buf, round & 1, sh, a) ? 1 : 0;
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) break;
      fence_after();
      const uint32_t taddr = tmem + buf * a.buf_cols + ((uint32_t)(quarter * 32) << 16);
      float* orow_p = a.out + job.out + (int64_t)row * a.mpad;
      const float sc = a.out_scale * (a.b_amax ? f16_inv_scale(__uint_as_float(*a.b_amax)) : 1.f);
      for (int c = c_begin; c < c_end; c += 8) {
        uint32_t r8[8], s8[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        tmem_ld8(taddr + c, r8);
        if (a.acc_b) tmem_ld8(taddr + a.acc_b + c, s8);
        tmem_wait_ld();
        float x[8];
        if (NA == 3 && a.c_a) {
          const int at = c - c_begin;
          if (at % 32 == 0 && at > 0) start.load(c, c_end, turn[warp - 2], o);
#pragma unroll
          for (int t = 0; t < 8; ++t) {
            const float v = (at & 16) ? ((at & 8) ? o[24 + t] : o[16 + t]) : ((at & 8) ? o[8 + t] : o[t]);
            r8[t] = __float_as_uint(__uint_as_float(r8[t]) - v);
          }
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) x[t] = sc * (__uint_as_float(r8[t]) + __uint_as_float(s8[t]));
        if (a.cl > 1) {   // the ring is free: this job is the CTA's only one
          int s0, s1;
          stages_of(job.nk, s0, s1);
          float4* dst = reinterpret_cast<float4*>(base + ((size_t)row * a.mpad + c) * 4);
          const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);   // (no stage: nothing was accumulated)
          dst[0] = s1 > s0 ? make_float4(x[0], x[1], x[2], x[3]) : z;
          dst[1] = s1 > s0 ? make_float4(x[4], x[5], x[6], x[7]) : z;
          continue;
        }
        float4* dst = reinterpret_cast<float4*>(orow_p + c);
        const bool in = RFF_SPAN(job.out + (int64_t)row * a.mpad + c, 8, a.out_elems);
        if (a.accumulate && in) {
          const float4 p0 = dst[0], p1 = dst[1];
          x[0] += p0.x; x[1] += p0.y; x[2] += p0.z; x[3] += p0.w;
          x[4] += p1.x; x[5] += p1.y; x[6] += p1.z; x[7] += p1.w;
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) mx = fmaxf(mx, fabsf(x[t]));
        if (in) {
          dst[0] = make_float4(x[0], x[1], x[2], x[3]);
          dst[1] = make_float4(x[4], x[5], x[6], x[7]);
        }
      }
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_acce + 8 * buf);   // the set is free for the job after next
      ++done_jobs;
    }
    if (a.amax && a.cl == 1) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      if (lane == 0 && mx > 0.f) atomicMax(a.amax, __float_as_uint(mx));
    }
  }
  // (the roles' single threads rejoin their warps; the columns go back before a cluster is waited for, see
  // simt.cuh)
  __syncwarp();
  fence_before();
  __syncthreads();
  fence_after();
  if (a.cl > 1) cluster_arrive();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.tmem_cols) : "memory");
  }
  if (a.cl > 1) {
    cluster_wait();
    const SgJob job = a.jobs[job0];
    if (!q_skip(job, a)) {
      const int rows = 128 / a.cl, n4 = rows * a.mpad / 4;
      const uint32_t src = smem_u32(base) + (uint32_t)(rank * rows * a.mpad * 4);
      float mx = 0.f;
      for (int e = threadIdx.x; e < n4; e += QNT) {
        float4 x = ld_cluster4(mapa_rank(src + 16 * e, 0));
        for (int r = 1; r < a.cl; ++r) {
          const float4 v = ld_cluster4(mapa_rank(src + 16 * e, r));
          x = make_float4(x.x + v.x, x.y + v.y, x.z + v.z, x.w + v.w);
        }
        const int64_t o = job.out + (int64_t)rank * rows * a.mpad + 4 * e;
        if (!RFF_SPAN(o, 4, a.out_elems)) continue;
        float4* dst = reinterpret_cast<float4*>(a.out + o);
        if (a.accumulate) {
          const float4 p0 = *dst;
          x = make_float4(x.x + p0.x, x.y + p0.y, x.z + p0.z, x.w + p0.w);
        }
        *dst = x;
        mx = fmaxf(mx, fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w))));
      }
      __syncwarp();
      if (a.amax) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0 && mx > 0.f) atomicMax(a.amax, __float_as_uint(mx));
      }
    }
    cluster_sync_all();   // nobody leaves while others read its shared memory
  }
}

// ---- the right-hand side, split three ways and transposed: rT_t[i][c][slot]
__global__ void k_rhs_split3T(const float* __restrict__ Wbar, const float* __restrict__ muij,
                              const float* __restrict__ Rpart, int nsplit, int R, int64_t fslots, int mpad,
                              const int32_t* __restrict__ feat_ok, const float* __restrict__ What,
                              __nv_bfloat16* __restrict__ r1, __nv_bfloat16* __restrict__ r2,
                              __nv_bfloat16* __restrict__ r3) {
  __shared__ float tile[32][33];
  const int i = blockIdx.z;
  const int64_t p0 = (int64_t)blockIdx.x * 32;
  const int c0 = blockIdx.y * 32;
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;   // 256 threads
  const int64_t nfe = fslots * mpad;
  for (int rr = ty; rr < 32; rr += 8) {
    const int64_t p = p0 + rr;
    const int c = c0 + tx;
    float v = 0.f;
    if (p < fslots && c < mpad && feat_ok[p] >= 0) {
      const int64_t e = p * mpad + c, t = (int64_t)i * nfe + e;
      v = Wbar[e] - muij[t];
      if (What) v -= What[t];
      for (int sp = 0; sp < nsplit; ++sp)
        if (RFF_IN((int64_t)sp * R * nfe + t, (int64_t)nsplit * R * nfe)) v += Rpart[(int64_t)sp * R * nfe + t];
    }
    tile[rr][tx] = v;
  }
  __syncthreads();
  for (int cc = ty; cc < 32; cc += 8) {
    const int c = c0 + cc;
    const int64_t p = p0 + tx;
    if (c < mpad && p < fslots) {
      const float x = tile[tx][cc];
      const __nv_bfloat16 h = __float2bfloat16_rn(x);
      const float rem = x - __bfloat162float(h);
      const __nv_bfloat16 m = __float2bfloat16_rn(rem);
      const __nv_bfloat16 l = __float2bfloat16_rn(rem - __bfloat162float(m));
      const int64_t o = ((int64_t)i * mpad + c) * fslots + p;
      if (!RFF_IN(o, (int64_t)R * mpad * fslots)) continue;
      r1[o] = h;
      r2[o] = m;
      r3[o] = l;
    }
  }
}

// ---- one block's Q (s x s, float64) into the three split arrays at row qrow
__global__ void k_split3_q(const double* __restrict__ Q, int s, int64_t ldq, int64_t qrow,
                           __nv_bfloat16* __restrict__ q1, __nv_bfloat16* __restrict__ q2,
                           __nv_bfloat16* __restrict__ q3) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= (int64_t)s * s) return;
  const int64_t r = t / s, c = t % s;
  const double x = Q[t];
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7ff);
  __nv_bfloat16 h, m, l;
  if (E >= 1023 - 64 && E <= 1023 + 64) {   // 2^-64 <= |x| < 2^65: every power below is a normal FP32
    // x = t + rs: t its leading 24 bits as an FP32 number and rs the remaining 29 (both exact,
    // built by integer instructions: this part's FP64 pipe runs at 1/64 of the FP32 rate);
    // then h = bf16(t), and m, l the BF16 terms of (t - h) + rs, whose FP32 rounding lies
    // below 2^-32 |x|
    const uint32_t sgn = (uint32_t)(b >> 32) & 0x80000000u;
    const float t32 = __uint_as_float(sgn | ((uint32_t)(E - 1023 + 127) << 23) | (uint32_t)((b >> 29) & 0x7fffffu));
    const float r32 = __uint2float_rn((uint32_t)(b & 0x1fffffffu)) * __uint_as_float((uint32_t)(E - 1075 + 127) << 23);
    h = __float2bfloat16_rn(t32);
    const float rem = __fadd_rn(__fsub_rn(t32, __bfloat162float(h)), sgn ? -r32 : r32);
    m = __float2bfloat16_rn(rem);
    l = __float2bfloat16_rn(__fsub_rn(rem, __bfloat162float(m)));
  } else {   // zero, tiny, huge or not finite: the FP64 route
    h = __double2bfloat16(x);
    const double rem = x - (double)__bfloat162float(h);
    m = __double2bfloat16(rem);
    l = __double2bfloat16(rem - (double)__bfloat162float(m));
  }
  const int64_t o = (qrow + r) * ldq + c;
  q1[o] = h;
  q2[o] = m;
  q3[o] = l;
}

template <int NA, int NB, int F16, int KC>
cudaError_t set_smem_attr() {
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  std::call_once(once, [] {
    attr = cudaFuncSetAttribute(k_split_gemm<NA, NB, F16, KC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                1024 + 216 * 1024 + 256);
  });
  return attr;
}

}  // namespace

cudaError_t launch_split3_q(const double* Q, int s, int64_t ldq, int64_t qrow, __nv_bfloat16* q1,
                            __nv_bfloat16* q2, __nv_bfloat16* q3, cudaStream_t st) {
  const int64_t n = (int64_t)s * s;
  if (n <= 0) return cudaSuccess;
  k_split3_q<<<(unsigned)ceil_div(n, 256), 256, 0, st>>>(Q, s, ldq, qrow, q1, q2, q3);
  return cudaGetLastError();
}

cudaError_t launch_rhs_split3T(const float* Wbar, const float* muij, const float* Rpart, int nsplit, int R,
                               int64_t fslots, int mpad, const int32_t* feat_ok, __nv_bfloat16* r1,
                               __nv_bfloat16* r2, __nv_bfloat16* r3, cudaStream_t st, const float* What) {
  dim3 grid((unsigned)ceil_div(fslots, 32), (unsigned)ceil_div(mpad, 32), (unsigned)R);
  k_rhs_split3T<<<grid, 256, 0, st>>>(Wbar, muij, Rpart, nsplit, R, fslots, mpad, feat_ok, What, r1, r2, r3);
  return cudaGetLastError();
}

cudaError_t split_gemm(const SgView& v) {
  if (v.njobs <= 0) return cudaSuccess;
  if (v.mpad > 256 || v.mpad < 16 || v.mpad % 16) return cudaErrorInvalidValue;
  if (!((v.na == 3 && v.nb == 3 && !v.f16) || (v.na == 2 && v.nb == 2 && v.f16))) return cudaErrorInvalidValue;
  QArgs a;
  memset(&a, 0, sizeof(a));
  cudaError_t e;
  const size_t budget = std::min<size_t>(v.smem_budget ? v.smem_budget : 216 * 1024, 216 * 1024);
  // 64-element stages only where two of them fit (m_pad = 256 with three terms does not)
  const int kc = (v.kc == 64 && 2 * (size_t)(v.na * 128 + v.nb * v.mpad) * 64 * 2 <= budget) ? 64 : 32;
  for (int s = 0; s < v.na; ++s)
    if ((e = tc_make_map_bf16(&a.tA[s], v.A[s], v.a_cols, v.a_rows, v.a_cols, 128, kc)) != cudaSuccess) return e;
  for (int s = 0; s < v.nb; ++s)
    if ((e = tc_make_map_bf16(&a.tB[s], v.B[s], v.b_cols, v.b_rows, v.b_cols, v.mpad, kc)) != cudaSuccess)
      return e;
  a.mpad = v.mpad;
  a.stage_bytes = (uint32_t)(v.na * 128 + v.nb * v.mpad) * kc * 2;
  a.ns = (int)std::min<size_t>(QMAXS, budget / a.stage_bytes);
  if (a.ns < 2) a.ns = 2;
  a.tmem_cols = v.mpad <= 32 ? 32 : v.mpad <= 64 ? 64 : v.mpad <= 128 ? 128 : 256;
  if (v.two_acc) {
    // the tensor cores' FP32 accumulator rounds toward zero at every accumulation: the
    // dominant hi.hi products get an accumulator of their own (K/16 accumulations instead of
    // NPROD K/16), the small products share the second, and the two are added in FP32
    a.acc_b = a.tmem_cols;
    a.tmem_cols *= 2;
  }
  a.jobs = v.jobs;
  a.njobs = v.njobs;
  a.out = v.out;
  a.out_elems = v.out_elems;
  a.out_scale = v.out_scale;
  a.b_amax = v.b_amax;
  a.amax = v.amax;
  a.bmask = v.bmask;
  a.accumulate = v.accumulate;
  a.err = tc_error_ptr();
  if (!a.err) return cudaErrorMemoryAllocation;
  a.timeout_cycles = 4000000000LL;   // about two seconds at the boost clock
  const size_t smem = 1024 + (size_t)a.ns * a.stage_bytes + 256;
  // the four instances: BF16 three-term or FP16 two-term operands, 32- or 64-element stages
  auto kern = [&]() -> const void* {
    if (v.na == 3) return kc == 64 ? (const void*)k_split_gemm<3, 3, 0, 64> : (const void*)k_split_gemm<3, 3, 0, 32>;
    return kc == 64 ? (const void*)k_split_gemm<2, 2, 1, 64> : (const void*)k_split_gemm<2, 2, 1, 32>;
  };
  if (v.na == 3)
    e = kc == 64 ? set_smem_attr<3, 3, 0, 64>() : set_smem_attr<3, 3, 0, 32>();
  else
    e = kc == 64 ? set_smem_attr<2, 2, 1, 64>() : set_smem_attr<2, 2, 1, 32>();
  if (e != cudaSuccess) return e;
  // one job per CTA, or (persistent) at most as many CTAs as fit on the device at once, each
  // taking every grid-th job; two accumulator sets when the tensor memory of the CTAs that
  // share an SM holds them
  a.buf_cols = a.tmem_cols;
  a.nbuf = 1;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern(), QNT, smem);
  if (e != cudaSuccess) return e;
  per_sm = std::min(std::max(per_sm, 1), std::max(1, 512 / (int)a.tmem_cols));
  const int64_t slots = (int64_t)device_sms() * per_sm;
  auto run = [&](int64_t grid, int cl) -> cudaError_t {
    a.cl = cl;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(grid * cl));
    cfg.blockDim = dim3(QNT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = v.st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cl;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (v.na == 3)
      return kc == 64 ? cudaLaunchKernelEx(&cfg, k_split_gemm<3, 3, 0, 64>, a)
                      : cudaLaunchKernelEx(&cfg, k_split_gemm<3, 3, 0, 32>, a);
    return kc == 64 ? cudaLaunchKernelEx(&cfg, k_split_gemm<2, 2, 1, 64>, a)
                    : cudaLaunchKernelEx(&cfg, k_split_gemm<2, 2, 1, 32>, a);
  };
  if (v.persistent) {
    if (2u * a.tmem_cols * (uint32_t)per_sm <= 512u) {
      a.nbuf = 2;
      a.tmem_cols *= 2;
    }
    return run(std::min<int64_t>(v.njobs, slots), 1);
  }
  // The jobs past the last whole wave would leave most SMs idle while each CTA walks its K stages at
  // the pace of the copies: clusters share those jobs' stages, as many CTAs as fit side by side
  // (where a partial result fits the ring's memory).  A sweep of four solves (16 to 64 jobs of K =
  // 1024 or 2048, m = 8): 47 -> 24 us a product, 12.4 -> 11.5 ms over 10 iterations; 48 jobs of K =
  // 1000: 50 iterations 17.7 -> 17.0 ms.  A product's chains of round-toward-zero accumulations get as
  // much shorter (K = 1024 over eight CTAs: emulated error 1.6e-6 -> 2.3e-7), so the solvers' errors
  // against float64 fall (60 drawn scoring cases 6.2e-6 -> 4.2e-6 in the geometric mean, sweeps of four
  // solves 6.2e-6 -> 4.5e-6 over all outputs), with the starts above also where a projection cancels;
  // some single outputs rise where the longer chain's bias cancelled another one (the sweep's largest
  // data set, D = 1024: 1.16e-6 -> 1.47e-6).  The streamed passes of 40,000 rows at D = 8192, 2 x 2 (pass 2:
  // 626 jobs on 304 slots): 10 iterations 14.2 -> 13.7 ms.
  const int64_t rest = v.njobs % slots, full = v.njobs - rest;
  int cl = 1;
  if ((size_t)128 * v.mpad * 4 <= (size_t)a.ns * a.stage_bytes)
    while (cl < 8 && 2 * cl * rest <= slots) cl *= 2;
  if (cl == 1 || rest == 0) return run(v.njobs, 1);
  if (full > 0) {
    a.njobs = (int)full;
    if ((e = run(full, 1)) != cudaSuccess) return e;
  }
  a.jobs = v.jobs + full;
  a.njobs = (int)rest;
  if (v.centre && v.two_acc && v.na == 3) {
    a.c_a = static_cast<const __nv_bfloat16*>(v.A[0]);
    a.c_b = static_cast<const __nv_bfloat16*>(v.B[0]);
    a.c_lda = v.a_cols;
    a.c_ldb = v.b_cols;
  }
  return run(rest, cl);
}

RFF_CHECK_UNIT(qgemm)

}  // namespace rff
