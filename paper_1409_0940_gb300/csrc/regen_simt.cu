// FP32 SIMT regeneration passes: the plain FP32 path (no tensor cores).
//
// Each CTA multiplies a fixed 128-row panel of one operand ("A") against a run of
// 128-row panels of the other ("B"), both holding rows of length K (the input
// dimension d, padded):
//     T   = A_panel . B_panel^T                       (X_i G_j or its transpose)
//     Z   = sqrt(2/D) cos(T + b)  masked to valid slots  (the transform T[X_i, j], Sec. 4;
//           the random Laplace map: Z = exp(-T) / sqrt(D))
//     acc += Z . M[B rows]                             (the chained product)
// and writes acc when a run ends.  With A = feature rows of G^T and B = data rows
// this is pass 1, R_ij = Z_ij^T V_ij (the Z_ij^T (Obar_ij + nu_i) term of eq. (gpWij));
// with A = data rows and B = feature rows it is pass 2, O'_ij = Z_ij W'_ij
// (eq. (gpOij)), and prediction when M is Wbar and the run spans all blocks.
//
// What bounds it: the FP32 pipe, with shared memory close behind.  A shared-memory load hands a
// warp 128 bytes per clock, however few addresses it reads, and 8 x 8 outputs per thread take 16
// words for 64 multiply-adds: exactly what the pipe needs at its full rate.  So the tile is 128 x
// 256 (two 128-row tiles of B), 8 x 16 outputs per thread (rows ty + 16 i, columns tx + 16 j): 24
// words for 128 multiply-adds.  A lone tile at the end of a run takes the 128 x 128 form.  The
// panels, and then the rows of M the chain multiplies, stream through one ring of two stages
// (32 K, 8,192 clocks of multiply-adds, each) filled by asynchronous copies across tiles, so that
// neither the copies nor the first K chunk of a tile is waited for.  For the chain a thread takes 8 rows (ty*4 + {0..3}, 64 + ty*4 +
// {0..3}) by m_pad/16 columns (tx + 16 q) of one 128-row half's Z tile in shared memory; its sums
// wait in tensor memory while the next T is formed.
// Measured: 50,001 rows, d = 784, D = 8192, m = 10: 21.2 -> 15.1 ms (44 TFLOP/s of the 73.6 that
// independent FFMA chains reach; issue slots 66 % busy: with two warps per scheduler a third of the
// clocks find none eligible, most of it register-port (dispatch) and shared-memory stalls); 20,000
// rows, d = 440, D = 8192, m = 147: pass 1 5.3 -> 4.1 ms, pass 2 9.9 -> 4.2 ms; 2000 rows, d = 16, D =
// 512, m = 1: pass 2 76 -> 13.5 us.  Packed multiply-adds (fma.rn.f32x2) measured 17.4 ms here.
#include "common.cuh"
#include "internal.h"
#include "simt.cuh"

#include <algorithm>

namespace rff {

namespace {

using namespace simt;

constexpr int BM = 128, BN = 128, BK = 32, NS = 2;
constexpr int LDK = row_stride(BK);
constexpr int ZLD = BM + 4;                       // Z^T row stride: 8 x 4 lanes store to distinct banks
constexpr int STAGE = (BM + 2 * BN) * LDK;        // floats: an A panel and two B panels of 32 K, or rows of M
// rows of M in a stage: as many of a tile's 128 as fit (fewer, longer steps between barriers)
__host__ __device__ constexpr int m_rows(int mq) { return mq <= 6 ? 128 : mq <= 13 ? 64 : 32; }
static_assert(m_rows(6) * 96 <= STAGE && m_rows(13) * 208 <= STAGE && m_rows(16) * 256 <= STAGE,
              "the rows of M fit a stage");
constexpr int PARTS = 8;                          // parts of a run of tiles (see pass 2)
enum { CHAIN, ADD, FF };                          // how the sums of a run are formed (see chain_tile)
// phases and validity (slot table entries) of a tile pair's B rows, two pairs deep: read from global
// memory where T becomes Z, their latency was 7 % of the kernel
struct Meta {
  float bias[2 * BN];
  int32_t ok[2 * BN];
};
constexpr size_t SMEM = ((size_t)NS * STAGE + (size_t)BN * ZLD) * 4 + 2 * sizeof(Meta);
static_assert(SMEM <= 232448 - 256, "the ring and the Z tile fit a CTA's shared memory");

__device__ __forceinline__ int chain_row(int ty, int i) { return i < 4 ? ty * 4 + i : 64 + ty * 4 + (i - 4); }

// What a tile reads: A rows a0.., B tiles of 128 rows from slot b0 on, M rows alike.
struct Operands {
  const float *A, *B, *M;   // A and M of this CTA's panel and block; B from row 0
  const float* b_bias;      // per B row, or null
  const int32_t* b_ok;      // per B row, < 0 = padding, or null
  int64_t lda, ldb;
  int K, mpad;
};

// The tiles t, t + 1, .. of parts p .. of a run of nt tiles in `parts` parts, taken two at a time
// within a part: width() of them at t.
struct Walk {
  int64_t t, end, nt;
  int p, p_end, parts;
  __device__ __forceinline__ void enter() {   // part p, or the first one after it that is not empty
    for (; p < p_end; ++p) {
      end = (p + 1) * nt / parts;
      if (t < end) return;
    }
  }
  __device__ __forceinline__ bool done() const { return p >= p_end; }
  __device__ __forceinline__ int width() const { return t + 1 < end ? 2 : 1; }
  __device__ __forceinline__ void step() {
    t += width();
    if (t >= end) {
      ++p;
      enter();
    }
  }
};
__device__ __forceinline__ Walk make_walk(int64_t nt, int parts, int p0, int p1) {
  Walk w{p0 * nt / parts, 0, nt, p0, p1, parts};
  w.enter();
  return w;
}

// The ring's producer side: every thread copies its share of each stage.  Steps run tile (or
// pair of tiles) by tile: nk panel stages and then, with a chain, 128 / MR stages of M per tile.
struct Feed {
  Walk w;
  int last;      // rows of the last tile that are read (64 or 128)
  int64_t b0;    // B row of tile 0
  int r;         // step within the tile
  int slot, pair;
};

// MR: rows of M per stage, 0 = no chain
template <int MR>
__device__ __forceinline__ void feed_step(Feed& f, const Operands& o, int nk, float* ring, Meta* meta) {
  if (!f.w.done()) {
    float* st = ring + f.slot * STAGE;
    const int tid = threadIdx.x, wd = f.w.width();
    const int64_t b = f.b0 + f.w.t * BN;
    const int rows = wd * BN - (f.w.t + wd == f.w.nt ? BN - f.last : 0);   // B rows of this tile pair
    if (f.r == 0 && tid < rows) {
      if (o.b_bias) cp_async4(&meta[f.pair].bias[tid], o.b_bias + b + tid);
      if (o.b_ok) cp_async4(&meta[f.pair].ok[tid], o.b_ok + b + tid);
    }
    if (f.r < nk) {
      constexpr int PIECES = BK / 4, ROWS = NT / PIECES;   // 16-byte pieces of a row, rows per round
      const int piece = 4 * (tid % PIECES), row = tid / PIECES;
      const float* a = o.A + row * o.lda + f.r * BK + piece;
      const float* bp = o.B + (b + row) * o.ldb + f.r * BK + piece;
      float* dst = st + row * LDK + piece;
#pragma unroll
      for (int q = 0; q < BM / ROWS; ++q) cp_async16(dst + q * ROWS * LDK, a + q * ROWS * o.lda);
#pragma unroll
      for (int q = 0; q < 2 * BN / ROWS; ++q)
        if (q * ROWS < rows) cp_async16(dst + (BM + q * ROWS) * LDK, bp + q * ROWS * o.ldb);
    } else {
      const float* src = o.M + (b + (int64_t)(f.r - nk) * MR) * o.mpad;
      const int n4 = min(MR, rows - (f.r - nk) * MR) * o.mpad / 4;
      for (int t = tid; t < n4; t += NT) cp_async16(st + 4 * t, src + 4 * t);
    }
    if (++f.r == nk + (MR ? wd * (BN / (MR ? MR : 1)) : 0)) {
      f.r = 0;
      f.pair ^= 1;
      f.w.step();
    }
    f.slot = f.slot + 1 == NS ? 0 : f.slot + 1;
  }
  cp_commit();
}

// acc[j][i] += A[ty + 16 i] . B[tx + 16 j] over 4 k4n elements of the stage, k in order
template <int NJ>
__device__ __forceinline__ void panel_fma(const float* __restrict__ st, int tx, int ty, int k4n, float (&acc)[16][8]) {
  const float* ap = st + ty * LDK;
  const float* bp = st + BM * LDK + tx * LDK;
#pragma unroll 1
  for (int k4 = 0; k4 < k4n; ++k4) {
    float a[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float4 v = *reinterpret_cast<const float4*>(ap + 16 * i * LDK + 4 * k4);
      a[i][0] = v.x; a[i][1] = v.y; a[i][2] = v.z; a[i][3] = v.w;
    }
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const float4 v = *reinterpret_cast<const float4*>(bp + 16 * j * LDK + 4 * k4);
      const float b[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[j][i] = fmaf(a[i][kk], b[kk], acc[j][i]);
    }
  }
}

// What becomes of T's elements: a thread turns the A rows 4 lane .. 4 lane + 3 into Z.
struct RowSide {
  uint32_t mask;      // bit i: A row 4 lane + i is valid
  float4 phase;       // their phases where the feature index is the A row (pass 1)
  bool on_a;
};
__device__ __forceinline__ RowSide row_side(const int32_t* __restrict__ ok, const float* __restrict__ bias, int64_t a0) {
  const int r = 4 * (threadIdx.x % 32);
  RowSide s{15u, make_float4(0.f, 0.f, 0.f, 0.f), bias != nullptr};
  if (ok) {
    const int4 v = *reinterpret_cast<const int4*>(ok + a0 + r);
    s.mask = (v.x >= 0 ? 1u : 0u) | (v.y >= 0 ? 2u : 0u) | (v.z >= 0 ? 4u : 0u) | (v.w >= 0 ? 8u : 0u);
  }
  if (bias) s.phase = *reinterpret_cast<const float4*>(bias + a0 + r);
  return s;
}

// Half H of T through the Z^T tile: T as it is, then, in a loop short enough for the instruction
// caches (64 cosines unrolled per half took a cold CTA longer to fetch than to run), the cosine with
// the feature phase (or exp(-T), the Laplace map), masked to valid rows and features.  The caller
// has a barrier before (the tile is free) and after (it is whole).
template <int H>
__device__ __forceinline__ void store_z(float* __restrict__ ZsT, const float (&acc)[16][8], int tx, int ty,
                                        const Meta& meta, bool have_ok, const RowSide& rs, float scale, int map) {
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int i = 0; i < 8; ++i) ZsT[(tx + 16 * j) * ZLD + ty + 16 * i] = acc[8 * H + j][i];
  __syncthreads();
  const int lane = threadIdx.x % 32;
#pragma unroll 1
  for (int n = threadIdx.x / 32; n < BN; n += NT / 32) {
    float4* zp = reinterpret_cast<float4*>(ZsT + n * ZLD + 4 * lane);
    const float4 v = *zp;
    const uint32_t mask = (!have_ok || meta.ok[H * BN + n] >= 0) ? rs.mask : 0u;
    float4 z;
    if (map == 1) {
      z = make_float4(expf(-v.x), expf(-v.y), expf(-v.z), expf(-v.w));
    } else {
      const float pb = rs.on_a ? 0.f : meta.bias[H * BN + n];
      z = make_float4(cos_rr(v.x + (rs.on_a ? rs.phase.x : pb)), cos_rr(v.y + (rs.on_a ? rs.phase.y : pb)),
                      cos_rr(v.z + (rs.on_a ? rs.phase.z : pb)), cos_rr(v.w + (rs.on_a ? rs.phase.w : pb)));
    }
    z.x = mask & 1u ? scale * z.x : 0.f;
    z.y = mask & 2u ? scale * z.y : 0.f;
    z.z = mask & 4u ? scale * z.z : 0.f;
    z.w = mask & 8u ? scale * z.w : 0.f;
    *zp = z;
  }
}

// acc2[q] += Z[chain_row(ty, .)][n] * M[n][tx + 16 q] over the MR rows n of a stage, n in order; a
// pair holds two consecutive rows
template <int MQ, int ROWS>
__device__ __forceinline__ void chain_fma(const float* __restrict__ ZsT, const float* __restrict__ Ms, int mpad, int tx,
                                          int ty, f32x2 (&acc2)[MQ][4]) {
#pragma unroll 4
  for (int n = 0; n < ROWS; ++n) {
    const ulonglong2 zl = *reinterpret_cast<const ulonglong2*>(ZsT + n * ZLD + ty * 4);
    const ulonglong2 zh = *reinterpret_cast<const ulonglong2*>(ZsT + n * ZLD + 64 + ty * 4);
#pragma unroll
    for (int q = 0; q < MQ; ++q) {
      const float mv = Ms[n * mpad + tx + 16 * q];
      const f32x2 m2 = pair2(mv, mv);
      acc2[q][0] = fma2(zl.x, m2, acc2[q][0]);
      acc2[q][1] = fma2(zl.y, m2, acc2[q][1]);
      acc2[q][2] = fma2(zh.x, m2, acc2[q][2]);
      acc2[q][3] = fma2(zh.y, m2, acc2[q][3]);
    }
  }
}

// The kernels' common body: T, Z and (chain) the products of every tile with M.
template <int MR>
struct Body {
  float *ring, *ZsT;
  Meta* meta;
  Operands o;
  Feed f;
  int nk, slot, pair, tx, ty;
  uint32_t park;

  // tiles of 128 B rows, tile 0 at row b0, walked by w
  __device__ __forceinline__ Body(float* smem, const Operands& op, int64_t b0, const Walk& w, int last_rows = BN)
      : ring(smem), ZsT(smem + NS * STAGE), meta(reinterpret_cast<Meta*>(ZsT + BN * ZLD)), o(op), f{w, last_rows, b0, 0, 0, 0},
        nk((op.K + BK - 1) / BK), slot(0), pair(0), tx(thread_tx()), ty(thread_ty()), park(0) {
#pragma unroll
    for (int s = 0; s < NS - 1; ++s) feed_step<MR>(f, o, nk, ring, meta);
  }
  // the next stage has landed; the one before it is free and is filled again
  __device__ __forceinline__ const float* next() {
    cp_wait<NS - 2>();
    __syncthreads();
    feed_step<MR>(f, o, nk, ring, meta);
    const float* st = ring + slot * STAGE;
    slot = slot + 1 == NS ? 0 : slot + 1;
    return st;
  }
  // T of one tile (NJ = 8) or two (NJ = 16)
  template <int NJ>
  __device__ __forceinline__ void form_t(float (&acc)[16][8]) {
#pragma unroll
    for (int j = 0; j < 16; ++j)
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[j][i] = 0.f;
    for (int r = 0; r < nk; ++r) {
      const float* st = next();
      panel_fma<NJ>(st, tx, ty, min(BK, o.K - r * BK) / 4, acc);
    }
  }
  // The tile or two at w: T, then half by half Z and its products with M (chain_tile)
  template <int MQ, int MODE>
  __device__ __forceinline__ void run(const Walk& w, const RowSide& rs, float scale, int map) {
    float acc[16][8];
    const int wd = w.width();
    if (wd == 2) form_t<16>(acc);
    else form_t<8>(acc);
    // (every thread is past the chain of the previous tile: nk >= 1 barriers ago)
    store_z<0>(ZsT, acc, tx, ty, meta[pair], o.b_ok, rs, scale, map);
    chain_tile<MQ, MODE>(w.t + 1 == w.nt ? f.last : BN);
    if (wd == 2) {
      __syncthreads();   // everyone is done with the first half's Z
      store_z<1>(ZsT, acc, tx, ty, meta[pair], o.b_ok, rs, scale, map);
      chain_tile<MQ, MODE>(w.t + 2 == w.nt ? f.last : BN);
    }
    pair ^= 1;
  }
  // The products of the Z tile's first `rows` rows (64 or 128; the first barrier in here makes it
  // whole) with M, 64 rows at a time, into the sums parked at words 0..
  //   CHAIN: one chain of multiply-adds per sum, through all tiles;
  //   ADD:   every 64 rows' sums are added to them;
  //   FF:    the same in float-float (TwoSum), the low parts at 8 MQ..
  template <int MQ, int MODE>
  __device__ __forceinline__ void chain_tile(int rows) {
    const float* st = nullptr;   // half a stage, a stage, or several per 64 rows
#pragma unroll 1
    for (int n0 = 0; n0 < rows; n0 += 64) {
      f32x2 acc2[MQ][4];
#pragma unroll
      for (int q = 0; q < MQ; ++q) {
        float h[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (MODE == CHAIN) unpark8(park + 8 * q, h);
#pragma unroll
        for (int i = 0; i < 4; ++i) acc2[q][i] = pair2(h[2 * i], h[2 * i + 1]);
      }
      if (MR >= 64) {
        if (n0 % MR == 0) st = next();
        chain_fma<MQ, 64>(ZsT + n0 * ZLD, st + n0 % MR * o.mpad, o.mpad, tx, ty, acc2);
      } else {
#pragma unroll 1
        for (int u = 0; u < 64; u += MR) {
          st = next();
          chain_fma<MQ, MR>(ZsT + (n0 + u) * ZLD, st, o.mpad, tx, ty, acc2);
        }
      }
#pragma unroll
      for (int q = 0; q < MQ; ++q) {
        float h[8], v[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) unpair2(acc2[q][i], v[2 * i], v[2 * i + 1]);
        if (MODE == CHAIN) {
          park8(park + 8 * q, v);
          continue;
        }
        unpark8(park + 8 * q, h);
        if (MODE == FF) {
          float l[8];
          unpark8(park + 8 * (MQ + q), l);
#pragma unroll
          for (int i = 0; i < 8; ++i) two_sum_into(h[i], l[i], v[i]);
          park8(park + 8 * (MQ + q), l);
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i) h[i] = __fadd_rn(h[i], v[i]);
        }
        park8(park + 8 * q, h);
      }
      tc5::tmem_wait_st();
    }
  }
  __device__ __forceinline__ void park_zeros(int words8) {
    const float z[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int w = 0; w < words8; ++w) park8(park + 8 * w, z);
    tc5::tmem_wait_st();
  }
};

// Pass 2 / predict.  A work item is 128 data rows against the feature slots of one column block
// (per_block: O'_ij to out + j * out_block_stride) or of all of them.  Its feature tiles form
// PARTS fixed parts, whose sums are added in order whether one CTA takes them all (cl = 1) or
// each CTA of a cluster takes one (cl = PARTS; with nt < PARTS tiles some parts are empty, and
// cl >= nt CTAs take PARTS / cl parts each, at most one of them not empty) and the sums meet
// through distributed shared memory, so a result does not depend on the split.  For m_pad <= 64 each 64-feature partial
// sum is folded into a float-float accumulator (TwoSum): a 4096-feature block then carries the
// error of one 64-term sum, not of a 4096-term one (the outer form's W' = c + Z^T P (V - Z c)
// takes the rounding of Z c with gain ~1 relative to |Z c|, which exceeds |W'|).
template <int MQ>
__global__ void __launch_bounds__(NT, 1) k_pass2_simt(const __grid_constant__ PassArgs p, int64_t item0, int cl) {
  constexpr bool COMP = MQ <= 4;
  constexpr int LOW = 8 * MQ;                    // parked words of the low parts
  constexpr int TOT = COMP ? 16 * MQ : 8 * MQ;   // and of the totals
  extern __shared__ __align__(16) float smem[];
  __shared__ uint32_t tmem_word;
  const uint32_t rank = cl > 1 ? tc5::cluster_rank() : 0;
  const int64_t units = p.per_block ? p.C : 1;
  const int64_t item = item0 + blockIdx.x / cl, a0 = item / units * BM;
  const int j = (int)(item % units);
  // row block of this tile: the chain operand W'_ij depends on it
  int rb = 0;
  while (rb + 1 < p.R && p.row_slot[rb + 1] <= a0) ++rb;
  if (p.per_block && p.bmask && !p.bmask[rb * p.C + j]) return;   // an inactive block (the whole cluster alike)
  const int64_t f0 = p.per_block ? p.col_slot[j] : 0;
  const int64_t nt = p.per_block ? ceil_div(p.col_size[j], BN) : p.g_rows / BN;
  if (!RFF_SPAN(a0, BM, p.x_rows) || !RFF_SPAN(f0, nt * BN, p.g_rows) ||
      !RFF_SPAN(rb * p.m_block_stride + f0 * p.mpad, nt * BN * p.mpad, p.m_elems) ||
      !RFF_SPAN(j * p.out_block_stride + a0 * p.mpad, BM * p.mpad, p.out_elems))
    return;
  if (threadIdx.x < 32) tc5::tmem_alloc<1>(tc5::smem_u32(&tmem_word), 512);
  const int p0 = cl > 1 ? (int)rank * (PARTS / cl) : 0, p1 = cl > 1 ? ((int)rank + 1) * (PARTS / cl) : PARTS;
  Walk w = make_walk(nt, PARTS, p0, p1);
  Body<m_rows(MQ)> b(smem, Operands{p.X + a0 * p.ldx, p.Gt, p.M + rb * p.m_block_stride, p.bias, p.feat_ok, p.ldx, p.ldg,
                                    p.K, p.mpad},
                     f0, w);
  const RowSide rs = row_side(p.row_ok, nullptr, a0);
  tc5::fence_before();
  __syncthreads();
  tc5::fence_after();
  b.park = park_base(tmem_word, 512);
  b.park_zeros((COMP ? 4 : 2) * MQ);
  while (!w.done()) {
    const int part = w.p;
    b.template run<MQ, COMP ? FF : ADD>(w, rs, p.scale, p.map);
    w.step();
    if (cl > 1 || w.p == part) continue;
    // the part's sum into the totals, and back to zero
#pragma unroll
    for (int q = 0; q < MQ; ++q) {
      float v[8], tot[8];
      unpark8(b.park + 8 * q, v);
      unpark8(b.park + TOT + 8 * q, tot);
      if (COMP) {
        float l[8], tl[8];
        unpark8(b.park + LOW + 8 * q, l);
        unpark8(b.park + TOT + LOW + 8 * q, tl);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          two_sum_into(tot[i], tl[i], v[i]);
          tl[i] = __fadd_rn(tl[i], l[i]);
          l[i] = 0.f;
        }
        park8(b.park + TOT + LOW + 8 * q, tl);
        park8(b.park + LOW + 8 * q, l);
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) tot[i] = __fadd_rn(tot[i], v[i]);
      }
      park8(b.park + TOT + 8 * q, tot);
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = 0.f;
      park8(b.park + 8 * q, v);
    }
    tc5::tmem_wait_st();
  }
  float* out = p.out + j * p.out_block_stride + a0 * p.mpad;
  cp_wait<0>();   // (only empty groups are left)
  if (cl == 1) {
#pragma unroll
    for (int q = 0; q < MQ; ++q) {
      float v[8];
      unpark8(b.park + TOT + 8 * q, v);
      if (COMP) {
        float l[8];
        unpark8(b.park + TOT + LOW + 8 * q, l);
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = __fadd_rn(v[i], l[i]);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) out[(int64_t)chain_row(b.ty, i) * p.mpad + b.tx + 16 * q] = v[i];
    }
    tmem_return(tmem_word, 512);
  } else {
    // this part's sums to shared memory (the ring's), then 16 rows per CTA over all parts
    __syncthreads();   // everyone is done reading the ring
    const int elems = BM * p.mpad;
#pragma unroll
    for (int q = 0; q < MQ; ++q) {
      float v[8];
      unpark8(b.park + 8 * q, v);
#pragma unroll
      for (int i = 0; i < 8; ++i) smem[chain_row(b.ty, i) * p.mpad + b.tx + 16 * q] = v[i];
      if (COMP) {
        unpark8(b.park + LOW + 8 * q, v);
#pragma unroll
        for (int i = 0; i < 8; ++i) smem[elems + chain_row(b.ty, i) * p.mpad + b.tx + 16 * q] = v[i];
      }
    }
    tmem_return_and_meet(tmem_word, 512);
    const int share = elems / cl;
    const uint32_t base = tc5::smem_u32(smem);
    for (int e = (int)rank * share + threadIdx.x; e < ((int)rank + 1) * share; e += NT) {
      float v[PARTS], l[PARTS];
#pragma unroll
      for (int r = 0; r < PARTS; ++r) {
        v[r] = r < cl ? ld_cluster(base + 4 * e, r) : 0.f;
        if (COMP) l[r] = r < cl ? ld_cluster(base + 4 * (elems + e), r) : 0.f;
      }
      float tot = 0.f, tl = 0.f;
#pragma unroll
      for (int r = 0; r < PARTS; ++r) {
        if (COMP) {
          two_sum_into(tot, tl, v[r]);
          tl = __fadd_rn(tl, l[r]);
        } else {
          tot = __fadd_rn(tot, v[r]);
        }
      }
      out[e] = COMP ? __fadd_rn(tot, tl) : tot;
    }
    tc5::cluster_sync_all();   // nobody leaves while others read its shared memory
  }
}

// Pass 1: one CTA per (128 feature slots, row block i, row split); runs over the
// data rows of its split (whole runs of 64 rows) in 128-row tiles, one chain of multiply-adds per
// sum.  Writes R-partials (features x m_pad).
template <int MQ>
__global__ void __launch_bounds__(NT, 1) k_pass1_simt(const __grid_constant__ PassArgs p) {
  extern __shared__ __align__(16) float smem[];
  __shared__ uint32_t tmem_word;
  const int64_t a0 = (int64_t)blockIdx.x * BM;  // feature slot tile
  const int i = blockIdx.y, split = blockIdx.z;
  // column block of this feature tile, and whether it holds any valid feature
  int j = 0;
  while (j + 1 < p.C && p.col_slot[j + 1] <= a0) ++j;
  if (a0 - p.col_slot[j] >= p.col_size[j]) return;
  if (p.bmask && !p.bmask[i * p.C + j]) return;   // inactive block: its partials are not read
  const int64_t nsteps = ceil_div(p.row_size[i], 64);
  const int64_t t0 = split * nsteps / p.nsplit, t1 = (split + 1) * nsteps / p.nsplit;
  const int64_t r0 = p.row_slot[i] + t0 * 64, tiles = ceil_div(t1 - t0, 2);
  const int64_t o = ((int64_t)split * p.R + i) * p.out_block_stride;
  if (!RFF_SPAN(a0, BM, p.g_rows) || !RFF_SPAN(r0, (t1 - t0) * 64, p.x_rows) ||
      !RFF_SPAN(j * p.m_block_stride + r0 * p.mpad, (t1 - t0) * 64 * p.mpad, p.m_elems) ||
      !RFF_SPAN(o + a0 * p.mpad, BM * p.mpad, p.out_elems))
    return;
  if (threadIdx.x < 32) tc5::tmem_alloc<1>(tc5::smem_u32(&tmem_word), 512);
  Walk w = make_walk(tiles, 1, 0, 1);
  Body<m_rows(MQ)> b(smem, Operands{p.Gt + a0 * p.ldg, p.X, p.M + j * p.m_block_stride, nullptr, p.row_ok, p.ldg, p.ldx,
                                    p.K, p.mpad},
                     r0, w, (t1 - t0) % 2 ? 64 : BN);
  const RowSide rs = row_side(p.feat_ok, p.bias, a0);
  tc5::fence_before();
  __syncthreads();
  tc5::fence_after();
  b.park = park_base(tmem_word, 512);
  b.park_zeros(MQ);
  for (; !w.done(); w.step()) b.template run<MQ, CHAIN>(w, rs, p.scale, p.map);
  cp_wait<0>();   // (only empty groups are left)
  float* out = p.out + o + a0 * p.mpad;
#pragma unroll
  for (int q = 0; q < MQ; ++q) {
    float v[8];
    unpark8(b.park + 8 * q, v);
#pragma unroll
    for (int ii = 0; ii < 8; ++ii) out[(int64_t)chain_row(b.ty, ii) * p.mpad + b.tx + 16 * q] = v[ii];
  }
  tmem_return(tmem_word, 512);
}

// half H of T as Z (or Z^T) to out, rows a0.., features b0..
template <int H>
__device__ __forceinline__ void write_z_half(const ZArgs& p, Body<0>& b, const float (&acc)[16][8], int64_t a0,
                                             int64_t b0) {
  __syncthreads();   // the Z tile is free
  store_z<H>(b.ZsT, acc, b.tx, b.ty, b.meta[0], p.feat_ok, row_side(p.row_ok, nullptr, a0), p.scale, p.map);
  __syncthreads();
  const int64_t nr = p.nr - (a0 - p.r0), nf = p.nf - (b0 - p.f0);   // of the window from this tile on
  if (p.trans) {
    float* out = p.out + (b0 - p.f0) * p.ldo + (a0 - p.r0);
    for (int t = threadIdx.x; t < BM * BN; t += NT) {
      const int r = t % BM, c = t / BM;
      if (r < nr && c < nf) out[c * p.ldo + r] = b.ZsT[c * ZLD + r];
    }
  } else {
    float* out = p.out + (a0 - p.r0) * p.ldo + (b0 - p.f0);
    // a warp takes 4 rows x 8 columns at a time: distinct banks, 32-byte runs
    for (int t = threadIdx.x; t < BM * BN; t += NT) {
      const int blk = t / 32, l = t % 32;
      const int r = blk / (BN / 8) * 4 + l / 8, c = blk % (BN / 8) * 8 + l % 8;
      if (r < nr && c < nf) out[r * p.ldo + c] = b.ZsT[c * ZLD + r];
    }
  }
}

// Materialise Z (or Z^T) for rows [r0, r0 + nr) and feature slots [f0, f0 + nf) into
// out (leading dimension ldo); one CTA per 128 rows x 128 `tiles` features (tiles = 1 or 2).
__global__ void __launch_bounds__(NT, 1) k_write_z_simt(const __grid_constant__ ZArgs p, int tiles) {
  extern __shared__ __align__(16) float smem[];
  const int64_t a0 = p.r0 + (int64_t)blockIdx.x * BM, b0 = p.f0 + (int64_t)blockIdx.y * tiles * BN;
  const int wd = tiles == 2 && b0 - p.f0 + BN < p.nf ? 2 : 1;
  Body<0> b(smem, Operands{p.X + a0 * p.ldx, p.Gt, nullptr, p.bias, p.feat_ok, p.ldx, p.ldg, p.K, 0}, b0, make_walk(wd, 1, 0, 1));
  float acc[16][8];
  if (wd == 2) b.form_t<16>(acc);
  else b.form_t<8>(acc);
  cp_wait<0>();
  write_z_half<0>(p, b, acc, a0, b0);
  if (wd == 2) write_z_half<1>(p, b, acc, a0, b0 + BN);
}

template <int MQ>
cudaError_t launch_pass2_mq(const PassArgs& p, int64_t items, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(k_pass2_simt<MQ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
  if (e != cudaSuccess) return e;
  // Whole waves of items go one to a CTA; the rest, which would leave SMs idle for a whole item's
  // time, goes to clusters of PARTS CTAs where those end sooner (an eighth of the tiles per
  // CTA; clusters of eight leave about an eighth of the SMs unused)
  const int64_t nsm = device_sms(), units = p.per_block ? p.C : 1;
  const int64_t nt = ceil_div(p.g_rows / BN, units);   // feature tiles of an item
  int64_t full = items / nsm * nsm, rest = items - full;
  const int cl = nt > 4 ? PARTS : nt > 2 ? 4 : 2;
  const int64_t split_cost = ceil_div(rest * cl, nsm * 7 / 8) * (2 * ceil_div(nt, cl) + 1);
  if (rest > 0 && split_cost >= 2 * nt + 1) {
    full = items;
    rest = 0;
  }
  if (full > 0) {
    k_pass2_simt<MQ><<<(unsigned)full, NT, SMEM, st>>>(p, 0, 1);
    if ((e = cudaGetLastError()) != cudaSuccess || rest == 0) return e;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(rest * cl));
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cl;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_pass2_simt<MQ>, p, full, cl);
}

template <int MQ>
cudaError_t launch_pass1_mq(const PassArgs& p, dim3 grid, cudaStream_t st) {
  const cudaError_t e =
      cudaFuncSetAttribute(k_pass1_simt<MQ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
  if (e != cudaSuccess) return e;
  k_pass1_simt<MQ><<<grid, NT, SMEM, st>>>(p);
  return cudaGetLastError();
}

}  // namespace

#define RFF_MQS RFF_MQ(1) RFF_MQ(2) RFF_MQ(3) RFF_MQ(4) RFF_MQ(5) RFF_MQ(6) RFF_MQ(7) RFF_MQ(8) \
  RFF_MQ(9) RFF_MQ(10) RFF_MQ(11) RFF_MQ(12) RFF_MQ(13) RFF_MQ(14) RFF_MQ(15) RFF_MQ(16)

cudaError_t launch_pass2_simt(const PassArgs& p, int64_t nrow_slots, cudaStream_t st) {
  if (nrow_slots % BM || p.g_rows % BN || p.K % 4 || p.K < 1) return cudaErrorInvalidValue;
  if (nrow_slots <= 0) return cudaSuccess;
  const int64_t items = nrow_slots / BM * (p.per_block ? p.C : 1);
  switch (p.mpad / 16) {
#define RFF_MQ(q) \
  case q:         \
    return launch_pass2_mq<q>(p, items, st);
    RFF_MQS
#undef RFF_MQ
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t launch_pass1_simt(const PassArgs& p, int64_t nfeat_slots, cudaStream_t st) {
  if (nfeat_slots % BM || p.K % 4 || p.K < 1) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)(nfeat_slots / BM), (unsigned)p.R, (unsigned)p.nsplit);
  switch (p.mpad / 16) {
#define RFF_MQ(q) \
  case q:         \
    return launch_pass1_mq<q>(p, grid, st);
    RFF_MQS
#undef RFF_MQ
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t launch_write_z_simt(const ZArgs& p, cudaStream_t st) {
  if (p.nr <= 0 || p.nf <= 0) return cudaSuccess;
  if (p.K % 4 || p.K < 1) return cudaErrorInvalidValue;
  const cudaError_t e = cudaFuncSetAttribute(k_write_z_simt, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
  if (e != cudaSuccess) return e;
  // Two tiles of features to a CTA (the panel of X is read once for both: 20,000 rows at d = 200, 2048
  // features 480 us), unless one each ends within a wave, where a pair is only the longer chain: 500 rows
  // at d = 33, 1000 features 23.8 -> 13.5 us, 1000 rows at d = 200, 2048 features 54 -> 32.  At two
  // waves of single tiles both are alike (5000 rows at d = 64, 512 features: 29 us as pairs).
  const int64_t rows = ceil_div(p.nr, BM), cols = ceil_div(p.nf, BN);
  const int tiles = rows * cols <= device_sms() ? 1 : 2;
  k_write_z_simt<<<dim3((unsigned)rows, (unsigned)ceil_div(cols, tiles)), NT, SMEM, st>>>(p, tiles);
  return cudaGetLastError();
}

RFF_CHECK_UNIT(regen_simt)

}  // namespace rff
