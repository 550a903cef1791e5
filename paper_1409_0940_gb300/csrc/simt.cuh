// Shared pieces of the FP32 SIMT kernels (regen_simt.cu, dense.cu): the thread layout of their
// 256-thread CTAs, asynchronous copies into a ring of shared-memory stages, and tensor memory as
// a per-thread parking place for accumulators.
//
// Thread layout: threads (ty, tx) in 16 x 16, a warp covering 4 ty x 8 tx, so that a warp's
// fragment reads are 4 or 8 distinct addresses on distinct banks, broadcast to the other lanes.
//
// Parking: a thread's 8 x 8 accumulators of one product, the fragments it multiplies and the
// accumulators of a second product do not fit in 255 registers together.  What a phase does not
// touch waits in tensor memory (256 words per thread of a 256-thread CTA that holds all 512
// columns: warp w owns the lanes 32 (w mod 4) .. and the columns from 256 (w / 4)); the words are
// private to the thread, so only its own stores and loads have to be ordered.
//
// Clusters and tensor memory: a CTA whose columns are taken waits in tcgen05.alloc until their
// holders give them back.  CTAs of two kernels that both held columns while they waited for the rest
// of their clusters could wait for one another on two SMs without end.  So a CTA of a cluster gives
// its columns back before it first waits for the cluster (tmem_return_and_meet): whoever holds columns
// finishes on its own, whatever else shares the SM.  (The tensor-core passes' CTA pairs hold theirs to
// the end: no two of them fit an SM's shared memory.)
#pragma once
#include "common.cuh"
#include "tcgen05.cuh"

namespace rff {
namespace simt {

constexpr int NT = 256;
// row stride (words) of a K-contiguous stage tile of BK elements a row, BK = 16 or 32: the 16-byte
// pieces of 8 consecutive rows lie on distinct banks
constexpr int row_stride(int bk) { return bk + 4; }

__device__ __forceinline__ int thread_ty() {
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  return (w >> 1) * 4 + (l >> 3);
}
__device__ __forceinline__ int thread_tx() {
  const int w = threadIdx.x / 32, l = threadIdx.x % 32;
  return (w & 1) * 8 + (l & 7);
}

__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc5::smem_u32(dst)), "l"(src) : "memory");
}
// bytes < 16: the rest of the 16 are zeros
__device__ __forceinline__ void cp_async16_fill(float* dst, const float* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(tc5::smem_u32(dst)), "l"(src), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(tc5::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// tensor memory of this thread: base address for words 0, 1, ... (cols: columns of the CTA)
__device__ __forceinline__ uint32_t park_base(uint32_t tmem, uint32_t cols) {
  const uint32_t w = threadIdx.x / 32;
  return tmem + ((w & 3) << 21) + (w >> 2) * (cols / 2);
}
__device__ __forceinline__ void park8(uint32_t taddr, const float (&v)[8]) { tc5::tmem_st8(taddr, v); }
__device__ __forceinline__ void unpark8(uint32_t taddr, float (&v)[8]) {   // complete after tmem_wait_ld
  uint32_t r[8];
  tc5::tmem_ld8(taddr, r);
  tc5::tmem_wait_ld();
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// every thread is done with the CTA's tensor memory: warp 0 gives it back
__device__ __forceinline__ void tmem_return(uint32_t tmem, uint32_t cols) {
  tc5::fence_before();
  __syncthreads();
  tc5::fence_after();
  if (threadIdx.x < 32) tc5::tmem_dealloc<1>(tmem, cols);
}

// the same, and the cluster is met: the columns go back while the others arrive
__device__ __forceinline__ void tmem_return_and_meet(uint32_t tmem, uint32_t cols) {
  tc5::fence_before();
  __syncthreads();
  tc5::fence_after();
  tc5::cluster_arrive();
  if (threadIdx.x < 32) tc5::tmem_dealloc<1>(tmem, cols);
  tc5::cluster_wait();
}

__device__ __forceinline__ float ld_cluster(uint32_t addr, uint32_t rank) {   // a CTA's shared memory in the cluster
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(tc5::mapa_rank(addr, rank)) : "memory");
  return v;
}

}  // namespace simt
}  // namespace rff
