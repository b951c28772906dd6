// Pieces shared by the kernels of the coarse even-odd GMRES: L2-coherent loads,
// the bounded grid barrier, L2 prefetch.
#pragma once

#include "common.cuh"
#include "kernels.h"

namespace ddamg {
namespace {

__device__ __forceinline__ cpx<float> ldc(const cpx<float>* p) {
  float2 t = __ldcg(reinterpret_cast<const float2*>(p));
  return mk(t.x, t.y);
}
__device__ __forceinline__ cpx<double> ldc(const cpx<double>* p) {
  double2 t = __ldcg(reinterpret_cast<const double2*>(p));
  return mk(t.x, t.y);
}

template <class T>
__device__ __forceinline__ T wsum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Grid barrier on a counter that only grows during a launch (zeroed before
// it): at its e-th barrier every CTA adds 1 and waits until the counter
// reaches e * gridDim.x.  The arrival is a fence followed by a relaxed
// reduction (no reply awaited), the wait an acquire load, so a barrier costs
// about one L2 round trip after the last arrival.  The wait is bounded (about
// a second); on time-out the CTA records DDAMG_ETIMEOUT and leaves, and the
// CTAs still waiting for it then time out at this or their next barrier.
__device__ inline unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__shared__ unsigned bar_epoch;       // barriers passed by this CTA in this launch

// thread 0 zeroes the count at kernel entry (a __syncthreads must follow
// before the first barrier)
__device__ inline void grid_barrier_reset() {
  if (threadIdx.x == 0) bar_epoch = 0;
}

// Split form: grid_arrive publishes this CTA's writes and counts it in;
// grid_wait returns once every CTA has arrived.  Between the two a CTA may do
// work that touches only its own shared memory and registers.
__device__ inline void grid_arrive(unsigned* bar) {
  __syncthreads();
  if (threadIdx.x == 0) {
    ++bar_epoch;
    __threadfence();                 // the CTA's writes (ordered by the bar.sync above) first
    asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
  }
}

__device__ inline bool grid_wait(unsigned* bar, int* status, long long limit) {
  __shared__ int ok_s;
  if (threadIdx.x == 0) {
    const unsigned target = bar_epoch * gridDim.x;
    int ok = 1;
    long long spins = 0;
    while ((int)(ld_acquire_gpu(bar) - target) < 0) {
      if (++spins > limit) {
        atomicExch(status, 6);
        ok = 0;
        break;
      }
    }
    ok_s = ok;
  }
  __syncthreads();
  return ok_s != 0;
}

__device__ inline bool grid_barrier(unsigned* bar, int* status, long long limit) {
  grid_arrive(bar);
  return grid_wait(bar, status, limit);
}

// L2 prefetch of `bytes` bytes at p (16-byte aligned, a multiple of 16) by
// the calling warp, in bulk prefetches of at most 32 KB per lane: the block
// operators of the next coarse site travel from HBM while this site's block
// product runs
__device__ __forceinline__ void prefetch_l2(const void* p, size_t bytes) {
  constexpr size_t PIECE = 32768;
  for (size_t off = (size_t)(threadIdx.x & 31) * PIECE; off < bytes; off += 32 * PIECE) {
    const size_t n = bytes - off < PIECE ? bytes - off : PIECE;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(static_cast<const char*>(p) + off),
                 "r"((unsigned)n)
                 : "memory");
  }
}

__host__ __device__ inline size_t al16(size_t v) { return (v + 15) / 16 * 16; }

}  // namespace

// the form for many right-hand sides (kernels_cgmres_wide.cu): its launch
// configuration (NR 0 where it does not apply), and its launch with
// work_bytes bytes of scratch
struct WideChoice {
  int NR, G, per, slots;
  size_t smem_bytes, work_bytes;
};
WideChoice cgmres_wide_choose(int dev, const Geom& g, int n2, int m, int nrhs);
cudaError_t cgmres_wide_launch(const WideChoice& c, const Geom& g, const CoarseSolveArgs& ca, const float* b, float* x,
                               int nrhs, void* work, int* iters, int* iters_acc, int* status, cudaStream_t st);

}  // namespace ddamg
