// frames_batched128.cu -- the M = 128 problems of a batched call in one
// persistent launch of the exchange-schedule kernel (frames_x3.cuh): the
// problems' frames, each problem's in its column-strip order, are one
// sequence that the blocks cut into equal runs; a block's run crosses into
// another problem a few times at most, and starts that problem as a launch of
// its own would (arguments, window, first copies).  Against one launch per
// problem this saves the launches' tails; against the thread-pair layout it
// replaces (64 values a thread, spills, per-element copies) the batch of 16
// problems went 5.21 -> 2.76 ms with the two fused launches around it
// (object_build_batch_kernel, finish_batch_kernel; one launch per problem: 3.01).
#include "frames_launch.h"
#include "frames_x3.cuh"

namespace mpbp {

namespace {

__global__ void __launch_bounds__(X3Cfg::T, 1) frames_x3_batch(const __grid_constant__ BatchArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[X3Cfg::T / 32];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_base;
  __shared__ X3Tables tab;
  __shared__ FrameArgs sp;   // the current problem's arguments
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i < a.nprob; i += blockDim.x)
      if (a.probs[i].arrivals) *a.probs[i].arrivals = 0u;
  X3Block b;
  x3_begin<true>(b, smem_raw, &mbar, &tmem_base, tab);
  const long long lo = (long long)a.nitems * blockIdx.x / gridDim.x;
  const long long hi = (long long)a.nitems * (blockIdx.x + 1) / gridDim.x;
  for (int k = 0; k < a.nprob; ++k) {
    const long long f0 = a.frame_base[k], n = a.probs[k].nframes;
    const int l = (int)(lo > f0 ? lo - f0 : 0);
    const int h = (int)(hi - f0 < n ? hi - f0 : n);
    double tot = 0.0;
    if (l < h && b.bs.ok) {
      constexpr int W = (int)(sizeof(FrameArgs) / sizeof(unsigned));
      static_assert(sizeof(FrameArgs) % sizeof(unsigned) == 0 && W <= X3Cfg::T, "word copy");
      if (threadIdx.x < W)
        reinterpret_cast<unsigned*>(&sp)[threadIdx.x] = reinterpret_cast<const unsigned*>(&a.probs[k])[threadIdx.x];
      tmem_fence_before_sync();   // the last run's window is read out before this one clears it
      __syncthreads();
      tmem_fence_after_sync();
      const double lsum = sp.bgT ? x3_run<true, false, true, false, false>(sp, a.tmaps + k, l, h, b, tab)
                                 : x3_run<true, false, false, false, false>(sp, a.tmaps + k, l, h, b, tab);
      tot = block_sum_d<X3Cfg::T>(lsum, red);   // barriers: sp may be overwritten
    } else if (l < h && threadIdx.x == 0) {
      // a wait ran out in an earlier problem: this one misses the block's frames too
      atomicOr(a.probs[k].err, kErrTimeout);
    }
    // every (problem, block) slot is written, so none needs clearing
    if (threadIdx.x == 0) a.frame_part[(long long)k * gridDim.x + blockIdx.x] = tot;
  }
  x3_end(b);
}

}  // namespace

bool batched128_prepare(int* blocks_per_sm) {
  *blocks_per_sm = 1;
  return cudaFuncSetAttribute(frames_x3_batch, cudaFuncAttributeMaxDynamicSharedMemorySize, X3Cfg::SMEM) == cudaSuccess;
}

cudaError_t batched128_launch(const BatchArgs& a, int grid, cudaStream_t s) {
  frames_x3_batch<<<grid, X3Cfg::T, X3Cfg::SMEM, s>>>(a);
  return cudaGetLastError();
}

}  // namespace mpbp
