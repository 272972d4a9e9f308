// fwd_batch.cu -- many frames' tensor-core forwards in one persistent launch
// (ndg_forward_batch); the tile itself is fwd_tile (fwd_h_tile.cuh).
#include "fwd_h_tile.cuh"

namespace ndg {

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long v;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(v));
  return v;
}

// One function per N, not inlined: the register allocation of one N's tile
// code then does not depend on the eleven others' (inlined, addresses of all
// of them were kept live and spilled).
template <int N>
__device__ __noinline__ void fwd_tile_fn(const FwdArgs* args, long long t) {
  const FwdArgs a = *args;
  fwd_tile<N>(a, t);
}

// Persistent CTAs (one per SM) over the (frame, tile) work list of a batch
// of frames of any N <= 12: a CTA takes the next item with an atomic
// cursor, renders that tile with fwd_tile<N> of the item's frame (so a
// frame's outputs equal those of its own fwd_h_kernel launch), and the CTA
// that completes a frame's last tile stamps the frame's completion time.
// Tensor memory is allocated once per CTA and reused by every tile.
__global__ void __launch_bounds__(kFwdThreads, 1) fwd_h_batch_kernel(FwdBatchArgs b) {
  __shared__ long long s_item;
  __shared__ int s_stop;
  const int tid = threadIdx.x;
  if (tid == 0) {
    s_stop = 0;
    if (b.stamps) atomicMin(&b.stamps[0], globaltimer_ns());
  }
  if (tid < 32) {
    tmem_alloc(&fwd_sync().tmem_base, 512);
    tmem_relinquish();
  }
  for (;;) {
    // s_item is rewritten only after the previous tile's closing barrier,
    // which every thread passes after reading it
    if (tid == 0) s_item = s_stop ? b.n_items : (long long)atomicAdd(b.cursor, 1ull);
    __syncthreads();
    const long long item = s_item;
    if (item >= b.n_items) break;
    int f = 0, hi = b.n_frames - 1;  // the frame whose item range holds item
    while (f < hi) {
      const int mid = (f + hi + 1) >> 1;
      if (b.tile_start[mid] <= item) f = mid;
      else hi = mid - 1;
    }
    const long long t = item - b.tile_start[f];
    switch (b.N[f]) {
      case 1: fwd_tile_fn<1>(b.frames + f, t); break;
      case 2: fwd_tile_fn<2>(b.frames + f, t); break;
      case 3: fwd_tile_fn<3>(b.frames + f, t); break;
      case 4: fwd_tile_fn<4>(b.frames + f, t); break;
      case 5: fwd_tile_fn<5>(b.frames + f, t); break;
      case 6: fwd_tile_fn<6>(b.frames + f, t); break;
      case 7: fwd_tile_fn<7>(b.frames + f, t); break;
      case 8: fwd_tile_fn<8>(b.frames + f, t); break;
      case 9: fwd_tile_fn<9>(b.frames + f, t); break;
      case 10: fwd_tile_fn<10>(b.frames + f, t); break;
      case 11: fwd_tile_fn<11>(b.frames + f, t); break;
      case 12: fwd_tile_fn<12>(b.frames + f, t); break;
      default: break;  // the host admits 1 <= N <= 12 only
    }
    if (tid == 0) {
      if (fwd_sync().s_abort) s_stop = 1;  // a timed-out wait: take no further items
      __threadfence();
      const unsigned long long nt = (unsigned long long)(b.tile_start[f + 1] - b.tile_start[f]);
      if (atomicAdd(&b.done[f], 1ull) + 1ull == nt && b.stamps) b.stamps[1 + f] = globaltimer_ns();
    }
  }
  if (tid < 32) {
    fence_after_sync();
    tmem_dealloc(fwd_sync().tmem_base, 512);
  }
}

int launch_fwd_tc_batch(const FwdBatchArgs& b, unsigned smem, int grid, cudaStream_t s) {
  if (b.n_items <= 0 || grid <= 0) return 0;
  cudaFuncSetAttribute(fwd_h_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  fwd_h_batch_kernel<<<(unsigned)grid, kFwdThreads, smem, s>>>(b);
  return 1;
}

}  // namespace ndg
