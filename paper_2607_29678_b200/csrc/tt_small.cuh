// A small text in one launch: the three kernels of a request as phases of one thread-block cluster.
//
// A text of a few tiles is nothing but a chain of dependent steps, and a good part of it was the way from one kernel to the
// next: the grid's end, the next one's release, its first loads.  A cluster's CTAs are placed together and wait for each other by a
// hardware barrier, so the phases follow without the GPU's scheduler in between.  Same code, same records in the workspace.
#pragma once
#include "tt_pretok_kernels.cuh"

// What bounds it is that chain: 4,000 characters take 6.5 us to the end of the look-ups, 8 to the end of the slowest piece's merges and 4
// for the scatter, 0.7 for each barrier.  Measured against three launches (us a call, back to back): 1,000 characters 22.9 ->
// 19.0, 4,000 20.8 -> 19.4, 8,000 of transcripts 20.7 -> 19.9, a conversation of 17 appends 866 -> 810-823.
// CTAs of the cluster: 16 (the largest; the device is asked whether it can place it) rather than the portable 8, because a text with many
// unsettled pieces needs the warps (8,000 characters with 4,096 merges: three launches 21.1, 8 CTAs 24.3, 16 CTAs 19.9).
// Tiles: 4, where 16 CTAs have as many warps as such a text has pieces; with 8 tiles (15,000 characters) it took 24.0, three launches 21.2.
constexpr int SMALL_CTAS = 16, SMALL_TILES = 4;
static_assert(SMALL_TILES <= SMALL_CTAS, "a CTA per tile");
constexpr size_t SMALL_SMEM_BYTES = MERGE_SMEM_REQUEST;
template <int PAT> using SmallFront = PretokShared<true, MERGE_THREADS, PAT>;
typedef ScatterShared<MERGE_THREADS> SmallScatter;

// All CTAs of the cluster are here, and what they wrote before is seen by all of them behind it.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

template <int PAT>
__global__ void __launch_bounds__(MERGE_THREADS, 1)
k_small(const __grid_constant__ PretokParams P, const __grid_constant__ FrontParams F, const __grid_constant__ PieceParams Q, const __grid_constant__ ScatterParams S) {
    extern __shared__ __align__(16) u64 s_buf[];              // SMALL_SMEM_BYTES, used by one phase after the other
    __shared__ u32 sc[SCR_WORDS];
    __shared__ LongShared LS;
    static_assert(sizeof(SmallFront<PAT>) <= SMALL_SMEM_BYTES && sizeof(SmallScatter) <= SMALL_SMEM_BYTES, "the phases share the buffer");
    cudaGridDependencySynchronize();                         // what was enqueued before this call is complete
    cudaTriggerProgrammaticLaunchCompletion();               // (not earlier: the calls behind this one would be placed one after the other, all waiting)
    pretok_tiles<true, MERGE_THREADS, PAT>(P, F, *reinterpret_cast<SmallFront<PAT>*>(s_buf));
    cluster_sync();
    merge_request(Q, s_buf, sc, LS);
    cluster_sync();
    scatter_tiles<MERGE_THREADS>(S, *reinterpret_cast<SmallScatter*>(s_buf));
}
