// k_ccl_batch.cu -- labeling many bond masks of different sizes at once.
//
// The tiles of all grids are numbered consecutively (a binary search of the
// grids' tile ranges, which the kernels get by value, maps a global tile to
// its grid), and each step of the stand-alone labeling path (local
// labeling, seam merge, final labels) runs as one launch over all tiles of
// all grids.  A grid's labels are the same as ccl_label gives for it
// alone: every grid has its own label array and scratch, and the steps only
// ever touch the grid of the tile at hand.
#include "label_tile.cuh"

namespace swccl {

__device__ __forceinline__ int job_of_tile(const CclBatchView& v, int gt) {
  int lo = 0, hi = v.n_jobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (gt < v.tile_end[mid]) hi = mid;
    else lo = mid + 1;
  }
  return lo;
}

template <int TH>
__global__ void __launch_bounds__(LABEL_THREADS, LABEL_CTAS_PER_SM) k_cclb_tile(const __grid_constant__ CclBatchView v) {
  __shared__ CclTileSmemT<TH> sm;
  wait_for_previous();
  const int gt = blockIdx.x;
  const CclJob& J = v.jobs[job_of_tile(v, gt)];
  ccl_label_tile<true, TH>(J.mask, J.labels, J.g, J.s, gt - J.tile0, sm);
}

__global__ void __launch_bounds__(MERGE_PER_TILE) k_cclb_merge(const __grid_constant__ CclBatchView v, int per) {
  __shared__ MergeSmem ms;
  wait_for_previous();
  const int gt0 = blockIdx.x * per;
  merge_tiles(ms, min(per, v.n_tiles - gt0),
              [&](int u) {
                const CclJob& J = v.jobs[job_of_tile(v, gt0 + u)];
                return MergeTile{&J.g, J.labels, J.s.seams, J.s.err, gt0 + u - J.tile0};
              },
              v.limit);
}

template <int TH>
__global__ void __launch_bounds__(FINAL_THREADS, FINAL_CTAS) k_cclb_final(const __grid_constant__ CclBatchView v) {
  __shared__ FinalSmem<TH> fs;
  wait_for_previous();
  const int gt = blockIdx.x;
  const CclJob& J = v.jobs[job_of_tile(v, gt)];
  final_labels_tile<TH>(J.labels, J.g, J.s, gt - J.tile0, fs, v.limit);
}

cudaError_t launch_ccl_batch(const CclBatchView& v, cudaStream_t st) {
  if (v.n_tiles == 0) return cudaSuccess;
  const int th = v.jobs[0].g.th;   // of all grids
  auto* tile = th == 8 ? k_cclb_tile<8> : th == 16 ? k_cclb_tile<16> : k_cclb_tile<TILE_H>;
  auto* final_labels = th == 8 ? k_cclb_final<8> : th == 16 ? k_cclb_final<16> : k_cclb_final<TILE_H>;
  cudaError_t e = launch_after(tile, v.n_tiles, LABEL_THREADS, st, v);
  if (e != cudaSuccess) return e;
  const int per = merge_tiles_per_cta(v.n_tiles);
  e = launch_after(k_cclb_merge, (unsigned)((v.n_tiles + per - 1) / per), MERGE_PER_TILE, st, v, per);
  if (e != cudaSuccess) return e;
  return launch_after(final_labels, v.n_tiles, FINAL_THREADS, st, v);
}

}  // namespace swccl
