// k_label.cu -- connected-component labeling of a packed bond mask.
//
// The paper's plan (Sec. II.B, II.C) is kept: label tiles independently,
// then consolidate labels across tile boundaries.  Its tile schemes
// (self-labeling, BFS, serial union-find) and its consolidation schemes
// (relaxation, hierarchical sewing) are replaced:
//
//  k_tile_label   one CTA per TILE_H x TILE_W tile, labeled by the tile engine
//                 (tile_engine.cuh).  Each site's label is the global index of
//                 its tile-local root (the tile component's minimum site index);
//                 roots are appended to a per-tile list, and the labels and
//                 bond bits of the four tile edges go to a compact seam record.
//  k_merge        the bonds leaving a tile (the periodic wrap included,
//                 Sec. II.C): union of the two tile roots on the
//                 global label array with atomicMin hooking.  A lane whose
//                 root pair equals its left neighbour's skips the union, so
//                 consecutive seam bonds of one cluster cost one union.
//  k_root_compress  for every tile root: label = final root (pointer
//                 jumping).  Because hooks always go to the smaller index,
//                 the final root is the cluster's minimum site index.  In a
//                 Swendsen-Wang sweep the final roots also draw their
//                 cluster's new state here (Sec. II.D), keyed by the root.
//  k_site_compress  label[i] = label[label[i]] for every site (the staged
//                 sweep's dump of canonical labels).
// The stand-alone labeling (launch_ccl) uses k_ccl_tile, a k_tile_label that
// keeps every site's tile root as a 16-bit local index in the tile's scratch
// and writes label entries only for the tile roots on the tile edge (their
// parent entries), then k_merge, then k_ccl_final: per tile, each edge root
// finds its cluster root once and every site takes its tile root's label from a
// shared-memory table -- every label written once, no gathers.
#include "label_tile.cuh"

namespace swccl {


__global__ void __launch_bounds__(LABEL_THREADS)
k_tile_label(const uint8_t* __restrict__ mask, int32_t* __restrict__ labels, Grid g, LabelScratch s) {
  __shared__ CclTileSmem sm;
  ccl_label_tile(mask, labels, g, s, blockIdx.x, sm);
}

cudaError_t launch_tile_label(const uint8_t* mask, int32_t* labels, const Grid& g,
                              const LabelScratch& s, cudaStream_t st) {
  k_tile_label<<<g.n_tiles(), LABEL_THREADS, 0, st>>>(mask, labels, g, s);
  return cudaGetLastError();
}

// Stand-alone labeling: local labeling with local-root labels, then (after
// the seam merge) the final labels of every tile in one pass.
template <int TH>
__global__ void __launch_bounds__(LABEL_THREADS, LABEL_CTAS_PER_SM)
k_ccl_tile(const uint8_t* mask, int32_t* labels, Grid g, LabelScratch s) {
  __shared__ CclTileSmemT<TH> sm;
  wait_for_previous();
  ccl_label_tile<true, TH>(mask, labels, g, s, blockIdx.x, sm);
}

template <int TH>
__global__ void __launch_bounds__(FINAL_THREADS, FINAL_CTAS)
k_ccl_final(int32_t* labels, Grid g, LabelScratch s, int limit) {
  __shared__ FinalSmem<TH> fs;
  wait_for_previous();
  final_labels_tile<TH>(labels, g, s, blockIdx.x, fs, limit);
}

cudaError_t launch_ccl(const uint8_t* mask, int32_t* labels, const Grid& g, const LabelScratch& s, cudaStream_t st) {
  auto* tile = g.th == 8 ? k_ccl_tile<8> : g.th == 16 ? k_ccl_tile<16> : k_ccl_tile<TILE_H>;
  auto* final_labels = g.th == 8 ? k_ccl_final<8> : g.th == 16 ? k_ccl_final<16> : k_ccl_final<TILE_H>;
  cudaError_t e = launch_after(tile, g.n_tiles(), LABEL_THREADS, st, mask, labels, g, s);
  if (e != cudaSuccess) return e;
  if ((e = launch_merge(labels, g, s, nullptr, nullptr, 0, 0, st)) != cudaSuccess) return e;
  const int limit = (int)std::min<int64_t>(g.n_sites() + 64, (int64_t)1 << 30);
  return launch_after(final_labels, g.n_tiles(), FINAL_THREADS, st, labels, g, s, limit);
}

// Critical percolation, 128-wide tiles, us per labeling with tiles of
// 32 / 16 / 8 rows: 28 x 64 14.5 / 14.4 / 14.2, 200 x 300 20.1 / 18.1 / 17.1,
// 512^2 21.5 / 19.2 / 18.7, 768^2 (576 tiles of 8 rows) 24.9 / 20.7 / 20.5, 900^2
// (456 of 16, 912 of 8) 26.5 / 22.5 / 23.2, 1280^2 (800 of 16) 27.7 / 24.8 / 31.1,
// 1440^2 (1080 of 16) 27.3 / 26.6 / 36.4, 2048^2 32.7 / 39.6 / 55.6.
int ccl_tile_rows(int64_t tiles8, int64_t tiles16) { return low_tile_rows(tiles8, tiles16); }

// ---------------------------------------------------------------------------
// Seam merge: one CTA per `per` consecutive tiles (merge_tiles).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(MERGE_PER_TILE)
k_merge(int32_t* labels, const __grid_constant__ Grid g, LabelScratch s, int per, int limit, SwCtl* adv,
        int64_t* obs, int obs_cap, int q) {
  __shared__ MergeSmem ms;
  wait_for_previous();
  if (adv && blockIdx.x == 0) {   // end of the drawing step: the next sweep's fills this sweep's observable slot
    const uint64_t sweep = adv->sweep;
    for (int k = threadIdx.x; k <= q; k += MERGE_PER_TILE) obs[(int64_t)(sweep % (uint64_t)obs_cap) * (q + 1) + k] = 0;
    __syncthreads();
    if (threadIdx.x == 0) adv->sweep = sweep + 1;
  }
  const int t0 = blockIdx.x * per;
  merge_tiles(ms, min(per, g.n_tiles() - t0), [&](int u) { return MergeTile{&g, labels, s.seams, s.err, t0 + u}; },
              limit);
}

cudaError_t launch_merge(int32_t* labels, const Grid& g, const LabelScratch& s, SwCtl* adv, int64_t* obs, int obs_cap,
                         int q, cudaStream_t st) {
  const int per = merge_tiles_per_cta(g.n_tiles());
  const int limit = (int)std::min<int64_t>(g.n_sites() + 64, (int64_t)1 << 30);
  return launch_after(k_merge, (unsigned)((g.n_tiles() + per - 1) / per), MERGE_PER_TILE, st, labels, g, s, per, limit,
                      adv, obs, obs_cap, q);
}

cudaError_t load_ccl_kernels() {
  cudaError_t e = cudaSuccess;
  auto load = [&](auto* kernel) {
    cudaFuncAttributes attr;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&attr, kernel);
  };
  load(k_ccl_tile<8>);
  load(k_ccl_tile<16>);
  load(k_ccl_tile<TILE_H>);
  load(k_merge);
  load(k_ccl_final<8>);
  load(k_ccl_final<16>);
  load(k_ccl_final<TILE_H>);
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}

// ---------------------------------------------------------------------------
// Root compression (+ root draws for a Swendsen-Wang sweep).
// ---------------------------------------------------------------------------
constexpr int ROOT_THREADS = 256;

__global__ void __launch_bounds__(ROOT_THREADS)
k_root_compress(int32_t* __restrict__ labels, Grid g, LabelScratch s, int8_t* __restrict__ spins,
                int q, uint64_t seed, const SwCtl* __restrict__ ctl, int limit) {
  root_compress_tile(labels, s, blockIdx.x, spins, q, seed, spins ? ctl->sweep : 0, limit);
}

cudaError_t launch_root_compress(int32_t* labels, const Grid& g, const LabelScratch& s,
                                 int8_t* spins, int q, uint64_t seed, const SwCtl* ctl,
                                 cudaStream_t st) {
  const int limit = (int)std::min<int64_t>(g.n_sites() + 64, (int64_t)1 << 30);
  k_root_compress<<<g.n_tiles(), ROOT_THREADS, 0, st>>>(labels, g, s, spins, q, seed, ctl, limit);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
__global__ void k_site_compress(int32_t* __restrict__ labels, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int r = labels[i];
    const int R = labels[r];
    if (R != r) labels[i] = R;
  }
}

cudaError_t launch_site_compress(int32_t* labels, int64_t n_sites, cudaStream_t st) {
  const int threads = 256;
  const int64_t blocks = std::min<int64_t>((n_sites + threads - 1) / threads, 152 * 32);
  k_site_compress<<<(unsigned)std::max<int64_t>(blocks, 1), threads, 0, st>>>(labels, n_sites);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
int64_t label_scratch_bytes(const Grid& g) {
  auto al = [](int64_t b) { return (b + 255) & ~(int64_t)255; };
  const int64_t nt = g.n_tiles();
  return 2 * al(nt * TILE_SITES * 4) + al(nt * 4) + al(nt * SeamLayout::INTS * 4) + al(4);
}

LabelScratch carve_label_scratch(const Grid& g, void* base, int* err) {
  auto al = [](int64_t b) { return (b + 255) & ~(int64_t)255; };
  const int64_t nt = g.n_tiles();
  char* p = static_cast<char*>(base);
  LabelScratch s;
  s.roots = reinterpret_cast<int32_t*>(p);
  p += al(nt * TILE_SITES * 4);
  s.work = reinterpret_cast<int32_t*>(p);
  p += al(nt * TILE_SITES * 4);
  s.root_counts = reinterpret_cast<int32_t*>(p);
  p += al(nt * 4);
  s.seams = reinterpret_cast<int32_t*>(p);
  p += al(nt * SeamLayout::INTS * 4);
  s.err = err ? err : reinterpret_cast<int*>(p);
  return s;
}

// The stand-alone labeling keeps 16-bit tile roots, edge-root bits and seam
// records only (2.4 bytes per site of the about 8.3 that label_scratch_bytes
// asks a caller for).
int64_t ccl_scratch_bytes(const Grid& g) {
  auto al = [](int64_t b) { return (b + 255) & ~(int64_t)255; };
  const int64_t nt = g.n_tiles(), sites = nt * g.th * TILE_W;
  return al(sites * 2) + al(sites / 8) + al(nt * SeamLayout::INTS * 4);
}

LabelScratch carve_ccl_scratch(const Grid& g, void* base, int* err) {
  auto al = [](int64_t b) { return (b + 255) & ~(int64_t)255; };
  const int64_t sites = (int64_t)g.n_tiles() * g.th * TILE_W;
  char* p = static_cast<char*>(base);
  LabelScratch s;
  s.work = reinterpret_cast<int32_t*>(p);
  p += al(sites * 2);
  s.roots = reinterpret_cast<int32_t*>(p);
  p += al(sites / 8);
  s.seams = reinterpret_cast<int32_t*>(p);
  s.root_counts = nullptr;
  s.err = err;
  return s;
}

}  // namespace swccl
