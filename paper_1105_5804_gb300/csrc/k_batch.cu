// k_batch.cu -- fused Swendsen-Wang sweeps of many independent lattices.
//
// A batch holds R chains of different sizes and temperatures (one SwRep
// each).  Their tiles are numbered consecutively; tile_rep[] maps a global
// tile to its chain.  Two schedules run the same three steps of the fused
// sweep (draw + label, seam merge, flip) over all tiles of all chains:
//
//  * phases: one launch per step over the global tile list (CUDA graph of
//    three kernels per sweep); kernel boundaries order the steps;
//  * persistent: one cooperative launch per sweep.  Each CTA walks the
//    global tile list step by step; a grid barrier separates the steps.  The
//    barrier's wait is bounded: if it does not complete within the time
//    limit, the kernel records SW_ERR_TIMEOUT and returns, so it can never
//    hang the device.
//
// Small lattices alone leave most SMs idle (L = 64 is two tiles); in one
// batch their tiles fill the machine.  Every chain draws from its own seed,
// so a chain's result is the same alone or in any batch.
#include <algorithm>

#include "low_tile.cuh"

namespace swccl {

namespace {

__device__ __forceinline__ bool batch_do_obs(const BatchCtl* ctl, uint64_t sweep) {
  return sweep > 0 && ctl->obs_done != (long long)(sweep - 1);
}

// Zero the observable slot of sweep s of every chain (the next sweep's draw
// step, or the observe kernel, fills it), then advance.  One CTA; the steps after
// it in the sweep count from the advanced counter.
__device__ __forceinline__ void batch_advance_block(const BatchView& b, BatchCtl* ctl, uint64_t s) {
  for (int r = 0; r < b.n_reps; ++r) {
    const SwRep& R = b.reps[r];
    int64_t* slot = R.obs + (int64_t)(s % (uint64_t)b.obs_cap) * (R.q + 1);
    for (int k = threadIdx.x; k <= R.q; k += blockDim.x) slot[k] = 0;
  }
  __syncthreads();
  if (threadIdx.x == 0) ctl->sweep = s + 1;
}

// Grid barrier for co-resident CTAs (cooperative launch).  Returns false if
// the wait ran out (limit_cycles of clock64()) or another CTA already
// failed; the error is recorded.  After a failure the barrier's counters are
// left as they are: the batch is not swept again (the host refuses).
__device__ __forceinline__ bool grid_barrier(BatchCtl* ctl, unsigned nblocks, long long limit_cycles) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    volatile unsigned* gen = &ctl->bar_gen;
    const unsigned my_gen = *gen;
    __threadfence();
    const unsigned arrived = atomicAdd(&ctl->bar_count, 1u) + 1u;
    if (arrived == nblocks) {
      atomicExch(&ctl->bar_count, 0u);
      __threadfence();
      atomicAdd(&ctl->bar_gen, 1u);
    } else {
      // the limit is tested before the flag, so a limit of 0 makes every
      // CTA but the last give up at once
      const long long t0 = clock64();
      for (;;) {
        if (clock64() - t0 >= limit_cycles) {
          atomicCAS(&ctl->err, 0, SW_ERR_TIMEOUT);
          ok = 0;
          break;
        }
        if (*gen != my_gen) break;
        __nanosleep(64);
      }
    }
    __threadfence();
    if (*reinterpret_cast<volatile int*>(&ctl->err) != 0) ok = 0;
  }
  __syncthreads();
  return ok != 0;
}

}  // namespace

// Initial state of every chain: its tiles' blocks (blockIdx.y of them per tile)
// share its sites, four per thread and step (L % 4 == 0), and the clearing of its
// observable ring, 16 bytes per thread and step.  The ring of a chain with many
// states is larger than a small lattice by far, so a batch of few tiles takes
// more blocks per tile, as many as fill the GPU (one chain, L = 16, q = 127,
// created in 37 us, 163 with one block for its 4 MB ring).
__global__ void __launch_bounds__(LABEL_THREADS) k_batch_init(BatchView b, int hot) {
  const SwRep& R = b.reps[b.tile_rep[blockIdx.x]];
  const int64_t tiles = R.g.n_tiles();
  const int64_t i0 = (blockIdx.x - R.tile0 + tiles * blockIdx.y) * LABEL_THREADS + threadIdx.x;
  const int64_t stride = tiles * gridDim.y * LABEL_THREADS;
  for (int64_t i = i0; i < R.g.n_sites() / 4; i += stride) {
    uint32_t w = 0u;
    if (hot) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        w |= (uint32_t)state_of(draw((uint32_t)(4 * i + k), 0, TAG_INIT, R.seed).x, R.q) << (8 * k);
    }
    reinterpret_cast<uint32_t*>(R.spins)[i] = w;
  }
  ulonglong2* ring = reinterpret_cast<ulonglong2*>(R.obs);   // 256-byte aligned, an even number of rows
  for (int64_t i = i0; i < (int64_t)b.obs_cap / 2 * (R.q + 1); i += stride) ring[i] = make_ulonglong2(0ull, 0ull);
}

// ---------------------------------------------------------------------------
// Phase kernels: one CTA per global tile (merge: per few tiles).
__global__ void __launch_bounds__(LABEL_THREADS, LABEL_CTAS_PER_SM) k_batch_label(BatchView b, const BatchCtl* ctl) {
  __shared__ LabelTileSmem ls;
  wait_for_previous();
  const uint64_t sweep = ctl->sweep;
  const bool do_obs = batch_do_obs(ctl, sweep);
  const int gt = blockIdx.x;
  const SwRep& R = b.reps[b.tile_rep[gt]];
  sw_label_tile(R, gt - R.tile0, sweep, do_obs, b.obs_cap, ls, SeedKey{(uint32_t)R.seed, (uint32_t)(R.seed >> 32)});
}

__global__ void __launch_bounds__(MERGE_PER_TILE) k_batch_merge(BatchView b, BatchCtl* ctl, int per) {
  __shared__ MergeSmem ms;
  wait_for_previous();
  if (blockIdx.x == 0) batch_advance_block(b, ctl, ctl->sweep);   // the next draw step fills this sweep's slots
  const int gt0 = blockIdx.x * per;
  merge_tiles(ms, min(per, b.n_tiles - gt0),
              [&](int u) {
                const SwRep& R = b.reps[b.tile_rep[gt0 + u]];
                return MergeTile{&R.g, R.gpar, R.s.seams, R.s.err, gt0 + u - R.tile0};
              },
              b.limit);
}

__global__ void __launch_bounds__(LABEL_THREADS, FLIP_CTAS_PER_SM) k_batch_flip(BatchView b, const BatchCtl* ctl) {
  __shared__ FlipTileSmem fs;
  wait_for_previous();
  const int gt = blockIdx.x;
  const SwRep& R = b.reps[b.tile_rep[gt]];
  sw_flip_tile(R, gt - R.tile0, ctl->sweep - 1, b.limit, fs, SeedKey{(uint32_t)R.seed, (uint32_t)(R.seed >> 32)});
}

// The same over the low tiles of a batch that has few tiles (low_tile.cuh).
// Tile gt of the batch: its chain with the grid and records of its low tiles,
// and the tile's number in the chain.
struct LowChain {
  SwRep R;
  int t;
};
template <int TH>
__device__ __forceinline__ LowChain low_chain(const BatchView& b, const LowBatch& low, int gt) {
  int lo = 0, hi = b.n_reps - 1;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (gt < low.end[mid]) hi = mid;
    else lo = mid + 1;
  }
  LowChain c;
  c.R = b.reps[lo];
  c.R.g.th = TH;
  c.R.g.tiles_y = (c.R.g.H + TH - 1) / TH;
  c.R.s.seams = c.R.s.work;   // see sweep_scratch
  c.t = gt - (lo > 0 ? low.end[lo - 1] : 0);
  return c;
}

template <int TH>
__global__ void __launch_bounds__(LABEL_THREADS)
k_batch_label_low(BatchView b, const __grid_constant__ LowBatch low, const BatchCtl* ctl) {
  __shared__ LowTileSmem<TH> ls;
  const LowChain c = low_chain<TH>(b, low, blockIdx.x);   // tables: not written by the kernels ahead
  wait_for_previous();
  const uint64_t sweep = ctl->sweep;
  sw_label_low_tile(c.R, c.t, sweep, batch_do_obs(ctl, sweep), b.obs_cap, ls,
                    SeedKey{(uint32_t)c.R.seed, (uint32_t)(c.R.seed >> 32)});
}

template <int TH>
__global__ void __launch_bounds__(MERGE_PER_TILE)
k_batch_merge_low(BatchView b, const __grid_constant__ LowBatch low, BatchCtl* ctl) {
  __shared__ MergeSmem ms;
  const LowChain c = low_chain<TH>(b, low, blockIdx.x);
  wait_for_previous();
  if (blockIdx.x == 0) batch_advance_block(b, ctl, ctl->sweep);
  merge_tiles(ms, 1, [&](int) { return MergeTile{&c.R.g, c.R.gpar, c.R.s.seams, c.R.s.err, c.t}; }, b.limit);
}

template <int TH>
__global__ void __launch_bounds__(LABEL_THREADS)
k_batch_flip_low(BatchView b, const __grid_constant__ LowBatch low, const BatchCtl* ctl) {
  __shared__ FlipTileSmemT<TH> fs;
  const LowChain c = low_chain<TH>(b, low, blockIdx.x);
  wait_for_previous();
  sw_flip_tile<TH>(c.R, c.t, ctl->sweep - 1, b.limit, fs, SeedKey{(uint32_t)c.R.seed, (uint32_t)(c.R.seed >> 32)});
}

__global__ void __launch_bounds__(LABEL_THREADS) k_batch_observe(BatchView b, BatchCtl* ctl) {
  __shared__ LabelTileSmem ls;
  const uint64_t done = ctl->sweep - 1;
  const int gt = blockIdx.x;
  const SwRep& R = b.reps[b.tile_rep[gt]];
  observe_tile(R, gt - R.tile0, done, b.obs_cap, ls);
  if (gt == 0 && threadIdx.x == 0) ctl->obs_done = (long long)done;
}

// ---------------------------------------------------------------------------
// Persistent kernel: the whole sweep in one cooperative launch.
union PersistentSmem {
  LabelTileSmem label;
  FlipTileSmem flip;
};

__global__ void __launch_bounds__(LABEL_THREADS, 4 * 256 / TILE_W) k_batch_persistent(BatchView b, BatchCtl* ctl, long long limit_cycles) {
  __shared__ PersistentSmem u;
  const uint64_t sweep = ctl->sweep;
  const bool do_obs = batch_do_obs(ctl, sweep);
  const unsigned nb = gridDim.x;
  // 1. draw bonds and label every tile
  for (int gt = blockIdx.x; gt < b.n_tiles; gt += nb) {
    const SwRep& R = b.reps[b.tile_rep[gt]];
    sw_label_tile(R, gt - R.tile0, sweep, do_obs, b.obs_cap, u.label,
                  SeedKey{(uint32_t)R.seed, (uint32_t)(R.seed >> 32)});
  }
  if (!grid_barrier(ctl, nb, limit_cycles)) return;
  // 2. seam merge: warp w of the CTA takes bonds 32w..32w+31 of a tile
  {
    constexpr int WARPS = LABEL_THREADS / 32, WPT = MERGE_PER_TILE / 32;
    const int64_t n_units = (int64_t)b.n_tiles * WPT;
    for (int64_t unit = (int64_t)blockIdx.x * WARPS + (threadIdx.x >> 5); unit < n_units;
         unit += (int64_t)nb * WARPS) {
      const int gt = (int)(unit / WPT), part = (int)(unit - (int64_t)gt * WPT);
      const SwRep& R = b.reps[b.tile_rep[gt]];
      merge_seam_bond(R.gpar, R.g, R.s, gt - R.tile0, part * 32 + (threadIdx.x & 31), b.limit);
    }
  }
  if (!grid_barrier(ctl, nb, limit_cycles)) return;
  // 3. flip every tile
  for (int gt = blockIdx.x; gt < b.n_tiles; gt += nb) {
    const SwRep& R = b.reps[b.tile_rep[gt]];
    sw_flip_tile(R, gt - R.tile0, sweep, b.limit, u.flip, SeedKey{(uint32_t)R.seed, (uint32_t)(R.seed >> 32)});
  }
  if (!grid_barrier(ctl, nb, limit_cycles)) return;
  if (blockIdx.x == 0) batch_advance_block(b, ctl, sweep);
}

// ---------------------------------------------------------------------------
cudaError_t launch_batch_init(const BatchView& b, int hot, cudaStream_t st) {
  constexpr int BLOCKS = 152 * 8 * 256 / TILE_W, MAX_PER_TILE = 64 * 256 / TILE_W;
  const int per_tile = std::max(1, std::min(MAX_PER_TILE, BLOCKS / b.n_tiles));
  k_batch_init<<<dim3(b.n_tiles, per_tile), LABEL_THREADS, 0, st>>>(b, hot);
  return cudaGetLastError();
}

cudaError_t launch_batch_label(const BatchView& b, const LowBatch& low, BatchCtl* ctl, cudaStream_t st) {
  if (low.th)
    return launch_after(low.th == 8 ? k_batch_label_low<8> : k_batch_label_low<16>, low.n_tiles, LABEL_THREADS, st, b, low,
                        ctl);
  return launch_after(k_batch_label, b.n_tiles, LABEL_THREADS, st, b, ctl);
}

cudaError_t launch_batch_merge(const BatchView& b, const LowBatch& low, BatchCtl* ctl, cudaStream_t st) {
  if (low.th)
    return launch_after(low.th == 8 ? k_batch_merge_low<8> : k_batch_merge_low<16>, low.n_tiles, MERGE_PER_TILE, st, b, low,
                        ctl);
  const int per = merge_tiles_per_cta(b.n_tiles);
  return launch_after(k_batch_merge, (unsigned)((b.n_tiles + per - 1) / per), MERGE_PER_TILE, st, b, ctl, per);
}

cudaError_t launch_batch_flip(const BatchView& b, const LowBatch& low, BatchCtl* ctl, cudaStream_t st) {
  if (low.th)
    return launch_after(low.th == 8 ? k_batch_flip_low<8> : k_batch_flip_low<16>, low.n_tiles, LABEL_THREADS, st, b, low,
                        ctl);
  return launch_after(k_batch_flip, b.n_tiles, LABEL_THREADS, st, b, ctl);
}

cudaError_t launch_batch_observe(const BatchView& b, BatchCtl* ctl, cudaStream_t st) {
  k_batch_observe<<<b.n_tiles, LABEL_THREADS, 0, st>>>(b, ctl);
  return cudaGetLastError();
}

int batch_persistent_blocks_per_sm() {
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_batch_persistent, LABEL_THREADS, 0) != cudaSuccess) return 0;
  return n;
}

cudaError_t launch_batch_persistent(const BatchView& b, BatchCtl* ctl, int blocks, long long limit_cycles,
                                    cudaStream_t st) {
  void* args[] = {(void*)&b, (void*)&ctl, (void*)&limit_cycles};
  return cudaLaunchCooperativeKernel((const void*)k_batch_persistent, dim3(blocks), dim3(LABEL_THREADS), args, 0, st);
}

}  // namespace swccl
