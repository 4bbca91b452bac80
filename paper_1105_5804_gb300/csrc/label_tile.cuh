// label_tile.cuh -- per-tile bodies of the stand-alone labeling path, shared
// by the single-grid kernels (k_label.cu) and the batched kernels over many
// grids (k_ccl_batch.cu): local labeling of a tile from the packed mask, root
// compression of a tile's root list, and the site pass that makes a tile's
// labels canonical.
#pragma once
#include "tile_engine.cuh"

namespace swccl {

// The even bits of a 64-bit word, packed into 32 bits (bit 2i -> bit i).
__device__ __forceinline__ uint32_t even_bits(unsigned long long x) {
  x &= 0x5555555555555555ull;
  x = (x | (x >> 1)) & 0x3333333333333333ull;
  x = (x | (x >> 2)) & 0x0F0F0F0F0F0F0F0Full;
  x = (x | (x >> 4)) & 0x00FF00FF00FF00FFull;
  x = (x | (x >> 8)) & 0x0000FFFF0000FFFFull;
  x = (x | (x >> 16)) & 0x00000000FFFFFFFFull;
  return (uint32_t)x;
}

// Mask bits of `nvalid` (1..32) consecutive sites from site0 on, site i in bits
// 2i (east) and 2i + 1 (north), the rest zero.  One 64-bit load where the
// sites start on a 32-site word; else three 32-bit words shifted into place
// (rows of any width start anywhere in a byte); single bytes only for a mask
// that is not 4-byte aligned and in its last word.
__device__ __forceinline__ unsigned long long mask_word(const uint8_t* __restrict__ mask, int64_t n_bytes,
                                                        int64_t site0, int nvalid) {
  const int64_t b0 = site0 >> 2;
  unsigned long long wd = 0ull;
  if ((site0 & 31) == 0 && (reinterpret_cast<uintptr_t>(mask) & 7) == 0 && b0 + 8 <= n_bytes) {
    wd = *reinterpret_cast<const unsigned long long*>(mask + b0);
  } else {
    const int off = 2 * (int)(site0 & 15);                  // first bit in its 32-bit word
    const int n_words = (off + 2 * nvalid + 31) >> 5;       // 1..3
    const int64_t w0 = site0 >> 4;
    if ((reinterpret_cast<uintptr_t>(mask) & 3) == 0 && 4 * (w0 + n_words) <= n_bytes) {
      const uint32_t* p = reinterpret_cast<const uint32_t*>(mask) + w0;
      const uint32_t a = p[0], b = n_words > 1 ? p[1] : 0u, c = n_words > 2 ? p[2] : 0u;
      wd = (unsigned long long)__funnelshift_r(a, b, off) | (unsigned long long)__funnelshift_r(b, c, off) << 32;
    } else {
      for (int i = 0; i < nvalid; ++i) wd |= (unsigned long long)site_bits(mask, site0 + i) << (2 * i);
    }
  }
  return nvalid < 32 ? wd & ((1ull << (2 * nvalid)) - 1ull) : wd;
}

// Local labeling of one tile for the stand-alone labeling path: every thread
// takes the bond bits of its row of its strip from the packed mask (bits of
// sites outside the grid and the east bond of the tile's last column
// cleared), the engine of tile_engine.cuh labels the tile, and the warps
// write their strips' labels (global index of the tile root, the minimum
// site index of its tile component), the tile's root list, and the seam
// record (labels and outgoing bond bits of the four tile edges).
// LOCAL (the stand-alone labeling path, finished by final_labels_tile): the
// label array receives only the parent entries of the tile roots whose
// component reaches the tile edge (label = own global index), which the
// seam merge and the final root walks use; every site's tile root goes, as
// a 16-bit local index, to the tile's slot of `work`, in tile row-major order;
// the root list holds local indices, with CCL_EDGE_ROOT set on the edge
// roots.  final_labels_tile writes every site's label.
constexpr int CCL_EDGE_ROOT = 1 << 30;
struct CclTileSmem {
  TileSmem tile;
  uint32_t edge_bits[TILE_SITES / 32];   // local roots on the tile edge
};
static_assert(TILE_SITES / 32 == LABEL_THREADS, "one edge word per thread");

template <bool LOCAL = false>
__device__ __forceinline__ void ccl_label_tile(const uint8_t* __restrict__ mask, int32_t* __restrict__ labels,
                                               const Grid& g, const LabelScratch& s, int t, CclTileSmem& cs) {
  TileSmem& sm = cs.tile;
  const uint16_t* par = sm.par;
  int* warp_roots = sm.warp_roots;

  const int ty = t / g.tiles_x, tx = t - ty * g.tiles_x;
  const int y0 = ty * TILE_H, x0 = tx * TILE_W;
  const int h = min(TILE_H, g.H - y0), w = min(TILE_W, g.W - x0);
  const int W = g.W;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int32_t* slot = s.roots + (int64_t)t * TILE_SITES;     // the root list
  cs.edge_bits[threadIdx.x] = 0u;                        // the engine's barriers order it before the marks

  // 1. bond bits of row `lane` of strip `warp`
  const int nvalid = min(max(w - 32 * warp, 0), 32);
  uint32_t we = 0u, wn = 0u, e_last = 0u;
  if (lane < h && nvalid > 0) {
    const unsigned long long wd =
        mask_word(mask, (g.n_sites() + 3) >> 2, (int64_t)(y0 + lane) * W + x0 + 32 * warp, nvalid);
    we = even_bits(wd);        // the mask interleaves east (even) and north (odd) bits
    wn = even_bits(wd >> 1);
  }
  if (nvalid > 0 && 32 * warp + nvalid == w) {   // east bonds leaving the tile
    const uint32_t bit = 1u << (nvalid - 1);
    e_last = __ballot_sync(FULL, (we & bit) != 0u);
    we &= ~bit;
  }

  // 2-4a. label the tile
  tile_engine(sm, we, wn, h, w, s.err);

  // 4b. the roots of my strip's sites, eight consecutive sites per thread and
  //     step, four threads a row.  LOCAL: as 16-bit local indices into the
  //     tile's slot of `work`.  Otherwise as global labels.  Bit 4j + k of mine
  //     flags site 2k of step j as a root, bit 16 + 4j + k site 2k + 1.
  const int lx0 = 32 * warp + 8 * (lane & 3);
  const int in = min(max(w - lx0, 0), 8);   // columns past the grid are no roots of the tile
  const uint32_t in_mask = ((1u << ((in + 1) >> 1)) - 1u) | ((1u << (in >> 1)) - 1u) << 16;
  uint16_t* lr = reinterpret_cast<uint16_t*>(s.work + (int64_t)t * TILE_SITES);
  uint32_t mine = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int ly = (lane >> 2) + 8 * j;
    if (ly >= h || in == 0) continue;   // the engine wrote no entries there
    const int sidx = local_of(ly, lx0);
    const uint4 r = roots_of(par, sidx);
    if (LOCAL) *reinterpret_cast<uint4*>(lr + ly * TILE_W + lx0) = r;
    const uint32_t own = (uint32_t)sidx * 0x00010001u + 0x00010000u;   // (sidx, sidx + 1)
    const uint32_t wv[4] = {r.x, r.y, r.z, r.w};
    uint32_t m = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) m |= zero_halves(wv[k] ^ (own + (uint32_t)k * 0x00020002u)) >> (15 - k);
    mine |= (m & in_mask) << (4 * j);
    if (!LOCAL) {
      int32_t* dst = labels + (int64_t)(y0 + ly) * W + x0 + lx0;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (k < in) dst[k] = tile_global((int)(wv[k >> 1] >> (16 * (k & 1)) & 0xFFFFu), y0, x0, W);
    }
  }

  // 5. my strip's part of the seam record; parent entries of edge roots; edge
  //    roots marked
  seam_strip(sm, s.seams + (int64_t)t * SeamLayout::INTS, labels, cs.edge_bits, wn, e_last, h, w, y0, x0, W);

  // 6. root list
  int cnt = __popc(mine), incl = cnt;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int v = __shfl_up_sync(FULL, incl, d);
    if (lane >= d) incl += v;
  }
  if (lane == 31) warp_roots[warp] = incl;
  __syncthreads();
  int base = 0, total = 0;
#pragma unroll
  for (int k = 0; k < LABEL_THREADS / 32; ++k) {
    const int c = warp_roots[k];
    base += (k < warp) ? c : 0;
    total += c;
  }
  base += incl - cnt;
  while (mine) {
    const int b = __ffs(mine) - 1;
    mine &= mine - 1;
    const int jk = b & 15;
    const int sidx = local_of((lane >> 2) + 8 * (jk >> 2), lx0) + 2 * (jk & 3) + (b >> 4);
    if (LOCAL) slot[base++] = sidx | (((cs.edge_bits[sidx >> 5] >> (sidx & 31)) & 1u) ? CCL_EDGE_ROOT : 0);
    else slot[base++] = tile_global(sidx, y0, x0, W);
  }
  if (threadIdx.x == 0) s.root_counts[t] = total;
  __syncthreads();
}

// Tile t's roots: label = final root; in a Swendsen-Wang sweep (spins set)
// final roots also draw their cluster's new state.  All threads call it.
__device__ __forceinline__ void root_compress_tile(int32_t* __restrict__ labels, const LabelScratch& s, int t,
                                                   int8_t* __restrict__ spins, int q, uint64_t seed, uint64_t sweep,
                                                   int limit) {
  const int n = __ldcg(s.root_counts + t);
  const int32_t* list = s.roots + (int64_t)t * TILE_SITES;
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const int r = __ldcg(list + k);
    const int R = g_find(labels, r, limit, s.err);
    if (R != r) atomicMin(labels + r, R);
    if (spins && R == r) spins[r] = (int8_t)state_of(draw((uint32_t)r, sweep, TAG_FLIP, seed).x, q);
  }
}

// Site pass of tile t: every label of the tile points at a tile root whose
// entry holds the final root after root compression; one jump makes the
// label canonical.
__device__ __forceinline__ void site_compress_tile(int32_t* __restrict__ labels, const Grid& g, int t) {
  const int ty = t / g.tiles_x, tx = t - ty * g.tiles_x;
  const int y0 = ty * TILE_H, x0 = tx * TILE_W;
  const int h = min(TILE_H, g.H - y0), w = min(TILE_W, g.W - x0);
  for (int k = threadIdx.x; k < TILE_SITES; k += blockDim.x) {
    const int ly = k >> TILE_W_LOG2, lx = k & (TILE_W - 1);
    if (ly < h && lx < w) {
      int32_t* p = labels + (int64_t)(y0 + ly) * g.W + x0 + lx;
      const int r = __ldcg(p);
      const int R = __ldcg(labels + r);
      if (R != r) *p = R;
    }
  }
}

// Final labels of tile t for the stand-alone path (after the seam merge, on
// what ccl_label_tile<true> wrote): each tile root (local root list) finds
// its cluster root R on the label array and stores it in `table` at its
// local index; then every site of the tile takes table[its tile root].
// A tile root's entry receives R (smaller than any value other walks may
// store there), so walks of other tiles through it stay valid.  All threads
// of the CTA call it; it synchronises the CTA.
__device__ __forceinline__ void final_labels_tile(int32_t* labels, const Grid& g, const LabelScratch& s, int t,
                                                  int32_t* table /* shared, TILE_SITES */, int limit) {
  const int ty = t / g.tiles_x, tx = t - ty * g.tiles_x;
  const int y0 = ty * TILE_H, x0 = tx * TILE_W;
  const int h = min(TILE_H, g.H - y0), w = min(TILE_W, g.W - x0);
  const int n = __ldcg(s.root_counts + t);
  const int32_t* list = s.roots + (int64_t)t * TILE_SITES;
  // 1. cluster roots of the tile roots: a root whose component stays inside
  //    the tile is its cluster's root; the others walk the label array, four
  //    walks of a thread in flight together
  constexpr int U = 4;
  for (int k0 = threadIdx.x; k0 < n; k0 += U * (int)blockDim.x) {
    int r[U], x[U];
    bool act[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = k0 + u * (int)blockDim.x;
      const int raw = k < n ? __ldcg(list + k) : 0;
      r[u] = raw & ~CCL_EDGE_ROOT;   // local index
      act[u] = k < n && (raw & CCL_EDGE_ROOT);
      x[u] = tile_global(r[u], y0, x0, g.W);
    }
    g_find_multi<U>(labels, x, act, limit, s.err);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (k0 + u * (int)blockDim.x < n) table[r[u]] = x[u];
  }
  __syncthreads();
  // 2. every site takes its tile root's cluster root; the tile roots are the
  //    16-bit local indices ccl_label_tile<true> left in the tile's slot
  //    of `work`, eight sites per 16-byte word, in tile row-major order; labels go
  //    out four sites per 16-byte store when rows start 16-byte aligned (a
  //    16-byte aligned array and W % 4 == 0; x0 is a multiple of TILE_W, so w
  //    is a multiple of 4 too)
  const uint16_t* lr = reinterpret_cast<const uint16_t*>(s.work + (int64_t)t * TILE_SITES);
  if ((g.W & 3) == 0 && (reinterpret_cast<uintptr_t>(labels) & 15) == 0) {
    for (int k = threadIdx.x; k < TILE_SITES / 8; k += blockDim.x) {
      const int sidx = 8 * k;
      const int ly = sidx >> TILE_W_LOG2, lx = sidx & (TILE_W - 1);
      if (ly >= h || lx >= w) continue;
      const uint4 v = __ldcg(reinterpret_cast<const uint4*>(lr + sidx));
      int32_t* p = labels + (int64_t)(y0 + ly) * g.W + x0 + lx;
      *reinterpret_cast<int4*>(p) =
          make_int4(table[v.x & 0xFFFFu], table[v.x >> 16], table[v.y & 0xFFFFu], table[v.y >> 16]);
      if (lx + 8 <= w)
        *reinterpret_cast<int4*>(p + 4) =
            make_int4(table[v.z & 0xFFFFu], table[v.z >> 16], table[v.w & 0xFFFFu], table[v.w >> 16]);
    }
  } else {
    for (int k = threadIdx.x; k < TILE_SITES; k += blockDim.x) {
      const int ly = k >> TILE_W_LOG2, lx = k & (TILE_W - 1);
      if (ly < h && lx < w) labels[(int64_t)(y0 + ly) * g.W + x0 + lx] = table[__ldcg(lr + k)];
    }
  }
  __syncthreads();
}

}  // namespace swccl
