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
__device__ __forceinline__ unsigned long long mask_word(const uint8_t* mask, int64_t n_bytes,
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

// Local labeling of one tile from a bond mask: every thread takes the bond bits
// of its row of its strip (bits of sites outside the grid and the east bond of
// the tile's last column cleared), the engine of tile_engine.cuh labels the
// tile, and the warps write their strips' sites and seam records (labels and
// outgoing bond bits of the four tile edges).
// LOCAL (the stand-alone labeling, finished by final_labels_tile): the label
// array receives only the parent entries of the tile roots whose component
// reaches the tile edge (label = own global index), which the seam merge and
// the final walks use; every site's tile root goes, as a 16-bit local index, to
// the tile's slot of `work`, in tile row-major order, and the edge-root bits to
// its slot of `roots`.
// Otherwise (the staged sweep) every site's label is written (global index of
// the tile root, the minimum site index of its tile component), and the tile's
// root list.
// Tile t's tile roots and edge-root bits in the scratch of the stand-alone
// labeling (carve_ccl_scratch); TH: rows of a tile.
template <int TH>
__device__ __forceinline__ uint16_t* ccl_roots(const LabelScratch& s, int t) {
  return reinterpret_cast<uint16_t*>(s.work) + (int64_t)t * (TH * TILE_W);
}
template <int TH>
__device__ __forceinline__ int32_t* ccl_edges(const LabelScratch& s, int t) {
  return s.roots + (int64_t)t * (TH * TILE_W / 32);
}

template <int TH>
struct CclTileSmemT {
  TileSmemT<TH> tile;
  uint32_t edge_bits[TH * TILE_W / 32];   // local roots on the tile edge
};
using CclTileSmem = CclTileSmemT<TILE_H>;
static_assert(TILE_SITES / 32 == LABEL_THREADS, "at most one edge word per thread");

template <bool LOCAL = false, int TH = TILE_H>
__device__ __forceinline__ void ccl_label_tile(const uint8_t* mask, int32_t* labels,
                                               const Grid& g, const LabelScratch& s, int t, CclTileSmemT<TH>& cs) {
  TileSmemT<TH>& sm = cs.tile;
  const uint16_t* par = sm.par;
  int* warp_roots = sm.warp_roots;

  const int ty = t / g.tiles_x, tx = t - ty * g.tiles_x;
  const int y0 = ty * TH, x0 = tx * TILE_W;
  const int h = min(TH, g.H - y0), w = min(TILE_W, g.W - x0);
  const int W = g.W;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x < TH * TILE_W / 32) cs.edge_bits[threadIdx.x] = 0u;                        // the engine's barriers order it before the marks

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

  // 4b. the roots of my strip's sites.  LOCAL: as 16-bit local indices into the
  //     tile's slot of `work`, eight consecutive sites per thread and step, four
  //     threads a row.  Otherwise as global labels, a lane per column, so that a
  //     warp stores a row's 32 labels as one line (eight consecutive labels per
  //     lane, stored one by one, touch 32 sectors a store: a staged sweep at
  //     L = 2048 85.3 us instead of 74.4); bit ly of mine flags site ly of my
  //     column as a root.
  uint32_t mine = 0;
  if (LOCAL) {
    const int lx0 = 32 * warp + 8 * (lane & 3);
#pragma unroll
    for (int j = 0; j < TH / 8; ++j) {
      const int ly = (lane >> 2) + 8 * j;
      if (ly >= h || lx0 >= w) continue;   // the engine wrote no entries there
      *reinterpret_cast<uint4*>(ccl_roots<TH>(s, t) + ly * TILE_W + lx0) = roots_of(par, local_of(ly, lx0));
    }
  } else if (32 * warp + lane < w) {
    int32_t* dst = labels + (int64_t)y0 * W + x0 + 32 * warp + lane;
#pragma unroll 8
    for (int ly = 0; ly < h; ++ly, dst += W) {
      const int site = local_of(ly, 32 * warp) + lane, r = root_of(par, site);
      *dst = tile_global(r, y0, x0, W);
      mine |= (uint32_t)(r == site) << ly;
    }
  }

  // 5. my strip's part of the seam record; parent entries of edge roots; edge
  //    roots marked
  seam_strip(par, s.seams + (int64_t)t * SeamLayout::INTS, labels, cs.edge_bits, wn, e_last, h, w, y0, x0, W);

  // 6. LOCAL: edge-root bits; otherwise the root list
  if (LOCAL) {
    __syncthreads();
    if (threadIdx.x < TH * TILE_W / 32) ccl_edges<TH>(s, t)[threadIdx.x] = (int32_t)cs.edge_bits[threadIdx.x];
    return;
  }
  int32_t* slot = s.roots + (int64_t)t * TILE_SITES;
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
  for (; mine; mine &= mine - 1) slot[base++] = (y0 + __ffs(mine) - 1) * W + x0 + 32 * warp + lane;
  if (threadIdx.x == 0) s.root_counts[t] = total;
  __syncthreads();
}

// Tile t's roots: label = final root; in a Swendsen-Wang sweep (spins set)
// final roots also draw their cluster's new state.  All threads call it.
__device__ __forceinline__ void root_compress_tile(int32_t* labels, const LabelScratch& s, int t,
                                                   int8_t* spins, int q, uint64_t seed, uint64_t sweep,
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

// Final labels of tile t for the stand-alone path (after the seam merge, on
// what ccl_label_tile<true> wrote): `table` holds every local index's label --
// first its own global index, the label of a component that stays in the tile;
// then each edge root finds its cluster root R on the label array -- and every
// site takes table[its tile root].  A walk compresses the entries it passes to
// smaller ones of the same tree, so walks of other tiles stay valid.  The tile
// roots of a thread's sites wait in registers while the table is filled and the
// edge roots walk; a tile has at most as many edge roots as sites on its
// perimeter, three per thread.  Labels go out as 16-byte words wherever the rows start (a row
// of any width, its roots shifted by up to three sites against the words they
// come in).  Bound by the latency of the walks, so what counts is tiles in
// flight: ten per SM, with a thread per column and no roots in shared memory,
// against eight of 256 threads with them: 4096^2 83.5 against 87.2 us per
// labeling, 8192^2 290 against 303, 5003 x 7001 176 against 181 (248 with every
// tile root listed and looked up and rows of odd width written site by site).
// All threads of the CTA call it.
constexpr int FINAL_THREADS = TILE_W;
constexpr int FINAL_CTAS = 1280 / FINAL_THREADS;   // 48 registers (1536: 84.2 us at 4096^2, 1024: 86.5)
template <int TH>
struct FinalSmem {
  alignas(16) int32_t table[TH * TILE_W];
  unsigned long long last[TH];             // tile roots of the rows' last four sites
  uint16_t list[2 * (TH + TILE_W)];
  int n_edge;
};
template <int TH>
__device__ __forceinline__ void final_labels_tile(int32_t* labels, const Grid& g, const LabelScratch& s, int t,
                                                  FinalSmem<TH>& fs, int limit) {
  constexpr int WORDS = TILE_W / 4, STEP = FINAL_THREADS / WORDS, PER = TH / STEP;
  const int ty = t / g.tiles_x, tx = t - ty * g.tiles_x;
  const int y0 = ty * TH, x0 = tx * TILE_W;
  const int h = min(TH, g.H - y0), w = min(TILE_W, g.W - x0);
  const int lane = threadIdx.x & 31;
  // 1. tile roots of my sites: of the rows row0 + STEP j, the aligned word q of
  //    four labels, whose first site is 4q less the sites that the row starts
  //    after a word
  const int q = threadIdx.x % WORDS, row0 = threadIdx.x / WORDS;
  const uint16_t* lr = ccl_roots<TH>(s, t);
  auto row_at = [&](int ly) { return labels + (int64_t)(y0 + ly) * g.W + x0; };
  auto shift_of = [&](const int32_t* row) { return (int)(reinterpret_cast<uintptr_t>(row) >> 2) & 3; };
  const bool whole = (g.W & 3) == 0 && (reinterpret_cast<uintptr_t>(labels) & 15) == 0;   // every row starts on a word
  unsigned long long roots[PER];
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int ly = row0 + STEP * j;
    roots[j] = ly < h && 4 * q < w ? reinterpret_cast<const unsigned long long*>(lr + ly * TILE_W)[q] : 0ull;
  }
  if (!whole) {
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int ly = row0 + STEP * j;
      if (q == WORDS - 1) fs.last[ly] = roots[j];
      unsigned long long before = __shfl_up_sync(FULL, roots[j], 1);
      if (WORDS > 32 && lane == 0 && q > 0 && ly < h && 4 * (q - 1) < w)
        before = reinterpret_cast<const unsigned long long*>(lr + ly * TILE_W)[q - 1];
      const int shift = shift_of(row_at(ly));
      if (shift) roots[j] = roots[j] << (16 * shift) | before >> (64 - 16 * shift);
    }
  }
  uint32_t edge = 0u;
  if (threadIdx.x < TH * TILE_W / 32) edge = (uint32_t)__ldcg(ccl_edges<TH>(s, t) + threadIdx.x);
  if (threadIdx.x == 0) fs.n_edge = 0;
  // 2. the table: own global indices
  for (int k = threadIdx.x; k < h * WORDS; k += FINAL_THREADS) {
    const int G = tile_global(4 * k, y0, x0, g.W);   // four local indices of a strip are four sites in a row
    *reinterpret_cast<int4*>(fs.table + 4 * k) = make_int4(G, G + 1, G + 2, G + 3);
  }
  __syncthreads();
  // 3. edge roots listed, then their cluster roots
  {
    const int cnt = __popc(edge);
    int incl = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(FULL, incl, d);
      if (lane >= d) incl += v;
    }
    int base = 0;
    if (lane == 31 && incl) base = atomicAdd(&fs.n_edge, incl);
    int at = __shfl_sync(FULL, base, 31) + incl - cnt;
    for (; edge; edge &= edge - 1, ++at) fs.list[at] = (uint16_t)(32 * threadIdx.x + high_bit(edge & -edge));
  }
  __syncthreads();
  for (int k = threadIdx.x; k < fs.n_edge; k += FINAL_THREADS) {
    const int r = fs.list[k];
    fs.table[r] = g_find(labels, fs.table[r], limit, s.err);
  }
  __syncthreads();
  // 4. every site takes its tile root's label
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int ly = row0 + STEP * j;
    if (ly >= h) break;
    int32_t* row = row_at(ly);
    auto label = [&](int i) { return fs.table[(int)(roots[j] >> (16 * i)) & 0xFFFF]; };
    const int shift = whole ? 0 : shift_of(row), lx = 4 * q - shift;
    if (lx >= 0 && lx + 4 <= w) {
      *reinterpret_cast<int4*>(row + lx) = make_int4(label(0), label(1), label(2), label(3));
    } else if (!whole) {   // else w is a multiple of 4 too
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (lx + i >= 0 && lx + i < w) row[lx + i] = label(i);
    }
    if (!whole && q == WORDS - 1)   // the word after the tile's last one
      for (int i = TILE_W - shift; i < w; ++i) row[i] = fs.table[(int)(fs.last[ly] >> (16 * (i & 3))) & 0xFFFF];
  }
}

}  // namespace swccl
