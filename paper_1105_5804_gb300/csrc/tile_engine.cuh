// tile_engine.cuh -- the tile-local labeling engine shared by the
// stand-alone labeling kernel (bond mask in memory), the fused
// Swendsen-Wang kernel (bonds drawn on the fly) and the simple-cubic kernel.
//
// Input: thread (lane, warp) holds the bond bits of row `lane` of the 32-column
// strip `warp` (we: bit i = east bond of site i of the strip; wn: bit i = its
// north bond), with bits of sites outside the grid and the east bond of the
// tile's last column cleared.  Output: par[] such that a site's tile root is
// the entry its entry names (root_of), the root being the smallest local index
// of the site's tile component.
//
// A row word is cut into runs of east-joined sites.  Every run is labelled by
// a union-find node: a run that no north bond from the row below reaches
// starts a fresh node (the local index of its first site); a run that is
// reached takes the label of the site below its first contact.  Runs reached
// from several runs below are joined afterwards.
//  1. per row word (lane = row), bit-parallel: the run starts S, the first
//     contact F of every reached run (the lowest north bond from below inside
//     the run), the starts U of unreached runs, and the extra contacts X: for
//     each run of the row below that the run touches, the lowest contact in
//     their overlap, other than F.  Overlaps are the segments of sites joined
//     east in both rows, so one contact per overlap keeps exactly one per
//     pair of runs.
//  2. warp c sweeps strip c from row 0 upwards, one site per lane, with the
//     labels of the row below in registers.  A lane finds its run's start
//     (the highest bit of S at or below it) and its run's anchor (the one
//     bit of F | U in the run: the first contact, or the start of an
//     unreached run; searched in the reversed word, where the lowest bit from
//     the start on is the highest of the remaining ones); the anchor lane's
//     candidate -- the label below it if it is a first contact, else its own
//     index -- is the run's label (one shuffle).  No union-find work happens
//     in the sweep.
//  3. the extra contacts are listed per warp and joined with a union-find in
//     shared memory (larger root hooked under the smaller), 32 at a time;
//     only the strip's own warp touches its nodes, so plain stores do;
//  4. after a barrier the east bonds from strip c into strip c + 1 are joined
//     (at most 32 per strip; compare-and-swap hooks);
//  5. after a barrier every hooked root takes its final root: the warp's list
//     and the strip roots of the strip's first and last column (only those can
//     have been hooked in step 4) cover the strip's nodes, so a warp goes on to
//     its own strip's sites without another barrier.
// What bounds the engine is instruction issue (about 70 % of the slots in the
// fused sweep) and the shared-memory pipe, so: 16-bit entries (six CTAs per SM
// instead of the five of 32-bit ones) laid out over all 32 banks (local_of;
// with plain rows the 64-byte strips fall into half of them: 37 against 23
// million conflicts at L = 8192), no shared atomics inside a strip, find loops
// with uniform branches and two steps per vote (the divergent form took twice
// the instructions), and only two barriers where the warps of a tile meet, so
// that their serial stretches overlap with other warps' arithmetic.  Fused
// sweep, critical Ising, L = 8192 (8192 tiles): 226 us for the whole labeling
// kernel against 259 us with 32-bit entries, atomicMin hooks, logged roots and
// four barriers; 95 us of it are the bond draws.
// The root is the smallest index of the tile component: the component's
// smallest site starts a run nothing reaches from below, so it is a node,
// and a smaller root never hooks under a larger one.
#pragma once
#include <climits>

#include "swccl_device.cuh"

namespace swccl {

constexpr int TILE_SITES = TILE_H * TILE_W;
constexpr int STRIPS = TILE_W / 32;
static_assert(LABEL_THREADS == TILE_W, "one warp per 32-column strip");
static_assert(TILE_H == 32, "one lane per row of a strip");
constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int SWEEP_UNROLL = 16;                // rows of the sweep per loop body (32: no faster, twice the code)

// ROWS: rows of the tile (32; the simple-cubic bricks have 16).
template <int ROWS>
struct TileSmemT {
  static constexpr int LIST_CAP = 8 * ROWS;     // contacts per warp and pass (the space of the sweep inputs)
  alignas(16) uint16_t par[ROWS * TILE_W];      // byte offsets (2 x local index); read eight sites at a time
  uint32_t be[ROWS * STRIPS];                   // east bonds, bit = lane of the strip
  uint32_t bn[ROWS * STRIPS];                   // north bonds
  union {
    alignas(16) uint4 rowinfo[STRIPS * ROWS];   // per row word, strip-major: S, F | U reversed, F (sweep inputs)
    uint16_t list[STRIPS * LIST_CAP];           // then: the warps' extra contacts to join
  };
  int warp_roots[LABEL_THREADS / 32];
};
using TileSmem = TileSmemT<TILE_H>;

// Global index of local index r of the tile at (y0, x0) of a W-wide grid.
__device__ __forceinline__ int tile_global(int r, int y0, int x0, int W) {
  return (y0 + local_y(r)) * W + x0 + local_x(r);
}

// Halves (16 bits) of x that are zero: bit 15 / bit 31 of the result.  A
// half is zero iff its low 15 bits plus 0x7FFF stay below bit 15 and its bit
// 15 is clear.
__device__ __forceinline__ uint32_t zero_halves(uint32_t x) {
  return ~(((x & 0x7FFF7FFFu) + 0x7FFF7FFFu) | x) & 0x80008000u;
}

// Tile root (local index) of the site with local index i.
__device__ __forceinline__ int root_of(const uint16_t* par, int i) { return sm_at(par, par[i]) >> 1; }

// The tile roots of eight consecutive sites from local index `sidx` on (a
// multiple of 8), two per word.
__device__ __forceinline__ uint4 roots_of(const uint16_t* par, int sidx) {
  const uint4 v = *reinterpret_cast<const uint4*>(par + sidx);
  auto two = [&](uint32_t w) { return (uint32_t)sm_at(par, w & 0xFFFFu) >> 1 | (uint32_t)sm_at(par, w >> 16) << 15; };
  return make_uint4(two(v.x), two(v.y), two(v.z), two(v.w));
}

// Position of the highest set bit (x != 0).
__device__ __forceinline__ int high_bit(uint32_t x) {
  int p;
  asm("bfind.u32 %0, %1;" : "=r"(p) : "r"(x));
  return p;
}

// Inclusive OR of the bits of x towards higher bits inside segments: bit i
// and bit i + 1 are in one segment iff bit i of j is set.
__device__ __forceinline__ uint32_t seg_or_up(uint32_t x, uint32_t j) {
  uint32_t m = j << 1;           // bit i: i - 1 and i joined
  x |= (x << 1) & m;
  m &= m << 1;                   // bit i: i - 2 .. i joined
  x |= (x << 2) & m;
  m &= m << 2;
  x |= (x << 4) & m;
  m &= m << 4;
  x |= (x << 8) & m;
  m &= m << 8;
  x |= (x << 16) & m;
  return x;
}

// The same towards lower bits.
__device__ __forceinline__ uint32_t seg_or_down(uint32_t x, uint32_t j) {
  uint32_t m = j;                // bit i: i and i + 1 joined
  x |= (x >> 1) & m;
  m &= m >> 1;
  x |= (x >> 2) & m;
  m &= m >> 2;
  x |= (x >> 4) & m;
  m &= m >> 4;
  x |= (x >> 8) & m;
  m &= m >> 8;
  x |= (x >> 16) & m;
  return x;
}

// Step 1 for the calling lane's row word (lane = row; all lanes call): `info`
// (S, F | U reversed, F) for the sweep, and the extra contacts X.
__device__ __forceinline__ uint32_t run_words(uint32_t we, uint32_t wn, int h, uint4& info) {
  const int lane = threadIdx.x & 31;
  const uint32_t e_below = __shfl_up_sync(FULL, we, 1);
  uint32_t c = __shfl_up_sync(FULL, wn, 1);   // contacts: north bonds of the row below into my row
  if (lane == 0 || lane >= h) c = 0u;
  const uint32_t S = ~(we << 1);               // run starts (bit 0 always)
  const uint32_t before = (seg_or_up(c, we) << 1) & (we << 1);     // a contact earlier in my run
  const uint32_t F = c & ~before;
  const uint32_t U = S & ~seg_or_down(c, we);                     // starts of runs without contact
  const uint32_t j2 = we & e_below;                               // joined east in both rows
  const uint32_t before2 = (seg_or_up(c, j2) << 1) & (j2 << 1);
  info = make_uint4(S, __brev(F | U), F, 0u);
  return c & ~before2 & ~F;
}

// Runs the engine.  we, wn: the calling thread's row word (row = lane, strip =
// warp), zero for rows >= h; w: columns of the tile (strips past them hold no
// sites and are skipped); rows past h are swept as rows of single sites, or with
// ALL_ROWS false not at all, their entries left unwritten (a rolled loop, for
// tiles of which h is a small part).  All threads call it.  On return the calling
// warp's strip is resolved: other strips' roots may be read after a
// __syncthreads().
template <bool ALL_ROWS = true, int ROWS>
__device__ __forceinline__ void tile_engine(TileSmemT<ROWS>& sm, uint32_t we, uint32_t wn, int h, int w, int* err) {
  constexpr int LIST_CAP = TileSmemT<ROWS>::LIST_CAP;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint16_t* par = sm.par;
  const int colbase = warp * 32;
  const bool strip = colbase < w;   // same for the whole warp
  const int row = local_of(lane, colbase);   // my row's first site in the strip
  uint16_t* list = sm.list + warp * LIST_CAP;
  int n_list = 0;
  int ends[2] = {0, 0};             // strip roots of my row's first and last site
  if (lane < ROWS) {
    sm.be[lane * STRIPS + warp] = we;
    sm.bn[lane * STRIPS + warp] = wn;
  }
  if (strip) {
  // 1. run structure of my row word against the row below
  uint4 info;
  const uint32_t X = run_words(we, wn, h, info);
  if (lane < ROWS) sm.rowinfo[warp * ROWS + lane] = info;
  __syncwarp();
  // 2. strip sweep.  Lane l takes column 31 - l: the anchor's column comes out
  //    as 31 - anchor, the lane to read from.
  {
    const int col = 31 - lane;
    const uint32_t upto = FULL >> lane;          // bits 0..col
    const uint32_t me = 1u << col;
    int lab_below = 0;
    auto sweep_row = [&](int ly) {
      const uint4 ri = sm.rowinfo[warp * ROWS + ly];
      const int start = high_bit(ri.x & upto);
      const int from = high_bit(ri.y & (FULL >> start));
      const int site = local_of(ly, colbase) + col;
      const int cand = (ri.z & me) ? lab_below : 2 * site;
      const int label = __shfl_sync(FULL, cand, from);
      par[site] = (uint16_t)label;
      lab_below = label;
    };
    if (ALL_ROWS) {
#pragma unroll SWEEP_UNROLL
      for (int ly = 0; ly < ROWS; ++ly) sweep_row(ly);
    } else {
#pragma unroll 1
      for (int ly = 0; ly < h; ++ly) sweep_row(ly);
    }
  }
  __syncwarp();

  // 3. joins inside the strip: list the sites of the extra contacts of my row
  //    (lane = row), join the labels on both ends 32 at a time, and leave the
  //    root that each join hooked in the contact's place.  A strip with more
  //    contacts than the list holds takes them in several passes.
  {
    const int cnt = __popc(X);
    int incl = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(FULL, incl, d);
      if (lane >= d) incl += v;
    }
    n_list = __shfl_sync(FULL, incl, 31);
    for (int first = 0; first < n_list; first += LIST_CAP) {
      int k = incl - cnt - first;
      for (uint32_t x = X; x; x &= x - 1, ++k)
        if ((unsigned)k < LIST_CAP) list[k] = (uint16_t)(row + high_bit(x & -x));
      __syncwarp();
      const int n = min(n_list - first, LIST_CAP);
      for (int j = lane; j - lane < n; j += 32) {
        int a = 2 * colbase, b = a;   // no contact: a node of the own strip (other strips' entries may not be written yet)
        if (j < n) {
          const int site = list[j];
          a = par[site];
          b = par[(site - TILE_W) ^ 32];   // the site below
        }
        const int hooked = sm_union_strip(par, a, b);
        if (j < n) list[j] = (uint16_t)hooked;   // -1: 0xFFFF, not an offset
      }
      __syncwarp();
    }
  }
  // strip roots of my row's ends (lanes past the tile's rows go along with row 0)
  ends[0] = par[lane < h ? row : colbase];
  ends[1] = par[lane < h ? row + 31 : colbase];
  sm_find_strip(par, ends);
  }
  __syncthreads();

  // 4. joins between strips: the east bond of my row into the next strip,
  //    unless the rows below join the same two runs
  if (warp < STRIPS - 1 && colbase + 32 < w) {
    bool join = lane < h && (we >> 31);
    if (join && lane > 0) {
      const int k0 = (lane - 1) * STRIPS + warp;
      if ((sm.be[k0] >> 31) && (sm.bn[k0] >> 31) && (sm.bn[k0 + 1] & 1u)) join = false;
    }
    if (__any_sync(FULL, join))
      sm_union_tile(par, ends[1], join ? (int)par[local_of(lane, colbase + 32)] : ends[1], err);
  }
  __syncthreads();

  // 5. final roots of the strip's hooked roots; a parent is replaced by an
  //    ancestor, so other walks through it stay valid
  if (strip) {
    int r[2] = {ends[0], ends[1]};
    sm_find_tile(par, r, err);
    sm_set(par, ends[0], r[0]);
    sm_set(par, ends[1], r[1]);
    if (n_list <= LIST_CAP) {
      for (int j = lane; j - lane < n_list; j += 32) {
        const int x = j < n_list ? (int)list[j] : 0xFFFF;
        int f[1] = {x != 0xFFFF ? x : r[0]};
        sm_find_tile(par, f, err);
        if (x != 0xFFFF) sm_set(par, x, f[0]);
      }
    } else {   // the list holds the last pass only: every site takes its root
      for (int ly = 0; ly < h; ++ly) {
        const int x = 2 * (local_of(ly, colbase) + lane);
        int f[1] = {x};
        sm_find_tile(par, f, err);
        sm_set(par, x, f[0]);
      }
    }
  }
  __syncwarp();
}

// The calling warp's part of the tile's seam record after the engine (tile
// roots on the tile edge, bonds leaving the tile), with the parent entries
// gpar[g] = g of those roots and their marks in edge_bits (TILE_SITES / 32
// words, zeroed before the engine).  wn: my row's north bonds; e_last: raw
// east bits of column w - 1 (bit = row) in the warp that holds that column.
__device__ __forceinline__ void seam_strip(const uint16_t* par, int32_t* rec, int32_t* gpar, uint32_t* edge_bits,
                                           uint32_t wn, uint32_t e_last, int h, int w, int y0, int x0, int W) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto edge_root = [&](bool ok, int i) -> int32_t {
    // global index of the tile root of local site i; the first of a run of
    // equal roots among consecutive lanes writes its parent entry and its mark
    const int r = ok ? root_of(par, i) : -1;
    const int left = __shfl_up_sync(FULL, r, 1);
    if (!ok) return -1;
    const int32_t gr = tile_global(r, y0, x0, W);
    if (lane == 0 || left != r) {
      gpar[gr] = gr;
      atomicOr(&edge_bits[r >> 5], 1u << (r & 31));
    }
    return gr;
  };
  if (warp == 0) rec[SeamLayout::COL_L + lane] = edge_root(lane < h, local_of(lane, 0));
  if (warp == (w - 1) >> 5) {
    rec[SeamLayout::COL_R + lane] = edge_root(lane < h, local_of(lane, w - 1));
    if (lane == 0) rec[SeamLayout::E_BITS] = (int32_t)e_last;
  }
  const int lx = 32 * warp + lane;
  rec[SeamLayout::ROW_B + lx] = edge_root(lx < w, local_of(0, lx));
  rec[SeamLayout::ROW_T + lx] = edge_root(lx < w, local_of(h - 1, lx));
  const uint32_t nb = __shfl_sync(FULL, wn, h - 1);
  if (lane == 0) rec[SeamLayout::N_BITS + warp] = (int32_t)nb;
}

// ---------------------------------------------------------------------------
// Seam merge (Sec. II.C): bond k of tile t leaves the tile east (k < TILE_H,
// row k) or north (k >= TILE_H, column k - TILE_H), the periodic wrap
// included.  If it is open, the two tile roots on its ends are joined on the
// global array `gpar` (atomicMin hooking, larger root under the smaller).  A
// lane whose root pair equals its left neighbour's skips the union, so runs
// of seam bonds of one cluster cost one union.  MERGE_PER_TILE is a multiple of
// 32, so a warp never spans two tiles.
constexpr int MERGE_PER_TILE = TILE_H + TILE_W;
static_assert(MERGE_PER_TILE % 32 == 0, "warps must not straddle tiles");

// The bond's bit and the roots at both ends, loaded together (the neighbour
// index wraps, so the loads stay inside the records even where the bond does
// not exist; then has is false).  Seam records are read through L2 (ld.cg): in
// a persistent kernel they were written by other SMs.
struct SeamBond {
  uint32_t bits;
  int a, b;
  bool has;
};
__device__ __forceinline__ SeamBond load_seam_bond(const Grid& g, const int32_t* seams, int t, int k) {
  const int ty = t / g.tiles_x, tx = t - ty * g.tiles_x;
  const int32_t* rec = seams + (int64_t)t * SeamLayout::INTS;
  SeamBond s;
  int tn, i_bits, i_a, i_b;
  if (k < TILE_H) {
    s.has = g.periodic || tx + 1 < g.tiles_x;
    tn = ty * g.tiles_x + (tx + 1 == g.tiles_x ? 0 : tx + 1);
    i_bits = SeamLayout::E_BITS;
    i_a = SeamLayout::COL_R + k;
    i_b = SeamLayout::COL_L + k;
  } else {
    const int lx = k - TILE_H;
    s.has = g.periodic || ty + 1 < g.tiles_y;
    tn = (ty + 1 == g.tiles_y ? 0 : ty + 1) * g.tiles_x + tx;
    i_bits = SeamLayout::N_BITS + (lx >> 5);
    i_a = SeamLayout::ROW_T + lx;
    i_b = SeamLayout::ROW_B + lx;
  }
  s.bits = (uint32_t)__ldcg(rec + i_bits);
  s.a = __ldcg(rec + i_a);
  s.b = __ldcg(seams + (int64_t)tn * SeamLayout::INTS + i_b);
  return s;
}
static_assert(TILE_H == 32, "bond k's bit is bit k % 32 of its word");

// Whether the calling lane has to join (lo, hi); all 32 lanes call together.
__device__ __forceinline__ bool seam_pair(const SeamBond& s, int k, int& lo, int& hi) {
  const bool valid = s.has && ((s.bits >> (k & 31)) & 1u) && s.a != s.b;
  lo = min(s.a, s.b);
  hi = max(s.a, s.b);
  const unsigned long long key = valid ? ((unsigned long long)(unsigned)lo << 32) | (unsigned)hi : ~0ull;
  const unsigned long long left = __shfl_up_sync(FULL, key, 1);
  return valid && ((threadIdx.x & 31) == 0 || left != key);
}

// Join lo < hi on gpar, trying the hook before any walk: most larger roots are
// still roots, and an entry that was hooked already is lowered if lo is
// smaller, its old parent then joined with lo as after a lost race.
__device__ __forceinline__ void seam_join(int32_t* gpar, int lo, int hi, int limit, int* err) {
  const int old = atomicMin(gpar + hi, lo);
  if (old != hi && old != lo) g_union(gpar, lo, old, limit, err);
}

// One bond per lane (the persistent batch kernel; all 32 lanes call together).
__device__ __forceinline__ void merge_seam_bond(int32_t* gpar, const Grid& g, const LabelScratch& s, int t, int k,
                                                int limit) {
  int lo, hi;
  if (seam_pair(load_seam_bond(g, s.seams, t, k), k, lo, hi)) seam_join(gpar, lo, hi, limit, s.err);
}

// The seam bonds of n <= MERGE_TILES consecutive tiles by one CTA of
// MERGE_PER_TILE threads (thread = bond): every thread loads its bond of all
// the tiles at once, the pairs to join (about one bond in six at criticality)
// go to a list, and the list is joined with all lanes busy.  With a union per
// lane where it stands, a warp ran its divergent walks for five lanes of 32 and
// issued 278 instructions; bound by the latency of the parent loads (L = 16384:
// 156 us then, 153 with the hook before the walk, 120 us as it is).  tile_of(u): grid, parents and scratch of tile u.
constexpr int MERGE_TILES = 2;
struct MergeSmem {
  int2 pairs[MERGE_TILES * MERGE_PER_TILE];
  uint8_t tile[MERGE_TILES * MERGE_PER_TILE];
  int n;
};
struct MergeTile {
  const Grid* g;
  int32_t* gpar;
  const int32_t* seams;
  int* err;
  int t;
};
template <class TileOf>
__device__ __forceinline__ void merge_tiles(MergeSmem& ms, int n, const TileOf& tile_of, int limit) {
  const int k = threadIdx.x, lane = threadIdx.x & 31;
  if (k == 0) ms.n = 0;
  SeamBond bond[MERGE_TILES];
#pragma unroll
  for (int u = 0; u < MERGE_TILES; ++u) {
    bond[u].has = false;
    if (u < n) {
      const MergeTile m = tile_of(u);
      bond[u] = load_seam_bond(*m.g, m.seams, m.t, k);
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < MERGE_TILES; ++u) {
    if (u >= n) break;
    int lo, hi;
    const bool join = seam_pair(bond[u], k, lo, hi);
    const uint32_t m = __ballot_sync(FULL, join);
    if (m == 0u) continue;
    int at = 0;
    if (lane == 0) at = atomicAdd(&ms.n, __popc(m));
    at = __shfl_sync(FULL, at, 0) + __popc(m & ((1u << lane) - 1u));
    if (join) {
      ms.pairs[at] = make_int2(lo, hi);
      ms.tile[at] = (uint8_t)u;
    }
  }
  __syncthreads();
  for (int j = threadIdx.x; j < ms.n; j += MERGE_PER_TILE) {
    const MergeTile m = tile_of(ms.tile[j]);
    seam_join(m.gpar, ms.pairs[j].x, ms.pairs[j].y, limit, m.err);
  }
}

// Tiles per CTA of a merge over n_tiles tiles: two where their bonds fill the
// GPU's 152 x 2048 threads more than once, one below (latency of one wave:
// L = 2048 13.2 against 13.9 us, L = 4096 19.4 against 16.6; three to six tiles
// are 2 % better at L = 16384 and up to 60 % worse at 4096).
inline int merge_tiles_per_cta(int64_t n_tiles) {
  return n_tiles * MERGE_PER_TILE > (int64_t)152 * 2048 ? MERGE_TILES : 1;
}

}  // namespace swccl
