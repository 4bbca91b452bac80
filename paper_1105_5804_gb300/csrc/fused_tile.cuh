// fused_tile.cuh -- per-tile bodies of the fused Swendsen-Wang sweep, shared
// by the single-lattice kernels (k_fused.cu) and the batched / persistent
// kernels over many lattices (k_batch.cu).  Description of the steps in
// k_fused.cu.
#pragma once
#include "tile_engine.cuh"

namespace swccl {

namespace fused {

constexpr int QREG_MAX = 8;

// Which of 32 consecutive sites of one row equal their east and north
// neighbours, and the observables of the spins read (bonds joining equal
// spins; sites per state for q <= QREG).
struct RowEqual {
  uint32_t east, north;     // bit i: site i equals its east / north neighbour
  int n_eq;                 // equal east and north neighbours among the sites
  int cnt[QREG_MAX];        // sites per state (q <= 8)
};

__device__ __forceinline__ void row_equal(const int8_t* spins, int L, int y, int x, int nvalid, int q,
                                          RowEqual& rb) {
  const int yn = (y + 1 == L) ? 0 : y + 1;
  const int64_t row = (int64_t)y * L, rown = (int64_t)yn * L;
  uint32_t s[8], n[8];
  const int nw = nvalid >> 2;   // whole 4-site words (L % 4 == 0)
  if (nw == 8 && (L & 15) == 0) {
    const uint4 a0 = *reinterpret_cast<const uint4*>(spins + row + x);
    const uint4 a1 = *reinterpret_cast<const uint4*>(spins + row + x + 16);
    const uint4 b0 = *reinterpret_cast<const uint4*>(spins + rown + x);
    const uint4 b1 = *reinterpret_cast<const uint4*>(spins + rown + x + 16);
    s[0] = a0.x; s[1] = a0.y; s[2] = a0.z; s[3] = a0.w; s[4] = a1.x; s[5] = a1.y; s[6] = a1.z; s[7] = a1.w;
    n[0] = b0.x; n[1] = b0.y; n[2] = b0.z; n[3] = b0.w; n[4] = b1.x; n[5] = b1.y; n[6] = b1.z; n[7] = b1.w;
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      s[k] = (k < nw) ? *reinterpret_cast<const uint32_t*>(spins + row + x + 4 * k) : 0u;
      n[k] = (k < nw) ? *reinterpret_cast<const uint32_t*>(spins + rown + x + 4 * k) : 0u;
    }
  }
  const int xe = (x + nvalid == L) ? 0 : x + nvalid;
  const uint32_t east_byte = (uint32_t)(uint8_t)spins[row + xe];
  uint32_t eq_e = 0, eq_n = 0;
#pragma unroll
  for (int c = 0; c < QREG_MAX; ++c) rb.cnt[c] = 0;
  if (q == 2 && nw == 8) {
    // Ising spins (bytes 0 or 1) packed one bit per site: the product puts
    // byte k's bit 0 at bit 24 + k, nothing else reaches bits 24..27
    uint32_t sb = 0u, nb = 0u;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      sb |= ((s[k] * 0x01020408u) >> 24) << (4 * k);
      nb |= ((n[k] * 0x01020408u) >> 24) << (4 * k);
    }
    eq_e = ~(sb ^ ((sb >> 1) | ((east_byte & 1u) << 31)));
    eq_n = ~(sb ^ nb);
    rb.n_eq = __popc(eq_e) + __popc(eq_n);
    rb.cnt[1] = __popc(sb);
    rb.cnt[0] = 32 - rb.cnt[1];
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (k < nw) {
        const uint32_t next = (k + 1 < nw) ? s[k + 1] : east_byte;
        eq_e |= eq4(s[k], (s[k] >> 8) | (next << 24)) << (4 * k);
        eq_n |= eq4(s[k], n[k]) << (4 * k);
      }
    }
    // observables of the spins read
    const uint32_t valid = nvalid == 32 ? 0xFFFFFFFFu : ((1u << nvalid) - 1u);
    rb.n_eq = __popc(eq_e & valid) + __popc(eq_n & valid);
    if (q == 2) {
      int ones = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) ones += (k < nw) ? __popc(s[k] & 0x01010101u) : 0;
      rb.cnt[0] = nvalid - ones;
      rb.cnt[1] = ones;
    } else if (q <= QREG_MAX) {
#pragma unroll
      for (int c = 0; c < QREG_MAX; ++c) {
        if (c >= q) break;
        int m = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) m += (k < nw) ? __popc(eq4(s[k], 0x01010101u * (uint32_t)c)) : 0;
        rb.cnt[c] = m;
      }
    }
  }
  rb.east = eq_e;
  rb.north = eq_n;
}

// e |= bit if r < thr: a compare and one predicated add.
__device__ __forceinline__ void set_if_below(uint32_t& e, uint32_t r, uint32_t thr, uint32_t bit) {
  asm("{ .reg .pred p; setp.lt.u32 p, %1, %2; @p add.u32 %0, %0, %3; }" : "+r"(e) : "r"(r), "r"(thr), "r"(bit));
}

// Open bonds of 32 consecutive sites from site index `site0` on (even; rule
// of Eq. 7): the bits of east / north (equal neighbours) whose draw is below
// T.  One Philox call per pair of sites i, i+1 (words: east i, north i, east
// i+1, north i+1).  Draws past the last valid site are dropped by the masks.
template <class Keys>
__device__ __forceinline__ void draw_bonds(uint32_t site0, int nvalid, uint64_t T, const Keys& keys, uint32_t sw_lo,
                                           uint32_t sw_hi, uint32_t& east, uint32_t& north) {
  if (T >= (1ull << 32)) return;         // p = 1: every bond between equal spins opens
  uint32_t e = 0u, n = 0u;
  if (T != 0) {
    const uint32_t thr = (uint32_t)T, c0 = site0 >> 1;
    constexpr int U = 16;   // sites per loop body (8: 5 % longer, 32: 4 %, its code misses the instruction cache)
#pragma unroll 1
    for (int i0 = 0; i0 < nvalid; i0 += U) {
      uint32_t eb = 0u, nb = 0u;
#pragma unroll
      for (int i = 0; i < U; i += 2) {
        const uint4 r = philox_draw(make_uint4(c0 + (uint32_t)((i0 + i) >> 1), sw_lo, sw_hi, TAG_BOND), keys);
        set_if_below(eb, r.x, thr, 1u << i);
        set_if_below(eb, r.z, thr, 2u << i);
        set_if_below(nb, r.y, thr, 1u << i);
        set_if_below(nb, r.w, thr, 2u << i);
      }
      e |= eb << i0;
      n |= nb << i0;
    }
  }
  east &= e;
  north &= n;
}

// Block-wide sums of n_eq and the state counts, added to the observable slot.
template <int NTHREADS>
__device__ __forceinline__ void add_observables(long long n_eq, const int* cnt, int q, int qreg, unsigned long long* slot,
                                unsigned long long* red /* shared, (1 + qreg) * NTHREADS/32 */,
                                int* hist /* shared, 128, already holds counts when qreg == 0 */) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int NW = NTHREADS / 32;
  unsigned long long v = (unsigned long long)n_eq;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(FULL, v, o);
  if (lane == 0) red[warp] = v;
#pragma unroll
  for (int k = 0; k < QREG_MAX; ++k) {
    if (k >= qreg) break;
    unsigned long long c = (unsigned long long)cnt[k];
    for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(FULL, c, o);
    if (lane == 0) red[(1 + k) * NW + warp] = c;
  }
  __syncthreads();
  if (threadIdx.x <= qreg) {
    unsigned long long tot = 0;
    for (int w = 0; w < NW; ++w) tot += red[threadIdx.x * NW + w];
    if (tot && (threadIdx.x == 0 || threadIdx.x - 1 < q)) atomicAdd(slot + threadIdx.x, tot);
  }
  if (qreg == 0) {
    for (int k = threadIdx.x; k < q; k += NTHREADS)
      if (hist[k]) atomicAdd(slot + 1 + k, (unsigned long long)hist[k]);
  }
}

// The two halves of add_observables, for a kernel that has a __syncthreads()
// between them anyway: every warp leaves its sums in `red` (at most 64 bonds
// and 32 sites per lane, so 32-bit sums are exact) ...
template <int NTHREADS>
__device__ __forceinline__ void observables_warp_sums(unsigned n_eq, const int* cnt, int qreg, unsigned* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int NW = NTHREADS / 32;
  const unsigned v = __reduce_add_sync(FULL, n_eq);
  if (lane == 0) red[warp] = v;
#pragma unroll
  for (int k = 0; k < QREG_MAX; ++k) {
    if (k >= qreg) break;
    const unsigned c = __reduce_add_sync(FULL, (unsigned)cnt[k]);
    if (lane == 0) red[(1 + k) * NW + warp] = c;
  }
}

// ... and, after a barrier, the block's totals are added to the slot.
template <int NTHREADS>
__device__ __forceinline__ void observables_commit(int q, int qreg, unsigned long long* slot, const unsigned* red,
                                                   const int* hist) {
  constexpr int NW = NTHREADS / 32;
  if (threadIdx.x <= qreg) {
    unsigned tot = 0;
    for (int w = 0; w < NW; ++w) tot += red[threadIdx.x * NW + w];
    if (tot && (threadIdx.x == 0 || threadIdx.x - 1 < q)) atomicAdd(slot + threadIdx.x, (unsigned long long)tot);
  }
  if (qreg == 0) {
    for (int k = threadIdx.x; k < q; k += NTHREADS)
      if (hist[k]) atomicAdd(slot + 1 + k, (unsigned long long)hist[k]);
  }
}

constexpr int QREG = QREG_MAX;   // state counts kept in registers for q <= QREG

}  // namespace fused
using namespace fused;

// The labeling kernel leaves a tile's edge-root bits in TILE_SITES / 32 words
// of the scratch (sweep_edges): bit r set iff local root r's component touches
// the tile edge, so that its cluster may continue in other tiles.  The flip and
// the few-cluster seed selection read them.
constexpr int EDGE_WORDS = TILE_SITES / 32;
__device__ __forceinline__ int32_t* sweep_edges(const LabelScratch& s, int t) { return s.roots + (int64_t)t * EDGE_WORDS; }
static_assert(EDGE_WORDS == LABEL_THREADS, "one edge word per thread");

struct LabelTileSmem {
  TileSmem tile;
  uint32_t edge_bits[EDGE_WORDS];                   // local roots on the tile edge
  unsigned long long red[(1 + QREG) * (LABEL_THREADS / 32)];
  int hist[128];
};

// The flip's shared memory, for tiles of TH rows.
template <int TH>
struct FlipTileSmemT {
  static constexpr int SITES = TH * TILE_W;
  static constexpr int LIST = SITES / 4;        // roots listed per pass (at criticality a tile has 0.14 per site)
  uint4 roots[SITES / 8];       // the tile roots of every thread's sites (pass-major, thread by thread)
  uint8_t ns[SITES];            // new state, indexed by local root
  uint16_t rlist[LIST];         // the tile's roots, edge roots first
  int warp_cnt[LABEL_THREADS / 32];
};
using FlipTileSmem = FlipTileSmemT<TILE_H>;

// One tile of the fused draw-and-label step (see k_fused.cu).  All threads
// of the CTA call it; it synchronises the CTA internally and on return.
template <class Keys>
__device__ __forceinline__ void sw_label_tile(const SwRep& R, int t, uint64_t sweep, bool do_obs, int obs_cap,
                                              LabelTileSmem& ls, const Keys& keys) {
  TileSmem& sm = ls.tile;
  unsigned* red = reinterpret_cast<unsigned*>(ls.red);
  int* hist = ls.hist;
  const int8_t* spins = R.spins;
  uint16_t* lroot = R.lroot;
  int32_t* gpar = R.gpar;
  const Grid& g = R.g;
  const LabelScratch& s = R.s;
  const int q = R.q;
  const uint64_t T = R.T;
  const int L = g.W;
  const int ty = t / g.tiles_x, tx = t - ty * g.tiles_x;
  const int y0 = ty * TILE_H, x0 = tx * TILE_W;
  const int h = min(TILE_H, L - y0), w = min(TILE_W, L - x0);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t* edge_bits = ls.edge_bits;
  edge_bits[threadIdx.x] = 0u;        // the engine's barriers order it before the marks
  if (q > QREG) {
    for (int k = threadIdx.x; k < 128; k += LABEL_THREADS) hist[k] = 0;
    __syncthreads();
  }

  // 1. bonds: warp c draws strip c, lane ly row ly; the observables are
  //    summed before the draws, so that their counters hold no registers
  //    across them
  const int nvalid = min(max(w - 32 * warp, 0), 32);
  const bool last_strip = nvalid > 0 && 32 * warp + nvalid == w;
  uint32_t we = 0u, wn = 0u, e_last = 0u;   // e_last: raw east bits of column w-1, bit = row
  {
    const bool in = lane < h && nvalid > 0;
    const int y = y0 + lane, x = x0 + 32 * warp;
    {
      RowEqual rb;
      rb.n_eq = 0;
#pragma unroll
      for (int k = 0; k < QREG; ++k) rb.cnt[k] = 0;
      if (in) {
        row_equal(spins, L, y, x, nvalid, q, rb);
        we = rb.east;
        wn = rb.north;
        if (do_obs && q > QREG) {
          const int8_t* p = spins + (int64_t)y * L + x;
          for (int j = 0; j < nvalid; ++j) atomicAdd(&hist[p[j]], 1);
        }
      }
      if (do_obs) observables_warp_sums<LABEL_THREADS>((unsigned)rb.n_eq, rb.cnt, q <= QREG ? q : 0, red);
    }
    if (in)
      draw_bonds((uint32_t)((int64_t)y * L + x), nvalid, T, keys, (uint32_t)sweep, (uint32_t)(sweep >> 32), we, wn);
    if (last_strip) {                 // east bonds leaving the tile
      const uint32_t bit = 1u << (nvalid - 1);
      e_last = __ballot_sync(FULL, (we & bit) != 0u);
      we &= ~bit;
    }
  }

  // 2. label the tile
  tile_engine(sm, we, wn, h, w, s.err);
  if (do_obs) {   // observables of the spins read (the previous sweep's result)
    unsigned long long* oslot =
        reinterpret_cast<unsigned long long*>(R.obs + (int64_t)((sweep - 1) % (uint64_t)obs_cap) * (q + 1));
    observables_commit<LABEL_THREADS>(q, q <= QREG ? q : 0, oslot, red, hist);
  }

  // 3. tile roots of my strip as 16-bit local indices: per step a thread
  //    takes eight consecutive sites (four threads a row) and stores 16
  //    bytes, or two halves where rows start only 8-byte aligned (L % 4 == 0;
  //    w is a multiple of 4, so four sites are all inside or all outside).
  //    Streaming stores: the roots are read once, after the merge, and leave
  //    L2 to spins, seam records and parents (L = 16384: this kernel 0.892 ->
  //    0.858 ms)
  {
    const int lx = 32 * warp + 8 * (lane & 3);
#pragma unroll 2
    for (int ly = lane >> 2; ly < h; ly += 8) {
      if (lx >= w) break;
      const uint4 r = roots_of(sm.par, local_of(ly, lx));
      uint16_t* dst = lroot + (int64_t)(y0 + ly) * L + x0 + lx;
      if ((L & 7) == 0) {   // then w is a multiple of 8 too
        __stcs(reinterpret_cast<uint4*>(dst), r);
      } else {
        *reinterpret_cast<uint2*>(dst) = make_uint2(r.x, r.y);
        if (lx + 8 <= w) *reinterpret_cast<uint2*>(dst + 4) = make_uint2(r.z, r.w);
      }
    }
  }

  // 4. my strip's part of the seam record; parent entries of edge roots; edge
  //    roots marked
  seam_strip(sm.par, s.seams + (int64_t)t * SeamLayout::INTS, gpar, edge_bits, wn, e_last, h, w, y0, x0, L);

  __syncthreads();
  // 5. edge-root bits; each thread reads and next clears only its own word
  sweep_edges(s, t)[threadIdx.x] = (int32_t)edge_bits[threadIdx.x];
}

// One tile of the fused flip step (see k_fused.cu).  All threads of the CTA
// call it; it synchronises the CTA internally and on return.
// Site ownership of the flip: with G = TILE_W / 8 column groups, thread k owns,
// in each pass j (four for a 32-row tile), the eight sites (row 8j + k / G,
// columns 8 (k % G) .. 8 (k % G) + 7) of the tile; their tile roots are one
// 16-byte word per pass.
constexpr int FLIP_GROUPS = TILE_W / 8;
static_assert(LABEL_THREADS / FLIP_GROUPS == 8, "site ownership");

// Local root (16 bits) of site i (0..7) of a pass word.
__device__ __forceinline__ int root_in(const uint4& v, int i) {
  const uint32_t wv = (i < 2) ? v.x : (i < 4) ? v.y : (i < 6) ? v.z : v.w;
  return (int)((wv >> (16 * (i & 1))) & 0xFFFFu);
}

// The flip of tile t (see k_fused.cu).  All threads of the CTA call it; it
// ends with a barrier.
// The tile roots wait in shared memory for the site pass (held in registers
// across the draws they spill at six CTAs per SM, read again through L2 they
// cost its traffic twice).  Edge roots, whose cluster root has to be found on
// gpar, come first in the list, so that each of the first threads has one walk
// whose first load is in flight while the thread draws its interior roots.
// Bound by instruction issue (74 % of the slots, 1.03 warp instructions per
// site, a third of them the draws); critical Ising, L = 16384: 0.298 ms against
// 0.389 ms with the roots read twice, flags looked up root by root and four
// walks per thread in step.  Above the critical temperature the draws are most
// of it (0.4 roots per site at 0.6 beta_c): L = 8192 there 146 us against 180 with
// every root listed and threads looking through their roots once per pass of
// the list (T = infinity 210 against 345).
// TH: rows of the lattice's tiles.
template <int TH = TILE_H, class Keys = SeedKey>
__device__ __forceinline__ void sw_flip_tile(const SwRep& R, int t, uint64_t sweep, int limit, FlipTileSmemT<TH>& fs,
                                             const Keys& keys) {
  constexpr int PASSES = TH / 8, FLIP_LIST = FlipTileSmemT<TH>::LIST;
  uint8_t* ns = fs.ns;
  int8_t* spins = R.spins;
  int32_t* gpar = R.gpar;
  const int q = R.q;
  int* err = R.s.err;
  const int L = R.g.W;
  const int ty = t / R.g.tiles_x, tx = t - ty * R.g.tiles_x;
  const int y0 = ty * TH, x0 = tx * TILE_W;
  const int h = min(TH, L - y0), w = min(TILE_W, L - x0);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int orow = threadIdx.x / FLIP_GROUPS, lx0 = 8 * (threadIdx.x % FLIP_GROUPS);   // my sites

  // 1. tile roots of my sites into shared memory (0xFFFF outside the tile; w
  //    is a multiple of 4: a group of eight sites is wholly inside, or its
  //    first four are; 16-byte loads need L % 8 == 0, 8-byte ones L % 4 == 0).
  //    Read through L2 because a persistent kernel wrote them on other SMs.
  uint4* const my_roots = fs.roots + threadIdx.x;   // pass j: my_roots[j LABEL_THREADS]
  const int id0 = local_of(orow, lx0);              // local index of my first site; pass j: id0 + 8 j TILE_W
  uint32_t edges = 0u;   // bit 8j + i: edge-root bit of site i of pass j
  {
    const uint8_t* eb = reinterpret_cast<const uint8_t*>(sweep_edges(R.s, t)) + (id0 >> 3);
    const uint16_t* src = R.lroot + (int64_t)(y0 + orow) * L + x0 + lx0;
    const int64_t step = (int64_t)8 * L;
#pragma unroll
    for (int j = 0; j < PASSES; ++j) edges |= (uint32_t)__ldcg(eb + j * TILE_W) << (8 * j);
    if ((L & 7) == 0 && h == TH && lx0 < w) {   // w is a multiple of 8
#pragma unroll
      for (int j = 0; j < PASSES; ++j) copy16_async(my_roots + j * LABEL_THREADS, src + j * step);
      copies_wait();   // a thread reads back only what it copied itself
    } else {
#pragma unroll
      for (int j = 0; j < PASSES; ++j) {
        uint4 v = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
        if (8 * j + orow < h && lx0 < w) {
          const uint2 a = __ldcg(reinterpret_cast<const uint2*>(src + j * step));
          v.x = a.x;
          v.y = a.y;
          if (lx0 + 8 <= w) {
            const uint2 c = __ldcg(reinterpret_cast<const uint2*>(src + j * step + 4));
            v.z = c.x;
            v.w = c.y;
          }
        }
        my_roots[j * LABEL_THREADS] = v;
      }
    }
  }

  // 2. my roots: a site is a tile root iff its entry is its own local index.
  //    Word k of pass j holds sites 2k and 2k + 1; both are compared at once.
  //    Bit 8j + i of mine flags site i of pass j.
  uint32_t mine;
  {
    uint32_t m = 0;   // bit 4j + k: site 2k of pass j, bit 16 + 4j + k: site 2k + 1
#pragma unroll
    for (int j = 0; j < PASSES; ++j) {
      const uint4 rv = my_roots[j * LABEL_THREADS];
      const uint32_t own = (uint32_t)(id0 + 8 * j * TILE_W) * 0x00010001u + 0x00010000u;   // (site, site + 1)
      const uint32_t wv[4] = {rv.x, rv.y, rv.z, rv.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) m |= zero_halves(wv[k] ^ (own + (uint32_t)k * 0x00020002u)) >> (15 - (4 * j + k));
    }
    mine = spread_bits(m & 0xFFFFu) | spread_bits(m >> 16) << 1;
  }
  const uint32_t on_edge = mine & edges;
  uint32_t inner = mine & ~edges;
  auto set_state = [&](int r, int G) {   // new state of the component with local root r and cluster root G
    const uint4 d = philox_draw(make_uint4((uint32_t)G, (uint32_t)sweep, (uint32_t)(sweep >> 32), TAG_FLIP), keys);
    ns[r] = (uint8_t)state_of(d.x, q);
  };
  auto root_at = [&](int n) { return id0 + n + (n & 24) * (TILE_W - 1); };   // local index of bit n's site
  // as many interior roots as every lane of the warp has are drawn where they
  // stand (hardly any at criticality, two in three at 0.6 beta_c); the list
  // spreads the others over the lanes
  for (int k = __reduce_min_sync(FULL, __popc(inner)); k > 0; --k) {
    const int n = high_bit(inner);
    inner ^= 1u << n;
    const int r = root_at(n);
    set_state(r, tile_global(r, y0, x0, L));
  }

  // 3. the tile's root list: edge roots, then the others (counts of both in
  //    one scan; a tile with more roots than the list holds takes several
  //    passes)
  const int cnt = __popc(on_edge) << 16 | __popc(inner);
  int incl = cnt;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int v = __shfl_up_sync(FULL, incl, d);
    if (lane >= d) incl += v;
  }
  if (lane == 31) fs.warp_cnt[warp] = incl;
  __syncthreads();
  int before = incl - cnt, total = 0;
#pragma unroll
  for (int k = 0; k < LABEL_THREADS / 32; ++k) {
    before += (k < warp) ? fs.warp_cnt[k] : 0;
    total += fs.warp_cnt[k];
  }
  const int n_edge = total >> 16, n_roots = n_edge + (total & 0xFFFF);
  const int at_edge = before >> 16, at_inner = n_edge + (before & 0xFFFF);

  for (int first = 0; first < n_roots; first += FLIP_LIST) {
    // my roots as local indices id0 + (site of a pass) + 8 (pass) TILE_W; a
    // thread whose roots all belong to another pass lists none
    auto list = [&](uint32_t bits, int at, bool fits) {
      if (!fits && (at >= FLIP_LIST || at + __popc(bits) <= 0)) return;
      while (bits) {
        const int n = high_bit(bits);
        bits ^= 1u << n;
        if (fits || (unsigned)at < FLIP_LIST) fs.rlist[at] = (uint16_t)root_at(n);
        ++at;
      }
    };
    if (n_roots <= FLIP_LIST) {
      list(on_edge, at_edge, true);
      list(inner, at_inner, true);
    } else {
      list(on_edge, at_edge - first, false);
      list(inner, at_inner - first, false);
    }
    __syncthreads();

    // 4. one draw per tile root, keyed by its cluster's final root
    const int n = min(n_roots - first, FLIP_LIST), ne = min(max(n_edge - first, 0), n);
    const int k0 = threadIdx.x;
    int r0 = 0, x = 0, p = 0;
    if (k0 < n) {
      r0 = fs.rlist[k0];
      p = x = tile_global(r0, y0, x0, L);
      if (k0 < ne) p = g_load(gpar + x);
    }
    for (int k = k0 + LABEL_THREADS; k < n; k += LABEL_THREADS) {
      const int r = fs.rlist[k];
      int G = tile_global(r, y0, x0, L);
      if (k < ne) G = g_find(gpar, G, limit, err);
      set_state(r, G);
    }
    if (k0 < n) set_state(r0, p == x ? x : g_find_from(gpar, x, p, limit, err));
    __syncthreads();
  }

  // 5. every site takes its tile root's state
  int8_t* dst = spins + (int64_t)(y0 + orow) * L + x0 + lx0;
  if (lx0 < w) {
#pragma unroll
    for (int j = 0; j < PASSES; ++j, dst += (int64_t)8 * L) {
      if (8 * j + orow >= h) break;
      const uint4 rv = my_roots[j * LABEL_THREADS];
      uint32_t lo = 0, hi = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) lo |= (uint32_t)ns[root_in(rv, i)] << (8 * i);
      if ((L & 7) == 0 || lx0 + 8 <= w) {
#pragma unroll
        for (int i = 0; i < 4; ++i) hi |= (uint32_t)ns[root_in(rv, 4 + i)] << (8 * i);
      }
      if ((L & 7) == 0) {
        *reinterpret_cast<uint2*>(dst) = make_uint2(lo, hi);
      } else {
        *reinterpret_cast<uint32_t*>(dst) = lo;   // 4-byte aligned: L % 4 == 0
        if (lx0 + 8 <= w) *reinterpret_cast<uint32_t*>(dst + 4) = hi;
      }
    }
  }
  __syncthreads();
}

// The flip of the few-cluster update (Sec. III, variant (c)).  Only clusters
// whose global root has its bit set in `sel` (seeded clusters) move: with FLIP
// draw w of the root, iff (uint64)w.y < P, to state (s + 1 + F_{q-1}(w.x)) mod q,
// s being the cluster's current state, that is by the same step on every site.
// Few clusters are seeded, and which of a tile's components belong to one can be
// seen without the sites' roots: the interior ones have their own bit set in
// sel, the others are edge roots (at most 576 of a tile's 8192 sites).  So a
// tile reads a bit per site of each kind, walks from its edge roots, and reads
// roots and spins only if some component of it moves.  Bound by instruction
// issue and the walks' latency; critical Ising, L = 4096, 16 x 16 seeds: 17 us
// against 53 with the state of every tile root looked up.
template <int TH>
struct FewFlipSmem {
  static constexpr int LIST = 1024;
  alignas(16) uint8_t step[TH * TILE_W];   // by local root; 0: stays
  uint16_t rlist[LIST];                    // the tile's edge roots, then its selected interior roots
  int warp_cnt[LABEL_THREADS / 32];
};

template <int TH, class Keys>
__device__ __forceinline__ void sw_flip_few_tile(const SwRep& R, int t, uint64_t sweep, int limit, FewFlipSmem<TH>& fs,
                                                 const Keys& keys, const uint32_t* sel, uint64_t P) {
  constexpr int LIST = FewFlipSmem<TH>::LIST, WORDS = TH * TILE_W / 32;
  int8_t* spins = R.spins;
  int32_t* gpar = R.gpar;
  const int q = R.q, L = R.g.W;
  int* err = R.s.err;
  const int ty = t / R.g.tiles_x, tx = t - ty * R.g.tiles_x;
  const int y0 = ty * TH, x0 = tx * TILE_W;
  const int h = min(TH, L - y0), w = min(TILE_W, L - x0);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

  // 1. roots that may move, 32 sites (a word of local indices) per thread
  uint32_t on_edge = 0u, inner = 0u;
  if (threadIdx.x < WORDS) {
    const int ly = local_y(32 * threadIdx.x), lx = local_x(32 * threadIdx.x);
    const int nv = ly < h ? min(max(w - lx, 0), 32) : 0;
    if (nv > 0) {
      const uint32_t G = (uint32_t)(y0 + ly) * (uint32_t)L + (uint32_t)(x0 + lx), at = G >> 5, off = G & 31u;
      on_edge = (uint32_t)sweep_edges(R.s, t)[threadIdx.x];
      const uint32_t lo = sel[at], hi = off + nv > 32 ? sel[at + 1] : 0u;
      inner = __funnelshift_r(lo, hi, off) & (FULL >> (32 - nv)) & ~on_edge;
    }
  }
  for (int k = threadIdx.x; k < TH * TILE_W / 16; k += LABEL_THREADS)
    reinterpret_cast<uint4*>(fs.step)[k] = make_uint4(0u, 0u, 0u, 0u);
  // 2. their list (counts of both kinds in one scan; several passes if it is full)
  const int cnt = __popc(on_edge) << 16 | __popc(inner);
  int incl = cnt;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int v = __shfl_up_sync(FULL, incl, d);
    if (lane >= d) incl += v;
  }
  if (lane == 31) fs.warp_cnt[warp] = incl;
  __syncthreads();
  int before = incl - cnt, total = 0;
#pragma unroll
  for (int k = 0; k < LABEL_THREADS / 32; ++k) {
    before += (k < warp) ? fs.warp_cnt[k] : 0;
    total += fs.warp_cnt[k];
  }
  const int n_edge = total >> 16, n_roots = n_edge + (total & 0xFFFF);
  bool moved = false;
  for (int first = 0; first < n_roots; first += LIST) {
    auto list = [&](uint32_t bits, int at) {
      while (bits) {
        const int n = high_bit(bits);
        bits ^= 1u << n;
        if ((unsigned)at < LIST) fs.rlist[at] = (uint16_t)(32 * threadIdx.x + n);
        ++at;
      }
    };
    list(on_edge, (before >> 16) - first);
    list(inner, n_edge + (before & 0xFFFF) - first);
    __syncthreads();
    // 3. the steps of the selected ones, keyed by their clusters' final roots
    const int n = min(n_roots - first, LIST), ne = min(max(n_edge - first, 0), n);
    for (int k = threadIdx.x; k < n; k += LABEL_THREADS) {
      const int r = fs.rlist[k];
      int G = tile_global(r, y0, x0, L);
      if (k < ne) {
        G = g_find(gpar, G, limit, err);
        if (!((sel[G >> 5] >> (G & 31)) & 1u)) continue;
      }
      const uint4 d = philox_draw(make_uint4((uint32_t)G, (uint32_t)sweep, (uint32_t)(sweep >> 32), TAG_FLIP), keys);
      if ((uint64_t)d.y < P) {
        fs.step[r] = (uint8_t)(1 + state_of(d.x, q - 1));
        moved = true;
      }
    }
    __syncthreads();
  }
  if (!__syncthreads_or(moved)) return;

  // 4. every site takes its tile root's step (s + step <= 252: four spins are
  //    added and reduced per word)
  const int orow = threadIdx.x / FLIP_GROUPS, lx0 = 8 * (threadIdx.x % FLIP_GROUPS);   // my sites, as in sw_flip_tile
  const uint32_t qq = 0x01010101u * (uint32_t)q;
  auto shift = [&](uint32_t s, uint32_t step) {
    const uint32_t v = __vadd4(s, step);
    return __vsub4(v, __vcmpgeu4(v, qq) & qq);
  };
  if (lx0 >= w) return;
#pragma unroll
  for (int j = 0; j < TH / 8; ++j) {
    const int ly = 8 * j + orow;
    if (ly >= h) break;
    const int64_t at = (int64_t)(y0 + ly) * L + x0 + lx0;
    const bool two = lx0 + 8 <= w;         // w is a multiple of 4
    uint4 rv = make_uint4(0u, 0u, 0u, 0u);
    if ((L & 7) == 0) {
      rv = __ldcs(reinterpret_cast<const uint4*>(R.lroot + at));
    } else {
      const uint2 a = *reinterpret_cast<const uint2*>(R.lroot + at);
      rv.x = a.x;
      rv.y = a.y;
      if (two) {
        const uint2 c = *reinterpret_cast<const uint2*>(R.lroot + at + 4);
        rv.z = c.x;
        rv.w = c.y;
      }
    }
    uint32_t lo = 0, hi = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      lo |= (uint32_t)fs.step[root_in(rv, i)] << (8 * i);
      hi |= (uint32_t)fs.step[root_in(rv, 4 + i)] << (8 * i);
    }
    uint32_t* dst = reinterpret_cast<uint32_t*>(spins + at);
    if (lo) dst[0] = shift(dst[0], lo);
    if (two && hi) dst[1] = shift(dst[1], hi);
  }
}

// Observables of the current spins of tile t (bonds joining equal spins, the
// tile's east and north bonds, and sites per state), added to the slot of
// sweep `done`.  All threads of the CTA call it.
__device__ __forceinline__ void observe_tile(const SwRep& R, int t, uint64_t done, int obs_cap, LabelTileSmem& ls) {
  const Grid& g = R.g;
  const int L = g.W, q = R.q;
  const int ty = t / g.tiles_x, tx = t - ty * g.tiles_x;
  const int y0 = ty * g.th, x0 = tx * TILE_W;
  const int h = min(g.th, L - y0), w = min(TILE_W, L - x0);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int k = threadIdx.x; k < 128; k += LABEL_THREADS) ls.hist[k] = 0;
  __syncthreads();
  long long n_eq = 0;
  int cnt[QREG];
#pragma unroll
  for (int k = 0; k < QREG; ++k) cnt[k] = 0;
  const int ly = lane, c = warp;
  const int nvalid = min(max(w - 32 * c, 0), 32);
  if (ly < h && nvalid > 0) {
    const int y = y0 + ly, x = x0 + 32 * c;
    const int yn = (y + 1 == L) ? 0 : y + 1;
    const int8_t* row = R.spins + (int64_t)y * L;
    const int8_t* rown = R.spins + (int64_t)yn * L;
    const int nw = nvalid >> 2;
    const int xe = (x + nvalid == L) ? 0 : x + nvalid;
    const uint32_t east_byte = (uint32_t)(uint8_t)row[xe];
    for (int k = 0; k < nw; ++k) {
      const uint32_t cur = *reinterpret_cast<const uint32_t*>(row + x + 4 * k);
      const uint32_t nor = *reinterpret_cast<const uint32_t*>(rown + x + 4 * k);
      const uint32_t next = (k + 1 < nw) ? *reinterpret_cast<const uint32_t*>(row + x + 4 * k + 4) : east_byte;
      n_eq += __popc(eq4(cur, (cur >> 8) | (next << 24))) + __popc(eq4(cur, nor));
      if (q <= QREG) {
#pragma unroll
        for (int s = 0; s < QREG; ++s)
          if (s < q) cnt[s] += __popc(eq4(cur, 0x01010101u * (uint32_t)s));
      } else {
        for (int j = 0; j < 4; ++j) atomicAdd(&ls.hist[(cur >> (8 * j)) & 0xFF], 1);
      }
    }
  }
  unsigned long long* oslot =
      reinterpret_cast<unsigned long long*>(R.obs + (int64_t)(done % (uint64_t)obs_cap) * (q + 1));
  add_observables<LABEL_THREADS>(n_eq, cnt, q, q <= QREG ? q : 0, oslot, ls.red, ls.hist);
  __syncthreads();
}


// ---------------------------------------------------------------------------
// Few-cluster seed selection (Sec. III, variant (c)): the seed of block b of
// the ell x ell block grid (side B = L / ell) is (bx B + F_B(w.x),
// by B + F_B(w.y)) with w the SEED draw (b, sweep); the bit of its cluster's
// global root is set in `sel`.  Runs between the merge and the flip.  If the
// seed's tile root is an edge root (its cluster may leave the tile), its
// global root is found on gpar; otherwise the tile root is the cluster's root.
__device__ __forceinline__ void few_select_seed(const SwRep& R, int ell, int64_t b, uint64_t sweep, uint32_t* sel,
                                                int limit) {
  const Grid& g = R.g;
  const int L = g.W;
  const int B = L / ell;
  const int by = (int)(b / ell), bx = (int)(b - (int64_t)by * ell);
  const uint4 w = philox(make_uint4((uint32_t)b, (uint32_t)sweep, (uint32_t)(sweep >> 32), TAG_SEED),
                         (uint32_t)R.seed, (uint32_t)(R.seed >> 32));
  const int x = bx * B + state_of(w.x, B), y = by * B + state_of(w.y, B);
  const int ty = y / g.th, tx = x / TILE_W;
  const int r = R.lroot[(int64_t)y * L + x];
  const int G = tile_global(r, ty * g.th, tx * TILE_W, L);
  const int32_t* edge_bits = sweep_edges(R.s, ty * g.tiles_x + tx);
  const bool edge = (__ldcg(edge_bits + (r >> 5)) >> (r & 31)) & 1;
  const int root = edge ? g_find(R.gpar, G, limit, R.s.err) : G;
  // most seeds of a critical lattice are in one cluster: only the first few set
  // its bit (a seed per site, L = 1024: 27 us, 290 with an atomic each)
  const uint32_t bit = 1u << (root & 31);
  if (!(__ldcg(sel + (root >> 5)) & bit)) atomicOr(sel + (root >> 5), bit);
}

}  // namespace swccl
