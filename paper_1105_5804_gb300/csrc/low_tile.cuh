// low_tile.cuh -- the draw-and-label step on tiles of TH = 8 or 16 rows.
//
// A small lattice has fewer 32 x 256 tiles than the GPU has SMs, and a tile's
// time is then the latency of its warps' serial chains (bonds of 32 sites per
// lane, 32 rows swept, list after list; an instruction every four or five
// cycles): 11 us at L = 256, where 8 SMs of 152 have work.  Lower tiles give
// the SMs that are left a share of it and make the chains shorter: a lane draws
// the bonds of 8 or 16 sites, all its Philox calls in step, and a strip sweeps
// 8 or 16 rows.  The seams they add cost the merge little, which is bound by
// the latency of its walks.  A whole sweep at L = 256: 25.5 us with 32 rows, 20.2
// with 8 (17.5 since the sweeps' launches overlap).  Everything but the bonds' division among the lanes is as in
// sw_label_tile.
#pragma once
#include "fused_tile.cuh"

namespace swccl {

template <int TH>
struct LowTileSmem {
  TileSmemT<TH> tile;
  uint32_t edge_bits[EDGE_WORDS];
  unsigned red[(1 + QREG) * (LABEL_THREADS / 32)];
  int hist[128];
};

template <int TH, class Keys>
__device__ __forceinline__ void sw_label_low_tile(const SwRep& R, int t, uint64_t sweep, bool do_obs, int obs_cap,
                                                  LowTileSmem<TH>& ls, const Keys& keys) {
  constexpr int SP = TH;                 // 32 / TH lanes per row, SP sites per lane
  constexpr int NW = LABEL_THREADS / 32;
  const int8_t* spins = R.spins;
  const int q = R.q;
  const uint64_t T = R.T;
  const int L = R.g.W;
  const int ty = t / R.g.tiles_x, tx = t - ty * R.g.tiles_x;
  const int y0 = ty * TH, x0 = tx * TILE_W;
  const int h = min(TH, L - y0), w = min(TILE_W, L - x0);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int uw = min(max(w - 32 * warp, 0), 32);
  ls.edge_bits[threadIdx.x] = 0u;        // the engine's barriers order it before the marks
  if (q > QREG) {
    for (int k = threadIdx.x; k < 128; k += LABEL_THREADS) ls.hist[k] = 0;
    __syncthreads();
  }

  // 1. bonds of my strip: lane (row, part) takes SP sites; observables of the
  //    spins read
  uint32_t e = 0u, nb = 0u;
  {
    const int row = lane % TH, part = lane / TH;
    const int nv = row < h ? min(max(uw - SP * part, 0), SP) : 0;
    const int y = y0 + row, x = x0 + 32 * warp + SP * part;
    const int64_t at = (int64_t)y * L + x, at_n = (int64_t)(y + 1 == L ? 0 : y + 1) * L + x;
    uint32_t s[SP / 4] = {}, n[SP / 4] = {}, east = 0u;
    if (nv > 0) {
#pragma unroll
      for (int j = 0; j < SP / 4; ++j) {
        if (4 * j < nv) {
          s[j] = *reinterpret_cast<const uint32_t*>(spins + at + 4 * j);
          n[j] = *reinterpret_cast<const uint32_t*>(spins + at_n + 4 * j);
        }
      }
      east = (uint8_t)spins[(int64_t)y * L + (x + nv == L ? 0 : x + nv)];
    }
    const uint32_t valid = (1u << nv) - 1u;
    int ones = 0;
    if (q == 2) {
      uint32_t sb = 0u, mb = 0u;
#pragma unroll
      for (int j = 0; j < SP / 4; ++j) {
        sb |= ((s[j] * 0x01020408u) >> 24) << (4 * j);
        mb |= ((n[j] * 0x01020408u) >> 24) << (4 * j);
      }
      e = ~(sb ^ ((sb | east << nv) >> 1)) & valid;
      nb = ~(sb ^ mb) & valid;
      ones = __popc(sb);
    } else {
#pragma unroll
      for (int j = 0; j < SP / 4; ++j) {
        const uint32_t next = 4 * j + 4 < nv ? s[(j + 1) % (SP / 4)] : east;
        e |= eq4(s[j], (s[j] >> 8) | next << 24) << (4 * j);
        nb |= eq4(s[j], n[j]) << (4 * j);
      }
      e &= valid;
      nb &= valid;
    }
    if (do_obs) {
      const unsigned v = __reduce_add_sync(FULL, (unsigned)(__popc(e) + __popc(nb)));
      if (lane == 0) ls.red[warp] = v;
      if (q == 2) {
        const unsigned v1 = __reduce_add_sync(FULL, (unsigned)ones);
        if (lane == 0) {
          ls.red[NW + warp] = (unsigned)(h * uw) - v1;
          ls.red[2 * NW + warp] = v1;
        }
      } else if (q <= QREG) {
        for (int k = 0; k < q; ++k) {
          const uint32_t same = 0x01010101u * (uint32_t)k;
          uint32_t is = 0u;
#pragma unroll
          for (int j = 0; j < SP / 4; ++j) is |= eq4(s[j], same) << (4 * j);
          const unsigned vk = __reduce_add_sync(FULL, (unsigned)__popc(is & valid));
          if (lane == 0) ls.red[(1 + k) * NW + warp] = vk;
        }
      } else {
        for (int j = 0; j < nv; ++j) atomicAdd(&ls.hist[(uint8_t)spins[at + j]], 1);
      }
    }
    if (T == 0) {
      e = nb = 0u;
    } else if (T < (1ull << 32)) {
      uint4 d[SP / 2];
#pragma unroll
      for (int i = 0; i < SP / 2; ++i)
        d[i] = make_uint4((uint32_t)(at >> 1) + i, (uint32_t)sweep, (uint32_t)(sweep >> 32), TAG_BOND);
      philox_draws(d, keys);
      uint32_t oe = 0u, on = 0u;
      const uint32_t thr = (uint32_t)T;
#pragma unroll
      for (int i = 0; i < SP / 2; ++i) {
        set_if_below(oe, d[i].x, thr, 1u << (2 * i));
        set_if_below(oe, d[i].z, thr, 2u << (2 * i));
        set_if_below(on, d[i].y, thr, 1u << (2 * i));
        set_if_below(on, d[i].w, thr, 2u << (2 * i));
      }
      e &= oe;
      nb &= on;
    }
    e <<= SP * part;                     // put the row words together
    nb <<= SP * part;
#pragma unroll
    for (int o = TH; o < 32; o *= 2) {
      e |= __shfl_xor_sync(FULL, e, o);
      nb |= __shfl_xor_sync(FULL, nb, o);
    }
    if (lane >= TH) e = nb = 0u;         // lane = row from here on
  }
  uint32_t e_last = 0u;                  // east bonds leaving the tile, bit = row
  if (uw > 0 && 32 * warp + uw == w) {
    const uint32_t bit = 1u << (uw - 1);
    e_last = __ballot_sync(FULL, (e & bit) != 0u);
    e &= ~bit;
  }

  // 2. label the tile
  tile_engine(ls.tile, e, nb, h, w, R.s.err);
  if (do_obs) {   // observables of the spins read (the previous sweep's result)
    unsigned long long* oslot =
        reinterpret_cast<unsigned long long*>(R.obs + (int64_t)((sweep - 1) % (uint64_t)obs_cap) * (q + 1));
    observables_commit<LABEL_THREADS>(q, q <= QREG ? q : 0, oslot, ls.red, ls.hist);
  }

  // 3. tile roots of my strip (as in sw_label_tile; kept in L2, which holds all
  //    of a small lattice)
  {
    const int lx = 32 * warp + 8 * (lane & 3);
#pragma unroll
    for (int j = 0; j < TH / 8; ++j) {
      const int ly = 8 * j + (lane >> 2);
      if (ly >= h || lx >= w) continue;
      const uint4 r = roots_of(ls.tile.par, local_of(ly, lx));
      uint16_t* dst = R.lroot + (int64_t)(y0 + ly) * L + x0 + lx;
      if ((L & 7) == 0) {   // then w is a multiple of 8 too
        *reinterpret_cast<uint4*>(dst) = r;
      } else {
        *reinterpret_cast<uint2*>(dst) = make_uint2(r.x, r.y);
        if (lx + 8 <= w) *reinterpret_cast<uint2*>(dst + 4) = make_uint2(r.z, r.w);
      }
    }
  }
  // 4. seam record; parent entries of edge roots; edge roots marked
  seam_strip(ls.tile.par, R.s.seams + (int64_t)t * SeamLayout::INTS, R.gpar, ls.edge_bits, nb, e_last, h, w, y0, x0, L);
  __syncthreads();
  // 5. edge-root bits; each thread reads and next clears only its own word
  sweep_edges(R.s, t)[threadIdx.x] = (int32_t)ls.edge_bits[threadIdx.x];
}

}  // namespace swccl
