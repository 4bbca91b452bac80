// k_cubic.cu -- the Swendsen-Wang sweep on the periodic simple-cubic lattice.
//
// The paper develops the method on the square lattice and notes that the
// three-dimensional case follows the same steps with six neighbours
// (Secs. II and II.B).  Box X x Y x Z, site i = (z Y + y) X + x; each site
// owns its bonds to the +x, +y and +z neighbours (periodic), drawn from one
// Philox call per site (tag BOND3, counter (i, sweep), word = direction) and
// open iff the two spins are equal and the word is below T (Eq. 7).
//
// One sweep is three kernels, the structure of the fused
// square-lattice sweep (k_fused.cu) carried to bricks of 32 x 8 x 16 sites:
//  k3_local    one CTA per brick: draws the bonds of its sites, labels every
//              (x, z) plane of the brick with the square-lattice tile engine
//              (a warp per plane), joins neighbouring planes by their +y
//              bonds, writes each site's brick root (the brick component's
//              smallest index) as a 16-bit local index, marks the roots whose
//              component touches the brick's faces (edge roots: bit words per
//              brick, and a parent entry gpar[G] = G at their global index
//              G), writes the open bonds that leave the brick as face words,
//              and counts the observables of the spins it read (the previous
//              sweep's);
//  k3_merge    one thread per face bond: if its bit is set, joins the brick
//              roots on its two ends on gpar with global atomics;
//  k3_flip     one CTA per brick: lists the brick's roots; an edge root looks
//              up its cluster root R on gpar, any other root is its own
//              cluster's root; one FLIP draw per root (keyed by R, Sec. II.D)
//              gives the state every site of the brick component takes.
//  k3_observe  counts the observables of the last sweep when they are read.
// HBM traffic per site: spins read 1 B and brick roots written 2 B (local),
// brick roots read 2 B and spins written 1 B (flip), plus the face sites,
// the edge-root and face bits (0.16 B) and the sparse parent entries.
#include "fused_tile.cuh"

namespace swccl {

constexpr int B3X = 32, B3Y = 8, B3Z = 16;
constexpr int B3_SITES = B3X * B3Y * B3Z;
constexpr int B3_THREADS = 256;
static_assert(B3_THREADS == B3X * B3Y, "thread (lx, ly) walks the brick along z");

__device__ __forceinline__ int64_t site3(const Box3& b, int x, int y, int z) {
  return ((int64_t)z * b.Y + y) * b.X + x;
}

// Words per brick: edge-root bits (one per local index), then the open bonds
// that leave the brick: +z of the last plane (bit lx of word ly), +y of the
// last plane (bit lx of word lz), +x of the last column (bit lz of word ly).
// Zero along an axis one brick long (those wraps are joined in the brick).
constexpr int B3_EDGE_WORDS = B3_SITES / 32;
constexpr int B3_FACE_Z = B3_EDGE_WORDS, B3_FACE_Y = B3_FACE_Z + B3Y, B3_FACE_X = B3_FACE_Y + B3Z;
constexpr int B3_WORDS = B3_FACE_X + B3Y;

struct Brick {
  int tbx, tby, tbz, x0, y0, z0, w, h, d;
};

__device__ __forceinline__ Brick brick_at(const Box3& b, int tbx, int tby, int tbz) {
  Brick k;
  k.tbx = tbx;
  k.tby = tby;
  k.tbz = tbz;
  k.x0 = tbx * B3X;
  k.y0 = tby * B3Y;
  k.z0 = tbz * B3Z;
  k.w = min(B3X, b.X - k.x0);
  k.h = min(B3Y, b.Y - k.y0);
  k.d = min(B3Z, b.Z - k.z0);
  return k;
}

__device__ __forceinline__ Brick brick_of(const Box3& b, int t) {
  const int u = t / b.bx;
  return brick_at(b, t - u * b.bx, u % b.by, u / b.by);
}

// A brick is labeled by the square-lattice tile engine (tile_engine.cuh) with
// row = lz and strip = ly, so each warp sweeps its (x, z) plane along z (the
// +x bonds are the engine's east bonds, the +z bonds its north bonds).
static_assert(B3X == 32 && B3Y == STRIPS && B3Z <= TILE_H && B3X * B3Y == TILE_W, "brick = engine tile");

// Local index of the site (lx, ly, lz) of a brick, and the global index of
// local index l of brick k.
__device__ __forceinline__ int brick_local(int lx, int ly, int lz) { return local_of(lz, ly * B3X + lx); }
__device__ __forceinline__ int64_t brick_global(const Box3& b, const Brick& k, int l) {
  const int c = local_x(l);
  return site3(b, k.x0 + c % B3X, k.y0 + c / B3X, k.z0 + local_y(l));
}

// +y contacts listed per plane and pass; of a plane's 512 sites about 120 have
// one at the critical point.
constexpr int Y_LIST = 256;

struct Local3Smem {
  TileSmemT<B3Z> tile;
  uint32_t edge[B3_EDGE_WORDS];
  union {
    uint32_t plane[B3Y][4][B3X];             // every plane's spins: byte z of word z / 4 of column lx
    uint16_t list[B3Y][Y_LIST];              // then: the +y contacts of every plane
  };
  alignas(16) uint8_t xface[B3Y][B3Z];       // spins of the column at x0 + w
  unsigned red[(1 + QREG) * (B3_THREADS / 32)];
  int hist[128];
};

// Transposes a 32 x 32 bit matrix held one row per lane.
__device__ __forceinline__ uint32_t transpose32(uint32_t x) {
  const int lane = threadIdx.x & 31;
  constexpr uint32_t M[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const int s = 16 >> i;
    const bool up = lane & s;
    const uint32_t y = __shfl_xor_sync(FULL, x, s);
    const uint32_t keep = up ? ~M[i] : M[i];
    x = (x & keep) | (__funnelshift_l(y, y, up ? 32 - s : s) & ~keep);
  }
  return x;
}

// Spins of the 16 sites along z at column (x, y) of brick k, four per word;
// zero past the brick's depth.
__device__ __forceinline__ void load_column(const int8_t* __restrict__ spins, const Box3& b, const Brick& k, int x,
                                            int y, bool in, uint32_t (&c)[4]) {
  const int64_t XY = (int64_t)b.X * b.Y;
  const int8_t* p = spins + site3(b, in ? x : 0, in ? y : 0, k.z0);
  uint32_t v[B3Z];
#pragma unroll
  for (int lz = 0; lz < B3Z; ++lz) v[lz] = (in && lz < k.d) ? (uint32_t)(uint8_t)p[lz * XY] : 0u;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    c[j] = v[4 * j] | v[4 * j + 1] << 8 | v[4 * j + 2] << 16 | v[4 * j + 3] << 24;
}

// Bit lz set iff byte lz of the columns a and b is equal.
__device__ __forceinline__ uint32_t eq_column(const uint32_t (&a)[4], const uint32_t (&b)[4]) {
  return eq4(a[0], b[0]) | eq4(a[1], b[1]) << 4 | eq4(a[2], b[2]) << 8 | eq4(a[3], b[3]) << 12;
}

// Local step of a brick.  Bound by instruction issue: 16 draws per thread
// (about 45 instructions each) and the engine; the comparisons work on four
// spins of a column per word, the bond bits of a column (one thread) become
// the engine's row words (one lane per row) by two bit-matrix transposes, and
// the +y bonds are joined in three rounds between disjoint pairs of plane
// groups, so that plain stores do (one warp per round and boundary, no shared
// atomics).
__global__ void __launch_bounds__(B3_THREADS, 6)
k3_local(const int8_t* __restrict__ spins, uint16_t* __restrict__ lroot, int32_t* __restrict__ gpar,
         uint32_t* __restrict__ words, Box3 b, int q, uint64_t T, const __grid_constant__ PhiloxKeys keys,
         const SwCtl* __restrict__ ctl, int64_t* obs, int obs_cap, int* err) {
  __shared__ Local3Smem ls;
  TileSmemT<B3Z>& sm = ls.tile;
  uint16_t* par = sm.par;
  const Brick k = brick_of(b, blockIdx.x);
  const int lane = threadIdx.x & 31, ly = threadIdx.x >> 5;
  wait_for_previous();
  const uint64_t sweep = ctl->sweep;
  const bool do_obs = sweep > 0 && ctl->obs_done != (long long)(sweep - 1);
  const bool plane = ly < k.h;               // the warp has a plane
  const bool col = plane && lane < k.w;      // the thread has a column
  const uint32_t depth = (1u << k.d) - 1u;   // bit lz: the brick has row lz
  if (threadIdx.x < B3_EDGE_WORDS) ls.edge[threadIdx.x] = 0u;
  if (q > QREG)
    for (int j = threadIdx.x; j < 128; j += B3_THREADS) ls.hist[j] = 0;

  // 1. spins of my column, of the columns past the brick (+x, +y) and of the
  //    row past it (+z); which neighbours are equal (bit = lz)
  uint32_t ex, ey, ez;
  {
    uint32_t c[4];
    load_column(spins, b, k, k.x0 + lane, k.y0 + ly, col, c);
    const int zf = k.z0 + k.d == b.Z ? 0 : k.z0 + k.d;
    const uint32_t top = col ? (uint32_t)(uint8_t)spins[site3(b, k.x0 + lane, k.y0 + ly, zf)] : 0u;
    const int xf = k.x0 + k.w == b.X ? 0 : k.x0 + k.w, yf = k.y0 + k.h == b.Y ? 0 : k.y0 + k.h;
    if (lane < B3Z)
      ls.xface[ly][lane] = plane && lane < k.d ? (uint8_t)spins[site3(b, xf, k.y0 + ly, k.z0 + lane)] : 0;
    uint32_t n[4];
    if (ly == k.h - 1) load_column(spins, b, k, k.x0 + lane, yf, col, n);   // the plane past the brick
#pragma unroll
    for (int j = 0; j < 4; ++j) ls.plane[ly][j][lane] = c[j];
    __syncthreads();
    if (ly < k.h - 1) {
#pragma unroll
      for (int j = 0; j < 4; ++j) n[j] = ls.plane[ly + 1][j][lane];
    }
    ey = plane ? eq_column(c, n) : 0u;
#pragma unroll
    for (int j = 0; j < 4; ++j) n[j] = __shfl_down_sync(FULL, c[j], 1);
    if (lane == k.w - 1) {
      const uint4 f = *reinterpret_cast<const uint4*>(ls.xface[ly]);
      n[0] = f.x;
      n[1] = f.y;
      n[2] = f.z;
      n[3] = f.w;
    }
    ex = eq_column(c, n);
    // the column moved down by one row, the row past the brick on top
#pragma unroll
    for (int j = 0; j < 4; ++j) n[j] = (c[j] >> 8) | (j < 3 ? c[j + 1] << 24 : 0u);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if ((k.d - 1) >> 2 == j) n[j] |= top << (8 * ((k.d - 1) & 3));
    ez = eq_column(c, n);
    const uint32_t mine = col ? depth : 0u;
    ex &= mine;
    ey &= mine;
    ez &= mine;
    if (do_obs) {
      int cnt[QREG];
#pragma unroll
      for (int s = 0; s < QREG; ++s) {
        const uint32_t same = 0x01010101u * (uint32_t)s;
        const uint32_t v[4] = {same, same, same, same};
        cnt[s] = s < q && q <= QREG ? __popc(eq_column(c, v) & mine) : 0;
      }
      if (q > QREG && col)
        for (int lz = 0; lz < k.d; ++lz)
          atomicAdd(&ls.hist[(uint8_t)spins[site3(b, k.x0 + lane, k.y0 + ly, k.z0 + lz)]], 1);
      observables_warp_sums<B3_THREADS>((unsigned)(__popc(ex) + __popc(ey) + __popc(ez)), cnt, q <= QREG ? q : 0,
                                        ls.red);
    }
  }

  // 2. open bonds of my column
  if (T == 0) {
    ex = ey = ez = 0u;
  } else if (T < (1ull << 32) && plane) {
    const uint32_t thr = (uint32_t)T, XY = (uint32_t)b.X * (uint32_t)b.Y;
    uint32_t site = (uint32_t)site3(b, k.x0 + lane, k.y0 + ly, k.z0);   // wraps past the box in lanes without a column
    uint32_t ox = 0u, oy = 0u, oz = 0u;
    constexpr int U = 8;
#pragma unroll 1
    for (int z0 = 0; z0 < k.d; z0 += U) {
      uint32_t bx = 0u, by = 0u, bz = 0u;
#pragma unroll
      for (int i = 0; i < U; ++i) {
        const uint4 r =
            philox_draw(make_uint4(site, (uint32_t)sweep, (uint32_t)(sweep >> 32), TAG_BOND3), keys);
        set_if_below(bx, r.x, thr, 1u << i);
        set_if_below(by, r.y, thr, 1u << i);
        set_if_below(bz, r.z, thr, 1u << i);
        site += XY;
      }
      ox |= bx << z0;
      oy |= by << z0;
      oz |= bz << z0;
    }
    ex &= ox;
    ey &= oy;
    ez &= oz;
  }

  // 3. row words (lane = row lz) of the plane's bonds: inside the brick for
  //    the engine and the +y joins, leaving it for the merge, wrapping inside
  //    it where the axis is one brick long
  const uint32_t xz = transpose32(ex | ez << 16);
  uint32_t yb = transpose32(ey);                                   // lanes 0 .. 15
  uint32_t we = lane < B3Z ? xz : 0u;
  uint32_t wn = __shfl_sync(FULL, xz, (lane & 15) + 16);
  if (lane >= B3Z) wn = 0u;
  const uint32_t last_x = 1u << (k.w - 1);
  const uint32_t x_out = __ballot_sync(FULL, (we & last_x) != 0u);  // bit = lz
  const uint32_t z_out = __shfl_sync(FULL, wn, k.d - 1);            // bit = lx
  we &= ~last_x;
  if (lane == k.d - 1) wn = 0u;
  const bool y_last = ly == k.h - 1;
  uint32_t* out = words + (int64_t)blockIdx.x * B3_WORDS;
  if (lane == 0) {
    out[B3_FACE_Z + ly] = b.bz > 1 ? z_out : 0u;
    out[B3_FACE_X + ly] = b.bx > 1 ? x_out : 0u;
  }
  if (y_last && lane < B3Z) out[B3_FACE_Y + lane] = b.by > 1 ? yb : 0u;

  // 4. the engine labels the planes (no bond joins two of its strips)
  tile_engine(sm, we, wn, k.d, B3X * k.h, err);
  __syncthreads();

  // 5. +y bonds between planes ly and ly + 1.  One contact per overlap of an
  //    x run with a run of the next plane is kept, and none whose row below
  //    has the bond too and +z bonds up on both sides.  Rounds: boundaries
  //    0 2 4 6, then 1 5, then 3 (each warp's pairs lie in planes that no other
  //    warp of the round touches).
  uint16_t* list = ls.list[ly];
  int n_list = 0;
  {
    uint32_t C = 0u;
    if (ly + 1 < k.h) {
      const uint32_t up_e = lane < B3Z ? sm.be[lane * STRIPS + ly + 1] : 0u;
      const uint32_t up_n = lane < B3Z ? sm.bn[lane * STRIPS + ly + 1] : 0u;
      const uint32_t j2 = we & up_e;
      const uint32_t implied = __shfl_up_sync(FULL, yb & wn & up_n, 1);
      C = yb & ~((seg_or_up(yb, j2) << 1) & (j2 << 1));
      if (lane > 0) C &= ~implied;
    }
    const int cnt = __popc(C);
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += v;
    }
    n_list = __shfl_sync(FULL, incl, 31);
    const int row = brick_local(0, ly, lane);
    const int my_round = !(ly & 1) ? 0 : (ly & 3) == 1 ? 1 : 2;
#pragma unroll 1
    for (int round = 0; round < 3; ++round) {
      if (round == my_round) {
        for (int first = 0; first < n_list; first += Y_LIST) {
          int at = incl - cnt - first;
          for (uint32_t x = C; x; x &= x - 1, ++at)
            if ((unsigned)at < Y_LIST) list[at] = (uint16_t)(row + high_bit(x & -x));
          __syncwarp();
          const int n = min(n_list - first, Y_LIST);
          for (int j = lane; j - lane < n; j += 32) {
            int a = 2 * brick_local(0, ly, 0), c = a;
            if (j < n) {
              const int site = list[j];
              const int lz = local_y(site);
              a = par[site];
              c = par[brick_local(0, ly + 1, lz) + (site & (B3X - 1))];
            }
            const int hooked = sm_union_strips(par, a, c, err);
            if (j < n) list[j] = (uint16_t)hooked;
          }
          __syncwarp();
        }
      }
      __syncthreads();
    }
  }
  // wraps of an axis one brick long
  const bool wraps = b.bx == 1 || b.by == 1 || b.bz == 1;
  if (wraps) {
    if (plane) {
      const int self = 2 * brick_local(0, ly, 0);
      if (b.bx == 1) {
        const bool on = lane < k.d && ((x_out >> lane) & 1u);
        sm_union_tile(par, on ? 2 * brick_local(k.w - 1, ly, lane) : self, on ? 2 * brick_local(0, ly, lane) : self,
                      err);
      }
      if (b.bz == 1) {
        const bool on = (z_out >> lane) & 1u;
        sm_union_tile(par, on ? 2 * brick_local(lane, ly, k.d - 1) : self, on ? 2 * brick_local(lane, ly, 0) : self,
                      err);
      }
      if (b.by == 1 && y_last) {
        for (int lz = 0; lz < k.d; ++lz) {
          const bool on = (__shfl_sync(FULL, yb, lz) >> lane) & 1u;
          sm_union_tile(par, on ? 2 * brick_local(lane, ly, lz) : self, on ? 2 * brick_local(lane, 0, lz) : self, err);
        }
      }
    }
    __syncthreads();
  }

  // 6. hooked roots take their final roots; a parent is replaced by an
  //    ancestor, so other walks through it stay valid.  A root hooked in any
  //    plane may be any warp's entry, so one list that did not hold all its
  //    joins (or a wrap, which is not listed) makes every site take its root.
  const bool listed = !__syncthreads_or(n_list > Y_LIST || wraps);
  if (plane) {
    const int self = 2 * brick_local(0, ly, 0);
    if (listed) {
      for (int j = lane; j - lane < n_list; j += 32) {
        const int x = j < n_list ? (int)list[j] : 0xFFFF;
        int f[1] = {x != 0xFFFF ? x : self};
        sm_find_tile(par, f, err);
        if (x != 0xFFFF) sm_set(par, x, f[0]);
      }
    } else {
      for (int lz = 0; lz < k.d; ++lz) {
        const int x = 2 * brick_local(lane, ly, lz);
        int f[1] = {x};
        sm_find_tile(par, f, err);
        sm_set(par, x, f[0]);
      }
    }
  }
  __syncthreads();

  // 7. brick roots of my plane's sites (site -> its plane's node -> that
  //    node's plane root -> the brick root), eight consecutive sites per
  //    thread and step; roots on the brick's faces marked; bit 4j + i of mine
  //    flags site 2i of step j as a root, bit 16 + 4j + i site 2i + 1
  const int lx0 = 8 * (lane & 3);
  const int in = plane ? min(max(k.w - lx0, 0), 8) : 0;
  uint32_t mine = 0;
  if (in > 0) {
    const uint32_t in_mask = ((1u << ((in + 1) >> 1)) - 1u) | ((1u << (in >> 1)) - 1u) << 16;
    auto mark = [&](uint32_t r) {
      const uint32_t bit = 1u << (r & 31);
      if (!(*reinterpret_cast<volatile uint32_t*>(&ls.edge[r >> 5]) & bit)) atomicOr(&ls.edge[r >> 5], bit);
    };
#pragma unroll
    for (int j = 0; j < B3Z / 8; ++j) {
      const int lz = (lane >> 2) + 8 * j;
      if (lz >= k.d) continue;
      const int l0 = brick_local(lx0, ly, lz);
      const uint4 v = *reinterpret_cast<const uint4*>(par + l0);
      auto two = [&](uint32_t w) {
        const int p0 = sm_at(par, w & 0xFFFFu), p1 = sm_at(par, w >> 16);
        return (uint32_t)sm_at(par, p0) >> 1 | (uint32_t)sm_at(par, p1) << 15;
      };
      const uint32_t wv[4] = {two(v.x), two(v.y), two(v.z), two(v.w)};
      uint16_t* dst = lroot + site3(b, k.x0 + lx0, k.y0 + ly, k.z0 + lz);
      if ((b.X & 7) == 0) {   // then k.w is a multiple of 8 too
        *reinterpret_cast<uint4*>(dst) = make_uint4(wv[0], wv[1], wv[2], wv[3]);
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (i < in) dst[i] = (uint16_t)(wv[i >> 1] >> (16 * (i & 1)));
      }
      const uint32_t own = (uint32_t)l0 * 0x00010001u + 0x00010000u;   // (l0, l0 + 1)
      uint32_t m = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) m |= zero_halves(wv[i] ^ (own + (uint32_t)i * 0x00020002u)) >> (15 - i);
      mine |= (m & in_mask) << (4 * j);
      if (ly == 0 || y_last || lz == 0 || lz == k.d - 1) {
        uint32_t left = 0xFFFFFFFFu;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint32_t r = (wv[i >> 1] >> (16 * (i & 1))) & 0xFFFFu;
          if (i < in && r != left) mark(r);
          left = r;
        }
      } else {
        if (lx0 == 0) mark(wv[0] & 0xFFFFu);
        if (lx0 + in == k.w && in > 0) mark((wv[(in - 1) >> 1] >> (16 * ((in - 1) & 1))) & 0xFFFFu);
      }
    }
  }
  if (do_obs) {
    unsigned long long* oslot =
        reinterpret_cast<unsigned long long*>(obs + (int64_t)((sweep - 1) % (uint64_t)obs_cap) * (q + 1));
    observables_commit<B3_THREADS>(q, q <= QREG ? q : 0, oslot, ls.red, ls.hist);
  }
  __syncthreads();
  // 8. parent entries of edge roots; the brick's edge bits for the flip
  while (mine) {
    const int bit = __ffs(mine) - 1;
    mine &= mine - 1;
    const int jk = bit & 15;
    const int l = brick_local(lx0, ly, (lane >> 2) + 8 * (jk >> 2)) + 2 * (jk & 3) + (bit >> 4);
    if ((ls.edge[l >> 5] >> (l & 31)) & 1u) {
      const int32_t G = (int32_t)brick_global(b, k, l);
      gpar[G] = G;
    }
  }
  if (threadIdx.x < B3_EDGE_WORDS) out[threadIdx.x] = ls.edge[threadIdx.x];
}

// One warp per face word of a brick (x: two words): z faces 0 .. 7 (bit lx of
// word ly), y face 8 .. 23 (bit lx of word lz), x face 24 .. 27 (bits lz of
// words ly, ly + 1).  A lane whose root pair equals its left neighbour's skips
// the union.  Bound by the latency of the root loads and parent walks.
constexpr int B3_MERGE_UNITS = B3Y + B3Z + B3Y / 2;
constexpr int MERGE3_THREADS = 256;

__global__ void __launch_bounds__(MERGE3_THREADS)
k3_merge(const uint16_t* __restrict__ lroot, int32_t* gpar, const uint32_t* __restrict__ words, Box3 b, int limit,
         SwCtl* ctl, int64_t* obs, int obs_cap, int q) {
  wait_for_previous();
  int* err = &ctl->err;
  if (blockIdx.x == 0) {   // the next sweep's local step fills this sweep's observable slot
    const uint64_t s = ctl->sweep;
    if ((int)threadIdx.x <= q) obs[(int64_t)(s % (uint64_t)obs_cap) * (q + 1) + threadIdx.x] = 0;
    __syncthreads();
    if (threadIdx.x == 0) ctl->sweep = s + 1;
  }
  const int64_t unit = blockIdx.x * (int64_t)(MERGE3_THREADS / 32) + (threadIdx.x >> 5);
  if (unit >= b.n_bricks() * B3_MERGE_UNITS) return;
  const int t = (int)(unit / B3_MERGE_UNITS), u = (int)(unit - (int64_t)t * B3_MERGE_UNITS);
  const int lane = threadIdx.x & 31;
  const uint32_t* wd = words + (int64_t)t * B3_WORDS;
  int lx = lane, ly = u, lz = 0, axis = 2;
  uint32_t bits;
  if (u < B3Y) {
    bits = wd[B3_FACE_Z + u] >> lane;
  } else if (u < B3Y + B3Z) {
    lz = u - B3Y;
    axis = 1;
    bits = wd[B3_FACE_Y + lz] >> lane;
  } else {
    ly = 2 * (u - B3Y - B3Z) + (lane >> 4);
    lz = lane & 15;
    axis = 0;
    bits = wd[B3_FACE_X + ly] >> lz;
  }
  bool valid = bits & 1u;
  if (!__any_sync(FULL, valid)) return;
  const Brick k = brick_of(b, t);
  if (axis == 2) lz = k.d - 1;
  if (axis == 1) ly = k.h - 1;
  if (axis == 0) lx = k.w - 1;
  const Brick kn = brick_at(b, axis == 0 ? (k.tbx + 1 == b.bx ? 0 : k.tbx + 1) : k.tbx,
                            axis == 1 ? (k.tby + 1 == b.by ? 0 : k.tby + 1) : k.tby,
                            axis == 2 ? (k.tbz + 1 == b.bz ? 0 : k.tbz + 1) : k.tbz);
  int ga = 0, gb = 0;
  if (valid) {   // the brick roots on the two ends (both edge roots)
    const int ra = lroot[site3(b, k.x0 + lx, k.y0 + ly, k.z0 + lz)];
    const int rb = lroot[site3(b, kn.x0 + (axis == 0 ? 0 : lx), kn.y0 + (axis == 1 ? 0 : ly),
                               kn.z0 + (axis == 2 ? 0 : lz))];
    ga = (int)brick_global(b, k, ra);
    gb = (int)brick_global(b, kn, rb);
  }
  valid = valid && ga != gb;
  const unsigned long long key =
      valid ? ((unsigned long long)(unsigned)min(ga, gb) << 32) | (unsigned)max(ga, gb) : ~0ull;
  const unsigned long long left = __shfl_up_sync(FULL, key, 1);
  if (valid && (lane == 0 || left != key)) g_union(gpar, ga, gb, limit, err);
}

// Flip of a brick: a thread owns the sites it wrote in k3_local's step 7 (two
// steps of eight consecutive sites of a row, one 16-byte load of roots each).
__global__ void __launch_bounds__(B3_THREADS, 6)
k3_flip(int8_t* __restrict__ spins, const uint16_t* __restrict__ lroot, int32_t* gpar,
        const uint32_t* __restrict__ words, Box3 b, int q, const __grid_constant__ PhiloxKeys keys,
        const SwCtl* __restrict__ ctl, int limit, int* err) {
  __shared__ uint16_t rlist[B3_SITES];
  __shared__ uint8_t ns[B3_SITES];
  __shared__ uint32_t edge[B3_EDGE_WORDS];
  __shared__ int warp_cnt[B3_THREADS / 32];
  const Brick k = brick_of(b, blockIdx.x);
  wait_for_previous();
  const uint64_t sweep = ctl->sweep - 1;   // the merge has advanced the counter
  const int lane = threadIdx.x & 31, ly = threadIdx.x >> 5, warp = ly;
  const int lx0 = 8 * (lane & 3);
  const int in = ly < k.h ? min(max(k.w - lx0, 0), 8) : 0;
  const bool whole = (b.X & 7) == 0;   // rows start 16-byte aligned, in is 0 or 8
  if (threadIdx.x < B3_EDGE_WORDS) edge[threadIdx.x] = words[(int64_t)blockIdx.x * B3_WORDS + threadIdx.x];
  // 1. brick roots of my sites (0xFFFF outside the brick), and which are roots
  uint4 roots[B3Z / 8];
  uint32_t mine = 0;
#pragma unroll
  for (int j = 0; j < B3Z / 8; ++j) {
    const int lz = (lane >> 2) + 8 * j;
    uint32_t v[4] = {0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu};
    if (lz < k.d && in > 0) {
      const uint16_t* src = lroot + site3(b, k.x0 + lx0, k.y0 + ly, k.z0 + lz);
      if (whole) {
        const uint4 r = *reinterpret_cast<const uint4*>(src);
        v[0] = r.x;
        v[1] = r.y;
        v[2] = r.z;
        v[3] = r.w;
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (i < in) v[i >> 1] = i & 1 ? (v[i >> 1] & 0xFFFFu) | (uint32_t)src[i] << 16 : 0xFFFF0000u | src[i];
      }
    }
    const uint32_t own = (uint32_t)brick_local(lx0, ly, lz) * 0x00010001u + 0x00010000u;
#pragma unroll
    for (int i = 0; i < 4; ++i) mine |= zero_halves(v[i] ^ (own + (uint32_t)i * 0x00020002u)) >> (15 - (4 * j + i));
    roots[j] = make_uint4(v[0], v[1], v[2], v[3]);
  }
  // 2. the brick's root list, edge roots flagged
  const int cnt = __popc(mine);
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(FULL, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) warp_cnt[warp] = incl;
  __syncthreads();
  int base = 0, n_roots = 0;
#pragma unroll
  for (int j = 0; j < B3_THREADS / 32; ++j) {
    base += (j < warp) ? warp_cnt[j] : 0;
    n_roots += warp_cnt[j];
  }
  base += incl - cnt;
  while (mine) {
    const int bit = __ffs(mine) - 1;
    mine &= mine - 1;
    const int jk = bit & 15;
    const int l = brick_local(lx0, ly, (lane >> 2) + 8 * (jk >> 2)) + 2 * (jk & 3) + (bit >> 4);
    rlist[base++] = (uint16_t)l | (((edge[l >> 5] >> (l & 31)) & 1u) ? EDGE_ROOT : (uint16_t)0);
  }
  __syncthreads();
  // 3. one draw per brick root, keyed by its cluster's root; a thread takes
  //    its roots two at a time, their parent walks in lock step
  constexpr int U = 2;
  for (int j0 = threadIdx.x; j0 < n_roots; j0 += U * B3_THREADS) {
    int r[U], R[U];
    bool act[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = j0 + u * B3_THREADS;
      const int raw = j < n_roots ? (int)rlist[j] : 0;
      r[u] = raw & ROOT_MASK;
      R[u] = (int)brick_global(b, k, r[u]);
      act[u] = j < n_roots && (raw & EDGE_ROOT);
    }
    g_find_multi<U>(gpar, R, act, limit, err);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (j0 + u * B3_THREADS >= n_roots) break;
      const uint4 w = philox_draw(make_uint4((uint32_t)R[u], (uint32_t)sweep, (uint32_t)(sweep >> 32), TAG_FLIP), keys);
      ns[r[u]] = (uint8_t)state_of(w.x, q);
    }
  }
  __syncthreads();
  // 4. every site takes its brick root's state
#pragma unroll
  for (int j = 0; j < B3Z / 8; ++j) {
    const int lz = (lane >> 2) + 8 * j;
    if (lz >= k.d || in == 0) continue;
    int8_t* dst = spins + site3(b, k.x0 + lx0, k.y0 + ly, k.z0 + lz);
    if (whole) {
      uint32_t lo = 0, hi = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        lo |= (uint32_t)ns[root_in(roots[j], i)] << (8 * i);
        hi |= (uint32_t)ns[root_in(roots[j], 4 + i)] << (8 * i);
      }
      *reinterpret_cast<uint2*>(dst) = make_uint2(lo, hi);
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (i < in) dst[i] = (int8_t)ns[root_in(roots[j], i)];
    }
  }
}

// Observables of the last sweep when they are read: a warp per row of sites,
// four sites per lane and step where rows are word aligned.
constexpr int OBS3_THREADS = 256;

__global__ void __launch_bounds__(OBS3_THREADS)
k3_observe(const int8_t* __restrict__ spins, Box3 b, int q, SwCtl* __restrict__ ctl, int64_t* obs, int obs_cap) {
  __shared__ unsigned long long red[(1 + QREG) * (OBS3_THREADS / 32)];
  __shared__ int hist[128];
  for (int k = threadIdx.x; k < 128; k += OBS3_THREADS) hist[k] = 0;
  __syncthreads();
  long long n_eq = 0;
  int cnt[QREG];
#pragma unroll
  for (int k = 0; k < QREG; ++k) cnt[k] = 0;
  const int lane = threadIdx.x & 31;
  const int rows = b.Y * b.Z;   // X Y Z <= 2^30
  const int step = (b.X & 3) == 0 ? 4 : 1;
  for (int r = blockIdx.x * (OBS3_THREADS / 32) + (threadIdx.x >> 5); r < rows; r += gridDim.x * (OBS3_THREADS / 32)) {
    const int z = r / b.Y, y = r - z * b.Y;
    const int8_t* p = spins + (int64_t)r * b.X;
    const int8_t* py = spins + site3(b, 0, y + 1 == b.Y ? 0 : y + 1, z);
    const int8_t* pz = spins + site3(b, 0, y, z + 1 == b.Z ? 0 : z + 1);
    for (int x = lane * step; x < b.X; x += 32 * step) {
      const int xe = x + step == b.X ? 0 : x + step;
      if (step == 4) {
        const uint32_t s = *reinterpret_cast<const uint32_t*>(p + x);
        const uint32_t e = (s >> 8) | (uint32_t)(uint8_t)p[xe] << 24;
        n_eq += __popc(eq4(s, e)) + __popc(eq4(s, *reinterpret_cast<const uint32_t*>(py + x))) +
                __popc(eq4(s, *reinterpret_cast<const uint32_t*>(pz + x)));
        if (q <= QREG) {
#pragma unroll
          for (int k = 0; k < QREG; ++k)
            if (k < q) cnt[k] += __popc(eq4(s, 0x01010101u * (uint32_t)k));
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i) atomicAdd(&hist[(s >> (8 * i)) & 0xFFu], 1);
        }
      } else {
        const int s = p[x];
        n_eq += (p[xe] == s) + (py[x] == s) + (pz[x] == s);
        if (q <= QREG) {
#pragma unroll
          for (int k = 0; k < QREG; ++k) cnt[k] += (s == k);
        } else {
          atomicAdd(&hist[s], 1);
        }
      }
    }
  }
  const uint64_t done = ctl->sweep - 1;
  unsigned long long* slot =
      reinterpret_cast<unsigned long long*>(obs + (int64_t)(done % (uint64_t)obs_cap) * (q + 1));
  add_observables<OBS3_THREADS>(n_eq, cnt, q, q <= QREG ? q : 0, slot, red, hist);
  if (blockIdx.x == 0 && threadIdx.x == 0) ctl->obs_done = (long long)done;
}

// Canonical labels of the last sweep: the cluster root of every site's brick root.
__global__ void k3_labels(const uint16_t* __restrict__ lroot, int32_t* gpar, const uint32_t* __restrict__ words,
                          Box3 b, int32_t* out, int limit, int* err) {
  const int64_t n = b.n();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % b.X);
    const int64_t yz = i / b.X;
    const int y = (int)(yz % b.Y), z = (int)(yz / b.Y);
    const int t = ((z / B3Z) * b.by + y / B3Y) * b.bx + x / B3X;
    const Brick k = brick_of(b, t);
    const int r = lroot[i];
    int R = (int)brick_global(b, k, r);
    if ((words[(int64_t)t * B3_WORDS + (r >> 5)] >> (r & 31)) & 1u) R = g_find(gpar, R, limit, err);
    out[i] = R;
  }
}

// ---------------------------------------------------------------------------
Box3 make_box3(int X, int Y, int Z) {
  Box3 b;
  b.X = X;
  b.Y = Y;
  b.Z = Z;
  b.bx = (X + B3X - 1) / B3X;
  b.by = (Y + B3Y - 1) / B3Y;
  b.bz = (Z + B3Z - 1) / B3Z;
  return b;
}

static int limit3(const Box3& b) { return (int)std::min<int64_t>(b.n() + 64, (int64_t)1 << 30); }

static unsigned stride_blocks(int64_t n, int threads) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + threads - 1) / threads, 152 * 16));
}

int64_t brick_words3(const Box3& b) { return b.n_bricks() * B3_WORDS; }

cudaError_t launch_sweep3(int8_t* spins, uint16_t* lroot, int32_t* gpar, uint32_t* words, const Box3& b, int q,
                          uint64_t T, uint64_t seed, SwCtl* ctl, int64_t* obs, int obs_cap, cudaStream_t st,
                          cudaEvent_t* ev) {
  cudaError_t e;
  int* err = &ctl->err;
  if (ev && (e = cudaEventRecord(ev[0], st)) != cudaSuccess) return e;
  const PhiloxKeys keys = philox_keys(seed);
  e = launch_after(k3_local, (unsigned)b.n_bricks(), B3_THREADS, st, spins, lroot, gpar, words, b, q, T, keys, ctl, obs,
                   obs_cap, err);
  if (e != cudaSuccess) return e;
  if (ev && (e = cudaEventRecord(ev[1], st)) != cudaSuccess) return e;
  // a box of one brick has no face bonds: one block only advances the counter
  constexpr int WARPS = MERGE3_THREADS / 32;
  const bool faces = b.bx > 1 || b.by > 1 || b.bz > 1;
  const int64_t blocks = faces ? (b.n_bricks() * B3_MERGE_UNITS + WARPS - 1) / WARPS : 1;
  e = launch_after(k3_merge, (unsigned)blocks, MERGE3_THREADS, st, lroot, gpar, words, b, limit3(b), ctl, obs, obs_cap, q);
  if (e != cudaSuccess) return e;
  if (ev && (e = cudaEventRecord(ev[2], st)) != cudaSuccess) return e;
  e = launch_after(k3_flip, (unsigned)b.n_bricks(), B3_THREADS, st, spins, lroot, gpar, words, b, q, keys, ctl, limit3(b),
                   err);
  if (e != cudaSuccess) return e;
  // the advance is part of the merge: its phase is empty
  if (ev && ((e = cudaEventRecord(ev[3], st)) != cudaSuccess || (e = cudaEventRecord(ev[4], st)) != cudaSuccess))
    return e;
  return cudaSuccess;
}

cudaError_t launch_observe3(const int8_t* spins, const Box3& b, int q, SwCtl* ctl, int64_t* obs, int obs_cap,
                            cudaStream_t st) {
  k3_observe<<<stride_blocks((int64_t)b.Y * b.Z, OBS3_THREADS / 32), OBS3_THREADS, 0, st>>>(spins, b, q, ctl, obs, obs_cap);
  return cudaGetLastError();
}

cudaError_t launch_labels3(const uint16_t* lroot, int32_t* gpar, const uint32_t* words, const Box3& b,
                           int32_t* out, int* err, cudaStream_t st) {
  k3_labels<<<stride_blocks(b.n(), 256), 256, 0, st>>>(lroot, gpar, words, b, out, limit3(b), err);
  return cudaGetLastError();
}

}  // namespace swccl
