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
//  k3_merge    one CTA per brick: lists the pairs of brick roots that its open
//              face bonds join, then joins them on gpar with global atomics;
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
static_assert(B3_THREADS == 32 * B3Y && 32 == 2 * B3Z, "a warp per plane, two lanes per row");

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
  uint16_t list[B3Y][Y_LIST];                // the +y contacts of every plane
  unsigned red[(1 + QREG) * (B3_THREADS / 32)];
  int hist[128];
};

// Sixteen consecutive spins from site i on, of which the first nv are wanted
// (the others are arbitrary).  whole: rows start 16-byte aligned and nv is 0 or
// 16; otherwise aligned words are shifted into place (a word is read only if it
// holds a wanted spin, so reads stay inside the array's last word).
__device__ __forceinline__ void load_row(const int8_t* spins, uint32_t i, int nv, bool whole,
                                         uint32_t (&c)[4]) {
  if (whole) {
    const uint4 v = nv > 0 ? *reinterpret_cast<const uint4*>(spins + i) : make_uint4(0u, 0u, 0u, 0u);
    c[0] = v.x;
    c[1] = v.y;
    c[2] = v.z;
    c[3] = v.w;
    return;
  }
  const int off = (int)(i & 3u);
  const uint32_t* p = reinterpret_cast<const uint32_t*>(spins + (i - off));
  uint32_t v[5];
#pragma unroll
  for (int j = 0; j < 5; ++j) v[j] = nv > 0 && 4 * j < off + nv ? p[j] : 0u;
#pragma unroll
  for (int j = 0; j < 4; ++j) c[j] = __funnelshift_r(v[j], v[j + 1], 8 * off);
}

// Bit i set iff byte i of the rows a and b is equal.
__device__ __forceinline__ uint32_t eq_row(const uint32_t (&a)[4], const uint32_t (&b)[4]) {
  return eq4(a[0], b[0]) | eq4(a[1], b[1]) << 4 | eq4(a[2], b[2]) << 8 | eq4(a[3], b[3]) << 12;
}

// Open bonds of row `lane` of a plane (bit = site), zero past its rows.
struct RowBonds {
  uint32_t x, y, z;
};

// Bonds, and observables of the spins read, of a plane of a flat brick (at most
// FLAT_D rows): the rows spread over all lanes, R consecutive sites of a row
// each, R being the power of two from the number of rows on.  With two lanes per
// row and sixteen sites per lane, as in a full brick, a brick of one row costs
// what a full one does: a sweep of 1000 x 1000 x 1 took 126 us, 78 this way (the
// 16 rows of the engine not swept and one-site axes not joined to themselves are
// part of it), x 2 138 and 97, x 4 153 and 122 (x 8 176 and 169, but 256 x 8 x 8
// without draws 16.1 and 17.4: bytes are loaded one by one here).
constexpr int FLAT_D = 4;
__device__ __forceinline__ RowBonds flat_bonds(const int8_t* spins, const Box3& b, const Brick& k, int q, uint64_t T,
                                               const PhiloxKeys& keys, uint64_t sweep, bool do_obs, unsigned* red,
                                               int* hist) {
  const int lane = threadIdx.x & 31, ly = threadIdx.x >> 5;
  const int R = k.d <= 2 ? k.d : 4;
  const int lz = lane & (R - 1), x0 = lane & ~(R - 1);   // my row, my first column
  const int y = k.y0 + ly, z = k.z0 + lz;
  const int n = ly < k.h && lz < k.d ? min(k.w - x0, R) : 0;
  const uint32_t first = (uint32_t)site3(b, k.x0 + x0, y, z);
  const uint32_t to_y = (y + 1 == b.Y ? -(uint32_t)y : 1u) * (uint32_t)b.X;
  const uint32_t to_z = (z + 1 == b.Z ? -(uint32_t)z : 1u) * ((uint32_t)b.X * (uint32_t)b.Y);
  const uint32_t thr = (uint32_t)T;
  RowBonds o = {0u, 0u, 0u};
  unsigned n_eq = 0u;
  unsigned long long states = 0ull;   // sites per state, 8 bits each (q <= QREG)
  if (do_obs && q > QREG) __syncthreads();   // the histogram is cleared
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    const uint32_t site = first + (uint32_t)i, bit = 1u << (x0 + i);
    const int x = k.x0 + x0 + i;
    const int s = spins[site];
    const bool ex = spins[x + 1 == b.X ? site - (uint32_t)x : site + 1u] == s, ey = spins[site + to_y] == s,
               ez = spins[site + to_z] == s;
    if (do_obs) {
      n_eq += (unsigned)ex + (unsigned)ey + (unsigned)ez;
      if (q <= QREG) states += 1ull << (8 * s);
      else atomicAdd(&hist[s], 1);
    }
    if (T == 0) continue;
    uint4 r = make_uint4(0u, 0u, 0u, 0u);
    if (T < (1ull << 32))
      r = philox_draw(make_uint4(site, (uint32_t)sweep, (uint32_t)(sweep >> 32), TAG_BOND3), keys);
    const bool all = T >= (1ull << 32);
    if (ex && (all || r.x < thr)) o.x |= bit;
    if (ey && (all || r.y < thr)) o.y |= bit;
    if (ez && (all || r.z < thr)) o.z |= bit;
  }
  __syncwarp();
  for (int u = R; u < 32; u *= 2) {
    o.x |= __shfl_xor_sync(FULL, o.x, u);
    o.y |= __shfl_xor_sync(FULL, o.y, u);
    o.z |= __shfl_xor_sync(FULL, o.z, u);
  }
  if (lane >= k.d) o = {0u, 0u, 0u};
  if (do_obs) {
    int cnt[QREG];
#pragma unroll
    for (int s = 0; s < QREG; ++s) cnt[s] = (int)(states >> (8 * s) & 0xFFu);
    observables_warp_sums<B3_THREADS>(n_eq, cnt, q <= QREG ? q : 0, red);
  }
  return o;
}

// Local step of a brick.  Bound by instruction issue and by the latency of the
// shared-memory walks: 16 draws per thread (about 45 instructions each), the
// engine and the +y joins take most of a warp's time, so eight CTAs per SM
// (32 registers) beat six.  A lane has half a row: its spins and those at +y and
// +z are three 16-byte loads (the neighbours' from L1), Ising spins packed one
// bit per site, others compared four per word, and the bond bits are row words
// already.  256^3, us: 185 with a thread per column (byte loads, neighbours' spins
// through shared memory, bit-matrix transposes), six CTAs and the +y joins in
// three rounds between disjoint planes (plain stores, but one to four warps of
// eight busy); 172 with joins by compare-and-swap all at once, 159 with rows, 153
// with eight CTAs, 142 with packed spins, 131 with the face roots looked up a lane
// per face site (before: by the sites' owners, a few lanes per warp) and parent
// entries written from the edge bits.
// FLAT: for boxes of at most FLAT_D rows in z, all of whose bricks are flat.  With
// a flat last layer behind full ones the other kernel is as fast or faster, since
// here the engine's sweep is a loop over the brick's rows instead of unrolled
// (256 x 256 x 17 42.2 us a sweep against 43.2 with the flat bricks told apart, x 24
// 42.8 against 44.3).
template <bool FLAT>
__global__ void __launch_bounds__(B3_THREADS, 8)
k3_local(const int8_t* spins, uint16_t* lroot, int32_t* gpar, uint32_t* words, Box3 b, int q, uint64_t T,
         const __grid_constant__ PhiloxKeys keys, const SwCtl* ctl, int64_t* obs, int obs_cap, int* err) {
  __shared__ Local3Smem ls;
  TileSmemT<B3Z>& sm = ls.tile;
  uint16_t* par = sm.par;
  const Brick k = brick_of(b, blockIdx.x);
  const int lane = threadIdx.x & 31, ly = threadIdx.x >> 5;
  wait_for_previous();
  const uint64_t sweep = ctl->sweep;
  const bool do_obs = sweep > 0 && ctl->obs_done != (long long)(sweep - 1);
  const bool plane = ly < k.h;               // the warp has a plane
  if (threadIdx.x < B3_EDGE_WORDS) ls.edge[threadIdx.x] = 0u;
  if (q > QREG)
    for (int j = threadIdx.x; j < 128; j += B3_THREADS) ls.hist[j] = 0;

  // 1. lane (lz, half) has sixteen sites of a row of its warp's plane: their
  //    spins, the rows at +y and +z and the spin at +x; which neighbours are
  //    equal (bit = site)
  const int lz = lane >> 1, half = lane & 1;
  const int nv = plane && lz < k.d ? min(max(k.w - 16 * half, 0), 16) : 0;
  const uint32_t row0 = (uint32_t)site3(b, k.x0, k.y0 + ly, k.z0 + lz);   // my row's first site; past the box without sites
  const uint32_t site0 = row0 + 16 * half;
  RowBonds row = {0u, 0u, 0u};
  if (FLAT) {
    row = flat_bonds(spins, b, k, q, T, keys, sweep, do_obs, ls.red, ls.hist);
  } else {
    uint32_t ex = 0u, ey = 0u, ez = 0u;
    {
      const bool whole = (b.X & 15) == 0;
      const int y = k.y0 + ly, z = k.z0 + lz, x1 = k.x0 + 16 * half + nv;
      uint32_t c[4], n[4], ny[4], nz[4];
      load_row(spins, site0, nv, whole, c);
      load_row(spins, site0 + (y + 1 == b.Y ? -(uint32_t)y : 1u) * (uint32_t)b.X, nv, whole, ny);
      load_row(spins, site0 + (z + 1 == b.Z ? -(uint32_t)z : 1u) * ((uint32_t)b.X * (uint32_t)b.Y), nv, whole, nz);
      const uint32_t next = nv > 0 ? (uint32_t)(uint8_t)spins[x1 == b.X ? row0 - k.x0 : row0 - k.x0 + x1] : 0u;
      const uint32_t mine = (1u << nv) - 1u;
      uint32_t ones = 0u;
      if (q == 2) {   // bytes 0 or 1, packed one bit per site
        auto pack = [](const uint32_t (&v)[4]) {
          return (v[0] * 0x01020408u) >> 24 | (v[1] * 0x01020408u) >> 24 << 4 | (v[2] * 0x01020408u) >> 24 << 8 |
                 (v[3] * 0x01020408u) >> 24 << 12;
        };
        ones = pack(c) & mine;
        ex = ~(ones ^ ((ones | next << nv) >> 1)) & mine;
        ey = ~(ones ^ pack(ny)) & mine;
        ez = ~(ones ^ pack(nz)) & mine;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          n[j] = __funnelshift_r(c[j], j < 3 ? c[j + 1] : next, 8);
          if (nv < 16 && (nv - 1) >> 2 == j) {
            const int sh = 8 * ((nv - 1) & 3);
            n[j] = (n[j] & ~(0xFFu << sh)) | next << sh;
          }
        }
        ex = eq_row(c, n) & mine;
        ey = eq_row(c, ny) & mine;
        ez = eq_row(c, nz) & mine;
      }
      if (do_obs) {
        int cnt[QREG] = {};
        if (q == 2) {
          cnt[1] = __popc(ones);
          cnt[0] = nv - cnt[1];
        } else if (q <= QREG) {
#pragma unroll
          for (int s = 0; s < QREG; ++s) {
            if (s >= q) break;
            const uint32_t same = 0x01010101u * (uint32_t)s;
            const uint32_t v[4] = {same, same, same, same};
            cnt[s] = __popc(eq_row(c, v) & mine);
          }
        }
        if (q > QREG) {
          __syncthreads();   // the histogram is cleared
          for (int i = 0; i < nv; ++i) atomicAdd(&ls.hist[(uint8_t)spins[site0 + i]], 1);
        }
        observables_warp_sums<B3_THREADS>((unsigned)(__popc(ex) + __popc(ey) + __popc(ez)), cnt, q <= QREG ? q : 0,
                                          ls.red);
      }
    }

    // 2. open bonds of my sites
    if (T == 0) {
      ex = ey = ez = 0u;
    } else if (T < (1ull << 32) && plane) {
      const uint32_t thr = (uint32_t)T;
      uint32_t ox = 0u, oy = 0u, oz = 0u;
      constexpr int U = 8;
#pragma unroll 1
      for (int i0 = 0; i0 < min(k.w, 16); i0 += U) {
        uint32_t bx = 0u, by = 0u, bz = 0u;
#pragma unroll
        for (int i = 0; i < U; ++i) {
          const uint4 r = philox_draw(
              make_uint4(site0 + (uint32_t)(i0 + i), (uint32_t)sweep, (uint32_t)(sweep >> 32), TAG_BOND3), keys);
          set_if_below(bx, r.x, thr, 1u << i);
          set_if_below(by, r.y, thr, 1u << i);
          set_if_below(bz, r.z, thr, 1u << i);
        }
        ox |= bx << i0;
        oy |= by << i0;
        oz |= bz << i0;
      }
      ex &= ox;
      ey &= oy;
      ez &= oz;
    }

    // row words (lane = row lz)
    auto row_word = [&](uint32_t e) {
      e <<= 16 * half;
      e |= __shfl_xor_sync(FULL, e, 1);
      e = __shfl_sync(FULL, e, 2 * (lane & 15));
      return lane < B3Z ? e : 0u;
    };
    row = {row_word(ex), row_word(ey), row_word(ez)};
  }

  // 3. the plane's bonds: inside the brick for the engine and the +y joins,
  //    leaving it for the merge, wrapping inside it where the axis is one brick
  //    long
  uint32_t we = row.x;
  uint32_t wn = row.z;
  const uint32_t yb = row.y;
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
  tile_engine<!FLAT>(sm, we, wn, k.d, B3X * k.h, err);
  __syncthreads();

  // 5. +y bonds between planes ly and ly + 1.  One contact per overlap of an
  //    x run with a run of the next plane is kept, and none whose row below
  //    has the bond too and +z bonds up on both sides.  Every join hooks one
  //    root, which takes the contact's place in the list.
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
    C = __shfl_sync(FULL, C, lz) >> (16 * half) & 0xFFFFu;   // my sixteen sites' contacts
    const int cnt = __popc(C);
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += v;
    }
    n_list = __shfl_sync(FULL, incl, 31);
    const int row = brick_local(16 * half, ly, lz);
    for (int first = 0; first < n_list; first += Y_LIST) {
      int at = incl - cnt - first;
      for (uint32_t x = C; x; x &= x - 1, ++at)
        if ((unsigned)at < Y_LIST) list[at] = (uint16_t)(row + high_bit(x & -x));
      __syncwarp();
      const int n = min(n_list - first, Y_LIST);
      for (int j = lane; j - lane < n; j += 32) {
        int a[1], c[1], hooked[1];
        a[0] = c[0] = 2 * brick_local(0, ly, 0);
        if (j < n) {
          const int site = list[j];
          a[0] = par[site];
          c[0] = par[brick_local(0, ly + 1, local_y(site)) + (site & (B3X - 1))];
        }
        sm_union_tile(par, a, c, hooked, err);
        if (j < n) list[j] = (uint16_t)hooked[0];
      }
      __syncwarp();
    }
    __syncthreads();
  }
  // wraps of an axis one brick long (of one site: its own neighbour)
  const bool wrap_x = b.bx == 1 && b.X > 1, wrap_y = b.by == 1 && b.Y > 1, wrap_z = b.bz == 1 && b.Z > 1;
  const bool wraps = wrap_x || wrap_y || wrap_z;
  if (wraps) {
    if (plane) {
      const int self = 2 * brick_local(0, ly, 0);
      if (wrap_x) {
        const bool on = lane < k.d && ((x_out >> lane) & 1u);
        sm_union_tile(par, on ? 2 * brick_local(k.w - 1, ly, lane) : self, on ? 2 * brick_local(0, ly, lane) : self,
                      err);
      }
      if (wrap_z) {
        const bool on = (z_out >> lane) & 1u;
        sm_union_tile(par, on ? 2 * brick_local(lane, ly, k.d - 1) : self, on ? 2 * brick_local(lane, ly, 0) : self,
                      err);
      }
      if (wrap_y && y_last) {
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
  //    thread and step
  const int lx0 = 8 * (lane & 3);
  const int in = plane ? min(max(k.w - lx0, 0), 8) : 0;
  if (in > 0) {
#pragma unroll
    for (int j = 0; j < B3Z / 8; ++j) {
      const int z = (lane >> 2) + 8 * j;
      if (z >= k.d) continue;
      const uint4 v = *reinterpret_cast<const uint4*>(par + brick_local(lx0, ly, z));
      auto two = [&](uint32_t w) {
        const int p0 = sm_at(par, w & 0xFFFFu), p1 = sm_at(par, w >> 16);
        return (uint32_t)sm_at(par, p0) >> 1 | (uint32_t)sm_at(par, p1) << 15;
      };
      const uint32_t wv[4] = {two(v.x), two(v.y), two(v.z), two(v.w)};
      uint16_t* dst = lroot + site3(b, k.x0 + lx0, k.y0 + ly, k.z0 + z);
      if ((b.X & 7) == 0) {   // then k.w is a multiple of 8 too
        *reinterpret_cast<uint4*>(dst) = make_uint4(wv[0], wv[1], wv[2], wv[3]);
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (i < in) dst[i] = (uint16_t)(wv[i >> 1] >> (16 * (i & 1)));
      }
    }
  }
  // 8. roots on the brick's faces marked, a lane per site: the first and last row
  //    of my plane, its first and last column (16 lanes each), rows ly and ly + 8
  //    of the first and the last plane (a flat brick has no row ly + 8); of a run
  //    of equal roots the first lane marks.  The lookups go in step.
  {
    constexpr int N = FLAT ? 5 : 7;
    const int z_of[7] = {0, k.d - 1, lane & 15, ly, ly, ly + 8, ly + 8};
    const int y_of[7] = {ly, ly, ly, 0, k.h - 1, 0, k.h - 1};
    int r[N];
#pragma unroll
    for (int u = 0; u < N; ++u) {
      const int x = u != 2 ? lane : lane < 16 ? 0 : k.w - 1;
      const bool ok = x < k.w && z_of[u] < k.d && (u > 2 || plane);
      r[u] = ok ? 2 * brick_local(x, y_of[u], z_of[u]) : -1;
    }
#pragma unroll
    for (int hop = 0; hop < 3; ++hop)   // site -> node -> plane root -> brick root
#pragma unroll
      for (int u = 0; u < N; ++u)
        if (r[u] >= 0) r[u] = sm_at(par, r[u]);
#pragma unroll
    for (int u = 0; u < N; ++u) {
      const int left = __shfl_up_sync(FULL, r[u], 1);
      const uint32_t bit = 1u << ((r[u] >> 1) & 31);
      uint32_t* word = &ls.edge[r[u] >= 0 ? r[u] >> 6 : 0];
      if (r[u] >= 0 && (lane == 0 || left != r[u]) && !(*reinterpret_cast<volatile uint32_t*>(word) & bit))
        atomicOr(word, bit);
    }
  }
  if (do_obs) {
    unsigned long long* oslot =
        reinterpret_cast<unsigned long long*>(obs + (int64_t)((sweep - 1) % (uint64_t)obs_cap) * (q + 1));
    observables_commit<B3_THREADS>(q, q <= QREG ? q : 0, oslot, ls.red, ls.hist);
  }
  __syncthreads();
  // 9. parent entries of edge roots, each by the owner of its site; the brick's
  //    edge bits for the flip
  if (in > 0) {
    const uint8_t* eb = reinterpret_cast<const uint8_t*>(ls.edge) + (brick_local(lx0, ly, lane >> 2) >> 3);
    const int32_t G0 = (int32_t)site3(b, k.x0 + lx0, k.y0 + ly, k.z0 + (lane >> 2));
    static_assert(B3Z == 16, "two steps of eight rows");
    for (uint32_t bits = eb[0] | (uint32_t)eb[TILE_W] << 8; bits; bits &= bits - 1) {
      const int i = high_bit(bits & -bits);
      const int32_t G = G0 + (i & 7) + (i & 8) * b.X * b.Y;
      gpar[G] = G;
    }
  }
  if (threadIdx.x < B3_EDGE_WORDS) out[threadIdx.x] = ls.edge[threadIdx.x];
}

// One CTA per brick, a warp per face word (x: two words): z faces 0 .. 7 (bit lx
// of word ly), y face 8 .. 23 (bit lx of word lz), x face 24 .. 27 (bits lz of
// words ly, ly + 1).  A lane whose root pair equals its left neighbour's skips
// the union; the others' pairs are listed and joined with all lanes busy (see
// merge_tiles).  Bound by the latency of the root loads and parent walks;
// 256^3: 37 us against 61 with a union per lane where its bond stands (blocks of
// 128 threads 40 us, of 448 45).  Flat bricks have few face bonds, and there what
// counts is bricks in flight: with more of them than blocks of 256 threads fit
// the GPU at once, blocks of 64 (2000 x 2000 x 1, 15750 bricks: 28.8 us against
// 35.9; 300 x 300 x 3, 380 bricks: 9.9 against 8.3).
constexpr int B3_MERGE_UNITS = B3Y + B3Z + B3Y / 2;
template <int MERGE3_THREADS>
__global__ void __launch_bounds__(MERGE3_THREADS)
k3_merge(const uint16_t* lroot, int32_t* gpar, const uint32_t* words, Box3 b, int limit,
         SwCtl* ctl, int64_t* obs, int obs_cap, int q) {
  constexpr int WARPS = MERGE3_THREADS / 32, UNITS = (B3_MERGE_UNITS + WARPS - 1) / WARPS;
  __shared__ int2 pairs[B3_MERGE_UNITS * 32];
  __shared__ int n_pairs;
  wait_for_previous();
  int* err = &ctl->err;
  if (blockIdx.x == 0) {   // the next sweep's local step fills this sweep's observable slot
    const uint64_t s = ctl->sweep;
    for (int j = threadIdx.x; j <= q; j += MERGE3_THREADS) obs[(int64_t)(s % (uint64_t)obs_cap) * (q + 1) + j] = 0;
    __syncthreads();
    if (threadIdx.x == 0) ctl->sweep = s + 1;
  }
  if (threadIdx.x == 0) n_pairs = 0;
  const int t = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t* wd = words + (int64_t)t * B3_WORDS;
  const Brick k = brick_of(b, t);
  uint32_t bit[UNITS];
  int ga[UNITS], gb[UNITS];
#pragma unroll
  for (int i = 0; i < UNITS; ++i) {
    const int u = warp + WARPS * i;
    bit[i] = u >= B3_MERGE_UNITS ? 0u
             : u < B3Y + B3Z     ? wd[B3_FACE_Z + u] >> lane
                                 : wd[B3_FACE_X + 2 * (u - B3Y - B3Z) + (lane >> 4)] >> (lane & 15);
  }
#pragma unroll
  for (int i = 0; i < UNITS; ++i) {
    const int u = warp + WARPS * i;
    ga[i] = gb[i] = 0;
    if (bit[i] & 1u) {   // the brick roots on the two ends (both edge roots)
      const int axis = u < B3Y ? 2 : u < B3Y + B3Z ? 1 : 0;
      const int lx = axis ? lane : k.w - 1;
      const int ly = axis == 2 ? u : axis == 1 ? k.h - 1 : 2 * (u - B3Y - B3Z) + (lane >> 4);
      const int lz = axis == 2 ? k.d - 1 : axis == 1 ? u - B3Y : lane & 15;
      const Brick kn = brick_at(b, axis == 0 ? (k.tbx + 1 == b.bx ? 0 : k.tbx + 1) : k.tbx,
                                axis == 1 ? (k.tby + 1 == b.by ? 0 : k.tby + 1) : k.tby,
                                axis == 2 ? (k.tbz + 1 == b.bz ? 0 : k.tbz + 1) : k.tbz);
      const int ra = lroot[site3(b, k.x0 + lx, k.y0 + ly, k.z0 + lz)];
      const int rb = lroot[site3(b, kn.x0 + (axis == 0 ? 0 : lx), kn.y0 + (axis == 1 ? 0 : ly),
                                 kn.z0 + (axis == 2 ? 0 : lz))];
      ga[i] = (int)brick_global(b, k, ra);
      gb[i] = (int)brick_global(b, kn, rb);
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < UNITS; ++i) {
    const int lo = min(ga[i], gb[i]), hi = max(ga[i], gb[i]);
    const bool valid = lo != hi;
    const unsigned long long key = valid ? ((unsigned long long)(unsigned)lo << 32) | (unsigned)hi : ~0ull;
    const unsigned long long left = __shfl_up_sync(FULL, key, 1);
    const bool join = valid && (lane == 0 || left != key);
    const uint32_t m = __ballot_sync(FULL, join);
    if (m == 0u) continue;
    int at = 0;
    if (lane == 0) at = atomicAdd(&n_pairs, __popc(m));
    at = __shfl_sync(FULL, at, 0) + __popc(m & ((1u << lane) - 1u));
    if (join) pairs[at] = make_int2(lo, hi);
  }
  __syncthreads();
  for (int j = threadIdx.x; j < n_pairs; j += MERGE3_THREADS) seam_join(gpar, pairs[j].x, pairs[j].y, limit, err);
}

// Flip of a brick: a thread owns the sites it wrote in k3_local's step 7 (two
// steps of eight consecutive sites of a row, one 16-byte load of roots each).
// Edge roots come first in the list, as in sw_flip_tile: the first walks' loads
// are in flight while the interior roots are drawn.  256^3: 54 us against 71 with
// flags looked up root by root and walks and draws in turn.
__global__ void __launch_bounds__(B3_THREADS, 6)
k3_flip(int8_t* spins, const uint16_t* lroot, int32_t* gpar,
        const uint32_t* words, Box3 b, int q, const __grid_constant__ PhiloxKeys keys,
        const SwCtl* ctl, int limit, int* err) {
  __shared__ uint16_t rlist[B3_SITES];
  __shared__ uint8_t ns[B3_SITES];
  __shared__ int warp_cnt[B3_THREADS / 32];
  const Brick k = brick_of(b, blockIdx.x);
  wait_for_previous();
  const uint64_t sweep = ctl->sweep - 1;   // the merge has advanced the counter
  const int lane = threadIdx.x & 31, ly = threadIdx.x >> 5, warp = ly;
  const int lx0 = 8 * (lane & 3);
  const int in = ly < k.h ? min(max(k.w - lx0, 0), 8) : 0;
  const bool whole = (b.X & 7) == 0;   // rows start 16-byte aligned, in is 0 or 8
  const int id0 = brick_local(lx0, ly, lane >> 2);   // local index of my first site; step j is 8 rows further
  const uint8_t* eb = reinterpret_cast<const uint8_t*>(words + (int64_t)blockIdx.x * B3_WORDS) + (id0 >> 3);
  // 1. brick roots of my sites (0xFFFF outside the brick), and which are roots
  //    and edge roots (bit 8j + i: site i of step j)
  uint4 roots[B3Z / 8];
  uint32_t m = 0, edges = 0;
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
    edges |= (uint32_t)eb[j * TILE_W] << (8 * j);
    const uint32_t own = (uint32_t)(id0 + 8 * j * TILE_W) * 0x00010001u + 0x00010000u;   // (site, site + 1)
#pragma unroll
    for (int i = 0; i < 4; ++i) m |= zero_halves(v[i] ^ (own + (uint32_t)i * 0x00020002u)) >> (15 - (4 * j + i));
    roots[j] = make_uint4(v[0], v[1], v[2], v[3]);
  }
  // 2. the brick's root list: edge roots, then the others (counts of both in
  //    one scan)
  const uint32_t mine = spread_bits(m & 0xFFFFu) | spread_bits(m >> 16) << 1;
  const uint32_t on_edge = mine & edges, inner = mine & ~edges;
  const int cnt = __popc(on_edge) << 16 | __popc(inner);
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(FULL, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) warp_cnt[warp] = incl;
  __syncthreads();
  int before = incl - cnt, total = 0;
#pragma unroll
  for (int j = 0; j < B3_THREADS / 32; ++j) {
    before += (j < warp) ? warp_cnt[j] : 0;
    total += warp_cnt[j];
  }
  const int n_edge = total >> 16, n_roots = n_edge + (total & 0xFFFF);
  auto list = [&](uint32_t bits, int at) {
    while (bits) {
      const int n = high_bit(bits);
      bits ^= 1u << n;
      rlist[at++] = (uint16_t)(id0 + n + (n & 24) * (TILE_W - 1));
    }
  };
  list(on_edge, before >> 16);
  list(inner, n_edge + (before & 0xFFFF));
  __syncthreads();
  // 3. one draw per brick root, keyed by its cluster's root.  A thread's first
  //    edge roots have their parents loaded before it draws its interior roots.
  auto set_state = [&](int r, int G) {
    const uint4 w = philox_draw(make_uint4((uint32_t)G, (uint32_t)sweep, (uint32_t)(sweep >> 32), TAG_FLIP), keys);
    ns[r] = (uint8_t)state_of(w.x, q);
  };
  constexpr int U = 3;   // of about 500 edge roots per brick at criticality (two: 56 us, four: as three)
  int x[U], p[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int j = threadIdx.x + u * B3_THREADS;
    x[u] = j < n_edge ? (int)brick_global(b, k, rlist[j]) : 0;
    p[u] = j < n_edge ? g_load(gpar + x[u]) : 0;
  }
  for (int j = n_edge + threadIdx.x; j < n_roots; j += B3_THREADS) {
    const int r = rlist[j];
    set_state(r, (int)brick_global(b, k, r));
  }
  g_find_multi<U>(gpar, x, p, limit, err);
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int j = threadIdx.x + u * B3_THREADS;
    if (j < n_edge) set_state(rlist[j], x[u]);
  }
  for (int j = threadIdx.x + U * B3_THREADS; j < n_edge; j += B3_THREADS) {
    const int r = rlist[j];
    set_state(r, g_find(gpar, (int)brick_global(b, k, r), limit, err));
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
  const bool flat = b.Z <= FLAT_D;
  e = launch_after(flat ? k3_local<true> : k3_local<false>, (unsigned)b.n_bricks(), B3_THREADS, st, spins, lroot, gpar,
                   words, b, q, T, keys, ctl, obs, obs_cap, err);
  if (e != cudaSuccess) return e;
  if (ev && (e = cudaEventRecord(ev[1], st)) != cudaSuccess) return e;
  // a box of one brick has no face bonds: one block only advances the counter
  const bool faces = b.bx > 1 || b.by > 1 || b.bz > 1;
  const int64_t blocks = faces ? b.n_bricks() : 1;
  const bool narrow = flat && blocks > 152 * 8;
  e = launch_after(narrow ? k3_merge<64> : k3_merge<256>, (unsigned)blocks, narrow ? 64u : 256u, st, lroot, gpar, words,
                   b, limit3(b), ctl, obs, obs_cap, q);
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
