// k_small.cu -- many Swendsen-Wang sweeps of a small lattice in one launch.
//
// A lattice up to SMALL_L = 112 on a side leaves the GPU all but empty, and its
// sweep is bound by latency: of the 14.3 us that a sweep at L = 64 takes as three
// kernels (k_fused.cu), most goes into launches and into loads and atomics that
// go through L2.  Here one block keeps the whole lattice in shared memory --
// int8 spins, and 16-bit union-find entries laid out like the sites, so that no
// seams, tile roots or global parents are needed -- and runs all n sweeps of a
// call.  The draws, the clusters' roots and the observables are those of the
// other paths, bit for bit.
//
// A warp owns a unit of 8 or 16 rows x 32 columns (the tile engine's strips with
// fewer rows: a unit's work is a serial chain).  A sweep:
//  1. lane (row, part): the bonds of 8 or 16 sites, and the observables of the
//     spins read (the previous sweep's); the parts are put together into row words;
//  2. the unit is labeled as in tile_engine.cuh (run words, row sweep, extra
//     contacts joined by the unit's own warp without atomics);
//  3. after a barrier, the bonds to the next unit east and north, wraps
//     included, are joined (compare-and-swap hooks);
//  4. after a barrier, the unit roots on the unit's four sides (only those can
//     have been hooked in step 3) take their final roots; the unit's cluster
//     roots are listed and draw their clusters' new states (FLIP draw keyed by
//     the root) into their own spins;
//  5. after a barrier, every site takes its root's spin.
// Bound by the latency of its chains up to about L = 80 (an instruction every
// five cycles in a warp, 4 warps per scheduler) and by issue above; the line
// (small_line) lies where one SM no longer keeps up with tiles spread over the
// GPU.  At the critical point, us per sweep here / as three kernels on low tiles:
// q = 2: L = 16 4.8 / 11.4, 64 7.8 / 14.3, 96 12.1 / 15.2, 100 15.1 / 15.5, 112
// 15.3 / 16.6, 116 16.8 / 17.0, 124 19.8 / 16.9; q = 3: 96 12.7 / 15.8, 112 16.2 /
// 16.6, 116 17.7 / 16.8.  More states mean more clusters, all drawn by one block,
// and past 8 their counts go by shared atomics: times as three kernels over times
// here at L = 96, 104, 112: q = 4 1.23, 0.98, 0.95; q = 6 1.03, 0.84, 0.87; q = 9
// 1.04, 0.88, 0.85; q = 20 0.83, 0.80, 0.80; q = 127 0.73, 0.66, 0.64 (L = 84: 1.29,
// 1.19, 1.35, 1.12, 0.99).  At 0.8 of the critical coupling the lines lie lower:
// q = 2 1.05, 0.88, 0.86; q = 3 0.96, 0.81, 0.78.
#include "fused_tile.cuh"

namespace swccl {

constexpr int SMALL_UNITS = 32;                               // one warp per unit
constexpr int SMALL_LIST = 128;                               // list entries per unit and pass

struct SmallUnit {
  union {
    alignas(16) uint4 rowinfo[16];      // sweep inputs, then
    uint16_t list[SMALL_LIST];          // the unit's list (contacts, hooked roots, cluster roots)
  };
  uint32_t be[16], bn[16];              // east and north bonds of the rows, bonds leaving the unit included
};

struct SmallSmem {
  SmallUnit unit[SMALL_UNITS];
  unsigned red[(1 + QREG) * SMALL_UNITS];
  int hist[128];
};

// Dynamic shared memory: SmallSmem, the entries (16 bits a site), the spins (8
// bits), both in rows of L + 4 (rows a multiple of 32 words long would put a
// unit's rows into one bank: step 1 at L = 128 took 5200 cycles instead of 1400).
__host__ __device__ inline int small_pitch(int L) { return L + 4; }
static size_t small_smem_bytes(int L) { return sizeof(SmallSmem) + (size_t)3 * L * small_pitch(L); }

// Units of H rows: 8 where that makes at most SMALL_UNITS of them (shorter
// chains, more warps: L = 64 8.1 against 9.9 us a sweep with 16), else 16.
static int small_units(int L, int H) { return ((L + 31) / 32) * ((L + H - 1) / H); }
static int small_rows(int L) { return small_units(L, 8) <= SMALL_UNITS ? 8 : 16; }
static_assert(((SMALL_L + 31) / 32) * ((SMALL_L + 15) / 16) <= SMALL_UNITS, "one warp per unit");

// Shared memory is read before it is written within each step (loads of all
// rows first, then the chain, then the stores): the compiler cannot tell the
// entries, spins and row words apart and would wait for every store.
// ISING: q = 2, spins packed one bit per site.
template <bool ISING, int SMALL_H>
__global__ void __launch_bounds__(32 * SMALL_UNITS)
k_sw_small(int8_t* spins_g, int L, int q, uint64_t T, const __grid_constant__ PhiloxKeys keys,
           SwCtl* ctl, int64_t* obs, int obs_cap, int n) {
  extern __shared__ __align__(16) unsigned char small_smem[];
  SmallSmem& ss = *reinterpret_cast<SmallSmem*>(small_smem);
  uint16_t* par = reinterpret_cast<uint16_t*>(small_smem + sizeof(SmallSmem));
  const int P = small_pitch(L);
  uint8_t* spins = small_smem + sizeof(SmallSmem) + (size_t)2 * L * P;
  wait_for_previous();
  const int units_x = (L + 31) / 32, units_y = (L + SMALL_H - 1) / SMALL_H, n_units = units_x * units_y;
  const int lane = threadIdx.x & 31, u = threadIdx.x >> 5;   // u < n_units: one warp per unit
  const int uy = u / units_x, ux = u - uy * units_x;
  const int y0 = uy * SMALL_H, x0 = ux * 32;
  const int h = min(SMALL_H, L - y0), w = min(32, L - x0);
  const int u_east = uy * units_x + (ux + 1 == units_x ? 0 : ux + 1);
  const int u_north = (uy + 1 == units_y ? 0 : uy + 1) * units_x + ux;
  const int x_east = ux + 1 == units_x ? 0 : x0 + 32, y_north = uy + 1 == units_y ? 0 : y0 + SMALL_H;
  SmallUnit& me = ss.unit[u];
  uint16_t* list = me.list;
  int* err = &ctl->err;
  const int qreg = q <= QREG ? q : 0;
  for (int i = threadIdx.x; i < L * L / 4; i += blockDim.x)
    *reinterpret_cast<uint32_t*>(spins + 4 * i + 4 * (4 * i / L)) = reinterpret_cast<const uint32_t*>(spins_g)[i];
  if (qreg == 0)
    for (int i = threadIdx.x; i < 128; i += blockDim.x) ss.hist[i] = 0;
  const uint64_t first = ctl->sweep;
  const bool pending = first > 0 && ctl->obs_done != (long long)(first - 1);   // the spins' observables not counted yet
  __syncthreads();

  constexpr int PARTS = 32 / SMALL_H, SP = 32 / PARTS;            // step 1: lanes per row, sites per lane
  const int row = lane & (SMALL_H - 1), part = lane / SMALL_H;
  const int y = y0 + row, x = x0 + SP * part;
  const int nv = row < h ? min(max(w - SP * part, 0), SP) : 0;   // my sites in step 1
  const int self = 2 * (y0 * P + x0);                             // a node of the unit
  for (int k = 0; k <= n; ++k) {
    const uint64_t sweep = first + (uint64_t)k;
    // 1. equal neighbours, observables of the spins, bonds
    uint32_t e = 0u, nb = 0u;
    {
      const bool count = k > 0 || pending;
      uint32_t c[SP / 4] = {}, m[SP / 4] = {}, east = 0u;
      if (nv > 0) {
        const uint8_t* p = spins + y * P + x;
        const uint8_t* pn = spins + (y + 1 == L ? 0 : y + 1) * P + x;
#pragma unroll
        for (int j = 0; j < SP / 4; ++j) {
          if (4 * j < nv) {
            c[j] = *reinterpret_cast<const uint32_t*>(p + 4 * j);
            m[j] = *reinterpret_cast<const uint32_t*>(pn + 4 * j);
          }
        }
        east = spins[y * P + (x + nv == L ? 0 : x + nv)];
      }
      const uint32_t valid = (1u << nv) - 1u;
      int ones = 0;
      if (ISING) {
        uint32_t sb = 0u, mb = 0u;   // spins of my sites and of the row north, one bit each
#pragma unroll
        for (int j = 0; j < SP / 4; ++j) {
          sb |= ((c[j] * 0x01020408u) >> 24) << (4 * j);
          mb |= ((m[j] * 0x01020408u) >> 24) << (4 * j);
        }
        e = ~(sb ^ ((sb | east << nv) >> 1)) & valid;
        nb = ~(sb ^ mb) & valid;
        ones = __popc(sb);
      } else {
#pragma unroll
        for (int j = 0; j < SP / 4; ++j) {
          const uint32_t next = 4 * j + 4 < nv ? c[(j + 1) % (SP / 4)] : east;
          e |= eq4(c[j], (c[j] >> 8) | next << 24) << (4 * j);
          nb |= eq4(c[j], m[j]) << (4 * j);
        }
        e &= valid;
        nb &= valid;
      }
      if (count) {
        const unsigned v = __reduce_add_sync(FULL, (unsigned)(__popc(e) + __popc(nb)));
        if (lane == 0) ss.red[u] = v;
        if (ISING) {
          const unsigned v1 = __reduce_add_sync(FULL, (unsigned)ones);
          if (lane == 0) {
            ss.red[SMALL_UNITS + u] = (unsigned)(h * w) - v1;
            ss.red[2 * SMALL_UNITS + u] = v1;
          }
        } else if (q <= QREG) {
          for (int s = 0; s < q; ++s) {
            const uint32_t same = 0x01010101u * (uint32_t)s;
            uint32_t is = 0u;
#pragma unroll
            for (int j = 0; j < SP / 4; ++j) is |= eq4(c[j], same) << (4 * j);
            const unsigned vs = __reduce_add_sync(FULL, (unsigned)__popc(is & valid));
            if (lane == 0) ss.red[(1 + s) * SMALL_UNITS + u] = vs;
          }
        } else {
#pragma unroll
          for (int j = 0; j < SP / 4; ++j)
            if (4 * j < nv)
#pragma unroll
              for (int i = 0; i < 4; ++i) atomicAdd(&ss.hist[(c[j] >> (8 * i)) & 0xFFu], 1);
        }
      }
    }
    if (k < n && T < (1ull << 32)) {
      uint32_t oe = 0u, on = 0u;
      if (T != 0) {
        uint4 d[SP / 2];
#pragma unroll
        for (int i = 0; i < SP / 2; ++i)
          d[i] = make_uint4((uint32_t)((y * L + x) >> 1) + i, (uint32_t)sweep, (uint32_t)(sweep >> 32), TAG_BOND);
        philox_draws(d, keys);
        const uint32_t thr = (uint32_t)T;
#pragma unroll
        for (int i = 0; i < SP / 2; ++i) {
          set_if_below(oe, d[i].x, thr, 1u << (2 * i));
          set_if_below(oe, d[i].z, thr, 2u << (2 * i));
          set_if_below(on, d[i].y, thr, 1u << (2 * i));
          set_if_below(on, d[i].w, thr, 2u << (2 * i));
        }
      }
      e &= oe;
      nb &= on;
    }
    e <<= SP * part;                               // put the row words together
    nb <<= SP * part;
#pragma unroll
    for (int o = SMALL_H; o < 32; o *= 2) {
      e |= __shfl_xor_sync(FULL, e, o);
      nb |= __shfl_xor_sync(FULL, nb, o);
    }
    const bool lower = lane < SMALL_H;             // lane = row
    if (lower) {
      me.be[row] = e;
      me.bn[row] = nb;
    } else {
      e = nb = 0u;
    }
    const uint32_t out_e = (e >> (w - 1)) & 1u;    // my row's bond to the next unit east
    e &= ~(1u << (w - 1));
    // 2. label the unit
    int n_list = 0;
    int ends[4] = {self, self, self, self};        // unit roots: my row's ends, my column's ends
    if (k < n) {
      uint4 info;
      const uint32_t X = run_words(e, nb, h, info);
      if (lower) me.rowinfo[row] = info;
      __syncwarp();
      {
        const int col = 31 - lane;
        const uint32_t upto = FULL >> lane, mine = 1u << col;
        uint32_t from[SMALL_H / 4];                // lane to read from (5 bits) and contact flag, a byte per row
#pragma unroll
        for (int r = 0; r < SMALL_H; ++r) {
          const uint4 ri = me.rowinfo[r];
          const int start = high_bit(ri.x & upto);
          const uint32_t f = (uint32_t)high_bit(ri.y & (FULL >> start)) | ((ri.z & mine) ? 32u : 0u);
          if (r % 4 == 0) from[r / 4] = f;
          else from[r / 4] |= f << (8 * (r % 4));
        }
        int site = 2 * (y0 * P + x0 + col), lab_below = 0;
#pragma unroll
        for (int r = 0; r < SMALL_H; ++r, site += 2 * P) {
          const uint32_t f = from[r / 4] >> (8 * (r % 4));
          const int label = __shfl_sync(FULL, (f & 32u) ? lab_below : site, (int)(f & 31u));
          if (r < h && col < w) sm_set(par, site, label);
          lab_below = label;
        }
      }
      __syncwarp();
      const int cnt = __popc(X);
      int incl = cnt;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(FULL, incl, d);
        if (lane >= d) incl += v;
      }
      n_list = __shfl_sync(FULL, incl, 31);
      for (int from = 0; from < n_list; from += SMALL_LIST) {
        int at = incl - cnt - from;
        for (uint32_t c = X; c; c &= c - 1, ++at)
          if ((unsigned)at < SMALL_LIST) list[at] = (uint16_t)(y * P + x0 + high_bit(c & -c));
        __syncwarp();
        const int m = min(n_list - from, SMALL_LIST);
        for (int j = lane; j - lane < m; j += 32) {
          int a = self, b = self;
          if (j < m) {
            const int site = list[j];
            a = par[site];
            b = par[site - P];
          }
          const int hooked = sm_union_strip(par, a, b);
          if (j < m) list[j] = (uint16_t)hooked;
        }
        __syncwarp();
      }
      // hooked roots take their unit root
      if (n_list <= SMALL_LIST) {
        for (int j = lane; j - lane < n_list; j += 32) {
          const int node = j < n_list ? (int)list[j] : 0xFFFF;
          int f[1] = {node != 0xFFFF ? node : self};
          sm_find_strip(par, f);
          if (node != 0xFFFF) sm_set(par, node, f[0]);
        }
      } else {   // the list holds the last pass only: every site does
        for (int i = 0; i < h; ++i) {
          const int node = lane < w ? 2 * ((y0 + i) * P + x0 + lane) : self;
          int f[1] = {node};
          sm_find_strip(par, f);
          sm_set(par, node, f[0]);
        }
      }
      __syncwarp();
      if (lane < h) {
        ends[0] = par[y * P + x0];
        ends[1] = par[y * P + x0 + w - 1];
      }
      if (lane < w) {
        ends[2] = par[y0 * P + x0 + lane];
        ends[3] = par[(y0 + h - 1) * P + x0 + lane];
      }
      sm_find_strip(par, ends);
    }
    __syncthreads();
    // observables: row of the sweep before (plain stores: this block alone
    // writes the row)
    if (k > 0 || pending) {
      int64_t* slot = obs + (int64_t)((sweep - 1) % (uint64_t)obs_cap) * (q + 1);
      for (int i = u; i <= qreg; i += n_units) {
        {
          const unsigned tot = __reduce_add_sync(FULL, lane < n_units ? ss.red[i * SMALL_UNITS + lane] : 0u);
          if (lane == 0) slot[i] = tot;
        }
      }
      if (qreg == 0)
        for (int i = threadIdx.x; i < q; i += blockDim.x) {
          slot[1 + i] = ss.hist[i];
          ss.hist[i] = 0;
        }
    }
    if (k == n) break;
    // 3. bonds to the units east and north
    {
      // lane = row: my row's bond east, unless the row below joins the same two runs
      bool join = lower && out_e;
      if (join && row > 0) {
        const uint32_t vert = (me.bn[row - 1] >> (w - 1)) & ss.unit[u_east].bn[row - 1] & (me.be[row - 1] >> (w - 1));
        if (vert & 1u) join = false;
      }
      int ja[2], jb[2];
      ja[0] = join ? ends[1] : self;
      jb[0] = join ? (int)par[y * P + x_east] : self;
      // lane = column: the last row's bond north, unless the column before joins the same two runs
      const uint32_t c = me.bn[h - 1];
      const uint32_t j2 = me.be[h - 1] & ss.unit[u_north].be[0] & ((1u << (w - 1)) - 1u);
      const uint32_t keep = c & ~((seg_or_up(c, j2) << 1) & (j2 << 1));
      join = (keep >> lane) & 1u;
      ja[1] = join ? ends[3] : self;
      jb[1] = join ? (int)par[y_north * P + x0 + lane] : self;
      sm_union_tile<SiteOrder>(par, ja, jb, err);
    }
    __syncthreads();
    // 4. final roots of the unit roots that may have been hooked; the unit's
    //    cluster roots draw
    {
      int r[4] = {ends[0], ends[1], ends[2], ends[3]};
      sm_find_tile(par, r, err);
#pragma unroll
      for (int i = 0; i < 4; ++i) sm_set(par, ends[i], r[i]);
    }
    __syncwarp();
    int roots[SMALL_H];                            // roots of my column's sites
    uint32_t is_root = 0u;
    {
      // site -> its run's node -> unit root -> cluster root
      const int site = 2 * (y0 * P + x0 + lane);
#pragma unroll
      for (int r = 0; r < SMALL_H; ++r) roots[r] = r < h && lane < w ? sm_at(par, site + 2 * r * P) : self;
#pragma unroll
      for (int r = 0; r < SMALL_H; ++r) roots[r] = sm_at(par, roots[r]);
#pragma unroll
      for (int r = 0; r < SMALL_H; ++r) roots[r] = sm_at(par, roots[r]);
#pragma unroll
      for (int r = 0; r < SMALL_H; ++r)
        if (r < h && lane < w && roots[r] == site + 2 * r * P) is_root |= 1u << r;
    }
    {
      const int cnt = __popc(is_root);
      int incl = cnt;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(FULL, incl, d);
        if (lane >= d) incl += v;
      }
      const int total = __shfl_sync(FULL, incl, 31);
      for (int from = 0; from < total; from += SMALL_LIST) {
        __syncwarp();
        int at = incl - cnt - from;
        for (uint32_t c = is_root; c; c &= c - 1, ++at)
          if ((unsigned)at < SMALL_LIST) list[at] = (uint16_t)((high_bit(c & -c) << 5) | lane);
        __syncwarp();
        const int m = min(total - from, SMALL_LIST);
        for (int j = lane; j < m; j += 64) {      // two draws per lane in step
          uint4 d[2];
          int at2[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int rc = list[min(j + 32 * i, m - 1)], ry = y0 + (rc >> 5), rx = x0 + (rc & 31);
            at2[i] = ry * P + rx;
            d[i] = make_uint4((uint32_t)(ry * L + rx), (uint32_t)sweep, (uint32_t)(sweep >> 32), TAG_FLIP);
          }
          philox_draws(d, keys);
#pragma unroll
          for (int i = 0; i < 2; ++i) spins[at2[i]] = (uint8_t)state_of(d[i].x, q);   // past the list: its last root again
        }
      }
    }
    __syncthreads();
    // 5. every site takes its root's spin
    {
      uint8_t state[SMALL_H];
#pragma unroll
      for (int r = 0; r < SMALL_H; ++r) state[r] = spins[roots[r] >> 1];
#pragma unroll
      for (int r = 0; r < SMALL_H; ++r)
        if (r < h && lane < w) spins[(y0 + r) * P + x0 + lane] = state[r];
    }
    __syncthreads();
  }

  for (int i = threadIdx.x; i < L * L / 4; i += blockDim.x)
    reinterpret_cast<uint32_t*>(spins_g)[i] = *reinterpret_cast<const uint32_t*>(spins + 4 * i + 4 * (4 * i / L));
  if (threadIdx.x == 0) {
    ctl->sweep = first + (uint64_t)n;
    ctl->obs_done = (long long)(first + (uint64_t)n - 1);
  }
}

cudaError_t small_prepare() {
  const int bytes = (int)small_smem_bytes(SMALL_L);
  cudaError_t e = cudaSuccess;
  for (auto* f : {k_sw_small<true, 8>, k_sw_small<false, 8>, k_sw_small<true, 16>, k_sw_small<false, 16>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  return e;
}

cudaError_t launch_sw_small(int8_t* spins, int L, int q, uint64_t T, uint64_t seed, SwCtl* ctl, int64_t* obs,
                            int obs_cap, int n, cudaStream_t st) {
  const int rows = small_rows(L);
  auto* kernel = rows == 8 ? (q == 2 ? k_sw_small<true, 8> : k_sw_small<false, 8>)
                           : (q == 2 ? k_sw_small<true, 16> : k_sw_small<false, 16>);
  return launch_after_smem(kernel, 1u, (unsigned)(32 * small_units(L, rows)), small_smem_bytes(L), st, spins, L, q, T,
                           philox_keys(seed), ctl, obs, obs_cap, n);
}

}  // namespace swccl
