// swccl_device.cuh -- device helpers shared by the sm_103a kernels of libswccl.
//
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11), the packed 2-bit bond
// mask, and lock-free union-find on shared and global memory.  The union
// rule hooks the larger root under the smaller one, so every tree's root is
// the minimum index in it; with labels initialised to their own index this
// makes the final root of a cluster its minimum site index, the canonical
// label that breadth-first search seeded in site order produces (Sec. II.B.1).
#pragma once
#include <cstdint>

#include "swccl_shared.h"

namespace swccl {

// ---------------------------------------------------------------------------
// Programmatic dependent launch.  A kernel launched with launch_after may be
// launched before the kernels ahead of it in the stream have ended, so that its
// launch overlaps them.  Every thread of such a kernel calls wait_for_previous
// first: it returns when the kernels ahead have completed and their writes are
// visible (at once in a kernel launched plainly).  Such a kernel, and the bodies
// it inlines, read what a kernel ahead of them may write through plain pointers
// or __ldcg: __restrict__ on a pointer that is only read, and __ldg, promise that
// the data does not change while the kernel runs and allow a read-only load
// ahead of the wait.  A sweep at L = 256 took 25.0
// us instead of 27.4 with it, 17.5 instead of 20.2 on low tiles where it also
// joins the sweeps.  The other half, a trigger that lets the next kernel's blocks
// become resident while this one's run, made everything slower (they take issue
// slots and place its blocks unevenly): L = 256 19.0 instead of 17.5 us, L = 2048
// 46 instead of 42, a labeling of 200 x 300 17.8 instead of 17.1, of 2048^2 34.1
// instead of 31.8.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
inline cudaError_t launch_after_smem(void (*kernel)(P...), unsigned blocks, unsigned threads, size_t smem,
                                     cudaStream_t st, A... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, P(args)...);
  if (e != cudaSuccess) cudaGetLastError();   // returned here, not left pending for the caller's next check
  return e;
}
template <class... P, class... A>
inline cudaError_t launch_after(void (*kernel)(P...), unsigned blocks, unsigned threads, cudaStream_t st, A... args) {
  return launch_after_smem(kernel, blocks, threads, 0, st, args...);
}

// ---------------------------------------------------------------------------
// Philox4x32-10.  Each round takes the two 32x32->64 products of the even
// counter words with the published multipliers; the high halves are mixed
// with the odd words and the round key, the key advances by the Weyl
// constants between rounds.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox(uint4 ctr, uint32_t key_lo, uint32_t key_hi) {
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    const unsigned long long pa = (unsigned long long)ctr.x * 0xD2511F53ull;
    const unsigned long long pb = (unsigned long long)ctr.z * 0xCD9E8D57ull;
    uint4 nxt;
    nxt.x = (uint32_t)(pb >> 32) ^ ctr.y ^ key_lo;
    nxt.y = (uint32_t)pb;
    nxt.z = (uint32_t)(pa >> 32) ^ ctr.w ^ key_hi;
    nxt.w = (uint32_t)pa;
    ctr = nxt;
    key_lo += 0x9E3779B9u;
    key_hi += 0xBB67AE85u;
  }
  return ctr;
}

// The ten round keys of a seed, computed once on the host and passed to a
// kernel by value (in constant memory, read directly by the XORs of each
// round), so that a kernel that makes many draws with one seed does not
// recompute the key schedule per call.
struct PhiloxKeys {
  uint32_t lo[10], hi[10];
};

__host__ __device__ inline PhiloxKeys philox_keys(uint64_t seed) {
  PhiloxKeys k;
  uint32_t lo = (uint32_t)seed, hi = (uint32_t)(seed >> 32);
  for (int r = 0; r < 10; ++r) {
    k.lo[r] = lo;
    k.hi[r] = hi;
    lo += 0x9E3779B9u;
    hi += 0xBB67AE85u;
  }
  return k;
}

// A seed whose key schedule is computed in every call (batches: one seed
// per lattice, read from device memory).
struct SeedKey {
  uint32_t lo, hi;
};

// Philox4x32-10 with the round keys given: the same rounds as philox().
__device__ __forceinline__ uint4 philox_draw(uint4 ctr, const PhiloxKeys& k) {
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    const unsigned long long pa = (unsigned long long)ctr.x * 0xD2511F53ull;
    const unsigned long long pb = (unsigned long long)ctr.z * 0xCD9E8D57ull;
    uint4 nxt;
    nxt.x = (uint32_t)(pb >> 32) ^ ctr.y ^ k.lo[round];
    nxt.y = (uint32_t)pb;
    nxt.z = (uint32_t)(pa >> 32) ^ ctr.w ^ k.hi[round];
    nxt.w = (uint32_t)pa;
    ctr = nxt;
  }
  return ctr;
}

// N draws in step, round by round: where only a few warps run, the independent
// chains hide each other's latency.
template <int N>
__device__ __forceinline__ void philox_draws(uint4 (&ctr)[N], const PhiloxKeys& k) {
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    unsigned long long pa[N], pb[N];
#pragma unroll
    for (int u = 0; u < N; ++u) pa[u] = (unsigned long long)ctr[u].x * 0xD2511F53ull;
#pragma unroll
    for (int u = 0; u < N; ++u) pb[u] = (unsigned long long)ctr[u].z * 0xCD9E8D57ull;
#pragma unroll
    for (int u = 0; u < N; ++u)
      ctr[u] = make_uint4((uint32_t)(pb[u] >> 32) ^ ctr[u].y ^ k.lo[round], (uint32_t)pb[u],
                          (uint32_t)(pa[u] >> 32) ^ ctr[u].w ^ k.hi[round], (uint32_t)pa[u]);
  }
}

template <int N>
__device__ __forceinline__ void philox_draws(uint4 (&ctr)[N], const SeedKey& k) {
  PhiloxKeys all;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    all.lo[r] = k.lo + (uint32_t)r * 0x9E3779B9u;
    all.hi[r] = k.hi + (uint32_t)r * 0xBB67AE85u;
  }
  philox_draws(ctr, all);
}

__device__ __forceinline__ uint4 philox_draw(uint4 ctr, const SeedKey& k) { return philox(ctr, k.lo, k.hi); }

__device__ __forceinline__ uint4 draw(uint32_t c0, uint64_t sweep, uint32_t tag, uint64_t seed) {
  return philox(make_uint4(c0, (uint32_t)sweep, (uint32_t)(sweep >> 32), tag), (uint32_t)seed,
                (uint32_t)(seed >> 32));
}

// New state of a cluster from a 32-bit word: floor(w q / 2^32).
__device__ __forceinline__ int state_of(uint32_t w, int q) {
  return (int)(((unsigned long long)w * (unsigned)q) >> 32);
}

// Two bits of site i in the packed mask: bit 0 east bond, bit 1 north bond.
__device__ __forceinline__ uint32_t site_bits(const uint8_t* mask, int64_t i) {
  return (uint32_t)(mask[i >> 2] >> (2 * (i & 3))) & 3u;
}

// Four byte lanes of a and b compared: bit k of the result is set iff byte k
// of a equals byte k of b.  Exact zero-byte test of a ^ b (no carry crosses a
// byte: each byte of (x & 0x7F..) + 0x7F.. is at most 0xFE), then the four
// flag bits are gathered by one multiply.
__device__ __forceinline__ uint32_t eq4(uint32_t a, uint32_t b) {
  const uint32_t x = a ^ b;
  const uint32_t y = ((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x;   // bit 7 of a byte set iff the byte is non-zero
  const uint32_t z = (~y & 0x80808080u) >> 7;                  // bit 0 of a byte set iff equal
  return (z * 0x00204081u) >> 21 & 0xFu;
}

// Bit i of x (i < 16) to bit 2i.
__device__ __forceinline__ uint32_t spread_bits(uint32_t x) {
  x = (x | (x << 8)) & 0x00FF00FFu;
  x = (x | (x << 4)) & 0x0F0F0F0Fu;
  x = (x | (x << 2)) & 0x33333333u;
  return (x | (x << 1)) & 0x55555555u;
}

// 16 bytes from global memory (through L2) to shared memory, asynchronously.
__device__ __forceinline__ void copy16_async(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Record a device-side failure without trapping: the first code wins.
__device__ __forceinline__ void set_error(int* err, int code) {
  if (err) atomicCAS(err, 0, code);
}

// ---------------------------------------------------------------------------
// Local indices.  A tile's sites are numbered row by row, with neighbouring
// 32-column strips swapped in odd rows: a strip's 16-bit entries (64 bytes a
// row) then alternate between the two halves of the 32 shared-memory banks
// instead of all falling into one.  Within a strip, and between different
// rows, local indices order like site indices; sites of one row compare by
// node_key.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int local_of(int ly, int lx) { return ly * TILE_W + (lx ^ ((ly & 1) << 5)); }
__device__ __forceinline__ int local_y(int r) { return r >> TILE_W_LOG2; }
__device__ __forceinline__ int local_x(int r) { return (r & (TILE_W - 1)) ^ ((r >> (TILE_W_LOG2 - 5)) & 32); }

// ---------------------------------------------------------------------------
// Union-find in shared memory on 16-bit entries.  A node id and an entry are
// byte offsets of entries (2 x local index), so that a walk step is one load
// with no address arithmetic.  A node's entry is the node itself (a root) or a
// node of a smaller site index in its component, so every walk ends.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int sm_at(const uint16_t* par, int x) {
  return *reinterpret_cast<const volatile uint16_t*>(reinterpret_cast<const char*>(par) + x);
}
__device__ __forceinline__ void sm_set(uint16_t* par, int x, int v) {
  *reinterpret_cast<volatile uint16_t*>(reinterpret_cast<char*>(par) + x) = (uint16_t)v;
}
// Orders nodes like their sites: twice the row-major index of the tile
// (TileOrder), or the node itself where entries are laid out like sites.
__device__ __forceinline__ int node_key(int x) { return x ^ ((x >> (TILE_W_LOG2 - 5)) & 64); }
struct TileOrder {
  static __device__ __forceinline__ int key(int x) { return node_key(x); }
};
struct SiteOrder {
  static __device__ __forceinline__ int key(int x) { return x; }
};

// The functions below are called by all 32 lanes of a warp together, each lane
// with valid nodes (one that has nothing to join or find passes any written
// node), and loop until every lane is done (a lane that is done reads its root
// again): uniform branches cost fewer instructions than 32 divergent walks,
// whose trees are shallow (0.8 steps per find at criticality).  No path
// compression; hooked roots are resolved at the end.

// The roots of N nodes of every lane, loads in flight together, two steps per
// vote.  Inside one strip node ids order like sites, so a walk that goes on
// only while entries decrease ends by itself; across strips the steps are
// counted, and on overrun (corrupted state) the error word is set and the walk
// stops.
constexpr int WALK_LIMIT = 1 << 15;   // more steps than any tree has nodes (16-bit byte offsets of 2-byte entries)
template <int N>
__device__ __forceinline__ void sm_find_strip(const uint16_t* par, int (&x)[N]) {
  bool more;
  do {
    int p[N];
#pragma unroll
    for (int u = 0; u < N; ++u) p[u] = sm_at(par, x[u]);
    more = false;
#pragma unroll
    for (int u = 0; u < N; ++u) {
      x[u] = sm_at(par, p[u]);
      more |= x[u] < p[u];
    }
  } while (__any_sync(0xFFFFFFFFu, more));
}
template <int N>
__device__ __forceinline__ void sm_find_tile(const uint16_t* par, int (&x)[N], int* err) {
  for (int steps = 0; steps <= WALK_LIMIT; ++steps) {
    int p[N];
#pragma unroll
    for (int u = 0; u < N; ++u) p[u] = sm_at(par, x[u]);
    bool more = false;
#pragma unroll
    for (int u = 0; u < N; ++u) {
      x[u] = sm_at(par, p[u]);
      more |= x[u] != p[u];
    }
    if (!__any_sync(0xFFFFFFFFu, more)) return;
  }
  set_error(err, SW_ERR_STATE);
}

// Join N pairs (a, b) of every lane (a == b: none) where other warps may join
// theirs at the same time.  The root of the larger site is hooked under the
// other by a compare-and-swap of the 32-bit word that holds its entry,
// repeated while only the entry beside it changed (it can be hooked once, so
// twice at most); if the root itself was hooked meanwhile, its new parent is
// joined in the next round, so no link is lost.  Every round lowers the larger
// operand, so at most WALK_LIMIT rounds run.  hooked[u]: the root that the pair
// hooked, or -1.
template <class Order = TileOrder, int N>
__device__ __forceinline__ void sm_union_tile(uint16_t* par, int (&a)[N], int (&b)[N], int (&hooked)[N], int* err) {
#pragma unroll
  for (int u = 0; u < N; ++u) hooked[u] = -1;
  for (int rounds = 0; rounds <= WALK_LIMIT; ++rounds) {
    int x[2 * N];
#pragma unroll
    for (int u = 0; u < N; ++u) {
      x[2 * u] = a[u];
      x[2 * u + 1] = b[u];
    }
    sm_find_tile(par, x, err);
    bool more = false;
#pragma unroll
    for (int u = 0; u < N; ++u) {
      a[u] = x[2 * u];
      b[u] = x[2 * u + 1];
      if (a[u] != b[u]) {
        const bool a_first = Order::key(a[u]) < Order::key(b[u]);
        const int lo = a_first ? a[u] : b[u], hi = a_first ? b[u] : a[u];
        unsigned* word = reinterpret_cast<unsigned*>(reinterpret_cast<char*>(par) + (hi & ~3));
        const int sh = 8 * (hi & 2);
        unsigned old = *reinterpret_cast<volatile unsigned*>(word);
        a[u] = b[u] = lo;
        for (;;) {
          const int cur = (int)((old >> sh) & 0xFFFFu);
          if (cur != hi) {   // hooked meanwhile
            b[u] = cur;
            break;
          }
          const unsigned seen = atomicCAS(word, old, old ^ ((unsigned)(lo ^ hi) << sh));
          if (seen == old) {
            hooked[u] = hi;
            break;
          }
          old = seen;
        }
        more |= a[u] != b[u];
      }
    }
    if (!__any_sync(0xFFFFFFFFu, more)) return;
  }
  set_error(err, SW_ERR_STATE);
}
template <class Order = TileOrder, int N>
__device__ __forceinline__ void sm_union_tile(uint16_t* par, int (&a)[N], int (&b)[N], int* err) {
  int hooked[N];
  sm_union_tile<Order>(par, a, b, hooked, err);
}
template <class Order = TileOrder>
__device__ __forceinline__ void sm_union_tile(uint16_t* par, int a, int b, int* err) {
  int x[1] = {a}, y[1] = {b};
  sm_union_tile<Order>(par, x, y, err);
}

// Join every lane's pair (a, b) (a == b: none) in one strip, whose trees no
// other warp changes meanwhile: no atomics.  In a round every lane finds the
// roots of its pair, then hooks the larger under the smaller with a plain
// store, then reads the entry back: of several lanes hooking one root a single
// one finds its own value and is done, the others go on to join their smaller
// root with the one that won (1.9 rounds of 1.6 steps on average at
// criticality).  Returns the root that the lane hooked, or -1 (lanes that
// stored the same value all name it).
__device__ __forceinline__ int sm_union_strip(uint16_t* par, int a, int b) {
  int hooked = -1;
  do {
    int x[2] = {a, b};
    sm_find_strip(par, x);
    a = min(x[0], x[1]);
    b = max(x[0], x[1]);
    __syncwarp();
    if (a != b) sm_set(par, b, a);
    __syncwarp();
    if (a != b) {
      const int won = sm_at(par, b);
      if (won == a) hooked = b;
      b = won;
    }
  } while (__any_sync(0xFFFFFFFFu, a != b));
  return hooked;
}

// ---------------------------------------------------------------------------
// Union-find on a global int32 array (the label array itself: the entry of a
// tile root is its parent pointer).  Loads bypass L1 (ld.cg) because other
// SMs update the array during the merge.  Bounded by `limit` steps: on
// overrun the error word is set and the walk stops.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int g_load(const int* p) { return __ldcg(p); }

__device__ __forceinline__ int g_find_from(int* lab, int x, int p, int limit, int* err) {   // p: the loaded parent of x
  int steps = 0;
  while (p != x) {
    const int gp = g_load(lab + p);
    if (gp != p) atomicMin(lab + x, gp);   // path halving; entries only ever decrease
    x = p;
    p = gp;
    if (++steps > limit) { set_error(err, SW_ERR_STATE); return x; }
  }
  return x;
}

__device__ __forceinline__ int g_find(int* lab, int x, int limit, int* err) {
  return g_find_from(lab, x, g_load(lab + x), limit, err);
}

// g_find of U nodes at once, p[u] being the loaded parent of x[u] (x[u] itself:
// no walk): the walks run in lock step so that their loads are in flight
// together.  x[u] is replaced by its root; same path halving and step limit as
// g_find.
template <int U>
__device__ __forceinline__ void g_find_multi(int* lab, int (&x)[U], int (&p)[U], int limit, int* err) {
  for (int steps = 0;; ++steps) {
    int gp[U];
    bool more = false;
#pragma unroll
    for (int u = 0; u < U; ++u) gp[u] = (p[u] != x[u]) ? g_load(lab + p[u]) : p[u];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (p[u] != x[u]) {
        if (gp[u] != p[u]) atomicMin(lab + x[u], gp[u]);
        x[u] = p[u];
        p[u] = gp[u];
        more = true;
      }
    }
    if (!more) return;
    if (steps > limit) {
      set_error(err, SW_ERR_STATE);
      return;
    }
  }
}

// Join the sets of a and b on the global array: atomicMin hooks the larger root
// under the smaller, a lost race is retried with the returned parent.  The two
// finds of a round walk in lock step, so that their loads are in flight together.
__device__ __forceinline__ void g_union(int* lab, int a, int b, int limit, int* err) {
  for (int rounds = 0; rounds <= limit; ++rounds) {
    int x[2] = {a, b};
    int p[2] = {g_load(lab + a), g_load(lab + b)};
    g_find_multi<2>(lab, x, p, limit, err);
    a = x[0];
    b = x[1];
    if (a == b) return;
    if (a > b) { const int t = a; a = b; b = t; }
    const int old = atomicMin(lab + b, a);
    if (old == b) return;
    b = old;
  }
  set_error(err, SW_ERR_STATE);
}

}  // namespace swccl
