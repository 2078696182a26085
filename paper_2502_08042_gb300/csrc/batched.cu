// Batched k-core peel for sm_103a: thousands of independent graphs, one launch.
//
// Input is a segmented CSR: graph g owns vertices [gv[g], gv[g+1]) of one
// global offsets array, and its adjacency lists hold graph-local ids. Each
// graph is peeled by one CTA with Algorithm 1's round structure and the
// online Peel of Algorithm 3, entirely inside the CTA:
//   * levels: the next level is the minimum induced degree of the live
//     vertices (found while the active list is compacted, so empty levels are
//     never visited); the frontier is the live vertices sitting at that level;
//   * subrounds: the arcs of the current frontier are processed edge-balanced
//     by all threads of the CTA (a block scan of the frontier's degrees, then
//     each warp takes 32-arc windows of the concatenated lists); a decrement that
//     returns k+1 lands its vertex on k and appends it to the next subround's
//     frontier; a barrier separates subrounds and levels;
//   * the induced degrees live in shared memory when the graph is small enough
//     (shared-memory atomics), those of a larger graph's first vertices in
//     shared memory and the rest in a per-graph slice of the workspace;
//     when every degree of the graph is below 2^16 they take 16 bits each
//     (twice as many vertices fit in shared memory, half the L2 footprint).
// Persistent CTAs take graphs from a device counter in descending order of
// arcs (longest-processing-time first), so the largest graphs start first;
// once the graphs are small, a 1,024-thread CTA splits into two teams that
// each peel graphs of their own.
// Nothing waits on another CTA: the kernel has no spin-waits.
//
// Measured (ms per batch, before the windows, the compile-time forms of d~,
// the split store and the teams / with them): 1,000 graphs of 1k..8k vertices
// 2.33 / 1.19, 512 of 1k..200k (617 M arcs, bound by its largest graphs) 20.6
// / 10.7, 1,500 of 1k..200k 28.9 / 14.2, 2,000 of 1k..40k 10.3 / 4.9.
//
// A small batch is bound by its largest graphs, each walked by one CTA while
// the others run out of work. The clustered form (batch_peel_cl) gives every
// graph with more arcs than a threshold (by default the batch's arcs per CTA)
// to a thread-block cluster of C CTAs: the cluster splits each list pass and
// each subround's frontier arcs among its CTAs, keeps the induced degrees in
// L2 and its counters in the first CTA's shared memory (reached through
// distributed shared memory), and closes every phase with the hardware cluster
// barrier. Once a cluster draws a graph below the threshold (the order is by
// arcs, so every later one is too), its CTAs go back to one graph each.
#include <cooperative_groups.h>

#include <climits>

#include "kcore_batched.h"
#include "kcore_device.cuh"
#include "kcore_search.h"

namespace kc {

// 32-arc windows a warp keeps in flight (bounded by the registers of three
// 512-thread or six 256-thread CTAs per SM)
template <int BLOCK>
constexpr int kBatchIlp = BLOCK >= 1024 ? 8 : 4;
constexpr int kScanItems = 8;  // active-list entries per thread per scan tile
constexpr int kPackShare = 8;  // the active list is rewritten when 1 / kPackShare of it is peeled

template <int BLOCK>
struct BatchShared {
  int pre[BLOCK];          // a chunk of frontier vertices: arcs ahead of each
  const int* list[BLOCK];  // the address of each one's first arc, less its pre
  int part[2][BLOCK / 32];  // block scan: two sets used in turn (one barrier per scan)
  int red[2][BLOCK / 32];
  int cnt[2];  // vertices appended to the next frontier (used in turn by the subrounds)
  GraphDesc gd;  // the graph being peeled (its nine pointers would take 18 registers)
  int g;
  int bad;  // this graph failed a bounds check: stop peeling it
  int base, base2;  // clustered peel: this CTA's output positions for the current tile
};

// A team: the BLOCK threads that peel one graph, the whole CTA or an aligned part
// of it, with a barrier of its own (named barrier 1 + the team's index).
template <int BLOCK>
__device__ __forceinline__ int team_tid() {
  static_assert((BLOCK & (BLOCK - 1)) == 0, "a power of two");
  return (int)(threadIdx.x & (BLOCK - 1));
}
template <int BLOCK>
__device__ __forceinline__ void team_sync() {
  asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)threadIdx.x / BLOCK), "n"(BLOCK) : "memory");
}

// Records a failed bounds check (first one wins: code, graph-local value) and
// flags the status; the access itself is skipped by the caller.
__device__ __forceinline__ void flag_bad(int* status, int code, long long value, int* bad) {
  if (atomicCAS(status, 0, ST_NOT_SIMPLE) == 0) {
    status[1] = code;
    status[2] = (int)(value & 0xffffffffll);
    status[3] = (int)(value >> 32);
  }
  *bad = 1;
}

// The sum of the first `warp` of the kW warps' values, and their total. By two
// warp reductions: every warp of the CTA runs this, and a scan's shuffles (one
// warp instruction per cycle and SM) cost more than the barrier it replaces.
template <int kW>
__device__ __forceinline__ int warps_ahead(const int* part, int* total) {
  const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) & (kW - 1);
  const unsigned p = lane < kW ? (unsigned)part[lane] : 0u;
  *total = (int)__reduce_add_sync(kFull, p);
  return (int)__reduce_add_sync(kFull, lane < warp ? p : 0u);
}

// Block-wide exclusive scan of one int per thread; returns the exclusive value,
// *total gets the sum. One barrier: every warp sums the warps' sums itself,
// and the sums alternate between two arrays (ph, toggled here), so the next
// scan's stores cannot meet this one's loads.
template <int BLOCK>
__device__ __forceinline__ int block_excl_scan(int x, BatchShared<BLOCK>& sh, int& ph, int* total) {
  constexpr int kW = BLOCK / 32;
  const int lane = threadIdx.x & 31, warp = team_tid<BLOCK>() >> 5;
  const int incl = warp_incl_scan(x, lane);
  int* part = sh.part[ph];
  ph ^= 1;
  if (lane == 31) part[warp] = incl;
  team_sync<BLOCK>();
  return warps_ahead<kW>(part, total) + incl - x;
}

// Block-wide minimum of two values (one barrier; the callers have another
// barrier between any two calls).
template <int BLOCK>
__device__ __forceinline__ void block_min2(int& x, int& y, BatchShared<BLOCK>& sh) {
  constexpr int kW = BLOCK / 32;
  const int lane = threadIdx.x & 31, warp = team_tid<BLOCK>() >> 5;
  x = __reduce_min_sync(kFull, x);
  y = __reduce_min_sync(kFull, y);
  if (lane == 0) {
    sh.red[0][warp] = x;
    sh.red[1][warp] = y;
  }
  team_sync<BLOCK>();
  x = __reduce_min_sync(kFull, lane < kW ? sh.red[0][lane] : INT_MAX);
  y = __reduce_min_sync(kFull, lane < kW ? sh.red[1][lane] : INT_MAX);
}

// The induced degrees d~ of one graph, in shared memory or in L2 (atomics are
// performed in L2, so a global d~ is never read through L1). Global d~
// accesses carry an evict-last hint and the once-read lists (active list,
// frontiers, adjacency) stream with evict-first loads and stores: with
// hundreds of large graphs in flight their state exceeds L2, and the d~ lines
// are the ones that are hit again.
// Narrow form: two 16-bit values per 32-bit word (vertex v in half v & 1 of
// word v >> 1). A vertex's d~ starts at its degree and falls by one per
// peeled neighbour (each arc is traversed once), so it stays in [0, degree]:
// with every degree below 2^16 a decrement never borrows from the other half.
// Where the words live: all in shared memory, all in global memory, or (a
// graph too large for shared memory) the first `cut` vertices in shared memory
// and the rest in global memory. One SM sends about one scattered global
// atomic per 1-2 cycles and several per cycle to shared memory, so every
// vertex kept there shortens a large graph's subrounds.
enum DegMode : int { kDegSmem = 0, kDegGlobal = 1, kDegSplit = 2 };
struct DegStore {
  int* w;       // the words, in global memory
  unsigned sa;  // in shared memory (shared-state address: a generic pointer would make
                // every access, the atomics above all, a generic one)
  int cut;      // vertices below are in shared memory (kDegSplit; even)
  int mode;
  bool narrow;
  uint64_t pol;
  template <bool kNarrow>
  __device__ static __forceinline__ int value(int x, int v) {
    return kNarrow ? ((unsigned)x >> ((v & 1) << 4)) & 0xffff : x;
  }
  template <bool kNarrow>
  __device__ static __forceinline__ int minus_one(int v) {
    return kNarrow && (v & 1) ? -65536 : -1;
  }
  template <bool kNarrow>
  __device__ __forceinline__ unsigned saddr(int v) const {
    return sa + 4u * (unsigned)(kNarrow ? v >> 1 : v);
  }
  // d~ of the vertices v[q] >= 0 (-1 where there is none), every load issued
  // before any result is used
  template <int kMode, bool kNarrow, int N>
  __device__ __forceinline__ void get_all(const int (&v)[N], int (&d)[N]) const {
#pragma unroll
    for (int q = 0; q < N; q++) {
      d[q] = -1;
      if (kMode != kDegGlobal && v[q] >= 0 && (kMode == kDegSmem || v[q] < cut))
        asm volatile("ld.shared.s32 %0, [%1];" : "=r"(d[q]) : "r"(saddr<kNarrow>(v[q])) : "memory");
      if (kMode != kDegSmem && v[q] >= 0 && (kMode == kDegGlobal || v[q] >= cut))
        d[q] = ld_cg_keep(w + (kNarrow ? v[q] >> 1 : v[q]), pol);
    }
#pragma unroll
    for (int q = 0; q < N; q++)
      if (v[q] >= 0) d[q] = value<kNarrow>(d[q], v[q]);
  }
  template <int N>
  __device__ __forceinline__ void get_all(const int (&v)[N], int (&d)[N]) const {
    if (mode == kDegSmem) narrow ? get_all<kDegSmem, true>(v, d) : get_all<kDegSmem, false>(v, d);
    else if (mode == kDegGlobal) narrow ? get_all<kDegGlobal, true>(v, d) : get_all<kDegGlobal, false>(v, d);
    else narrow ? get_all<kDegSplit, true>(v, d) : get_all<kDegSplit, false>(v, d);
  }
  // decrements d~[u[q]] by one for the slots q with q * 32 < left; old[q]: the
  // value before (0 for the other slots)
  template <int kMode, bool kNarrow, int N>
  __device__ __forceinline__ void dec_all(const int (&u)[N], int (&old)[N], int left) const {
#pragma unroll
    for (int q = 0; q < N; q++) {
      old[q] = 0;
      if (kMode != kDegGlobal && q * 32 < left && (kMode == kDegSmem || u[q] < cut))
        asm volatile("atom.shared.add.s32 %0, [%1], %2;"
                     : "=r"(old[q])
                     : "r"(saddr<kNarrow>(u[q])), "r"(minus_one<kNarrow>(u[q]))
                     : "memory");
      if (kMode != kDegSmem && q * 32 < left && (kMode == kDegGlobal || u[q] >= cut))
        old[q] = atom_add_keep(w + (kNarrow ? u[q] >> 1 : u[q]), minus_one<kNarrow>(u[q]), pol);
    }
#pragma unroll
    for (int q = 0; q < N; q++)
      if (q * 32 < left) old[q] = value<kNarrow>(old[q], u[q]);
  }
  // initial values: one word (narrow: vertices 2i and 2i + 1, degree d1 of
  // the second, 0 past the end)
  __device__ __forceinline__ void put_word(int i, int d0, int d1) const {
    const int x = narrow ? (d0 | (d1 << 16)) : d0;
    if (mode == kDegSmem || (mode == kDegSplit && i < (narrow ? cut >> 1 : cut)))
      asm volatile("st.shared.s32 [%0], %1;" ::"r"(sa + 4u * (unsigned)i), "r"(x) : "memory");
    else st_keep(w + i, x, pol);
  }
};

// A chunk of up to BLOCK frontier vertices at `F`: thread tid gives its vertex
// coreness k (set_core) and the chunk's arcs are laid out one after another
// (sh.pre, sh.list). Returns the chunk's arcs. Two barriers; the chunk's
// arrays may be reused after the caller's next barrier.
template <int BLOCK>
__device__ __forceinline__ int load_chunk(const GraphDesc& gd, const int* F, int cnum, int n, int k, bool set_core,
                                          int* status, BatchShared<BLOCK>& sh, int& ph) {
  const int tid = team_tid<BLOCK>();
  int len = 0;
  long long st = 0;
  if (tid < cnum) {
    const int v = __ldcg(F + tid);
    if ((unsigned)v < (unsigned)n) {
      if (set_core) gd.core[v] = k;
      st = gd.off[v];
      const long long e = gd.off[v + 1];
      if (st < 0 || e < st || e > gd.m || e - st >= n) flag_bad(status, 2, v, &sh.bad);
      else len = (int)(e - st);
      // A vertex peeled at a level above 0 has arcs, except in a graph that is
      // not symmetric, where a 16-bit d~ can be decremented below 0 and come
      // round. The map from arcs to lists (chunk_arcs) relies on it.
      if (len == 0 && k > 0) flag_bad(status, 4, v, &sh.bad);
    } else {
      flag_bad(status, 3, v, &sh.bad);
    }
  }
  int total;
  const int ex = block_excl_scan(len, sh, ph, &total);
  sh.pre[tid] = ex;
  sh.list[tid] = gd.adj + (st - ex);
  team_sync<BLOCK>();
  return total;
}

// Arcs [jlo, jhi) of the chunk: each warp takes a contiguous run of 32-arc
// windows. The vertex a window starts in is found once per run (two ballots
// over sh.pre); inside the run the vertices that start in a window form a bit
// mask (one warp reduction), so an arc's vertex is a population count. What
// bounds a chunk is the issue rate of one SM's warps, so the loop holds few
// instructions per window: no search, no check of an arc's index (load_chunk
// checked the lists; after a failed check nothing is read), the form of d~
// fixed at compile time, and d~ decremented unread: a vertex at or below k is
// already in a frontier (or peeled), never returns k + 1, and its d~ is only
// compared with levels above k afterwards. All loads are issued before any
// result is checked (a check that can branch to flag_bad between two loads
// makes each wait for the one before), and the crossing vertices of kBatchIlp
// windows are appended to Fn with one atomic. Every list of a chunk holds an
// arc (load_chunk reports one that does not): two lists that start at the same
// arc would count as one in the bit mask, and the arcs after them would be
// read past their lists' ends.
template <int BLOCK, int kIlp, int kMode, bool kNarrow>
__device__ __forceinline__ void chunk_arcs(const GraphDesc& gd, const DegStore& D, int n, int k, unsigned jlo,
                                           unsigned jhi, int cnum, int* Fn, int* counter, int* status, BatchShared<BLOCK>& sh) {
  constexpr int kW = BLOCK / 32;
  const int lane = threadIdx.x & 31, warp = team_tid<BLOCK>() >> 5;
  // (positions go up to 2^31 - 2, and an iteration's reach past it: unsigned)
  const unsigned run = ((((jhi - jlo + 31) >> 5) + kW - 1) / kW) << 5;  // arcs per warp
  unsigned j0 = jlo + warp * run;
  const unsigned jend = min(jhi, j0 + run);
  if (j0 >= jend || __any_sync(kFull, sh.bad)) return;
  int idx;  // last vertex that starts at or before j0
  {
    const int x = lane * kW;
    unsigned m = __ballot_sync(kFull, x < cnum && (unsigned)sh.pre[x] <= j0);
    const int c = m ? (31 - __clz(m)) * kW : 0;
    m = __ballot_sync(kFull, lane < kW && c + lane < cnum && (unsigned)sh.pre[c + lane] <= j0);
    idx = m ? c + 31 - __clz(m) : c;
  }
  const unsigned le = lanemask_lt() | (1u << lane);
  for (; j0 < jend; j0 += kIlp * 32) {
    int u[kIlp];
    // the starts inside the iteration: one read gives the next 32; when they
    // reach past it, the windows' masks do not depend on each other
    const int e0 = idx + 1 + lane;
    const unsigned d0 = e0 < cnum ? (unsigned)sh.pre[e0] - j0 : 0x7fffffffu;
    const bool few = __shfl_sync(kFull, d0, 31) >= kIlp * 32u;
#pragma unroll
    for (int q = 0; q < kIlp; q++) {
      u[q] = 0;
      if (j0 + q * 32 < jend) {
        unsigned d = d0 - q * 32u;
        if (!few) {
          const int e = idx + 1 + lane;
          d = e < cnum ? (unsigned)sh.pre[e] - (j0 + q * 32) : 32u;
        }
        const unsigned m = __reduce_or_sync(kFull, d < 32u ? 1u << d : 0u);
        const int mine = idx + __popc(m & le);
        idx += __popc(m);
        const unsigned j = j0 + q * 32 + lane;
        if (j < jend) u[q] = ld_stream_s32(sh.list[mine] + j);
      }
    }
    const int left = (int)(jend - j0) - lane;
    bool bad = false;  // an id outside [0, n)
#pragma unroll
    for (int q = 0; q < kIlp; q++) bad |= (unsigned)u[q] >= (unsigned)n;
    if (__any_sync(kFull, bad)) {
      if (bad) flag_bad(status, 5, j0, &sh.bad);
      return;
    }
    int old[kIlp];
    D.dec_all<kMode, kNarrow>(u, old, left);
    int cnt = 0;
#pragma unroll
    for (int q = 0; q < kIlp; q++) cnt += old[q] == k + 1 ? 1 : 0;
    cnt = (int)__reduce_add_sync(kFull, (unsigned)cnt);
    if (cnt) {
      int pos = 0;
      if (lane == 0) pos = atomicAdd(counter, cnt);
      pos = __shfl_sync(kFull, pos, 0);
      if (pos + cnt > n) {  // cannot happen: every vertex lands on k at most once per level
        if (lane == 0) flag_bad(status, 7, pos, &sh.bad);
        return;
      }
#pragma unroll
      for (int q = 0; q < kIlp; q++) {
        const unsigned m = __ballot_sync(kFull, old[q] == k + 1);
        if (old[q] == k + 1) {
          Fn[pos + __popc(m & lanemask_lt())] = u[q];
          // its offsets are read next: from L2 then, not from DRAM
          asm volatile("prefetch.global.L2 [%0];" ::"l"(gd.off + u[q]));
        }
        pos += __popc(m);
      }
    }
  }
}

template <int BLOCK>
__device__ __forceinline__ void chunk_arcs(const GraphDesc& gd, const DegStore& D, int n, int k, unsigned jlo,
                                           unsigned jhi, int cnum, int* Fn, int* counter, int* status, BatchShared<BLOCK>& sh) {
  // at most one window per warp: without the slots of further windows, whose
  // instructions alone would be most of a small graph's phase
#define KC_ARCS2(ILP, MODE)                                                                                     \
  (D.narrow ? chunk_arcs<BLOCK, ILP, MODE, true>(gd, D, n, k, jlo, jhi, cnum, Fn, counter, status, sh)             \
            : chunk_arcs<BLOCK, ILP, MODE, false>(gd, D, n, k, jlo, jhi, cnum, Fn, counter, status, sh))
#define KC_ARCS(MODE)                           \
  do {                                          \
    if (jhi - jlo <= BLOCK) KC_ARCS2(1, MODE);  \
    else KC_ARCS2(kBatchIlp<BLOCK>, MODE);      \
  } while (0)
  if (D.mode == kDegSmem) KC_ARCS(kDegSmem);
  else if (D.mode == kDegGlobal) KC_ARCS(kDegGlobal);
  else KC_ARCS(kDegSplit);
#undef KC_ARCS2
#undef KC_ARCS
}

// A tile of BLOCK * kScanItems list entries: a warp takes consecutive entries,
// 32 per slot, so its loads and the stores of what it keeps are consecutive.
// (Eight entries per thread side by side in the output put every lane of a
// store in a sector of its own: 4,700 of a tile's 10,700 cycles.) A short tile
// fills fewer slots, not fewer warps.
struct TileMap {
  int first, end, rows;  // this thread's first entry, the tile's end, the slots filled
  template <int BLOCK>
  __device__ __forceinline__ static TileMap at(int base, int len) {
    const int rows = min(kScanItems, (len - base + BLOCK - 1) / BLOCK);
    return TileMap{base + (team_tid<BLOCK>() >> 5) * (32 * rows) + (int)(threadIdx.x & 31), min(len, base + BLOCK * rows),
                   rows};
  }
  // the list index of slot q, or -1
  __device__ __forceinline__ int entry(int q) const {
    const int i = first + q * 32;
    return q < rows && i < end ? i : -1;
  }
};

// The kept (d >= keep_from) and taken (d == take_at) entries of a tile, packed
// taken << 16 | kept: *total for the tile, *own for this warp; returns those
// ahead of it.
template <int BLOCK>
__device__ __forceinline__ int tile_count(const int (&d)[kScanItems], int keep_from, int take_at,
                                          BatchShared<BLOCK>& sh, int& ph, int* total, int* own) {
  constexpr int kW = BLOCK / 32;
  const int lane = threadIdx.x & 31, warp = team_tid<BLOCK>() >> 5;
  int sum = 0;
#pragma unroll
  for (int q = 0; q < kScanItems; q++) sum += (d[q] >= keep_from ? 1 : 0) + (d[q] == take_at ? 1 << 16 : 0);
  sum = (int)__reduce_add_sync(kFull, (unsigned)sum);
  *own = sum;
  int* part = sh.part[ph];
  ph ^= 1;
  if (lane == 0) part[warp] = sum;
  team_sync<BLOCK>();
  return warps_ahead<kW>(part, total);
}

// Writes the entries v[q] of the lanes with want(d[q]) to out, in list order.
template <typename Want>
__device__ __forceinline__ void tile_write(const int (&v)[kScanItems], const int (&d)[kScanItems], int* out, Want want) {
#pragma unroll
  for (int q = 0; q < kScanItems; q++) {
    const bool w = want(d[q]);
    const unsigned m = __ballot_sync(kFull, w);
    if (w) __stcs(out + __popc(m & lanemask_lt()), v[q]);
    out += __popc(m);
  }
}

// One pass over the active list after level k: entries with D > k survive
// into `out` (nullptr: the list stays as it is; their minimum goes to *dmin);
// among them, those at exactly k+1
// are also written to F (the next frontier if level k+1 is not empty).
// Returns the survivors; *nf gets the number written to F.
template <int BLOCK>
__device__ int compact_active(const int* A, int la, int n, int* out, int* F, const DegStore& D, int k,
                              BatchShared<BLOCK>& sh, int& ph, int* dmin, int* nf) {
  int written = 0, wf = 0, lmin = INT_MAX;
  for (int base = 0; base < la; base += BLOCK * kScanItems) {
    const TileMap tm = TileMap::at<BLOCK>(base, la);
    int v[kScanItems];
#pragma unroll
    for (int q = 0; q < kScanItems; q++) {
      const int i = tm.entry(q);
      v[q] = -1;
      if (i >= 0) {
        int x = __ldcs(A + i);
        v[q] = (unsigned)x < (unsigned)n ? x : -1;  // ids are < n by construction; checked anyway
      }
    }
    int d[kScanItems];
    D.get_all(v, d);
#pragma unroll
    for (int q = 0; q < kScanItems; q++)
      if (d[q] > k) lmin = min(lmin, d[q]);  // (no entry: -1)
    int tot, own;
    const int at = tile_count(d, k + 1, k + 1, sh, ph, &tot, &own);
    if (out) tile_write(v, d, out + written + (at & 0xffff), [k](int x) { return x > k; });
    if (own >> 16) tile_write(v, d, F + wf + (at >> 16), [k](int x) { return x == k + 1; });
    written += tot & 0xffff;
    wf += tot >> 16;
  }
  int none = INT_MAX;
  block_min2(lmin, none, sh);  // its barrier also publishes the writes above
  *dmin = lmin;
  *nf = wf;
  return written;
}

// Selection of the frontier: entries of A with D[v] == k.
template <int BLOCK>
__device__ int select_frontier(const int* A, int la, int n, int* F, const DegStore& D, int k,
                               BatchShared<BLOCK>& sh, int& ph) {
  int written = 0;
  for (int base = 0; base < la; base += BLOCK * kScanItems) {
    const TileMap tm = TileMap::at<BLOCK>(base, la);
    int v[kScanItems];
#pragma unroll
    for (int q = 0; q < kScanItems; q++) {
      const int i = tm.entry(q);
      v[q] = -1;
      if (i >= 0) {
        int x = __ldcs(A + i);
        v[q] = (unsigned)x < (unsigned)n ? x : -1;  // ids are < n by construction; checked anyway
      }
    }
    int d[kScanItems];
    D.get_all(v, d);
    int tot, own;
    const int at = tile_count(d, INT_MAX, k, sh, ph, &tot, &own);
    if (own) tile_write(v, d, F + written + (at >> 16), [k](int x) { return x == k; });
    written += tot >> 16;
  }
  team_sync<BLOCK>();  // the frontier is read by other threads next
  return written;
}

// Peels one graph with the whole CTA (see the file comment).
template <int BLOCK>
__device__ void peel_one_graph(int smem_deg_max, int* status, int* sdeg, BatchShared<BLOCK>& sh) {
  const GraphDesc& gd = sh.gd;
  const int tid = team_tid<BLOCK>();
  if (gd.n <= 0) {
    if (tid == 0) *gd.kmax = 0;
    team_sync<BLOCK>();
    return;
  }
  const int n = (int)gd.n;

  // degrees: their minimum (the first level) and maximum (whether 16 bits
  // hold them), then the store, the initial values and the identity active list
  if (tid == 0) {
    sh.bad = 0;
    sh.cnt[0] = 0;
    sh.cnt[1] = 0;
  }
  team_sync<BLOCK>();
  int ph = 0;  // which of the two sets of block-scan sums the next scan uses
  int lmin = INT_MAX, lmax = 0;
  for (int v = tid; v < n; v += BLOCK) {
    long long o0 = gd.off[v], o1 = gd.off[v + 1];
    if (o0 < 0 || o1 < o0 || o1 > gd.m || o1 - o0 >= n) {
      flag_bad(status, 1, v, &sh.bad);
      o1 = o0;
    }
    const int d = (int)(o1 - o0);
    lmin = min(lmin, d);
    lmax = max(lmax, d);
  }
  int k = lmin, dmax = -lmax;
  block_min2(k, dmax, sh);
  dmax = -dmax;
  if (sh.bad) {  // malformed offsets: leave this graph (its outputs are undefined)
    if (tid == 0) *gd.kmax = -1;
    team_sync<BLOCK>();
    return;
  }
  const bool narrow = dmax < 65536;
  const int chunk = chunk_vertices(BLOCK, dmax);
  const int fit = narrow ? 2 * smem_deg_max : smem_deg_max;  // vertices that fit in shared memory
  const DegStore D{gd.deg, (unsigned)__cvta_generic_to_shared(sdeg), fit,
                   n <= fit ? kDegSmem : (fit > 0 ? kDegSplit : kDegGlobal), narrow, l2_evict_last_policy()};
  const int nw = narrow ? (n + 1) / 2 : n;
  for (int i = tid; i < nw; i += BLOCK) {
    const int v0 = narrow ? 2 * i : i;
    const int d0 = (int)(gd.off[v0 + 1] - gd.off[v0]);
    const int d1 = narrow && v0 + 1 < n ? (int)(gd.off[v0 + 2] - gd.off[v0 + 1]) : 0;
    D.put_word(i, d0, d1);
  }
  for (int v = tid; v < n; v += BLOCK) __stcs(gd.A0 + v, v);
  team_sync<BLOCK>();
  bool odd = false;  // the active list is in A1
  int peeled = 0;    // its entries peeled since it was written
  int la = n;
  int kmax = 0;
  int r = 0;  // subrounds: frontier counter r & 1 counts this one's appends
  int nf = select_frontier<BLOCK>(gd.A0, la, n, gd.F0, D, k, sh, ph);
  for (;;) {
    bool fodd = false;  // the frontier is in F1
    while (nf > 0) {
      peeled += nf;
      for (int c0 = 0; c0 < nf; c0 += chunk) {
        const int cnum = min(chunk, nf - c0);
        const int total = load_chunk<BLOCK>(gd, (fodd ? gd.F1 : gd.F0) + c0, cnum, n, k, true, status, sh, ph);
        // every thread has read the last subround's counter: clear it for the next
        if (tid == 0 && c0 == 0) sh.cnt[(r + 1) & 1] = 0;
        chunk_arcs<BLOCK>(gd, D, n, k, 0, total, cnum, fodd ? gd.F0 : gd.F1, &sh.cnt[r & 1], status, sh);
        team_sync<BLOCK>();
      }
      nf = sh.cnt[r & 1];
      if (nf > n) nf = 0;  // cannot happen: every vertex lands on k at most once per level
      r++;
      fodd = !fodd;
    }
    kmax = k;
    // The minimum induced degree of the vertices left is the next non-empty
    // level; vertices at k+1 are collected on the way in case that level is
    // the next one. The list is rewritten without the peeled vertices once
    // they are kPackShare of it: a deep graph's levels peel a percent or two
    // each, and the stores are a third of a tile's time.
    const bool pack = (long long)peeled * kPackShare >= la;
    int dmin;
    const int left = compact_active<BLOCK>(odd ? gd.A1 : gd.A0, la, n, pack ? (odd ? gd.A0 : gd.A1) : nullptr, gd.F0, D, k,
                                           sh, ph, &dmin, &nf);
    if (left == 0) break;
    if (pack) {
      la = left;
      odd = !odd;
      peeled = 0;
    }
    if (dmin != k + 1) nf = select_frontier<BLOCK>(odd ? gd.A1 : gd.A0, la, n, gd.F0, D, dmin, sh, ph);
    k = dmin;
  }
  if (tid == 0) *gd.kmax = kmax;
  team_sync<BLOCK>();
}

// ------------------------------------------------------------------ clustered form
namespace cg = cooperative_groups;

// Counters of a cluster, kept in its first CTA. Each phase (the work between
// two cluster barriers) accumulates into slot[phase % 3] -- [0] and [1]
// counts, [2] a minimum, [3] a maximum -- which every CTA reads after the
// barrier that ends the phase; the first CTA clears the slot of the next phase
// at the start of each phase (its last readers passed a barrier since).
struct ClusterCtl {
  int g;    // graph drawn for the cluster
  int bad;  // the graph failed a bounds check
  int slot[3][4];
};

template <int BLOCK, int C>
struct ClusterPeel {
  cg::cluster_group cl;
  ClusterCtl* lc;  // the first CTA's counters
  BatchShared<BLOCK>& sh;
  int* status;
  int r;       // this CTA's rank in the cluster
  int ph = 0;  // phase index (the same in every CTA)
  int sp = 0;  // which of the two sets of block-scan sums the next scan uses

  __device__ ClusterPeel(ClusterCtl* lead, BatchShared<BLOCK>& s, int* st)
      : cl(cg::this_cluster()), lc(lead), sh(s), status(st), r((int)cg::this_cluster().block_rank()) {}

  __device__ int* slot(int p) const { return lc->slot[p % 3]; }
  __device__ void clear(int p) const {
    int* x = slot(p);
    x[0] = 0;
    x[1] = 0;
    x[2] = INT_MAX;
    x[3] = 0;
  }
  __device__ bool first() const { return r == 0 && threadIdx.x == 0; }
  // ends a phase: this CTA's bounds-check failure goes to the cluster flag,
  // then the cluster barrier (release / acquire: the phase's stores, global
  // and distributed shared, are seen by every CTA after it)
  __device__ void next_phase() {
    __syncthreads();  // every thread's flag_bad of this phase is seen by thread 0
    if (threadIdx.x == 0 && sh.bad) atomicOr(&lc->bad, 1);
    cl.sync();
    ph++;
    if (first()) clear(ph + 1);
  }
  // this CTA's part [lo, hi) of a range of len entries
  __device__ long long part_lo(long long len) const { return len * r / C; }
  __device__ long long part_hi(long long len) const { return len * (r + 1) / C; }

  // entries of A with D == k go to F (count in this phase's slot[0])
  __device__ void select(const int* A, int la, int n, int* F, const DegStore& D, int k) {
    const int lo = (int)part_lo(la), hi = (int)part_hi(la);
    for (int base = lo; base < hi; base += BLOCK * kScanItems) {
      const TileMap tm = TileMap::at<BLOCK>(base, hi);
      int v[kScanItems];
#pragma unroll
      for (int q = 0; q < kScanItems; q++) {
        const int i = tm.entry(q);
        v[q] = -1;
        if (i >= 0) {
          const int x = __ldcg(A + i);  // written by other CTAs of the cluster
          v[q] = (unsigned)x < (unsigned)n ? x : -1;
        }
      }
      int d[kScanItems];
      D.get_all(v, d);
      int tot, own;
      const int at = tile_count(d, INT_MAX, k, sh, sp, &tot, &own);
      if (threadIdx.x == 0) sh.base = tot ? atomicAdd(&slot(ph)[0], tot >> 16) : 0;
      __syncthreads();
      if (own) tile_write(v, d, F + sh.base + (at >> 16), [k](int x) { return x == k; });
      __syncthreads();  // sh.base is reused by the next tile
    }
  }

  // entries of A with D > k survive into out (count slot[0], minimum slot[2]);
  // those at k + 1 also go to F (count slot[1])
  __device__ void compact(const int* A, int la, int n, int* out, int* F, const DegStore& D, int k) {
    const int lo = (int)part_lo(la), hi = (int)part_hi(la);
    int lmin = INT_MAX;
    for (int base = lo; base < hi; base += BLOCK * kScanItems) {
      const TileMap tm = TileMap::at<BLOCK>(base, hi);
      int v[kScanItems];
#pragma unroll
      for (int q = 0; q < kScanItems; q++) {
        const int i = tm.entry(q);
        v[q] = -1;
        if (i >= 0) {
          const int x = __ldcg(A + i);
          v[q] = (unsigned)x < (unsigned)n ? x : -1;
        }
      }
      int d[kScanItems];
      D.get_all(v, d);
#pragma unroll
      for (int q = 0; q < kScanItems; q++)
        if (d[q] > k) lmin = min(lmin, d[q]);  // (no entry: -1)
      int tot, own;
      const int at = tile_count(d, k + 1, k + 1, sh, sp, &tot, &own);
      if (threadIdx.x == 0) {
        const int bk = (tot & 0xffff) ? atomicAdd(&slot(ph)[0], tot & 0xffff) : 0;
        const int bf = (tot >> 16) ? atomicAdd(&slot(ph)[1], tot >> 16) : 0;
        sh.base = bk;
        sh.base2 = bf;
      }
      __syncthreads();
      tile_write(v, d, out + sh.base + (at & 0xffff), [k](int x) { return x > k; });
      if (own >> 16) tile_write(v, d, F + sh.base2 + (at >> 16), [k](int x) { return x == k + 1; });
      __syncthreads();
    }
    int none = INT_MAX;
    block_min2(lmin, none, sh);
    if (threadIdx.x == 0 && lmin != INT_MAX) atomicMin(&slot(ph)[2], lmin);
  }

  // Peels one graph with the whole cluster (Algorithm 1's levels and
  // subrounds, the online Peel of Algorithm 3, as peel_one_graph does in one CTA).
  __device__ void peel(const GraphDesc& gd) {
    const int tid = threadIdx.x;
    if (first()) {
      lc->bad = 0;
      clear(0);
      clear(1);
      clear(2);
    }
    if (tid == 0) sh.bad = 0;
    ph = 0;
    cl.sync();
    const int n = (int)gd.n;
    const long long* O = gd.off;
    // phase: degrees (least and largest)
    int lmin = INT_MAX, lmax = 0;
    for (long long v = (long long)r * BLOCK + tid; v < n; v += (long long)C * BLOCK) {
      long long o0 = O[v], o1 = O[v + 1];
      if (o0 < 0 || o1 < o0 || o1 > gd.m || o1 - o0 >= n) {
        flag_bad(status, 1, v, &sh.bad);
        o1 = o0;
      }
      lmin = min(lmin, (int)(o1 - o0));
      lmax = max(lmax, (int)(o1 - o0));
    }
    lmax = -lmax;
    block_min2(lmin, lmax, sh);
    lmax = -lmax;
    if (tid == 0) {
      atomicMin(&slot(ph)[2], lmin);
      atomicMax(&slot(ph)[3], lmax);
    }
    next_phase();
    int k = slot(ph - 1)[2];
    const int dmax = slot(ph - 1)[3];
    if (lc->bad) {  // malformed offsets: leave this graph (its outputs are undefined)
      if (first()) *gd.kmax = -1;
      return;
    }
    const bool narrow = dmax < 65536;
    const int chunk = chunk_vertices(BLOCK, dmax);
    const DegStore D{gd.deg, 0u, 0, kDegGlobal, narrow, l2_evict_last_policy()};
    // phase: initial induced degrees, the identity active list
    const int nw = narrow ? (n + 1) / 2 : n;
    for (long long i = (long long)r * BLOCK + tid; i < nw; i += (long long)C * BLOCK) {
      const int v0 = narrow ? 2 * (int)i : (int)i;
      const int d0 = (int)(O[v0 + 1] - O[v0]);
      const int d1 = narrow && v0 + 1 < n ? (int)(O[v0 + 2] - O[v0 + 1]) : 0;
      D.put_word((int)i, d0, d1);
    }
    for (long long v = (long long)r * BLOCK + tid; v < n; v += (long long)C * BLOCK) gd.A0[v] = (int)v;
    next_phase();
    int* A = gd.A0;
    int* An = gd.A1;
    int la = n, kmax = 0;
    select(A, la, n, gd.F0, D, k);
    next_phase();
    int nf = slot(ph - 1)[0];
    for (;;) {
      int* Fc = gd.F0;
      int* Fn = gd.F1;
      while (nf > 0) {
        // a large frontier: the CTAs take whole chunks of frontier vertices in turn; a small one: every CTA walks every chunk and takes
        // its share of the chunk's arcs (the first CTA writes their coreness)
        const bool whole = nf >= 2 * C * chunk;
        for (int c0 = whole ? r * chunk : 0; c0 < nf; c0 += whole ? C * chunk : chunk) {
          const int cnum = min(chunk, nf - c0);
          const int total = load_chunk<BLOCK>(gd, Fc + c0, cnum, n, k, whole || r == 0, status, sh, sp);
          chunk_arcs<BLOCK>(gd, D, n, k, whole ? 0 : (int)part_lo(total), whole ? total : (int)part_hi(total), cnum, Fn,
                            &slot(ph)[0], status, sh);
          __syncthreads();  // the chunk's arrays are reused by the next one
        }
        next_phase();
        nf = slot(ph - 1)[0];
        if (nf > n) nf = 0;  // cannot happen: every vertex lands on k at most once per level
        if (lc->bad) {
          if (first()) *gd.kmax = -1;
          return;
        }
        int* t = Fc;
        Fc = Fn;
        Fn = t;
      }
      kmax = k;
      compact(A, la, n, An, gd.F0, D, k);
      next_phase();
      la = slot(ph - 1)[0];
      nf = slot(ph - 1)[1];
      const int dmin = slot(ph - 1)[2];
      int* t = A;
      A = An;
      An = t;
      if (la == 0) break;
      if (dmin != k + 1) {
        select(A, la, n, gd.F0, D, dmin);
        next_phase();
        nf = slot(ph - 1)[0];
      }
      k = dmin;
    }
    if (first()) *gd.kmax = kmax;
  }
};

// Where a kernel's graphs come from: a batch's segmented CSR, or descriptors in
// a device table (graphs in separate allocations, as the server holds them;
// the launch lists the table slots to process). find() looks up the graph at
// position gi of the processing order, desc() describes it.
struct Found {
  long long g, v0, n, arcs;  // graph (or slot), first vertex, vertices, arcs
};
struct BatchSource {
  const BatchArgs& a;
  __device__ __forceinline__ long long count() const { return a.G; }
  __device__ __forceinline__ int* next() const { return a.next_graph; }
  __device__ __forceinline__ int* status() const { return a.status; }
  __device__ __forceinline__ int smem() const { return a.smem_deg_max; }
  __device__ __forceinline__ long long team_arcs() const { return a.team_arcs; }
  // false: a failed check, recorded by the thread that reports it
  __device__ __forceinline__ bool find(long long gi, bool report, int* bad, Found* f) const {
    f->g = a.order ? a.order[gi] : gi;
    if (f->g < 0 || f->g >= a.G) {  // the order is a permutation of [0, G); checked anyway
      if (report) flag_bad(a.status, 8, f->g, bad);
      return false;
    }
    f->v0 = a.gv[f->g];
    f->n = a.gv[f->g + 1] - f->v0;
    if (f->v0 < 0 || f->n < 0 || f->v0 + f->n > a.N) {  // graph outside the vertex range
      if (report) {
        flag_bad(a.status, 9, f->g, bad);
        a.kmax[f->g] = -1;
      }
      return false;
    }
    f->arcs = a.off[f->v0 + f->n] - a.off[f->v0];
    return true;
  }
  __device__ __forceinline__ GraphDesc desc(const Found& f) const {
    return GraphDesc{a.off + f.v0, a.adj,       a.core + f.v0, a.kmax + f.g, a.deg + f.v0, a.A0 + f.v0,
                     a.A1 + f.v0,  a.F0 + f.v0, a.F1 + f.v0,   f.n,          a.m};
  }
};
struct ListSource {
  const GraphDesc* table;
  const SlotList& list;
  int* next_;
  int* status_;
  int smem_deg_max;
  long long team_arcs_;
  __device__ __forceinline__ long long count() const { return list.count; }
  __device__ __forceinline__ int* next() const { return next_; }
  __device__ __forceinline__ int* status() const { return status_; }
  __device__ __forceinline__ int smem() const { return smem_deg_max; }
  __device__ __forceinline__ long long team_arcs() const { return team_arcs_; }
  __device__ __forceinline__ bool find(long long gi, bool, int*, Found* f) const {
    f->g = list.slot[gi];
    const GraphDesc& d = table[f->g];
    f->v0 = 0;
    f->n = d.n;
    f->arcs = d.n > 0 ? d.off[d.n] - d.off[0] : 0;
    return true;
  }
  __device__ __forceinline__ GraphDesc desc(const Found& f) const { return table[f.g]; }
};

// Draws graph after graph for the team and peels them. first >= 0: a graph the
// CTA drew already. With stop_below > 0, returns the position of the first
// graph of fewer arcs, unpeeled; -1 once the graphs are exhausted.
template <int BLOCK, typename Source>
__device__ long long peel_drawn(const Source& src, int smem_deg_max, int* sdeg, BatchShared<BLOCK>& sh, long long first,
                                long long stop_below) {
  const int tid = team_tid<BLOCK>();
  for (;;) {
    if (tid == 0) sh.g = first >= 0 ? (int)first : atomicAdd(src.next(), 1);
    first = -1;
    team_sync<BLOCK>();
    const long long gi = sh.g;
    team_sync<BLOCK>();
    if (gi >= src.count()) return -1;
    Found f;
    if (!src.find(gi, tid == 0, &sh.bad, &f)) continue;
    // (0: never. A malformed graph may count fewer than no arcs: it is peeled
    // here all the same, so that peel_one_graph's checks report it)
    if (stop_below > 0 && f.arcs < stop_below) return gi;
    if (tid == 0) sh.gd = src.desc(f);
    team_sync<BLOCK>();
    peel_one_graph<BLOCK>(smem_deg_max, src.status(), sdeg, sh);
  }
}

// A 1,024-thread CTA peels whole graphs while they are large (team_arcs arcs
// or more; the order is by arcs) and from the first smaller one on splits into
// teams of kTeam threads, each drawing graphs of its own with its share of the
// shared memory: a small graph's phases are short dependent chains that leave
// most of an SM idle.
constexpr int kTeam = 512;
template <int BLOCK>
constexpr int kTeams = BLOCK >= 1024 ? BLOCK / kTeam : 1;
template <int BLOCK>
union CtaShared {
  BatchShared<BLOCK> whole;
  BatchShared<BLOCK / kTeams<BLOCK>> team[kTeams<BLOCK>];
};
template <int BLOCK, typename Source>
__device__ void peel_cta(const Source& src, int* sdeg, CtaShared<BLOCK>& sh, long long first) {
  constexpr int T = kTeams<BLOCK>;
  const long long gi = peel_drawn<BLOCK>(src, src.smem(), sdeg, sh.whole, first, T > 1 ? src.team_arcs() : 0);
  if constexpr (T > 1) {
    if (gi < 0) return;
    __syncthreads();
    const int t = threadIdx.x / kTeam, share = src.smem() / T;
    peel_drawn<kTeam>(src, share, sdeg + t * share, sh.team[t], t == 0 ? gi : -1, 0);
  }
}

// The clustered form: clusters of C CTAs for the graphs of at least big_arcs
// arcs (see the file comment). A cluster draws graphs together while they are
// big; from the first graph below the threshold on, its CTAs draw their own
// (the first CTA starts with that graph).
template <int BLOCK, int C, typename Source>
__device__ void peel_cluster(const Source& src, int* sdeg, CtaShared<BLOCK>& sh, ClusterCtl& ctl, long long big_arcs) {
  cg::cluster_group cl = cg::this_cluster();
  ClusterCtl* lc = cl.map_shared_rank(&ctl, 0);
  const bool lead = cl.block_rank() == 0;
  for (;;) {
    if (lead && threadIdx.x == 0) ctl.g = atomicAdd(src.next(), 1);
    cl.sync();
    const long long gi = lc->g;
    cl.sync();  // every CTA has read the draw before the next one
    if (gi >= src.count()) return;
    Found f;
    if (!src.find(gi, lead && threadIdx.x == 0, &sh.whole.bad, &f)) continue;
    if (!(f.n > 0 && f.n < INT_MAX && f.arcs >= big_arcs)) {
      peel_cta<BLOCK>(src, sdeg, sh, lead ? gi : -1);
      return;
    }
    if (threadIdx.x == 0) sh.whole.gd = src.desc(f);
    __syncthreads();
    ClusterPeel<BLOCK, C> cp(lc, sh.whole, src.status());
    cp.peel(sh.whole.gd);
  }
}

template <int BLOCK>
__global__ void __launch_bounds__(BLOCK, (BLOCK >= 1024 ? 1 : 2048 / BLOCK * 3 / 4)) batch_peel(BatchArgs a) {
  extern __shared__ int sdeg[];
  __shared__ CtaShared<BLOCK> sh;
  peel_cta<BLOCK>(BatchSource{a}, sdeg, sh, -1);
}

template <int BLOCK, int C>
__global__ void __cluster_dims__(C, 1, 1) __launch_bounds__(BLOCK, (BLOCK >= 1024 ? 1 : 2048 / BLOCK / 2))
    batch_peel_cl(BatchArgs a, long long big_arcs) {
  extern __shared__ int sdeg[];
  __shared__ CtaShared<BLOCK> sh;
  __shared__ ClusterCtl ctl;
  peel_cluster<BLOCK, C>(BatchSource{a}, sdeg, sh, ctl, big_arcs);
}

// (the launch lists the slots largest first)
template <int BLOCK>
__global__ void __launch_bounds__(BLOCK, (BLOCK >= 1024 ? 1 : 2048 / BLOCK / 2))
    desc_peel(const GraphDesc* table, const __grid_constant__ SlotList list, int* next, int smem_deg_max, int* status,
              long long team_arcs) {
  extern __shared__ int sdeg[];
  __shared__ CtaShared<BLOCK> sh;
  peel_cta<BLOCK>(ListSource{table, list, next, status, smem_deg_max, team_arcs}, sdeg, sh, -1);
}

template <int BLOCK, int C>
__global__ void __cluster_dims__(C, 1, 1) __launch_bounds__(BLOCK, (BLOCK >= 1024 ? 1 : 2048 / BLOCK / 2))
    desc_peel_cl(const GraphDesc* table, const __grid_constant__ SlotList list, int* next, int smem_deg_max, int* status,
                 long long team_arcs, long long big_arcs) {
  extern __shared__ int sdeg[];
  __shared__ CtaShared<BLOCK> sh;
  __shared__ ClusterCtl ctl;
  peel_cluster<BLOCK, C>(ListSource{table, list, next, status, smem_deg_max, team_arcs}, sdeg, sh, ctl, big_arcs);
}

// Order of graphs: descending number of arcs (ties by index). One CTA sorts
// keys (~arcs << 24 | g) bitonically in shared memory; batches larger than
// kMaxSortGraphs keep their given order.
__global__ void __launch_bounds__(1024) batch_order(const long long* gv, const long long* off,
                                                    long long G, int* order) {
  extern __shared__ unsigned long long key[];
  int P = 1;
  while (P < G) P <<= 1;
  for (int i = threadIdx.x; i < P; i += blockDim.x) {
    if (i < G) {
      unsigned long long arcs = (unsigned long long)(off[gv[i + 1]] - off[gv[i]]);
      if (arcs > 0xffffffffffull) arcs = 0xffffffffffull;
      key[i] = ((0xffffffffffull - arcs) << 24) | (unsigned long long)i;
    } else {
      key[i] = ~0ull;
    }
  }
  __syncthreads();
  for (int size = 2; size <= P; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = threadIdx.x; i < P; i += blockDim.x) {
        int j = i ^ stride;
        if (j > i) {
          bool up = (i & size) == 0;
          unsigned long long x = key[i], y = key[j];
          if ((x > y) == up) {
            key[i] = y;
            key[j] = x;
          }
        }
      }
      __syncthreads();
    }
  }
  for (int i = threadIdx.x; i < G; i += blockDim.x) order[i] = (int)(key[i] & 0xffffffull);
}

// ------------------------------------------------------------------ host side
namespace {
template <int BLOCK>
cudaError_t launch_block(const BatchArgs& a, int grid, size_t smem, cudaStream_t stream) {
  cudaError_t e = cudaFuncSetAttribute(batch_peel<BLOCK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  batch_peel<BLOCK><<<grid, BLOCK, smem, stream>>>(a);
  return cudaGetLastError();
}
template <int BLOCK, int C>
cudaError_t launch_cluster(const BatchArgs& a, int grid, size_t smem, long long big_arcs, cudaStream_t stream) {
  cudaError_t e = cudaFuncSetAttribute(batch_peel_cl<BLOCK, C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  grid = grid / C * C;
  if (grid < C) grid = C;
  batch_peel_cl<BLOCK, C><<<grid, BLOCK, smem, stream>>>(a, big_arcs);
  return cudaGetLastError();
}
template <int BLOCK>
int occupancy_block(size_t smem) {
  int nb = 0;
  cudaFuncSetAttribute(batch_peel<BLOCK>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, batch_peel<BLOCK>, BLOCK, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return nb;
}
}  // namespace

namespace {
template <int C>
cudaError_t desc_launch_cl(const GraphDesc* table, const SlotList& list, int* next, int smem_deg_max, int* status,
                           int grid, size_t smem, long long team_arcs, long long big_arcs, cudaStream_t stream) {
  cudaError_t e = cudaFuncSetAttribute(desc_peel_cl<1024, C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  grid = std::max(C, grid / C * C);
  desc_peel_cl<1024, C><<<grid, 1024, smem, stream>>>(table, list, next, smem_deg_max, status, team_arcs, big_arcs);
  return cudaGetLastError();
}
}  // namespace

cudaError_t desc_launch(const GraphDesc* table, const SlotList& list, int* next, int smem_deg_max,
                        int* status, int grid, size_t smem, cudaStream_t stream, long long team_arcs, int cluster,
                        long long big_arcs) {
  switch (cluster) {
    case 2: return desc_launch_cl<2>(table, list, next, smem_deg_max, status, grid, smem, team_arcs, big_arcs, stream);
    case 4: return desc_launch_cl<4>(table, list, next, smem_deg_max, status, grid, smem, team_arcs, big_arcs, stream);
    case 8: return desc_launch_cl<8>(table, list, next, smem_deg_max, status, grid, smem, team_arcs, big_arcs, stream);
  }
  cudaError_t e = cudaFuncSetAttribute(desc_peel<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  desc_peel<1024><<<grid, 1024, smem, stream>>>(table, list, next, smem_deg_max, status, team_arcs);
  return cudaGetLastError();
}

size_t desc_static_smem() { return sizeof(CtaShared<1024>); }

__global__ void batch_single_gv_kernel(long long* gv, long long n) {
  gv[0] = 0;
  gv[1] = n;
}

cudaError_t batch_single_gv(long long* gv, long long n, cudaStream_t stream) {
  batch_single_gv_kernel<<<1, 1, 0, stream>>>(gv, n);
  return cudaGetLastError();
}

int batch_occupancy(int block, size_t smem) {
  switch (block) {
    case 256: return occupancy_block<256>(smem);
    case 512: return occupancy_block<512>(smem);
    case 1024: return occupancy_block<1024>(smem);
  }
  return 0;
}

size_t batch_static_smem(int block) {
  switch (block) {
    case 256: return sizeof(CtaShared<256>);
    case 512: return sizeof(CtaShared<512>);
    case 1024: return sizeof(CtaShared<1024>);
  }
  return 0;
}

cudaError_t batch_launch(const BatchArgs& a, int block, int grid, size_t smem, bool sort_graphs,
                         cudaStream_t stream, int cluster, long long big_arcs) {
  if (sort_graphs && a.order) {
    int P = 1;
    while (P < a.G) P <<= 1;
    size_t ss = sizeof(unsigned long long) * (size_t)P;
    cudaError_t e = cudaFuncSetAttribute(batch_order, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ss);
    if (e != cudaSuccess) return e;
    batch_order<<<1, 1024, ss, stream>>>(a.gv, a.off, a.G, (int*)a.order);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (cluster > 1) {
    const int key = block * 16 + cluster;
    switch (key) {
      case 512 * 16 + 2: return launch_cluster<512, 2>(a, grid, smem, big_arcs, stream);
      case 512 * 16 + 4: return launch_cluster<512, 4>(a, grid, smem, big_arcs, stream);
      case 512 * 16 + 8: return launch_cluster<512, 8>(a, grid, smem, big_arcs, stream);
      case 1024 * 16 + 2: return launch_cluster<1024, 2>(a, grid, smem, big_arcs, stream);
      case 1024 * 16 + 4: return launch_cluster<1024, 4>(a, grid, smem, big_arcs, stream);
      case 1024 * 16 + 8: return launch_cluster<1024, 8>(a, grid, smem, big_arcs, stream);
    }
    return cudaErrorInvalidValue;
  }
  switch (block) {
    case 256: return launch_block<256>(a, grid, smem, stream);
    case 512: return launch_block<512>(a, grid, smem, stream);
    case 1024: return launch_block<1024>(a, grid, smem, stream);
  }
  return cudaErrorInvalidValue;
}

}  // namespace kc
