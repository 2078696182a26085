// CSR build on sm_103a: edge list -> simple undirected CSR.
//
// The paper symmetrises directed inputs (Sec. 6.1, "Datasets"); the peel needs
// a simple graph. Steps, all on the device:
//   1. keys: each pair (a, b) with a != b gives the arcs a->b and b->a as
//      integers (a << B) | b with B = bits of n-1; self-loops and ids out of
//      range become a sentinel that sorts last (ids out of range also set an
//      error status). The keys are not stored: the first radix pass (which
//      need not be stable) makes them from the edge arrays as it reads them.
//   2. stable LSD radix sort of the keys over their 2B significant bits, 8-bit
//      digits. Each CTA owns a contiguous chunk; a pass is an upsweep (digit
//      histogram per CTA), a scan of each digit's row of the 256 x CTAs
//      histogram (one CTA per digit), and a downsweep that ranks each
//      4,096-key tile in shared memory and writes runs of equal digits
//      contiguously, while the next tile's lines are prefetched. A key's rank
//      within its warp and digit comes from one pass over the warp's rows: the
//      lanes holding a digit or their bits into the warp's counter for it.
//   3. unique + emit: keys equal to their predecessor are dropped; the rest
//      are written in order as adj[] (low B bits), and the first arc of each
//      source vertex fixes offsets[] (vertices without arcs take the next
//      vertex's offset). Each warp walks a chunk of its own in rows of 32 keys;
//      the predecessor comes from the next lower lane or row and the positions
//      from warp ballots, so no key passes through shared memory.
// A single graph, and a batch for which it means fewer keys to move, takes the
// edge route through steps 1-3: each pair (a, b) with a != b gives ONE key
// (min << B) | max (global ids); sorting these E keys by both
// fields gives every vertex's upper neighbours in order (A), and a stable
// sort of A by its low B bits (the larger endpoint) gives every vertex's
// lower neighbours in order (B). A vertex's list is its lower neighbours
// followed by its upper ones, both ascending, so emission writes the CSR from
// A and B directly: 2B + B digit passes over E keys instead of 2B over 2E.
// Repeats stay in A as adjacent equal keys and are dropped on emission; the
// first pass of B's sort drops them (and the sentinels), and the rest of B's
// buffer holds sentinels written beforehand, which every stable pass keeps
// behind the real keys.
//
// Lists come out ascending and duplicate-free, the canonical form of the CPU
// builder, so the two are comparable bit for bit.
#include <algorithm>
#include <climits>

#include "kcore_csr.h"
#include "kcore_device.cuh"

namespace kc {

constexpr int kCsrBlock = 256;
constexpr unsigned long long kSentinel = ~0ull;

// Keys (source << Bd) | target. Single graph: ids in [0, n), source = id.
// Batch (gv != nullptr): edge i belongs to the graph g with eoff[g] <= i <
// eoff[g+1]; its ids are graph-local in [0, gv[g+1] - gv[g]); the source part
// is the global id gv[g] + local, the target part stays local.
struct EdgeList {
  const int* src;
  const int* dst;
  long long n;
  int Bd;
  const long long* gv;
  const long long* eoff;
  long long G;
  int* status;
};

// a batch: the last graph g in [glo, ghi) with eoff[g] <= i
__device__ __forceinline__ long long graph_of(const EdgeList& es, long long i, long long glo, long long ghi) {
  long long lo = glo, hi = ghi;
  while (hi - lo > 1) {
    const long long mid = (lo + hi) >> 1;
    if (es.eoff[mid] <= i) lo = mid;
    else hi = mid;
  }
  return lo;
}

// a batch: the graphs [*glo, *ghi) that hold edges [e0, e1) (a CTA's chunk;
// one binary search each for its first and last edge, by thread 0, shared
// through *glo / *ghi in shared memory; the caller synchronises)
__device__ __forceinline__ void chunk_graphs(const EdgeList& es, long long e0, long long e1, long long* glo,
                                             long long* ghi) {
  if (threadIdx.x == 0) {
    *glo = es.gv && e0 < e1 ? graph_of(es, e0, 0, es.G) : 0;
    *ghi = es.gv && e0 < e1 ? graph_of(es, e1 - 1, *glo, es.G) + 1 : es.G;
  }
}

// the arcs of edge i = (a, b): keys 2i (a -> b) and 2i + 1 (b -> a); a batch's
// edge i lies in one of the graphs [glo, ghi)
__device__ __forceinline__ void edge_keys(const EdgeList& es, long long i, int a, int b, unsigned long long& k0,
                                          unsigned long long& k1, long long glo = 0, long long ghi = 0) {
  long long base = 0, lim = es.n;
  if (es.gv) {
    const long long g = ghi - glo == 1 ? glo : graph_of(es, i, glo, ghi > glo ? ghi : es.G);
    base = es.gv[g];
    lim = es.gv[g + 1] - base;
  }
  k0 = k1 = kSentinel;
  if ((unsigned long long)(unsigned)a >= (unsigned long long)lim ||
      (unsigned long long)(unsigned)b >= (unsigned long long)lim) {
    atomicCAS(es.status, 0, 1);
  } else if (a != b) {
    k0 = ((unsigned long long)(base + a) << es.Bd) | (unsigned long long)b;
    k1 = ((unsigned long long)(base + b) << es.Bd) | (unsigned long long)a;
  }
}

// edge i = (a, b) as one key (min << B) | max; a batch's (kBatch) with global
// ids, its edge i in one of the graphs [glo, ghi)
template <bool kBatch>
__device__ __forceinline__ unsigned long long edge_canon(const EdgeList& es, long long i, int a, int b, long long glo,
                                                         long long ghi) {
  long long base = 0, lim = es.n;
  if constexpr (kBatch) {
    const long long g = ghi - glo == 1 ? glo : graph_of(es, i, glo, ghi);
    base = es.gv[g];
    lim = es.gv[g + 1] - base;
  }
  if ((unsigned long long)(unsigned)a >= (unsigned long long)lim ||
      (unsigned long long)(unsigned)b >= (unsigned long long)lim) {
    atomicCAS(es.status, 0, 1);
    return kSentinel;
  }
  if (a == b) return kSentinel;
  return ((unsigned long long)(base + min(a, b)) << es.Bd) | (unsigned long long)(base + max(a, b));
}

// Where a pass's keys come from: a key array, the edge list as two arcs per
// edge (the first pass of the arc route), the edge list as one key per edge
// (the first pass of the edge route; kCanonB: a batch's), or a sorted key array
// without its sentinels and without keys equal to their predecessor (the
// first pass of B's sort).
enum KeySrc : int { kKeys = 0, kArcs = 1, kCanon = 2, kKeysDrop = 3, kCanonB = 4 };

// digit of a pass: bits [shift, shift + 8) of the key, masked by dmask (the
// last pass over a field narrower than a multiple of 8 bits keeps only its bits)
__device__ __forceinline__ int digit_of(unsigned long long k, int shift, int dmask) {
  return (int)((k >> shift) & (unsigned long long)dmask);
}

// Per-CTA digit histogram of its chunk: hist[d * G + g]. kArcs: the keys are
// made from the edge list, two per edge (chunks hold whole edges: chunk and lo
// are even); kCanon: one per edge.
template <int kSrc>
__global__ void __launch_bounds__(kCsrBlock) rs_upsweep(const unsigned long long* keys, EdgeList es,
                                                        long long N, long long chunk, int shift, int dmask,
                                                        unsigned* hist) {
  wait_predecessor();
  __shared__ unsigned cnt[kCsrBlock / 32][256];
  const int tid = threadIdx.x, warp = tid >> 5;
  for (int i = tid; i < (kCsrBlock / 32) * 256; i += kCsrBlock) (&cnt[0][0])[i] = 0;
  __syncthreads();
  long long lo = (long long)blockIdx.x * chunk, hi = min(N, lo + chunk);
  if constexpr (kSrc == kCanon || kSrc == kCanonB) {
    __shared__ long long cg_lo, cg_hi;
    if constexpr (kSrc == kCanonB) {
      chunk_graphs(es, lo, max(lo, hi), &cg_lo, &cg_hi);
      __syncthreads();
    }
    const long long glo = kSrc == kCanonB ? cg_lo : 0, ghi = kSrc == kCanonB ? cg_hi : 0;
    constexpr int kU = 4;
    for (long long e0 = lo + tid; e0 < hi; e0 += kU * kCsrBlock) {
      int a[kU], b[kU];
#pragma unroll
      for (int u = 0; u < kU; u++) {
        const long long e = e0 + u * kCsrBlock;
        a[u] = e < hi ? __ldcs(es.src + e) : 0;
        b[u] = e < hi ? __ldcs(es.dst + e) : 0;
      }
#pragma unroll
      for (int u = 0; u < kU; u++)
        if (e0 + u * kCsrBlock < hi)
          atomicAdd(&cnt[warp][digit_of(edge_canon<kSrc == kCanonB>(es, e0 + u * kCsrBlock, a[u], b[u], glo, ghi), shift, dmask)],
                    1u);
    }
  } else if constexpr (kSrc == kArcs) {
    __shared__ long long cg_lo, cg_hi;
    chunk_graphs(es, lo / 2, hi > lo ? hi / 2 : lo / 2, &cg_lo, &cg_hi);
    __syncthreads();
    const long long glo = cg_lo, ghi = cg_hi;
    constexpr int kU = 4;  // edges per thread per step, loaded before any count
    for (long long e0 = lo / 2 + tid; e0 < hi / 2; e0 += kU * kCsrBlock) {
      int a[kU], b[kU];
#pragma unroll
      for (int u = 0; u < kU; u++) {
        const long long e = e0 + u * kCsrBlock;
        a[u] = e < hi / 2 ? __ldcs(es.src + e) : 0;
        b[u] = e < hi / 2 ? __ldcs(es.dst + e) : 0;
      }
#pragma unroll
      for (int u = 0; u < kU; u++) {
        const long long e = e0 + u * kCsrBlock;
        if (e < hi / 2) {
          unsigned long long k0, k1;
          edge_keys(es, e, a[u], b[u], k0, k1, glo, ghi);
          atomicAdd(&cnt[warp][digit_of(k0, shift, dmask)], 1u);
          atomicAdd(&cnt[warp][digit_of(k1, shift, dmask)], 1u);
        }
      }
    }
  } else if constexpr (kSrc == kKeysDrop) {
    for (long long i = lo + tid; i < hi; i += kCsrBlock) {
      const unsigned long long x = keys[i], p = i > 0 ? keys[i - 1] : kSentinel;
      if (x != kSentinel && x != p) atomicAdd(&cnt[warp][digit_of(x, shift, dmask)], 1u);
    }
  } else {
    for (long long i = lo + tid; i < hi; i += kCsrBlock) atomicAdd(&cnt[warp][digit_of(keys[i], shift, dmask)], 1u);
  }
  __syncthreads();
  unsigned s = 0;
  for (int w = 0; w < kCsrBlock / 32; w++) s += cnt[w][tid];
  hist[(long long)tid * gridDim.x + blockIdx.x] = s;
}

// Exclusive scans of uint32 rows into uint64: CTA r (1024 threads) scans
// in[r * len, (r + 1) * len) into out[] at the same place and, if totals is
// given, writes the row's sum to totals[r].
__global__ void __launch_bounds__(1024) scan_u32_to_u64(const unsigned* in, unsigned long long* out,
                                                        long long len, unsigned long long* totals) {
  wait_predecessor();
  __shared__ unsigned long long part[32];
  __shared__ unsigned long long carry;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  in += (long long)blockIdx.x * len;
  out += (long long)blockIdx.x * len;
  if (tid == 0) carry = 0;
  __syncthreads();
  for (long long base = 0; base < len; base += 1024) {
    long long i = base + tid;
    unsigned long long x = i < len ? in[i] : 0;
    unsigned long long incl = warp_incl_scan(x, lane);
    if (lane == 31) part[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      unsigned long long p = part[lane];
      unsigned long long pi = warp_incl_scan(p, lane);
      part[lane] = pi - p;
    }
    __syncthreads();
    unsigned long long c = carry;
    if (i < len) out[i] = c + part[warp] + incl - x;
    __syncthreads();
    if (tid == 1023) carry = c + part[warp] + incl;
    __syncthreads();
  }
  if (totals && tid == 0) totals[blockIdx.x] = carry;
}

// Stable scatter of one radix pass. Each CTA walks its chunk tile by tile, in
// order. offs[d * G + g] counts the keys of digit d in the chunks before g,
// rowtot[d] all keys of digit d; so the CTA's first key of digit d goes after
// every key of a smaller digit and the digit-d keys of earlier chunks.
// kArcs / kCanon / kCanonB: the first pass, whose keys are made from the edge
// list (a tile is 2,048 edges / 4,096 edges; the order within a tile does not
// matter in the first pass).
// Pos: the type of an output position (32 bits when there are at most 2^32
// keys: positions are then computed modulo 2^32).
static_assert(kCsrBlock == 256, "one thread per 8-bit digit");
constexpr int kSortKeys = 16;                     // keys per thread per tile
constexpr int kSortTile = kCsrBlock * kSortKeys;  // 4,096
template <int kSrc, typename Pos>
__global__ void __launch_bounds__(kCsrBlock, 3) rs_downsweep(const unsigned long long* in, EdgeList es,
                                                          unsigned long long* out, long long N,
                                                          long long chunk, int shift, int dmask,
                                                          const unsigned long long* offs,
                                                          const unsigned long long* rowtot) {
  wait_predecessor();
  constexpr int kW = kCsrBlock / 32, kRow = kSortKeys * 32;  // keys of a warp's part of a tile
  // The warps' digit counters (x: the lanes of the current row that hold the
  // digit, y: keys counted) are done with before the exchange buffer is
  // written, so they share its memory.
  __shared__ __align__(16) union {
    unsigned long long buf[kSortTile];
    uint2 cnt[kW][256];
  } sm;
  __shared__ unsigned wofs[kW][256];  // tile offset of each (warp, digit)'s first key
  __shared__ Pos dstb[256];  // output position of the tile's first key of digit d, minus its tile offset
  __shared__ unsigned long long part64[kW];
  __shared__ unsigned part[kW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = gridDim.x;
  const unsigned lt = lanemask_lt();
  // run: where this CTA's next key of digit tid goes
  unsigned long long run;
  {
    const unsigned long long rt = rowtot[tid];
    const unsigned long long incl = warp_incl_scan(rt, lane);
    if (lane == 31) part64[warp] = incl;
    __syncthreads();
    unsigned long long before = 0;
    for (int w = 0; w < warp; w++) before += part64[w];
    run = before + incl - rt + offs[(long long)tid * G + blockIdx.x];
  }
  const long long lo = (long long)blockIdx.x * chunk, hi = min(N, lo + chunk);
  __shared__ long long cg_lo, cg_hi;  // a batch's first pass: the graphs of this chunk's edges
  if constexpr (kSrc == kArcs) chunk_graphs(es, lo / 2, hi > lo ? hi / 2 : lo / 2, &cg_lo, &cg_hi);
  if constexpr (kSrc == kCanonB) chunk_graphs(es, lo, max(lo, hi), &cg_lo, &cg_hi);
  for (long long ts = lo; ts < hi; ts += kSortTile) {
    const int tn = (int)min((long long)kSortTile, hi - ts);
    unsigned long long k[kSortKeys];
    unsigned rk[kSortKeys / 2];  // ranks below 4,096: two per word
    // key it of this thread is key j_of(it) of the tile, a row of 32 keys per
    // warp and it (kArcs: arc it & 1 of the tile's edge el_of(it))
    auto j_of = [&](int it) { return warp * kRow + it * 32 + lane; };
    auto el_of = [&](int it) { return warp * (kRow / 2) + (it >> 1) * 32 + lane; };
    unsigned dropped = 0;  // kKeysDrop: bit it set for a dropped key
    auto valid = [&](int it) {
      return kSrc == kArcs ? el_of(it) < tn / 2 : (j_of(it) < tn && !((dropped >> it) & 1u));
    };
    // every load of the tile before any use
    if constexpr (kSrc == kCanon || kSrc == kCanonB) {
      int x[kSortKeys], y[kSortKeys];
#pragma unroll
      for (int it = 0; it < kSortKeys; it++) {
        x[it] = valid(it) ? __ldcs(es.src + ts + j_of(it)) : 0;
        y[it] = valid(it) ? __ldcs(es.dst + ts + j_of(it)) : 0;
      }
      if (kSrc == kCanonB && ts == lo) __syncthreads();  // cg_lo, cg_hi
#pragma unroll
      for (int it = 0; it < kSortKeys; it++)
        k[it] = valid(it) ? edge_canon<kSrc == kCanonB>(es, ts + j_of(it), x[it], y[it], kSrc == kCanonB ? cg_lo : 0,
                                                        kSrc == kCanonB ? cg_hi : 0)
                          : 0;
    } else if constexpr (kSrc == kArcs) {
      int x[kSortKeys / 2], y[kSortKeys / 2];
#pragma unroll
      for (int it = 0; it < kSortKeys; it += 2) {
        x[it / 2] = valid(it) ? __ldcs(es.src + ts / 2 + el_of(it)) : 0;
        y[it / 2] = valid(it) ? __ldcs(es.dst + ts / 2 + el_of(it)) : 0;
      }
      if (ts == lo) __syncthreads();  // cg_lo, cg_hi
#pragma unroll
      for (int it = 0; it < kSortKeys; it += 2) {
        k[it] = k[it + 1] = 0;
        if (valid(it)) edge_keys(es, ts / 2 + el_of(it), x[it / 2], y[it / 2], k[it], k[it + 1], cg_lo, cg_hi);
      }
    } else {
#pragma unroll
      for (int it = 0; it < kSortKeys; it++) k[it] = j_of(it) < tn ? __ldcs(in + ts + j_of(it)) : kSentinel;
      if constexpr (kSrc == kKeysDrop) {
        const long long first = ts + warp * kRow;
        unsigned long long last = lane == 0 && first > 0 && first < N ? __ldcg(in + first - 1) : kSentinel;
#pragma unroll
        for (int it = 0; it < kSortKeys; it++) {
          const unsigned long long up = __shfl_up_sync(kFull, k[it], 1);
          const unsigned long long p = lane > 0 ? up : last;
          if (k[it] == kSentinel || k[it] == p) dropped |= 1u << it;
          last = __shfl_sync(kFull, k[it], 31);
        }
      }
    }
    // the next tile's lines start their way from DRAM (one 16-key line per thread)
    static_assert(kSortTile / 16 == kCsrBlock, "one line per thread");
    if ((kSrc == kKeys || kSrc == kKeysDrop) && ts + kSortTile + tid * 16 < hi)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(in + ts + kSortTile + tid * 16));
    __syncthreads();  // the last tile's keys are written out: the counters may take their place
    for (int i = tid; i < kW * 256 / 2; i += kCsrBlock) reinterpret_cast<uint4*>(sm.cnt)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    // A key's rank among its warp's keys of the same digit, in key order (rows
    // in order, lanes in order within a row). The lanes of a digit find each
    // other by or-ing their bits into its counter and reading it back (a method
    // of public GPU radix sorts, CUB's among them): about 11 cycles of the SM
    // per row of 32 random digits, where match.any takes 40 and eight ballots 16
    // (one CTA of 256 threads x 5 per SM, measured). The first pass of a build
    // need not be stable: a counter's old value is rank enough.
#pragma unroll
    for (int it = 0; it < kSortKeys; it++) {
      const bool v = valid(it);
      uint2* c = &sm.cnt[warp][digit_of(k[it], shift, dmask)];
      unsigned r = 0;
      if constexpr (kSrc == kCanon || kSrc == kCanonB || kSrc == kArcs) {
        if (v) r = atomicAdd(&c->y, 1u);
      } else {
        if (v) atomicOr(&c->x, 1u << lane);
        __syncwarp();
        const uint2 mc = *c;
        __syncwarp();
        r = mc.y + __popc(mc.x & lt);
        if (v && (mc.x & lt) == 0) *c = make_uint2(0u, mc.y + __popc(mc.x));
        __syncwarp();
      }
      if (it & 1) rk[it >> 1] |= r << 16;
      else rk[it >> 1] = r;
    }
    __syncthreads();
    // per digit (thread d): tile count, exclusive offsets over digits, then
    // over warps
    unsigned tc = 0;
#pragma unroll
    for (int w = 0; w < kW; w++) tc += sm.cnt[w][tid].y;
    const unsigned incl = warp_incl_scan(tc, lane);
    if (lane == 31) part[warp] = incl;
    __syncthreads();
    const unsigned p8 = lane < kW ? part[lane] : 0;
    const unsigned pi = warp_incl_scan(p8, lane);
    const unsigned lo_d = __shfl_sync(kFull, pi - p8, warp) + incl - tc;
    const int tk = (int)__shfl_sync(kFull, pi, kW - 1);  // keys of the tile that are written
    unsigned acc = lo_d;
#pragma unroll
    for (int w = 0; w < kW; w++) {
      wofs[w][tid] = acc;
      acc += sm.cnt[w][tid].y;
    }
    dstb[tid] = (Pos)(run - lo_d);  // modulo 2^64 (2^32): adding a tile offset of digit tid lands at or after run
    run += tc;
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kSortKeys; it++)
      if (valid(it))
        sm.buf[wofs[warp][digit_of(k[it], shift, dmask)] + ((rk[it >> 1] >> (16 * (it & 1))) & 0xffffu)] = k[it];
    __syncthreads();
#pragma unroll 4
    for (int j = tid; j < tk; j += kCsrBlock) {
      const unsigned long long key = sm.buf[j];
      out[(unsigned long long)(Pos)(dstb[digit_of(key, shift, dmask)] + (Pos)j)] = key;
    }
  }
}

// The unique-key passes: a warp walks its own contiguous chunk of keys,
// kURows rows of 32 at a time, all loaded before any is compared; a key's
// neighbours come from the next lanes and rows. Nothing is shared between
// warps, so there is no barrier (a CTA-wide tile needed three per 1,024 keys:
// 278 M keys were counted in 0.55 ms and emitted in 1.82, now 0.40 and 1.16).
constexpr int kURows = 8;
constexpr int kUTile = kURows * 32;

struct WarpKeys {
  unsigned long long x[kURows];
  unsigned long long prev, next;  // the keys before and after the tile (kSentinel: none)
  // keys [ts, ts + kUTile) of k[0, hi), hi <= N; prev holds the key before ts
  __device__ __forceinline__ void load(const unsigned long long* k, long long ts, long long hi, long long N, int lane) {
#pragma unroll
    for (int q = 0; q < kURows; q++) {
      const long long i = ts + q * 32 + lane;
      x[q] = i < hi ? __ldcs(k + i) : kSentinel;
    }
    next = ts + kUTile < N ? k[ts + kUTile] : kSentinel;
  }
  __device__ __forceinline__ unsigned long long pred(int q, int lane) const {
    const unsigned long long up = __shfl_up_sync(kFull, x[q], 1);
    const unsigned long long last = q > 0 ? __shfl_sync(kFull, x[q > 0 ? q - 1 : 0], 31) : prev;
    return lane > 0 ? up : last;
  }
  __device__ __forceinline__ unsigned long long succ(int q, int lane) const {
    const unsigned long long dn = __shfl_down_sync(kFull, x[q], 1);
    const unsigned long long first = q < kURows - 1 ? __shfl_sync(kFull, x[q < kURows - 1 ? q + 1 : q], 0) : next;
    return lane < 31 ? dn : first;
  }
  __device__ __forceinline__ void step() { prev = __shfl_sync(kFull, x[kURows - 1], 31); }
};

// A batch's edge route: the first vertex of the graph that holds vertex v, for
// the ids that leave as graph-local ones. A warp's keys run through the graphs
// in order, so the last graph found serves most of them.
struct GraphBase {
  const long long* gv;
  long long G, from, to;  // the graph at hand: vertices [from, to)
  __device__ __forceinline__ GraphBase(const long long* gv_, long long G_) : gv(gv_), G(G_), from(0), to(0) {}
  __device__ __forceinline__ long long of(long long v) {
    if (v < from || v >= to) {
      long long lo = 0, hi = G;  // the last graph with gv[g] <= v
      while (hi - lo > 1) {
        const long long mid = (lo + hi) >> 1;
        if (gv[mid] <= v) lo = mid;
        else hi = mid;
      }
      from = gv[lo];
      to = gv[lo + 1];
    }
    return from;
  }
};

// Unique keys of each warp's chunk (a key differing from its predecessor).
__global__ void __launch_bounds__(kCsrBlock) csr_count_unique(const unsigned long long* k, long long N,
                                                              long long chunk, unsigned* cnt) {
  wait_predecessor();
  const int lane = threadIdx.x & 31;
  const long long w = (long long)blockIdx.x * (kCsrBlock / 32) + (threadIdx.x >> 5);
  const long long lo = w * chunk, hi = min(N, lo + chunk);
  unsigned c = 0;
  WarpKeys t;
  t.prev = lo > 0 && lo < hi ? k[lo - 1] : kSentinel;
  for (long long ts = lo; ts < hi; ts += kUTile) {
    t.load(k, ts, hi, N, lane);
#pragma unroll
    for (int q = 0; q < kURows; q++) {
      const unsigned long long p = t.pred(q, lane);
      c += t.x[q] != kSentinel && t.x[q] != p ? 1 : 0;
    }
    t.step();
  }
  c = warp_sum(c);
  if (lane == 0) cnt[w] = c;
}

// Ordered emission of the unique keys. A unique key's position ("before":
// unique keys ahead of it) is the warp's base, plus the unique keys of earlier
// rows and lower lanes (ballots). A key's group is its high field (the source,
// or the smaller endpoint).
//   kEmitAll: adj[pos] = low B bits; the first arc of each source fixes
//     offsets[] for that source and every source without arcs just below it;
//     the last arc fills the offsets of the sources above it.
//   kEmitUpper (sequence A): vertex u's upper neighbours go after its lower
//     ones: adj[pos + starts[u + 1]] = larger endpoint, and offsets[x] = A's
//     unique keys with smaller endpoint below x (csr_finish_offsets adds
//     starts[x]); m = twice A's unique keys. gv: a batch's ids leave graph-local.
enum EmitMode : int { kEmitAll = 0, kEmitUpper = 2 };
template <int kMode>
__global__ void __launch_bounds__(kCsrBlock) csr_emit(const unsigned long long* k, long long N, long long chunk, int B,
                                                      long long n, const unsigned long long* base, int* adj,
                                                      long long* off, long long* m_out, const unsigned long long* starts,
                                                      long long* tail, const long long* __restrict__ gv, long long G) {
  wait_predecessor();
  const int lane = threadIdx.x & 31;
  GraphBase gb(gv, G);
  const long long w = (long long)blockIdx.x * (kCsrBlock / 32) + (threadIdx.x >> 5);
  const unsigned long long mask = (1ull << B) - 1;
  const unsigned lt = lanemask_lt();
  const long long lo = w * chunk, hi = min(N, lo + chunk);
  if (lo >= hi) return;
  unsigned long long running = base[w];
  WarpKeys t;
  t.prev = lo > 0 ? k[lo - 1] : kSentinel;
  for (long long ts = lo; ts < hi; ts += kUTile) {
    t.load(k, ts, hi, N, lane);
    // the lookups of each key (kEmitUpper: the lower neighbours of u come
    // first), all issued before any store
    unsigned long long look[kURows];
#pragma unroll
    for (int q = 0; q < kURows; q++)
      look[q] = kMode == kEmitUpper && t.x[q] != kSentinel ? starts[(long long)(t.x[q] >> B) + 1] : 0;
#pragma unroll
    for (int q = 0; q < kURows; q++) {
      const unsigned long long x = t.x[q], p = t.pred(q, lane), sk = t.succ(q, lane);
      const bool u = x != kSentinel && x != p;
      const unsigned bal = __ballot_sync(kFull, u);
      const unsigned long long before = running + __popc(bal & lt);
      running += __popc(bal);
      const long long s = (long long)(x >> B);  // the key's group
      if (u) {
        long long id = (long long)(x & mask);
        if (kMode == kEmitUpper && gv) id -= gb.of(s);
        adj[before + look[q]] = (int)id;
        const long long ps = p == kSentinel ? -1 : (long long)(p >> B);
        for (long long v = ps + 1; v <= s; v++) off[v] = (long long)before;
      }
      // the last valid key (unique or a repeat) closes the groups above its own
      if (x != kSentinel && sk == kSentinel) {
        const long long m_val = (long long)before + (u ? 1 : 0);
        if constexpr (kMode == kEmitAll) {
          for (long long v = s + 1; v <= n; v++) off[v] = m_val;
          *m_out = m_val;
        } else {
          // the groups above the last one are finished by csr_finish_offsets
          tail[0] = s;
          tail[1] = m_val;
          *m_out = 2 * m_val;
        }
      }
    }
    t.step();
  }
}

// Sequence B: its E' = tail[1] keys, unique and ordered by (larger, smaller)
// endpoint, then sentinels. starts[x] = keys of B whose larger endpoint is
// below x, for x in [0, n] (cleared beforehand: the groups up to the first key's
// need no store; the last key records its group in tail[0] and E' in tail[1]).
__global__ void csr_lower_starts(const unsigned long long* Bq, long long E, int B, long long n,
                                 unsigned long long* starts, long long* tail) {
  wait_predecessor();
  constexpr int kU = 4;  // keys per thread per step, all loaded first
  const unsigned long long mask = (1ull << B) - 1;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i0 = blockIdx.x * (long long)blockDim.x + threadIdx.x; i0 < E; i0 += kU * stride) {
    unsigned long long x[kU], xp[kU], xn[kU];
#pragma unroll
    for (int u = 0; u < kU; u++) {
      const long long i = i0 + u * stride;
      x[u] = i < E ? __ldcs(Bq + i) : kSentinel;
      xp[u] = i < E && i > 0 ? Bq[i - 1] : kSentinel;
      xn[u] = i + 1 < E ? Bq[i + 1] : kSentinel;
    }
#pragma unroll
    for (int u = 0; u < kU; u++) {
      const long long i = i0 + u * stride;
      if (x[u] == kSentinel) continue;
      const long long g = (long long)(x[u] & mask);
      if (i > 0) {
        const long long gp = (long long)(xp[u] & mask);  // a key: sentinels only follow the keys
        for (long long v = gp + 1; v <= g; v++) starts[v] = (unsigned long long)i;
      }
      if (xn[u] == kSentinel) {
        tail[0] = g;
        tail[1] = i + 1;
      }
    }
  }
}

// starts[v] = E' for the groups above the last key's group s = tail[0], in parallel.
__global__ void csr_fill_starts(const long long* tail, long long n, unsigned long long* starts) {
  wait_predecessor();
  const long long s = tail[0], m_val = tail[1];
  for (long long v = s + 1 + blockIdx.x * (long long)blockDim.x + threadIdx.x; v <= n;
       v += (long long)gridDim.x * blockDim.x)
    starts[v] = (unsigned long long)m_val;
}

// The lower neighbours: B's key i (u, v) is v's (i - starts[v])-th lower
// neighbour, and v's list opens with them.
__global__ void csr_lower_emit(const unsigned long long* Bq, long long E, int B, const long long* off,
                               const unsigned long long* starts, int* adj, const long long* __restrict__ gv,
                               long long G) {
  wait_predecessor();
  GraphBase gb(gv, G);
  constexpr int kU = 4;  // keys per thread per step, all loaded first, then all their lookups
  const unsigned long long mask = (1ull << B) - 1;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i0 = blockIdx.x * (long long)blockDim.x + threadIdx.x; i0 < E; i0 += kU * stride) {
    unsigned long long x[kU], at[kU];
#pragma unroll
    for (int u = 0; u < kU; u++) {
      const long long i = i0 + u * stride;
      x[u] = i < E ? __ldcs(Bq + i) : kSentinel;
    }
#pragma unroll
    for (int u = 0; u < kU; u++) {
      const long long v = (long long)(x[u] & mask);
      at[u] = x[u] != kSentinel ? (unsigned long long)off[v] - starts[v] : 0;
    }
#pragma unroll
    for (int u = 0; u < kU; u++)
      if (x[u] != kSentinel) {
        long long id = (long long)(x[u] >> B);
        if (gv) id -= gb.of(id);
        adj[at[u] + (unsigned long long)(i0 + u * stride)] = (int)id;
      }
  }
}

// offsets[v] = (A's unique keys with smaller endpoint below v) + starts[v]:
// csr_emit<kEmitUpper> wrote the first term for v up to the last valid key's
// group tail[0]; above it the term is tail[1], A's unique keys in all.
__global__ void csr_finish_offsets(const long long* tail, long long n, long long* off,
                                   const unsigned long long* starts) {
  wait_predecessor();
  const long long s = tail[0], m_val = tail[1];
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v <= n; v += (long long)gridDim.x * blockDim.x)
    off[v] = (v > s ? m_val : off[v]) + (long long)starts[v];
}

// ------------------------------------------------------------------ host side
static int bits_for(long long n) {
  int B = 1;
  while ((1ll << B) < n) B++;
  return B;
}

CsrLayout csr_layout(long long n, long long E, int sms, long long max_graph_n, bool allow_edges) {
  CsrLayout L{};
  long long N = 2 * E;
  L.N = N;
  L.Bs = bits_for(n);
  // batched: one spare code so that no valid (local) target has all bits set
  // and a valid key can never equal the sentinel in the sorted bits
  L.B = max_graph_n > 0 ? bits_for(max_graph_n + 1) : L.Bs;
  // A single graph takes the edge route, a batch the route with fewer keys to
  // move: 2B + B digit passes over E edge keys with global ids, or one sort of
  // 2E arcs by (global source, local target). 256 graphs of 1k..200k vertices
  // (139 M edges; 9 passes over E against 6 over 2E): 14.1 ms by arcs, 12.9 ms
  // by edges.
  const int edge_passes = (2 * L.Bs + 7) / 8 + (L.Bs + 7) / 8, arc_passes = (L.Bs + L.B + 7) / 8;
  // A short batch's passes are launches, not keys: the route with fewer passes
  // (16 graphs of 1k..4k vertices: 0.249 ms by arcs, 0.265 by edges).
  L.by_edges = max_graph_n <= 0 || (allow_edges && E > (long long)sms * 3 * kSortTile && edge_passes < 2 * arc_passes);
  if (L.by_edges) L.B = L.Bs;
  // Three CTAs per SM (80 registers per thread), each sorting 4,096-key tiles:
  // 16 keys per thread share a tile's barriers and its scan of the counters.
  // Measured on 67 M random 44-bit keys (us per downsweep): 2,048-key tiles
  // ranked by match.any, five CTAs 512; ranked through shared memory: 8 keys
  // per thread, five CTAs 390, six 455 (spills); 12 keys, four CTAs 325; 14
  // keys, four 335 (spills); 16 keys, three 305; ballots in place of the
  // shared-memory masks 350.
  // (1,024-key tiles for a list of less than one 4,096-key tile per CTA: 0.332
  // against 0.318 ms for 1.0 M edges, not kept.)
  const long long keys = L.by_edges ? E : N;
  auto ctas_of = [&](long long k) {
    return std::max<long long>(1, std::min<long long>((long long)sms * 3, (k + kSortTile - 1) / kSortTile));
  };
  const long long G = ctas_of(keys);
  L.grid = (int)G;
  L.chunk = std::max<long long>(1, (keys + G * kSortTile - 1) / (G * kSortTile)) * kSortTile;
  // unique-key passes: a chunk of whole 256-key tiles per warp, eight CTAs per SM
  auto warps_of = [&](long long k) {
    return std::max<long long>(1, std::min<long long>((long long)sms * 64, (k + kUTile - 1) / kUTile));
  };
  const long long warps = warps_of(keys);
  L.ugrid = (int)((warps + kCsrBlock / 32 - 1) / (kCsrBlock / 32));
  L.uchunk = std::max<long long>(1, (keys + warps * kUTile - 1) / (warps * kUTile)) * kUTile;
  size_t off = 0;
  auto al = [](size_t x) { return (x + 255) / 256 * 256; };
  L.status = off;
  off = al(off + 256);
  // 2E keys per buffer: the arc route's sequence, or the edge route's two
  L.keys0 = off;
  off = al(off + 8 * (size_t)N);
  L.keys1 = off;
  off = al(off + 8 * (size_t)N);
  // sized for 2E keys on either route: a batch's workspace is at most a single graph's
  const size_t counts = std::max<size_t>(256 * (size_t)ctas_of(N), (size_t)warps_of(N) + kCsrBlock / 32);
  L.hist = off;
  off = al(off + 4 * counts);
  L.offs = off;
  off = al(off + 8 * counts);
  L.rowtot = off;
  off = al(off + 8 * 256);
  L.starts = off;  // the edge route: starts of the lower-neighbour lists
  off = al(off + (L.by_edges ? 8 * (size_t)(n + 1) : 8));
  L.total = off;
  return L;
}

// Launches a kernel of the chain. early: it starts while the one before it
// drains (every kernel of this file begins with wait_predecessor, and reads what
// its predecessors wrote by ordinary loads: the read-only path, __ldg or const
// __restrict__, is for data that stays as it is while the kernel is resident). A list of at
// most one tile per CTA is some thirty launches of a few microseconds, whose
// start-up that takes off the critical path: 1.0 M edges 0.310 -> 0.279 ms. A
// longer list's kernels fill the GPU, and waiting CTAs only take their room
// (67 M edges 5.04 -> 5.24 ms), so they start in turn.
template <typename... P, typename... A>
static cudaError_t after(bool early, void (*kernel)(P...), int grid, int block, cudaStream_t stream, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(block);
  c.stream = stream;
  c.attrs = &at;
  c.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&c, kernel, (P)args...);
}

cudaError_t csr_build_launch(const CsrLayout& L, char* ws, long long n, long long E, const int* src,
                             const int* dst, const long long* gv, const long long* eoff, long long ngraphs,
                             long long* off_out, int* adj_out, long long* m_out, cudaStream_t stream) {
  cudaError_t e;
  int* status = (int*)(ws + L.status);
  unsigned long long* k0 = (unsigned long long*)(ws + L.keys0);
  unsigned long long* k1 = (unsigned long long*)(ws + L.keys1);
  unsigned* hist = (unsigned*)(ws + L.hist);
  unsigned long long* offs = (unsigned long long*)(ws + L.offs);
  unsigned long long* rowtot = (unsigned long long*)(ws + L.rowtot);
  if ((e = cudaMemsetAsync(status, 0, 256, stream)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(off_out, 0, 8 * (size_t)(n + 1), stream)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(m_out, 0, 8, stream)) != cudaSuccess) return e;
  if (E == 0) return cudaSuccess;
  const int G = L.grid;
  const bool early = L.chunk == kSortTile;
  const EdgeList es{src, dst, n, L.B, gv, eoff, ngraphs, status};
  // one radix pass: upsweep, row scans, downsweep
  auto pass = [&](int src_kind, const unsigned long long* in, unsigned long long* out, long long N, long long chunk,
                  int shift, int dmask) {
#define KC_UP(S) e = after(early, rs_upsweep<S>, G, kCsrBlock, stream, in, es, N, chunk, shift, dmask, hist)
    switch (src_kind) {
      case kKeys: KC_UP(kKeys); break;
      case kArcs: KC_UP(kArcs); break;
      case kCanon: KC_UP(kCanon); break;
      case kCanonB: KC_UP(kCanonB); break;
      default: KC_UP(kKeysDrop); break;
    }
#undef KC_UP
    e = after(early, scan_u32_to_u64, 256, 1024, stream, hist, offs, G, rowtot);
    // 32-bit positions when the keys number at most 2^32
    const bool narrow = N <= (1ll << 32);
#define KC_RUN(S, P) e = after(early, rs_downsweep<S, P>, G, kCsrBlock, stream, in, es, out, N, chunk, shift, dmask, offs, rowtot)
#define KC_DOWN(S)                    \
  if (narrow) KC_RUN(S, unsigned);    \
  else KC_RUN(S, unsigned long long); \
  break
    switch (src_kind) {
      case kKeys: KC_DOWN(kKeys);
      case kArcs: KC_DOWN(kArcs);
      case kCanon: KC_DOWN(kCanon);
      case kCanonB: KC_DOWN(kCanonB);
      default: KC_DOWN(kKeysDrop);
    }
#undef KC_RUN
#undef KC_DOWN
  };
  if (L.by_edges) {
    // the edge route: A = the E edge keys sorted by (min, max); B = A stably
    // sorted by max. A ping-pongs between the first halves of the two key
    // buffers, B between their second halves
    unsigned long long *a0 = k0, *a1 = k1, *b0 = k0 + E, *b1 = k1 + E;
    const int passes_a = (2 * L.B + 7) / 8;
    for (int p = 0; p < passes_a; p++) {
      pass(p == 0 ? (gv ? kCanonB : kCanon) : kKeys, a0, a1, E, L.chunk, 8 * p, 0xff);
      std::swap(a0, a1);
    }
    const unsigned long long* A = a0;
    // B: A without sentinels and repeats, stably by the larger endpoint; the
    // first pass writes E' <= E keys over a buffer of sentinels
    if ((e = cudaMemsetAsync(b1, 0xff, 8 * (size_t)E, stream)) != cudaSuccess) return e;
    const int passes_b = (L.B + 7) / 8;
    for (int p = 0; p < passes_b; p++) {
      const int bits = std::min(8, L.B - 8 * p);
      pass(p == 0 ? kKeysDrop : kKeys, p == 0 ? A : b0, b1, E, L.chunk, 8 * p, (1 << bits) - 1);
      std::swap(b0, b1);
    }
    const unsigned long long* Bq = b0;
    unsigned long long* starts = (unsigned long long*)(ws + L.starts);
    // B's last key's group and E' (0, 0 when no key is valid: the fills then
    // write what the cleared arrays hold)
    long long* tail = (long long*)(ws + L.status + 64);
    const int fill_grid = (int)std::min<long long>((n + kCsrBlock) / kCsrBlock, 4 * (long long)G);
    const int key_grid = (int)std::min<long long>((E + 4 * kCsrBlock - 1) / (4 * kCsrBlock), 8 * (long long)G);
    if ((e = cudaMemsetAsync(starts, 0, 8 * (size_t)(n + 1), stream)) != cudaSuccess) return e;
    e = after(early, csr_lower_starts, key_grid, kCsrBlock, stream, Bq, E, L.B, n, starts, tail);
    e = after(early, csr_fill_starts, fill_grid, kCsrBlock, stream, tail, n, starts);
    e = after(early, csr_count_unique, L.ugrid, kCsrBlock, stream, A, E, L.uchunk, hist);
    e = after(early, scan_u32_to_u64, 1, 1024, stream, hist, offs, L.ugrid * (kCsrBlock / 32), nullptr);
    e = after(early, csr_emit<kEmitUpper>, L.ugrid, kCsrBlock, stream, A, E, L.uchunk, L.B, n, offs, adj_out, off_out, m_out,
                                                     starts, tail, gv, ngraphs);
    e = after(early, csr_finish_offsets, fill_grid, kCsrBlock, stream, tail, n, off_out, starts);
    e = after(early, csr_lower_emit, key_grid, kCsrBlock, stream, Bq, E, L.B, off_out, starts, adj_out, gv, ngraphs);
    return cudaGetLastError();
  }
  // the arc route: two arcs per edge, sorted by (global source, local target)
  const long long N = L.N;
  const int passes = (L.Bs + L.B + 7) / 8;
  for (int p = 0; p < passes; p++) {
    pass(p == 0 ? kArcs : kKeys, k0, k1, N, L.chunk, 8 * p, 0xff);
    std::swap(k0, k1);
  }
  e = after(early, csr_count_unique, L.ugrid, kCsrBlock, stream, k0, N, L.uchunk, hist);
  e = after(early, scan_u32_to_u64, 1, 1024, stream, hist, offs, L.ugrid * (kCsrBlock / 32), nullptr);
  e = after(early, csr_emit<kEmitAll>, L.ugrid, kCsrBlock, stream, k0, N, L.uchunk, L.B, n, offs, adj_out, off_out, m_out, nullptr,
                                                  nullptr, nullptr, 0);
  return cudaGetLastError();
}

}  // namespace kc
