// kcore_validate_csr: checks on the device that a CSR is the simple undirected
// graph the peel requires (Sec. 2: an undirected graph without self-loops or
// parallel edges; the input format of every decomposition entry point).
//
// Three launches. The first checks the offsets: monotone, off[0] = 0 and
// off[n] = m. The second, only if they are sound, is a grid-stride pass over
// the arcs, a warp taking rows of 32. Per arc: the neighbour id is in
// [0, n), differs from the source, and is larger than the previous entry of
// the same list (ascending lists, hence no repeats). Symmetry: of an edge's two
// arcs, the one that points at the endpoint of smaller degree (ties: smaller
// id) is searched for in that endpoint's list, and these arcs are counted. With
// every one of them answered by an arc the other way and exactly m / 2 of them,
// no arc is left without its reverse (lists hold no repeats). When the count is
// off, the third launch searches for the other arcs' reverses to name one. The
// first failure is recorded (check code, vertex, arc); the rest of the pass
// still runs but records nothing more.
//
// What bounds it are the scattered reads: an arc's neighbour's offsets, and the
// steps of a search. Searching half the arcs, each in the shorter list, and
// keeping several searches of a lane in flight took R-MAT scale 20 (31.4 M
// arcs) from 1.19 to 0.67 ms.
#include <cuda_runtime.h>

#include <climits>

#include "kcore_device.cuh"
#include "kcore_peel.h"
#include "kcore_search.h"

namespace kc {

namespace {

__device__ __forceinline__ void record(int* st, int code, long long v, long long arc) {
  if (atomicCAS(st, 0, code) == 0) {
    long long* p = (long long*)(st + 2);
    p[0] = v;
    p[1] = arc;
  }
}

// Pass 1: the offsets. Monotone, within [0, m], off[0] = 0 and off[n] = m.
__global__ void __launch_bounds__(256) csr_validate_offsets(long long n, long long m, const long long* off,
                                                            int* st) {
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long nthreads = (long long)gridDim.x * blockDim.x;
  for (long long v = tid; v < n; v += nthreads) {
    const long long a = off[v], b = off[v + 1];
    if (a < 0 || b < a || b > m) record(st, 1, v, a);
  }
  if (tid == 0) {
    if (off[0] != 0) record(st, 2, 0, off[0]);
    else if (off[n] != m) record(st, 2, n, off[n]);
  }
}

constexpr int kRows = 4;                // rows of 32 arcs a warp has in flight
constexpr int kWarpArcs = 32 * kRows * 4;  // arcs it takes at a time: the first one's source is searched for once

// The source of arc j: the last v in [0, n) with off[v] <= j. A 32-way search
// by the warp (every lane gets the result).
__device__ __forceinline__ long long warp_source(const long long* off, long long j, long long n, int lane) {
  long long lo = 0, hi = n;  // off[lo] <= j < off[hi]
  while (hi - lo > 1) {
    const long long step = (hi - lo + 31) >> 5;
    const long long at = lo + (lane + 1) * step;
    const int c = __popc(__ballot_sync(kFull, at < hi && off[at] <= j));
    lo += c * step;
    hi = min(hi, lo + step);
  }
  return lo;
}

// The source of this lane's arc j0 + lane, given that of arc j0 - 1 or j0
// (warp-uniform v): the lists that start after v, 32 at a time (lists may be
// empty), and per lane how many of them start at or before its arc.
__device__ __forceinline__ long long row_source(const long long* off, long long n, long long v, long long j, int lane) {
  long long mine = v;
  for (bool more = true;; v += 32) {
    const long long s = off[min(v + 1 + lane, n)];
    int L = 0;
#pragma unroll
    for (int st = 16; st > 0; st >>= 1)
      if (__shfl_sync(kFull, s, L + st - 1) <= j) L += st;
    const bool all = __shfl_sync(kFull, s, 31) <= j;  // (off[n] = m is past every arc, so this ends)
    if (more) mine = v + (all ? 32 : L);
    more = more && all;
    if (!__any_sync(kFull, more)) return mine;
  }
}

// Passes 2 and 3: the arcs, only once pass 1 found the offsets sound (the
// launch boundary orders them, so every offset read below is within [0, m]).
// kRest: the third pass, which searches for the arcs the second did not.
template <bool kRest>
__global__ void __launch_bounds__(256) csr_validate_arcs(long long n, long long m, const long long* off,
                                                         const int* adj, int* st, unsigned long long* count) {
  if (*((volatile int*)st) != 0) return;
  if (kRest && 2 * *((volatile unsigned long long*)count) == (unsigned long long)m) return;
  const long long nthreads = (long long)gridDim.x * blockDim.x;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = nthreads >> 5;
  const int lane = threadIdx.x & 31;
  int searched = 0;
  for (long long base = warp * kWarpArcs; base < m; base += nwarps * kWarpArcs) {
    const long long end = min(base + kWarpArcs, m);
    long long vr = warp_source(off, base, n, lane);  // the source of the next row's first arc, or of the one before
    int last = base > 0 ? adj[base - 1] : 0;         // the entry before the next row
    for (long long row = base; row < end; row += 32 * kRows) {
      // every read of the group before any check
      int u[kRows], v[kRows], before[kRows];
      long long o0[kRows];  // the neighbours' lists
      int len[kRows], dv[kRows];
#pragma unroll
      for (int q = 0; q < kRows; q++) u[q] = row + q * 32 + lane < end ? adj[row + q * 32 + lane] : 0;
#pragma unroll
      for (int q = 0; q < kRows; q++) {
        const long long j0 = row + q * 32, j = min(j0 + lane, end - 1);
        v[q] = -1;
        before[q] = -1;
        dv[q] = 0;
        if (j0 >= end) continue;
        const long long x = row_source(off, n, vr, j, lane);
        const long long s = off[x];
        dv[q] = (int)min(off[x + 1] - s, (long long)INT_MAX);
        const int up = __shfl_up_sync(kFull, u[q], 1);
        if (j > s) before[q] = lane > 0 ? up : last;
        last = __shfl_sync(kFull, u[q], 31);
        vr = __shfl_sync(kFull, x, 31);
        if (j0 + lane < end) v[q] = (int)x;
      }
#pragma unroll
      for (int q = 0; q < kRows; q++) {
        const bool ok = v[q] >= 0 && (unsigned)u[q] < (unsigned)n;
        o0[q] = ok ? off[u[q]] : 0;
        len[q] = ok ? (int)min(off[u[q] + 1] - o0[q], (long long)INT_MAX) : 0;
      }
      // the reverse arc: position of the source in the neighbour's list
      int lo[kRows], hi[kRows];
      unsigned left = 0;  // bit q: arc q is searched for
#pragma unroll
      for (int q = 0; q < kRows; q++) {
        lo[q] = 0;
        hi[q] = 0;
        if (v[q] < 0) continue;
        const long long j = row + q * 32 + lane;
        const int bad = (unsigned)u[q] >= (unsigned)n ? 3 : (u[q] == v[q] ? 4 : (before[q] >= u[q] ? 5 : 0));
        if (bad) {
          record(st, bad, v[q], j);
          continue;
        }
        const bool small = len[q] < dv[q] || (len[q] == dv[q] && u[q] < v[q]);
        if (small != kRest) {
          left |= 1u << q;
          hi[q] = len[q];
          searched++;
        }
      }
      // the lane's searches step together: one read of each per round
      while (left) {
        int y[kRows];
#pragma unroll
        for (int q = 0; q < kRows; q++)
          y[q] = ((left >> q) & 1u) && lo[q] < hi[q] ? adj[o0[q] + middle(lo[q], hi[q])] : 0;
#pragma unroll
        for (int q = 0; q < kRows; q++) {
          if (!((left >> q) & 1u)) continue;
          const int mid = middle(lo[q], hi[q]);
          if (lo[q] >= hi[q]) record(st, 6, v[q], row + q * 32 + lane);
          if (lo[q] >= hi[q] || y[q] == v[q]) left &= ~(1u << q);
          else if (y[q] < v[q]) lo[q] = mid + 1;
          else hi[q] = mid;
        }
      }
      __syncwarp();
    }
  }
  if (!kRest) {
    searched = warp_sum(searched);
    if (lane == 0 && searched) atomicAdd(count, (unsigned long long)searched);
  }
}

}  // namespace

cudaError_t validate_launch(long long n, long long m, const long long* off, const int* adj, int* st, int sms,
                            cudaStream_t stream) {
  unsigned long long* count = (unsigned long long*)(st + 8);
  cudaError_t e = cudaMemsetAsync(st, 0, 64, stream);
  if (e != cudaSuccess) return e;
  csr_validate_offsets<<<sms * 4, 256, 0, stream>>>(n, m, off, st);
  e = cudaGetLastError();
  if (e != cudaSuccess || m == 0) return e;
  csr_validate_arcs<false><<<sms * 8, 256, 0, stream>>>(n, m, off, adj, st, count);
  csr_validate_arcs<true><<<sms * 8, 256, 0, stream>>>(n, m, off, adj, st, count);
  return cudaGetLastError();
}

}  // namespace kc
