// Host-side declarations of the CSR build.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

#include <algorithm>

namespace kc {

struct CsrLayout {
  size_t status, keys0, keys1, hist, offs, rowtot, starts, total;
  long long N;      // keys = 2 * edges
  long long chunk;  // radix passes: keys per CTA (whole 4,096-key tiles)
  int grid;
  long long uchunk; // unique-key passes: keys per warp
  int ugrid;
  bool by_edges;    // the edge route (one key per edge), else the arc route
  int B;            // bits of the target (local) id in a key
  int Bs;           // bits of the source (global) id in a key
};

// max_graph_n > 0: batched build (targets are graph-local ids below max_graph_n);
// allow_edges false: the arc route, which needs 8 n bytes less
CsrLayout csr_layout(long long n, long long E, int sms, long long max_graph_n = 0, bool allow_edges = true);
cudaError_t csr_build_launch(const CsrLayout& L, char* ws, long long n, long long E, const int* src,
                             const int* dst, const long long* gv, const long long* eoff, long long G,
                             long long* off_out, int* adj_out, long long* m_out, cudaStream_t stream);

}  // namespace kc
