// Batched persistent blocked Floyd-Warshall (internal; see batch.cu).
#pragma once
#include <cstddef>
#include <cstdint>
#include <vector>

#include <cuda_runtime.h>

#include "fw_launch.h"

namespace apsp {

// Default bound on every dependency wait of the batched kernel (polls with a
// 64 ns sleep between them: on the order of a second).
constexpr int64_t kDefaultSpinLimit = int64_t(1) << 24;

struct BatchGraph {
  const int32_t *W;  // input, leading dimension ldw (W == D allowed)
  int32_t *D;        // result, leading dimension ldd
  int32_t *M;        // the matrix the rounds run on: D, or a copy with 16-byte rows
  uint32_t *colT;    // 64 x ldT panel buffer (32-bit words), then a DiagBuf
  int *in_status;    // device word the input checks are ORed into
  int64_t n, ldw, ldd, ld, ldT;  // ld: of M
  int q;             // rounds
  int chunks;        // Phase-2 tasks per round
  int tiles_x, tiles;  // Phase-3 tasks per round
  int cnt_base;      // first of this graph's 3 * q done-counters
  int pair_base;     // first of its 64 x 64 tile pairs (input and output passes)
  int vec;           // 16-byte vector access allowed (on M)
  int asym;          // device-written: 1 = W is not symmetric
  int status;        // device-written: 4 = a wait timed out
};

struct BatchSeg {  // tasks [first, first + count) = (graph, round, phase, 0 .. count-1)
  long long first;
  int graph, round, phase, count;
};

// One graph of a batch as the caller sees it.
struct BatchInput {
  const int32_t *W;
  int32_t *D;
  int64_t n, ldw, ldd;
  int *in_status;
  bool copy;  // solve in a copy with 16-byte rows when D has none
};

struct BatchPlan {
  std::vector<BatchGraph> graphs;
  std::vector<BatchSeg> segs;
  long long total = 0;
  int ncounters = 0, pairs = 0;
  // The plan of `in` (n > 0 each) on the workspace at `base`, and its size in
  // bytes; base == nullptr only sizes it.
  size_t build(const std::vector<BatchInput> &in, char *base);
};

// Panel-buffer leading dimension for a graph of n vertices (words per row; 64 rows).
inline int64_t batch_panel_ld(int64_t n) { return ((n > 0 ? n : 1) + 255) / 256 * 256; }
// Bytes of the panel buffer and the closed diagonal block (DiagBuf) behind it.
inline int64_t batch_panel_bytes(int64_t n) { return 64 * batch_panel_ld(n) * 4 + (int64_t)kDiagBufBytes; }
// Bytes of the copy with 16-byte rows of an n x n int32 matrix.
inline int64_t batch_copy_bytes(int64_t n) { return n * ((n + 3) / 4 * 4) * 4 + 256; }

// Uploads the plan into its `workspace` and launches, on s, the input pass
// (checks, copies, symmetry), the persistent kernel and the output pass.  gate (nullable): round 0 of every
// graph also waits for *gate >= 1.  err |= 4 when a wait timed out; the graph's
// status (at (*graphs_dev)[i].status after the stream syncs) says which.
cudaError_t launch_batch(BatchPlan &plan, void *workspace, cudaStream_t s, int64_t spin_limit, const int *gate,
                         int *err, BatchGraph **graphs_dev, int64_t *launches);

}  // namespace apsp
