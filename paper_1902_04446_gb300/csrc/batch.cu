// Batched persistent blocked Floyd-Warshall: many graphs of uneven n in one
// launch (the rounds are Alg. 3/4's; the paper solves one graph at a time).
//
// Every graph's rounds are cut into tasks:
//   phase 0  P1  closes the round's diagonal block into the graph's DiagBuf
//                (round 0 from the matrix, later rounds by next_diag);
//   phase 1  P2  one chunk of the panels (panel_chunk);
//   phase 2  P3  one 128 x 128 tile.
// The task list is in dependency order, step by step: every active graph's
// P2(r), then every P1(r + 1), then every P3(r), with P1(0) in the step before.  Resident CTAs
// take task ids from a device counter and wait for the task's dependencies on
// per-(graph, round, phase) counters:
//   P2(r)      <- P1(r), and P3(r - 1): the tiles hold the panels' values and
//                 read the panel buffer that P2(r) rewrites;
//   P1(r + 1)  <- P2(r): it applies round r's update to its block itself, so
//                 the closure runs beside the round's tiles;
//   P3(r)      <- P2(r).
// A task waits only on tasks with smaller ids, which running CTAs already hold,
// so the launch always progresses.  Every wait is bounded: past the limit the
// graph is marked timed out, its remaining tasks are skipped but still counted.
// Data written earlier in the same launch is read through L2 only
// (ld.global.cg); producers publish with __threadfence + atomicAdd.
//
// Before the rounds one pass over pairs of mirrored 64 x 64 blocks checks every
// input, copies it where it has to be copied, and notes whether it is
// symmetric; a symmetric graph then computes only the tiles that touch the
// upper triangle.  A graph whose D has no 16-byte rows is solved in a copy that
// has: 4-byte accesses at every tile edge and row cost more than the copy.  The
// last pass writes the lower triangles and the copies' results.
// Measured (64 undirected graphs, n log-uniform in 128 .. 1024): 2.64 ms with
// every round's closure after its tiles, 256-word panel chunks, general mode
// and element-wise access to unaligned rows; 1.14 ms in this form.
#include <algorithm>
#include <cstdint>
#include <vector>

#include <cuda_runtime.h>

#include "batch.h"
#include "fw_panels.cuh"
#include "fw_passes.cuh"
#include "fw_tasks.cuh"

namespace apsp {

namespace {

constexpr int BK = 64;
constexpr int NT = 256;
constexpr int P2_XW = 32;  // panel chunk: 64 x 32 words (64: 64 graphs of 128 - 1024 4 % faster, small batches 5 % slower)
constexpr int SMEM_BYTES = 2 * BK * 128 * 4;  // the largest task (P3)
static_assert(SMEM_BYTES >= (int)sizeof(PanelSmem<OpI32, P2_XW>) && SMEM_BYTES >= (int)sizeof(NextDiagSmem<OpI32>),
              "shared memory");

__device__ __forceinline__ int ld_volatile(const int *p) { return *reinterpret_cast<const volatile int *>(p); }

__device__ __forceinline__ DiagBuf *diag_of(const BatchGraph &g) {
  return reinterpret_cast<DiagBuf *>(g.colT + 64 * g.ldT);
}

// Each task kind is compiled as its own function so that its register
// allocation does not add to the others' under the kernel's 128-register cap.
__device__ __noinline__ void task_p1(const BatchGraph &g, int round, uint8_t *smem, int tid) {
  auto &sm = *reinterpret_cast<NextDiagSmem<OpI32> *>(smem);
  const int64_t q0 = (int64_t)round * BK;
  if (round > 0) {
    next_diag<OpI32, CtaBar>(g.M, g.ld, g.n, q0 - BK, q0, g.colT, g.ldT,
                             g.asym ? nullptr : reinterpret_cast<const int32_t *>(g.colT), g.vec, diag_of(g), sm, tid);
    return;
  }
  int v[4][4];
  load_block<OpI32, 64, true>(g.M, g.ld, g.n, 0, v, tid);
  close_block<OpI32, 64, CtaBar>(sm.p1, v, tid);
  store_diag<OpI32>(diag_of(g), v, tid);
}
__device__ __noinline__ void task_p2(const BatchGraph &g, int64_t p0, int idx, uint8_t *smem, int tid) {
  panel_chunk<OpI32, P2_XW, NT>(g.M, g.ld, g.n, p0, g.colT, g.ldT, nullptr, diag_of(g), g.vec, !g.asym, idx,
                                *reinterpret_cast<PanelSmem<OpI32, P2_XW> *>(smem), tid);
}
__device__ __noinline__ void task_p3(const BatchGraph &g, int64_t p0, int64_t p1, int idx, uint8_t *smem, int tid) {
  int ty, tx;
  if (g.asym) {
    ty = idx / g.tiles_x;
    tx = idx % g.tiles_x;
  } else {  // the tiles (ty, tx) with tx >= ty, row by row
    ty = 0;
    for (; idx >= g.tiles_x - ty; ++ty) idx -= g.tiles_x - ty;
    tx = ty + idx;
  }
  p3_task<OpI32, BK, true>(g.M, g.ld, g.n, p0, p1, g.colT, g.ldT, (int64_t)ty * 128, (int64_t)tx * 128, g.vec != 0,
                           reinterpret_cast<uint32_t *>(smem), tid,
                           g.asym ? nullptr : reinterpret_cast<const int32_t *>(g.colT));
}

// Waits (thread 0) until *dep reaches target; false when the limit ran out.
__device__ __forceinline__ bool wait_count(const int *dep, int target, long long spin_limit) {
  for (long long spins = 0; ld_volatile(dep) < target; ++spins) {
    if (spins > spin_limit) return false;
    __nanosleep(64);
  }
  return true;
}

__global__ void __launch_bounds__(NT, 2)
    fw_batch_kernel(BatchGraph *G, const BatchSeg *__restrict__ segs, int nsegs, unsigned long long *head, int *cnt,
                    long long spin_limit, const int *gate, int *err) {
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ long long s_task;
  __shared__ int s_seg, s_ok;
  const int tid = threadIdx.x;
  const long long total = segs[nsegs - 1].first + segs[nsegs - 1].count;
  for (;;) {
    if (tid == 0) {
      const long long task = (long long)atomicAdd(head, 1ull);
      s_task = task;
      if (task < total) {
        int lo = 0, hi = nsegs - 1;  // last segment with first <= task
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (segs[mid].first <= task) lo = mid;
          else hi = mid - 1;
        }
        s_seg = lo;
        const BatchSeg sg = segs[lo];
        const BatchGraph &g = G[sg.graph];
        int ok = ld_volatile(&G[sg.graph].status) == 0;
        if (ok) {
          const int *c = cnt + g.cnt_base + sg.round * 3;  // this round's counters; the previous round's lie before
          if (sg.phase == 0) {
            if (sg.round > 0) ok = wait_count(c - 3 + 1, g.chunks, spin_limit);
            else if (gate) ok = wait_count(gate, 1, spin_limit);
          } else if (sg.phase == 1) {
            ok = wait_count(c, 1, spin_limit);
            if (ok && sg.round > 0) ok = wait_count(c - 3 + 2, g.tiles, spin_limit);
          } else {
            ok = wait_count(c + 1, g.chunks, spin_limit);
          }
          if (!ok) {
            atomicOr(&G[sg.graph].status, 4);
            atomicOr(err, 4);
          }
          __threadfence();
        }
        s_ok = ok;
      }
    }
    __syncthreads();
    const long long task = s_task;
    if (task >= total) break;
    const BatchSeg sg = segs[s_seg];
    if (s_ok) {
      const BatchGraph &g = G[sg.graph];
      const int idx = (int)(task - sg.first);
      const int64_t p0 = (int64_t)sg.round * BK;
      const int64_t p1 = (p0 + BK < g.n) ? p0 + BK : g.n;
      if (sg.phase == 0) task_p1(g, sg.round, smem, tid);
      else if (sg.phase == 1) task_p2(g, p0, idx, smem, tid);
      else task_p3(g, p0, p1, idx, smem, tid);
    }
    __syncthreads();  // every thread's writes of this task are done
    if (tid == 0) {
      __threadfence();
      atomicAdd(cnt + G[sg.graph].cnt_base + sg.round * 3 + sg.phase, 1);
    }
  }
}

__device__ __forceinline__ int graph_of_pair(const BatchGraph *G, int count, int p) {
  int lo = 0, hi = count - 1;  // last graph with pair_base <= p
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (G[mid].pair_base <= p) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Checks, copies (W != M) and compares the mirrored blocks of one pair: the
// conventions of input_pairs_kernel (status |= 1 invalid, 2 range).
__global__ void __launch_bounds__(256) batch_input_kernel(BatchGraph *G, int count) {
  __shared__ int32_t tile[64][65];
  const int gi = graph_of_pair(G, count, blockIdx.x);
  const BatchGraph &g = G[gi];
  int R, C;
  pair_of((int)blockIdx.x - g.pair_base, R, C);
  const int tx = threadIdx.x % 64, ty = threadIdx.x / 64;
  int bad = 0, asym = 0;
  auto take = [&](int64_t r, int64_t c) {
    const int32_t e = g.W[r * g.ldw + c];
    if (e < 0 || (r == c && e != 0)) bad |= 1;
    if (e > OpI32::inf_elem()) bad |= 2;
    if (g.W != g.M) g.M[r * g.ld + c] = e;
    return e;
  };
#pragma unroll 4
  for (int k = ty; k < 64; k += 4) {  // block (C, R), on or above the diagonal
    const int64_t r = C * 64 + k, c = R * 64 + tx;
    if (r < g.n && c < g.n) tile[k][tx] = take(r, c);
  }
  __syncthreads();
#pragma unroll 4
  for (int k = ty; k < 64; k += 4) {  // block (R, C)
    const int64_t r = R * 64 + k, c = C * 64 + tx;
    if (r < g.n && c < g.n) asym |= (R == C ? tile[k][tx] : take(r, c)) != tile[tx][k];
  }
  if (bad) atomicOr(g.in_status, bad);
  if (__syncthreads_or(asym) && threadIdx.x == 0) atomicOr(&G[gi].asym, 1);
}

// After the input pass: the tasks that a symmetric graph has (one panel of
// chunks, the upper tiles), and every segment's first task.  One CTA.
__global__ void __launch_bounds__(1024) batch_plan_kernel(BatchGraph *G, int count, BatchSeg *segs, int nsegs) {
  __shared__ long long warp_sum[32];
  __shared__ long long carry;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < count; i += blockDim.x)
    if (!G[i].asym) {
      G[i].chunks /= 2;
      if (G[i].q > 1) G[i].tiles = G[i].tiles_x * (G[i].tiles_x + 1) / 2;
    }
  if (tid == 0) carry = 0;
  __syncthreads();
  for (int b = 0; b < nsegs; b += (int)blockDim.x) {
    const int i = b + tid;
    long long c = 0;
    if (i < nsegs) {
      const BatchGraph &g = G[segs[i].graph];
      c = segs[i].phase == 0 ? 1 : segs[i].phase == 1 ? g.chunks : g.tiles;
    }
    long long x = c;  // inclusive scan
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane >= d) x += y;
    }
    if (lane == 31) warp_sum[warp] = x;
    __syncthreads();
    if (warp == 0) {
      long long y = warp_sum[lane];
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const long long z = __shfl_up_sync(0xffffffffu, y, d);
        if (lane >= d) y += z;
      }
      warp_sum[lane] = y;
    }
    __syncthreads();
    const long long base = carry + (warp > 0 ? warp_sum[warp - 1] : 0);
    if (i < nsegs) {
      segs[i].first = base + x - c;
      segs[i].count = (int)c;
    }
    __syncthreads();
    if (tid == 0) carry += warp_sum[31];
    __syncthreads();
  }
}

// The result from M: D's lower blocks from the upper ones of a symmetric
// graph, and all of D when the graph was solved in a copy.
__global__ void __launch_bounds__(256) batch_output_kernel(const BatchGraph *G, int count) {
  __shared__ int32_t tile[64][65];
  const BatchGraph &g = G[graph_of_pair(G, count, blockIdx.x)];
  const bool copy = g.M != g.D, sym = g.asym == 0;
  if (!copy && !sym) return;
  int R, C;
  pair_of((int)blockIdx.x - g.pair_base, R, C);
  const int tx = threadIdx.x % 64, ty = threadIdx.x / 64;
#pragma unroll 4
  for (int k = ty; k < 64; k += 4) {
    const int64_t r = C * 64 + k, c = R * 64 + tx;
    if (r < g.n && c < g.n) {
      const int32_t e = g.M[r * g.ld + c];
      tile[k][tx] = e;
      if (copy && (R != C || !sym || c >= r)) g.D[r * g.ldd + c] = e;
    }
  }
  __syncthreads();
#pragma unroll 4
  for (int k = ty; k < 64; k += 4) {
    const int64_t r = R * 64 + k, c = C * 64 + tx;
    if (r >= g.n || c >= g.n) continue;
    if (sym) {
      if (c < r) g.D[r * g.ldd + c] = tile[tx][k];
    } else if (R != C) {
      g.D[r * g.ldd + c] = g.M[r * g.ld + c];
    }
  }
}

int sm_count_now() {
  int dev = 0, c = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&c, cudaDevAttrMultiProcessorCount, dev);
  return c > 0 ? c : 1;
}

size_t pad256(size_t b) { return (b + 255) / 256 * 256; }

}  // namespace

size_t BatchPlan::build(const std::vector<BatchInput> &in, char *base) {
  graphs.clear();
  segs.clear();
  ncounters = 0;
  pairs = 0;
  int maxq = 0;
  for (const BatchInput &x : in) {
    BatchGraph g{};
    g.W = x.W;
    g.D = x.D;
    g.in_status = x.in_status;
    g.n = x.n;
    g.ldw = x.ldw;
    g.ldd = x.ldd;
    const bool aligned = reinterpret_cast<uintptr_t>(x.D) % 16 == 0 && x.ldd % 4 == 0;
    g.vec = aligned || x.copy ? 1 : 0;
    g.ld = aligned || !x.copy ? x.ldd : (x.n + 3) / 4 * 4;
    g.ldT = batch_panel_ld(x.n);
    g.q = (int)((x.n + BK - 1) / BK);
    g.chunks = (int)(2 * panel_chunks<OpI32, P2_XW>(x.n));
    g.tiles_x = (int)((x.n + 127) / 128);
    g.tiles = g.q == 1 ? 0 : g.tiles_x * g.tiles_x;
    g.cnt_base = ncounters;
    g.pair_base = pairs;
    ncounters += 3 * g.q;
    pairs += g.q * (g.q + 1) / 2;
    maxq = std::max(maxq, g.q);
    graphs.push_back(g);
  }
  // Where each graph's rounds lie among the maxq steps of the list: the graph
  // with the most rounds takes all of them, the others (most rounds first) the
  // window that holds the least work so far, so that every step has tiles enough
  // to hide the largest graphs' chains of dependent tasks.
  std::vector<int> order(graphs.size()), start(graphs.size(), 0);
  for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return graphs[a].q > graphs[b].q; });
  std::vector<double> load(maxq, 0.0);
  for (int i : order) {
    const BatchGraph &g = graphs[i];
    double sum = 0.0, best = 0.0;
    for (int t = 0; t < maxq; ++t) {
      sum += load[t];
      if (t >= g.q) sum -= load[t - g.q];
      if (t + 1 == g.q || (t + 1 > g.q && sum < best)) {
        best = sum;
        start[i] = t + 1 - g.q;
      }
    }
    const double work = g.tiles + 0.25 * g.chunks;  // a chunk costs about a quarter of a tile
    for (int r = 0; r < g.q; ++r) load[start[i] + r] += work;
  }
  long long first = 0;
  auto add = [&](int t, int phase) {  // step t: round t - start (phase 0: the closure for the next round)
    for (int i : order) {
      const BatchGraph &g = graphs[i];
      const int r = t - start[i] + (phase == 0 ? 1 : 0);
      const int count = r < 0 || r >= g.q ? 0 : phase == 0 ? 1 : phase == 1 ? g.chunks : g.tiles;
      if (count == 0) continue;
      segs.push_back(BatchSeg{first, i, r, phase, count});
      first += count;
    }
  };
  add(-1, 0);
  for (int t = 0; t < maxq; ++t) {
    add(t, 1);
    add(t, 0);
    add(t, 2);
  }
  total = first;
  // workspace: graphs, segments, counters and the task counter, then per graph
  // the panel buffer with its DiagBuf and the copy
  size_t off = pad256(graphs.size() * sizeof(BatchGraph)) + pad256(segs.size() * sizeof(BatchSeg)) +
               pad256(ncounters * sizeof(int) + sizeof(unsigned long long));
  for (size_t i = 0; i < graphs.size(); ++i) {
    BatchGraph &g = graphs[i];
    g.colT = reinterpret_cast<uint32_t *>(base + off);
    off += pad256((size_t)batch_panel_bytes(g.n));
    g.M = g.D;
    if (g.ld != g.ldd || (in[i].copy && reinterpret_cast<uintptr_t>(g.D) % 16 != 0)) {
      g.M = reinterpret_cast<int32_t *>(base + off);
      off += pad256((size_t)g.n * g.ld * 4);
    }
  }
  return off;
}

cudaError_t launch_batch(BatchPlan &plan, void *workspace, cudaStream_t s, int64_t spin_limit, const int *gate,
                         int *err, BatchGraph **graphs_dev, int64_t *launches) {
  if (plan.total == 0) return cudaSuccess;
  char *w = static_cast<char *>(workspace);
  BatchGraph *G = reinterpret_cast<BatchGraph *>(w);
  w += pad256(plan.graphs.size() * sizeof(BatchGraph));
  BatchSeg *S = reinterpret_cast<BatchSeg *>(w);
  w += pad256(plan.segs.size() * sizeof(BatchSeg));
  unsigned long long *head = reinterpret_cast<unsigned long long *>(w);
  int *cnt = reinterpret_cast<int *>(head + 1);
  cudaError_t e;
  e = cudaMemcpyAsync(G, plan.graphs.data(), plan.graphs.size() * sizeof(BatchGraph), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  e = cudaMemcpyAsync(S, plan.segs.data(), plan.segs.size() * sizeof(BatchSeg), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(head, 0, sizeof(unsigned long long) + (size_t)plan.ncounters * sizeof(int), s);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(fw_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
  if (e != cudaSuccess) return e;
  const int count = (int)plan.graphs.size();
  // Graphs of one round have no tiles, and their panel chunks write the whole
  // closed block: the symmetry test changes nothing then, and without copies
  // there is nothing left to write at the end (one graph of 64 vertices 32 - 39 us
  // with all four launches, 26 with two).
  bool rounds = false, copies = false;
  for (const BatchGraph &g : plan.graphs) {
    rounds = rounds || g.q > 1;
    copies = copies || g.M != g.D;
  }
  batch_input_kernel<<<(unsigned)plan.pairs, 256, 0, s>>>(G, count);
  if (rounds) batch_plan_kernel<<<1, 1024, 0, s>>>(G, count, S, (int)plan.segs.size());
  const long long grid = std::min<long long>(2LL * sm_count_now(), plan.total);
  fw_batch_kernel<<<(unsigned)grid, NT, SMEM_BYTES, s>>>(G, S, (int)plan.segs.size(), head, cnt,
                                                         spin_limit > 0 ? spin_limit : kDefaultSpinLimit, gate, err);
  if (rounds || copies) batch_output_kernel<<<(unsigned)plan.pairs, 256, 0, s>>>(G, count);
  if (launches) *launches += 2 + (rounds ? 1 : 0) + (rounds || copies ? 1 : 0);
  if (graphs_dev) *graphs_dev = G;
  return cudaGetLastError();
}

}  // namespace apsp
