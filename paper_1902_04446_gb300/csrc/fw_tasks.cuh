// Phase bodies of one round of blocked Floyd-Warshall (the paper's Sec. 4.4/4.5,
// Alg. 3 and 4), as device functions shared by the per-round kernels and the
// single launch (fw_kernels.cu), the 64-wide rounds (fw_panels.cuh) and the
// batched persistent kernel (batch.cu).
//
// Round k covers vertices [p0, p1) = [k*BK, min(n, (k+1)*BK)); w = p1 - p0.
//   phase1_body   Floyd-Warshall closure of D_kk (Table 1 FloydWarshall); also
//                 writes D_kk transposed into the panel buffer colT.
//   p2_row_task   D_kJ = min(D_kJ, D_kk (x) D_kJ) for one column chunk J.
//   p2_col_task   D_Ik = min(D_Ik, D_Ik (x) D_kk) for one row chunk I; writes
//                 the updated block transposed into colT.
//   p3_task       D_IJ = min(D_IJ, D_Ik (x) D_kJ) for one output tile, rows and
//                 columns of the panel excluded (Table 1 MatProd + MatMin).
// CG = true reads everything through L2 (ld.global.cg), which is required when
// the producer of the data ran earlier in the same launch.
#pragma once
#include <type_traits>

#include "fw_device.cuh"

namespace apsp {

// Barrier policy of the phase bodies: the whole CTA (the per-round and batch
// kernels), or, in the warp-specialized Phase-3 kernel that runs next-round
// tasks on its consumer warps while the producer warp goes on, a bounded
// barrier over those warps (GroupBar in fw_kernels.cu).
struct CtaBar {
  __device__ __forceinline__ static void sync() { __syncthreads(); }
};

template <bool CG, class T>
__device__ __forceinline__ T ld_elem(const T *p) {
  if constexpr (CG) return __ldcg(p);
  else return *p;
}

// ---------------------------------------------------------------- Phase 1
// 256 threads: thread (by, bx) of a 16 x 16 grid owns the PT x PT block of rows
// by*PT + r, columns bx*PT + c (PT = BK / 16) in registers; the pivot's row and
// column pass through shared memory, double buffered.
template <class Op, int BK>
struct P1Smem {
  alignas(16) typename Op::scalar row[2][BK];
  alignas(16) typename Op::scalar col[2][BK];
};

template <class S>
__device__ __forceinline__ S bits_scalar(int w) {
  if constexpr (std::is_same<S, float>::value) return __int_as_float(w);
  else return w;
}
__device__ __forceinline__ int scalar_bits(int x) { return x; }
__device__ __forceinline__ int scalar_bits(float x) { return __float_as_int(x); }

// N (2 or 4) consecutive scalars by one shared-memory access; p is aligned to N of them.
template <int N, class S>
__device__ __forceinline__ void lds_vec(S (&x)[N], const S *p) {
  static_assert(sizeof(S) == 4 && (N == 2 || N == 4), "8- or 16-byte accesses");
  if constexpr (N == 4) {
    const int4 q = *reinterpret_cast<const int4 *>(p);
    const int w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int i = 0; i < N; ++i) x[i] = bits_scalar<S>(w[i]);
  } else {
    const int2 q = *reinterpret_cast<const int2 *>(p);
    x[0] = bits_scalar<S>(q.x);
    x[1] = bits_scalar<S>(q.y);
  }
}
template <int N, class S>
__device__ __forceinline__ void sts_vec(S *p, const S (&x)[N]) {
  if constexpr (N == 4)
    *reinterpret_cast<int4 *>(p) = make_int4(scalar_bits(x[0]), scalar_bits(x[1]), scalar_bits(x[2]), scalar_bits(x[3]));
  else
    *reinterpret_cast<int2 *>(p) = make_int2(scalar_bits(x[0]), scalar_bits(x[1]));
}

// v = min(v, a0 + b0, a1 + b1): the add-min twice, or (alt) both sums and one
// three-input minimum, which takes half the ALU instructions (integer sums on
// the FMA pipe; see tile_minplus).
template <class Op>
__device__ __forceinline__ typename Op::scalar s_update2(typename Op::scalar v, typename Op::scalar a0,
                                                         typename Op::scalar b0, typename Op::scalar a1,
                                                         typename Op::scalar b1, bool alt, uint32_t one) {
  if constexpr (Op::DTYPE == 2) return fmin3(v, a0 + b0, a1 + b1);
  else if (alt)
    return __vimin3_s32(v, (int)add_fma_pipe((uint32_t)a0, (uint32_t)b0, one),
                        (int)add_fma_pipe((uint32_t)a1, (uint32_t)b1, one));
  else return Op::s_addmin(a1, b1, Op::s_addmin(a0, b0, v));
}

// Closes the BK x BK block held block by block in v, in place: Floyd-Warshall,
// one pivot and one barrier a step.  A step reads the pivot's row and column
// (one 16-byte access each), updates the thread's block, and its owners write
// the next pivot's row and column into the other buffer.
// The closure is on every round's critical path and runs on one SM, bound by
// the ALU (PT^2 add-mins a thread, 64 cycles a pivot at width 64) and the
// latency of one shared-memory read and one barrier.  Taking several pivots a
// step saves barriers but adds work to every thread, and each was measured
// slower: cycles for 64 x 64, int32 -- one pivot 8.5 thousand, two 9.0
// (redundant pivot-column updates), four 11.7 - 12.1 (closing the corner in
// every thread), pivot rows handed from warp to warp instead of barriers 13.6.
template <class Op, int BK, class Bar>
__device__ __forceinline__ void close_block(P1Smem<Op, BK> &sm, typename Op::scalar (&v)[BK / 16][BK / 16], int tid) {
  using S = typename Op::scalar;
  constexpr int PT = BK / 16;
  static_assert(PT % 2 == 0, "the buffers alternate within a thread block");
  const int by = tid / 16, bx = tid % 16;
  auto publish = [&](int nb, int t, int buf) {  // row and column t of thread block nb
    if (by == nb) sts_vec<PT>(&sm.row[buf][bx * PT], v[t]);
    if (bx == nb) {
      S w[PT];
#pragma unroll
      for (int r = 0; r < PT; ++r) w[r] = v[r][t];
      sts_vec<PT>(&sm.col[buf][by * PT], w);
    }
  };
  publish(0, 0, 0);
  Bar::sync();
#pragma unroll 1
  for (int p = 0; p < 16; ++p) {
#pragma unroll
    for (int h = 0; h < PT; ++h) {
      S a[PT], b[PT];
      lds_vec<PT>(a, &sm.col[h & 1][by * PT]);
      lds_vec<PT>(b, &sm.row[h & 1][bx * PT]);
#pragma unroll
      for (int r = 0; r < PT; ++r)
#pragma unroll
        for (int c = 0; c < PT; ++c) v[r][c] = Op::s_addmin(a[r], b[c], v[r][c]);
      publish(h + 1 < PT ? p : p + 1, (h + 1) % PT, (h + 1) & 1);  // block 16: nobody's
      Bar::sync();
    }
  }
}

// Thread (by, bx)'s part of the BK x BK diagonal block at p0 (INF outside the
// matrix): one access per row, and no branch between them, for a block inside a
// matrix with 16-byte rows.
template <class Op, int BK, bool CG>
__device__ __forceinline__ void load_block(const typename Op::elem *__restrict__ D, Layout L, int64_t n, int64_t p0,
                                           typename Op::scalar (&v)[BK / 16][BK / 16], int tid) {
  using E = typename Op::elem;
  constexpr int PT = BK / 16;
  const int64_t r0 = p0 + (tid / 16) * PT, c0 = p0 + (tid % 16) * PT;
  const E *base = D + L.off(p0, p0);
  if constexpr (PT == 4) {
    if (p0 + BK <= n && ((reinterpret_cast<uintptr_t>(base) | (uint64_t)L.ld * sizeof(E)) & 15) == 0) {
      const E *q = base + (r0 - p0) * L.ld + (c0 - p0);
      if constexpr (Op::EPW == 1) {
        uint4 w[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) w[r] = ld16<CG>(q + r * L.ld);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) v[r][c] = Op::to_s(bits_elem<Op>(chunk_get<Op>(w[r], c)));
      } else {
        uint2 w[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) w[r] = CG ? __ldcg(reinterpret_cast<const uint2 *>(q + r * L.ld))
                                              : __ldg(reinterpret_cast<const uint2 *>(q + r * L.ld));
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          v[r][0] = Op::to_s((E)(w[r].x & 0xFFFFu));
          v[r][1] = Op::to_s((E)(w[r].x >> 16));
          v[r][2] = Op::to_s((E)(w[r].y & 0xFFFFu));
          v[r][3] = Op::to_s((E)(w[r].y >> 16));
        }
      }
      return;
    }
  }
#pragma unroll
  for (int r = 0; r < PT; ++r)
#pragma unroll
    for (int c = 0; c < PT; ++c)
      v[r][c] = Op::to_s((r0 + r < n && c0 + c < n) ? ld_elem<CG>(D + L.off(r0 + r, c0 + c)) : Op::inf_elem());
}

// PT consecutive words from PT scalars (an aligned 8- or 16-byte store).
template <class Op, int PT>
__device__ __forceinline__ void store_words(uint32_t *p, const typename Op::scalar (&x)[PT]) {
  uint32_t w[PT];
#pragma unroll
  for (int i = 0; i < PT; ++i) w[i] = Op::dup(Op::from_s(x[i]));
  if constexpr (PT == 4) *reinterpret_cast<uint4 *>(p) = make_uint4(w[0], w[1], w[2], w[3]);
  else *reinterpret_cast<uint2 *>(p) = make_uint2(w[0], w[1]);
}

template <class Op, int BK, int NT, bool CG, class Bar = CtaBar>
__device__ __forceinline__ void phase1_body(typename Op::elem *__restrict__ D, Layout L, int64_t n, int64_t p0,
                                            uint32_t *__restrict__ colT, int64_t ldT, P1Smem<Op, BK> &sm, int tid,
                                            typename Op::elem *__restrict__ rowP = nullptr) {
  using S = typename Op::scalar;
  constexpr int PT = BK / 16;
  static_assert(BK % 16 == 0 && NT == 256, "phase 1 layout");
  S v[PT][PT];
  load_block<Op, BK, CG>(D, L, n, p0, v, tid);
  close_block<Op, BK, Bar>(sm, v, tid);
  const int i0 = (tid / 16) * PT, j0 = (tid % 16) * PT;
#pragma unroll
  for (int r = 0; r < PT; ++r)
#pragma unroll
    for (int c = 0; c < PT; ++c) {
      const int64_t row = p0 + i0 + r, col = p0 + j0 + c;
      if (row < n && col < n) D[L.off(row, col)] = Op::from_s(v[r][c]);
      // symmetric mode: the panel as elements (row t = D[p0 + t][.])
      if (rowP) rowP[(i0 + r) * ldT + col] = Op::from_s(v[r][c]);
    }
#pragma unroll
  for (int c = 0; c < PT; ++c) {
    S x[PT];
#pragma unroll
    for (int r = 0; r < PT; ++r) x[r] = v[r][c];
    store_words<Op>(colT + (j0 + c) * ldT + p0 + i0, x);
  }
}

// ---------------------------------------------------------------- Phase 2
// Row panel chunk: output rows [p0, p0+BK), words [col0/EPW, col0/EPW + BNW).
// A = D_kk (from colT), B = C = the chunk itself.  Shared memory: BK*BK + BK*BNW words.
//
// Symmetric mode (sym != nullptr, undirected input): only columns >= p1 are
// updated (the upper triangle); the results also go to the symmetric panel
// (colT words, and sym->rowP elements for packed 16-bit) and, for columns
// below sym->band_end, to the lower-triangle column-panel element D[x][p0+t]
// (those lie in diagonal-band Phase-3 tiles, which are updated in full).
template <class Op>
struct SymPanel {
  typename Op::elem *rowP;  // BK x ldT elements (packed 16-bit only; nullptr otherwise)
  int64_t band_end;         // end of the Phase-3 tile column band that holds the diagonal block
};

// Per-element publication of a chunk that straddles p1 or n (out of line: rare).
template <class Op>
__device__ __noinline__ void sym_publish_slow(typename Op::elem *D, Layout L, int64_t n, int64_t p0, int64_t p1,
                                              uint32_t *colT, int64_t ldT, const SymPanel<Op> *sym, int t,
                                              int64_t x0, uint4 w4) {
  constexpr int E = 4 * Op::EPW;
  for (int e = 0; e < E; ++e) {
    const int64_t x = x0 + e;
    if (x < p1 || x >= n) continue;
    const typename Op::elem v = bits_elem<Op>(chunk_get<Op>(w4, e));
    colT[(int64_t)t * ldT + x] = Op::dup(v);
    if (sym->rowP) sym->rowP[(int64_t)t * ldT + x] = v;
    if (x < sym->band_end && p0 + t < n) D[L.off(x, p0 + t)] = v;
  }
}

// Lower-triangle band elements D[x][p0+t] of a full chunk (out of line: only
// the chunks next to the diagonal block have any).
template <class Op>
__device__ __noinline__ void sym_band_store(typename Op::elem *D, Layout L, int64_t col, int64_t band_end, int64_t x0,
                                            uint4 w4) {
  constexpr int E = 4 * Op::EPW;
  for (int e = 0; e < E; ++e)
    if (x0 + e < band_end) D[L.off(x0 + e, col)] = bits_elem<Op>(chunk_get<Op>(w4, e));
}

template <class Op, int BK, int BNW, int NT, bool CG, int TN = 8, class Bar = CtaBar>
__device__ __forceinline__ void p2_row_task(typename Op::elem *__restrict__ D, Layout L, int64_t n, int64_t p0,
                                            int64_t p1, uint32_t *__restrict__ colT, int64_t ldT, int64_t col0,
                                            bool vec, uint32_t *smem, int tid, const SymPanel<Op> *sym = nullptr) {
  using Map = TileMap<BK, BNW, TN>;
  static_assert(Map::THREADS == NT, "row tile");
  uint32_t *As = smem;
  uint32_t *Bs = smem + BK * BK;
  const int tx = tid % Map::TX, ty = tid / Map::TX;
  uint32_t acc[8][TN];
  load_As_colT<BK, BK, NT, CG>(As, colT, ldT, p0, tid);
  load_Bs_rows<Op, BNW, BK, NT, CG>(Bs, D, L, n, n, p0, col0, vec, tid);
  load_acc<Op, BK, BNW, CG, TN>(D, L, n, n, p0, col0, vec, acc, ty, tx);
  Bar::sync();
  tile_minplus<Op, BK, BNW, BK, TN>(As, Bs, acc, ty, tx);
  if (!sym) {
    store_acc<Op, BK, BNW, TN>(D, L, n, n, p0, col0, 0, 0, p0, p1, vec, acc, ty, tx);
    return;
  }
  store_acc<Op, BK, BNW, TN>(D, L, n, n, p0, col0, 0, 0, 0, p1, vec, acc, ty, tx);
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int t = Map::row(ty, r);
#pragma unroll
    for (int h = 0; h < Map::NH; ++h) {
      const int64_t x0 = col0 + (int64_t)Map::wcol(tx, h) * Op::EPW;  // first element of these 4 words
      constexpr int E = 4 * Op::EPW;
      const uint4 w4 = make_uint4(acc[r][4 * h + 0], acc[r][4 * h + 1], acc[r][4 * h + 2], acc[r][4 * h + 3]);
      if (x0 >= p1 && x0 + E <= n) {
        // the whole chunk is right of the diagonal block: 16-byte panel stores
        uint32_t *cw = colT + (int64_t)t * ldT + x0;
        if constexpr (Op::EPW == 1) {
          *reinterpret_cast<uint4 *>(cw) = w4;
        } else {
          *reinterpret_cast<uint4 *>(cw) = make_uint4(Op::dup(w4.x & 0xFFFFu), Op::dup(w4.x >> 16),
                                                      Op::dup(w4.y & 0xFFFFu), Op::dup(w4.y >> 16));
          *reinterpret_cast<uint4 *>(cw + 4) = make_uint4(Op::dup(w4.z & 0xFFFFu), Op::dup(w4.z >> 16),
                                                          Op::dup(w4.w & 0xFFFFu), Op::dup(w4.w >> 16));
          *reinterpret_cast<uint4 *>(sym->rowP + (int64_t)t * ldT + x0) = w4;
        }
        if (x0 < sym->band_end && p0 + t < n) sym_band_store<Op>(D, L, p0 + t, sym->band_end, x0, w4);
      } else if (x0 + E > p1 && x0 < n) {
        sym_publish_slow<Op>(D, L, n, p0, p1, colT, ldT, sym, t, x0, w4);
      }
    }
  }
}

// Symmetric mode: only rows < p0 are updated (the upper triangle); the
// panel_finalize pass then copies colT[t][x < p0] to the element panel and to
// the row panel's lower-triangle elements in the diagonal band.
// Transposed colT store of 4 rows of which some lie in the panel (out of line: rare).
static __device__ __noinline__ void colT_store_partial(uint32_t *dst, int64_t rb, int64_t p0, int64_t xr1, uint32_t q0,
                                                uint32_t q1, uint32_t q2, uint32_t q3) {
  const uint32_t q4[4] = {q0, q1, q2, q3};
  for (int q = 0; q < 4; ++q)
    if (rb + q < p0 || rb + q >= xr1) dst[q] = q4[q];
}

template <class Op, int BK, int BM, int NT, bool CG, int TN = 8, class Bar = CtaBar>
__device__ __forceinline__ void p2_col_task(typename Op::elem *__restrict__ D, Layout L, int64_t n, int64_t p0,
                                            int64_t p1, uint32_t *__restrict__ colT, int64_t ldT, int64_t row0,
                                            bool vec, uint32_t *smem, int tid, const SymPanel<Op> *sym = nullptr) {
  constexpr int BNW = BK / Op::EPW;
  using Map = TileMap<BM, BNW, TN>;
  static_assert(Map::THREADS == NT, "col tile");
  uint32_t *As = smem;
  uint32_t *Bs = smem + BK * BM;
  const int tx = tid % Map::TX, ty = tid / Map::TX;
  uint32_t acc[8][TN];
  load_As_transposed<Op, BM, BK, NT, CG>(As, D, L, n, n, row0, p0, vec, tid);
  load_Bs_rows<Op, BNW, BK, NT, CG>(Bs, D, L, n, n, p0, p0, vec, tid);
  load_acc<Op, BM, BNW, CG, TN>(D, L, n, n, row0, p0, vec, acc, ty, tx);
  Bar::sync();
  tile_minplus<Op, BM, BNW, BK, TN>(As, Bs, acc, ty, tx);
  // symmetric mode stores rows < p0 only
  const int64_t xr1 = sym ? INT64_MAX : p1;
  store_acc<Op, BM, BNW, TN>(D, L, n, n, row0, p0, p0, xr1, 0, 0, vec, acc, ty, tx);
  // transposed copy: colT[t][row0 + i] = word(D_Ik[i][t]) for rows outside [p0, p1)
#pragma unroll
  for (int h = 0; h < Map::NH; ++h) {
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const int ib = Map::row(ty, 4 * g);  // 4 consecutive rows ib .. ib+3
      const int64_t rb = row0 + ib;
      const bool all_out = (rb + 3 < p0) || (rb >= xr1);
#pragma unroll
      for (int cw = 0; cw < 4; ++cw) {
        const int w = Map::wcol(tx, h) + cw;
#pragma unroll
        for (int lane = 0; lane < Op::EPW; ++lane) {
          const int t = w * Op::EPW + lane;
          uint32_t q4[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint32_t word = acc[4 * g + q][4 * h + cw];
            q4[q] = (Op::EPW == 2) ? Op::dup(bits_elem<Op>(lane ? (word >> 16) : (word & 0xFFFFu))) : word;
          }
          uint32_t *dst = colT + (int64_t)t * ldT + rb;
          if (all_out) *reinterpret_cast<uint4 *>(dst) = make_uint4(q4[0], q4[1], q4[2], q4[3]);
          else colT_store_partial(dst, rb, p0, xr1, q4[0], q4[1], q4[2], q4[3]);

        }
      }
    }
  }
}

// ---------------------------------------------------------------- Phase 3 (one tile)
// Output tile rows [row0, row0+128), words [col0/EPW, +128); 256 threads;
// shared memory 2 * BK * 128 words.
// symB (nullable): symmetric mode, B rows come from this BK x ldT panel of
// elements instead of D's row panel.
template <class Op, int BK, bool CG>
__device__ __forceinline__ void p3_task(typename Op::elem *__restrict__ D, Layout L, int64_t n, int64_t p0,
                                        int64_t p1, const uint32_t *__restrict__ colT, int64_t ldT, int64_t row0,
                                        int64_t col0, bool vec, uint32_t *smem, int tid,
                                        const typename Op::elem *symB = nullptr) {
  constexpr int BM = 128, BNW = 128, NT = 256;
  using Map = TileMap<BM, BNW>;
  uint32_t *As = smem;
  uint32_t *Bs = smem + BK * BM;
  const int tx = tid % Map::TX, ty = tid / Map::TX;
  uint32_t acc[8][8];
  load_As_colT<BM, BK, NT, CG>(As, colT, ldT, row0, tid);
  if (symB)
    load_Bs_rows<Op, BNW, BK, NT, CG>(Bs, symB, ldT, BK, ldT, 0, col0, true, tid);
  else
    load_Bs_rows<Op, BNW, BK, NT, CG>(Bs, D, L, n, n, p0, col0, vec, tid);
  load_acc<Op, BM, BNW, CG>(D, L, n, n, row0, col0, vec, acc, ty, tx);
  __syncthreads();
  tile_minplus<Op, BM, BNW, BK>(As, Bs, acc, ty, tx);
  if (vec && row0 + BM <= n && col0 + BNW * Op::EPW <= n && (row0 + BM <= p0 || row0 >= p1) &&
      (col0 + BNW * Op::EPW <= p0 || col0 >= p1))
    store_acc_interior<Op, BM, BNW>(D, L, row0, col0, acc, ty, tx);
  else
    store_acc<Op, BM, BNW>(D, L, n, n, row0, col0, p0, p1, p0, p1, vec, acc, ty, tx);
}

}  // namespace apsp
