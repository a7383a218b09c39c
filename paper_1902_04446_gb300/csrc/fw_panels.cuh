// The 64-wide rounds' panels (the paper's Sec. 4.4/4.5, Alg. 3 and 4): Phase 2
// as one kernel of narrow chunks, and the closure of the next round's diagonal
// block as a task of this round's Phase 3.
//
// With one launch per phase, a round of a small or mid-size matrix was bound
// by the chain diagonal closure -> panels -> tiles: at n = 2048 38 us, of which
// the tiles' add-mins need 7.  Here a round is two launches:
//   fw_panels   relaxes every chunk of the panels with the closed diagonal
//               block (16 words wide, so that a small n still fills the GPU),
//               and publishes them: D, colT, and in symmetric mode the element
//               panel and the band elements below the diagonal;
//   Phase 3     whose first CTA, before its tiles, applies this round's update
//               to the next diagonal block and closes it (next_diag), into a
//               side buffer that the next fw_panels reads and copies into D.
// Closing into the side buffer keeps D's block to one writer: the Phase-3 tile
// that holds it.
#pragma once
#include "fw_launch.h"
#include "fw_tasks.cuh"
#include "tma.cuh"

namespace apsp {

// A closed 64 x 64 diagonal block as A-operand words, in both orders:
// t[s][i] = word(D[p0 + i][p0 + s]), n[s][i] = word(D[p0 + s][p0 + i]);
// entries outside the matrix are INF.
struct alignas(16) DiagBuf {
  uint32_t t[64][64];
  uint32_t n[64][64];
};
static_assert(sizeof(DiagBuf) == kDiagBufBytes, "placed after the 64 panel rows of a 64-wide round");

template <class Op>
__device__ __forceinline__ typename Op::elem word_elem(uint32_t w) {
  return bits_elem<Op>(Op::EPW == 2 ? (w & 0xFFFFu) : w);
}

template <class Op>
__device__ __forceinline__ void store_diag(DiagBuf *out, const typename Op::scalar (&v)[4][4], int tid) {
  const int i0 = (tid / 16) * 4, j0 = (tid % 16) * 4;
#pragma unroll
  for (int r = 0; r < 4; ++r) store_words<Op>(&out->n[i0 + r][j0], v[r]);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const typename Op::scalar x[4] = {v[0][c], v[1][c], v[2][c], v[3][c]};
    store_words<Op>(&out->t[j0 + c][i0], x);
  }
}

// Closes D's diagonal block at p0 into `out` (256 threads).
template <class Op>
__global__ void __launch_bounds__(256) fw_diag(const typename Op::elem *__restrict__ D, Layout L, int64_t n, int64_t p0,
                                               DiagBuf *__restrict__ out) {
  __shared__ P1Smem<Op, 64> sm;
  typename Op::scalar v[4][4];
  const int tid = threadIdx.x;
  pdl_trigger();
  pdl_wait();
  load_block<Op, 64, true>(D, L, n, p0, v, tid);
  close_block<Op, 64, CtaBar>(sm, v, tid);
  store_diag<Op>(out, v, tid);
}

// Closed D block copied back (a matrix of one round has no fw_panels).
template <class Op>
__global__ void diag_to_matrix(typename Op::elem *__restrict__ D, Layout L, int64_t n, int64_t p0,
                               const DiagBuf *__restrict__ diag) {
  pdl_trigger();
  pdl_wait();
  for (int idx = threadIdx.x; idx < 64 * 64; idx += blockDim.x) {
    const int64_t r = p0 + idx / 64, c = p0 + idx % 64;
    if (r < n && c < n) D[L.off(r, c)] = word_elem<Op>(__ldcg(&diag->n[idx / 64][idx % 64]));
  }
}

// Barrier of the 256 threads that run next_diag inside a larger CTA.
struct Bar256 {
  __device__ __forceinline__ static void sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
};

template <class Op>
struct NextDiagSmem {
  P1Smem<Op, 64> p1;
  alignas(16) typename Op::scalar a[64][64];  // a[t][i]: this round's column panel at the next block's rows
  alignas(16) typename Op::scalar b[64][64];  // b[t][j]: its row panel at the next block's columns
};

// The next round's diagonal block (at q0) after this round's update, closed,
// into `out`; 256 threads.  D's block may or may not hold this round's update
// yet (its Phase-3 tile runs meanwhile): the minimum is the same.
// symB: symmetric mode's panel (64 x ldT elements), else nullptr and the row
// panel is D's rows p0 ...
template <class Op, class Bar>
__device__ __noinline__ void next_diag(const typename Op::elem *__restrict__ D, Layout L, int64_t n, int64_t p0,
                                       int64_t q0, const uint32_t *__restrict__ colT, int64_t ldT,
                                       const typename Op::elem *__restrict__ symB, int vec,
                                       DiagBuf *__restrict__ out, NextDiagSmem<Op> &sm, int tid) {
  using S = typename Op::scalar;
  constexpr int E4 = 4 * Op::EPW, BIT = 64 * 64 / E4 / 256;
  S v[4][4];
  {
    // all loads first: the panels' 64 x 64 parts and this thread's part of the
    // block.  Rows and columns past the matrix read as INF.
    uint4 ta[4], tb[BIT];
    const uint32_t *pa = colT + (int64_t)(tid / 16) * ldT + q0 + (tid % 16) * 4;  // panel rows are aligned words
#pragma unroll
    for (int k = 0; k < 4; ++k) ta[k] = ld16<true>(pa + (int64_t)k * 16 * ldT);
    if ((symB || vec) && q0 + 64 <= n) {
      // no branch between the loads: with one each they are a chain of latencies
      const typename Op::elem *pb = (symB ? symB : D + L.off(p0, 0)) + q0 + (tid % (64 / E4)) * E4;
      const int64_t row = symB ? ldT : L.ld;
#pragma unroll
      for (int k = 0; k < BIT; ++k) tb[k] = ld16<true>(pb + (int64_t)((tid + k * 256) / (64 / E4)) * row);
    } else {
#pragma unroll
      for (int k = 0; k < BIT; ++k) {
        const int t = (tid + k * 256) / (64 / E4);
        const int64_t x = q0 + (tid % (64 / E4)) * E4;
        tb[k] = symB ? load_chunk<Op, true>(symB, ldT, 64, n, t, x, true)
                     : load_chunk<Op, true>(D, L, n, n, p0 + t, x, vec != 0);
      }
    }
    load_block<Op, 64, true>(D, L, n, q0, v, tid);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int t = (tid + k * 256) / 16, i = (tid % 16) * 4;
      const uint32_t w[4] = {ta[k].x, ta[k].y, ta[k].z, ta[k].w};
      S x[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) x[e] = Op::to_s(q0 + i + e < n ? word_elem<Op>(w[e]) : Op::inf_elem());
      sts_vec<4>(&sm.a[t][i], x);
    }
#pragma unroll
    for (int k = 0; k < BIT; ++k) {
      const int t = (tid + k * 256) / (64 / E4), i = (tid % (64 / E4)) * E4;
#pragma unroll
      for (int g = 0; g < E4; g += 4) {
        S x[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) x[e] = Op::to_s(bits_elem<Op>(chunk_get<Op>(tb[k], g + e)));
        sts_vec<4>(&sm.b[t][i + g], x);
      }
    }
  }
  Bar::sync();
  const int by = tid / 16, bx = tid % 16;
  const uint32_t one = kOne;
#pragma unroll 4
  for (int t = 0; t < 64; t += 2) {
    S a[2][4], b[2][4];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      lds_vec<4>(a[k], &sm.a[t + k][by * 4]);
      lds_vec<4>(b[k], &sm.b[t + k][bx * 4]);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) v[r][c] = s_update2<Op>(v[r][c], a[0][r], b[0][c], a[1][r], b[1][c], (r + c) & 1, one);
  }
  close_block<Op, 64, Bar>(sm.p1, v, tid);
  store_diag<Op>(out, v, tid);
}

// ---------------------------------------------------------------- panels
// One chunk of the panels per CTA: XW words (XE = XW * EPW elements) of
// columns x0 .. x0 + XE of the row panel, or as many rows of the column panel.
// Both are out[t][x] = min(S[t][x], min_s A[s][t] + S[s][x]) on the chunk held
// as S[t][x]: row panel S[t][x] = D[p0 + t][x] and A = diag.t, column panel
// S[t][x] = D[x][p0 + t] (loaded and stored transposed) and A = diag.n.
//   symmetric mode (chunks 0 .. nx-1): a chunk is a column chunk left of the diagonal block, a row
//     chunk right of it (only the upper triangle is kept), and its result is
//     the symmetric panel: colT words, rowP elements (packed 16-bit), and in
//     the tile band of the diagonal block both D[p0 + t][x] and D[x][p0 + t];
//   otherwise chunks 0 .. nx-1 are row chunks, nx .. 2 nx - 1 column chunks
//     (their result also goes to colT).
// The diagonal block's own chunks copy the closed block.  A chunk never
// straddles the diagonal block (XE divides 64).
constexpr int PANEL_THREADS = 128;
template <class Op, int XW>
__host__ __device__ constexpr int64_t panel_chunks(int64_t n) {  // of one panel
  return (n + XW * Op::EPW - 1) / (XW * Op::EPW);
}
template <class Op, int XW>
struct PanelSmem {
  uint32_t a[64][64];
  uint32_t s[64][XW + 4];  // the chunk's words
};

// NT threads (128 or 256), whole-CTA barriers.
template <class Op, int XW, int NT>
__device__ __forceinline__ void panel_chunk(typename Op::elem *__restrict__ D, Layout L, int64_t n, int64_t p0,
                                            uint32_t *__restrict__ colT, int64_t ldT,
                                            typename Op::elem *__restrict__ rowP, const DiagBuf *__restrict__ diag,
                                            int vec, int sym, int chunk, PanelSmem<Op, XW> &sm, int tid) {
  using E = typename Op::elem;
  constexpr int EPW = Op::EPW, XE = XW * EPW, TXN = NT / 16, CW = XW / TXN;  // CW words per thread and row
  constexpr int E4 = 4 * EPW;
  static_assert(64 % XE == 0, "a chunk never straddles the diagonal block");
  static_assert(CW % 2 == 0, "words in pairs");
  const int64_t band_start = p0 / (128 * EPW) * (128 * EPW), band_end = band_start + 128 * EPW;
  const int nx = (int)((n + XE - 1) / XE);
  if (sym && chunk >= nx) return;
  const bool second = chunk >= nx;
  const int64_t x0 = (int64_t)(chunk - (second ? nx : 0)) * XE;
  const bool on_diag = x0 >= p0 && x0 < p0 + 64;
  const bool col = sym ? x0 < p0 : second;
  const bool to_colT = sym || col;
  const bool wr_row = sym ? x0 >= band_start : !col;
  const bool wr_col = sym ? x0 < band_end : col;
  if (on_diag) {
    // all loads first: taken one at a time they made this the round's slowest
    // CTA (packed 16-bit n = 4096: 1847 us per solve, 1699 in this form)
    constexpr int IT = 64 * (XE / 4) / NT;
    const int d0 = (int)(x0 - p0);
    uint4 wn[IT], wt[IT];
#pragma unroll
    for (int k = 0; k < IT; ++k) {
      const int idx = tid + k * NT, t = idx / (XE / 4), x = idx % (XE / 4) * 4;
      wn[k] = __ldcg(reinterpret_cast<const uint4 *>(&diag->n[t][d0 + x]));
      wt[k] = __ldcg(reinterpret_cast<const uint4 *>(&diag->t[t][d0 + x]));
    }
#pragma unroll
    for (int k = 0; k < IT; ++k) {
      const int idx = tid + k * NT, t = idx / (XE / 4), x = idx % (XE / 4) * 4;
      if (to_colT) *reinterpret_cast<uint4 *>(colT + (int64_t)t * ldT + x0 + x) = wt[k];
      const uint32_t w[4] = {wn[k].x, wn[k].y, wn[k].z, wn[k].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const E v = word_elem<Op>(w[e]);
        if (!col && p0 + t < n && x0 + x + e < n) D[L.off(p0 + t, x0 + x + e)] = v;
        if (sym && EPW == 2) rowP[(int64_t)t * ldT + x0 + x + e] = v;
      }
    }
    return;
  }
  // ---- operands: the closed block, and the chunk (all loads first).  A column
  // chunk is loaded 32 bytes of one row per thread, consecutive threads in
  // consecutive rows: full sectors from memory, and the transposed element
  // stores of a warp fall into consecutive words (16 bytes a thread along the
  // rows made them conflict 8-fold).
  constexpr int AIT = 64 * 16 / NT;
  constexpr int SIT = 64 * (XW / 4) / NT;  // 16-byte pieces per thread
  constexpr int PB = SIT < 2 ? SIT : 2;    // pieces of one row that a thread takes in a row
  static_assert(SIT % PB == 0, "pieces");
  const uint32_t *A = col ? &diag->n[0][0] : &diag->t[0][0];
  // column chunk: row and first column of this thread's piece k
  auto col_piece = [&](int k, int &x, int &t) {
    const int u = tid + (k / PB) * NT;
    x = u % XE;
    t = (u / XE * PB + k % PB) * E4;
  };
  uint4 va[AIT], vs[SIT];
#pragma unroll
  for (int k = 0; k < AIT; ++k) va[k] = __ldcg(reinterpret_cast<const uint4 *>(A) + tid + k * NT);
  const bool whole = vec && x0 + XE <= n && p0 + 64 <= n;  // no branch between the loads then
#pragma unroll
  for (int k = 0; k < SIT; ++k) {
    if (!col) {
      const int idx = tid + k * NT;
      const int64_t r = p0 + idx / (XW / 4), c = x0 + (idx % (XW / 4)) * E4;
      if (whole) vs[k] = ld16<true>(D + L.off(r, c));
      else vs[k] = load_chunk<Op, true>(D, L, n, n, r, c, vec);
    } else {
      int x, t;
      col_piece(k, x, t);
      if (whole) vs[k] = ld16<true>(D + L.off(x0 + x, p0 + t));
      else vs[k] = load_chunk<Op, true>(D, L, n, n, x0 + x, p0 + t, vec);
    }
  }
#pragma unroll
  for (int k = 0; k < AIT; ++k) *(reinterpret_cast<uint4 *>(sm.a) + tid + k * NT) = va[k];
  E *se = reinterpret_cast<E *>(sm.s);           // the chunk as elements
  constexpr int SE = (XW + 4) * EPW;             // elements per row of it
#pragma unroll
  for (int k = 0; k < SIT; ++k) {
    if (!col) {
      const int idx = tid + k * NT;
      *reinterpret_cast<uint4 *>(&sm.s[idx / (XW / 4)][(idx % (XW / 4)) * 4]) = vs[k];
    } else {
      int x, t;
      col_piece(k, x, t);
#pragma unroll
      for (int e = 0; e < E4; ++e) se[(t + e) * SE + x] = bits_elem<Op>(chunk_get<Op>(vs[k], e));
    }
  }
  __syncthreads();
  // ---- out = min(S, A (x) S): 4 rows x CW words per thread
  const int ty = tid / TXN, tx = tid % TXN;
  uint32_t acc[4][CW];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < CW; ++c) acc[r][c] = sm.s[4 * ty + r][tx * CW + c];
  const uint32_t one = kOne;
#pragma unroll 4
  for (int k = 0; k < 64; k += 2) {
    uint32_t a[2][4], b[2][CW];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint4 av = *reinterpret_cast<const uint4 *>(&sm.a[k + h][4 * ty]);
      a[h][0] = av.x; a[h][1] = av.y; a[h][2] = av.z; a[h][3] = av.w;
#pragma unroll
      for (int c = 0; c < CW; c += 2) {
        const uint2 bv = *reinterpret_cast<const uint2 *>(&sm.s[k + h][tx * CW + c]);
        b[h][c] = bv.x;
        b[h][c + 1] = bv.y;
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < CW; ++c) acc[r][c] = word_update2<Op>(acc[r][c], a[0][r], b[0][c], a[1][r], b[1][c], (r + c) & 1, one);
  }
  // ---- results
  const int64_t xw = x0 + (int64_t)tx * CW * EPW;  // first element of this thread's words
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int t = 4 * ty + r;
#pragma unroll
    for (int c = 0; c < CW; c += 2) {
      const int64_t x = xw + c * EPW;
      const uint2 w2 = make_uint2(acc[r][c], acc[r][c + 1]);
      if (to_colT) {
        uint32_t *cw = colT + (int64_t)t * ldT + x;
        if constexpr (EPW == 1) *reinterpret_cast<uint2 *>(cw) = w2;
        else
          *reinterpret_cast<uint4 *>(cw) = make_uint4(Op::dup(w2.x & 0xFFFFu), Op::dup(w2.x >> 16),
                                                      Op::dup(w2.y & 0xFFFFu), Op::dup(w2.y >> 16));
      }
      if (sym && EPW == 2) *reinterpret_cast<uint2 *>(rowP + (int64_t)t * ldT + x) = w2;
      if (wr_row && p0 + t < n) {
        E *dp = D + L.off(p0 + t, x);
        if (vec && x + 2 * EPW <= n) {
          *reinterpret_cast<uint2 *>(dp) = w2;
        } else {
#pragma unroll
          for (int e = 0; e < 2 * EPW; ++e) {
            const uint32_t w = e < EPW ? w2.x : w2.y;
            if (x + e < n) dp[e] = bits_elem<Op>(EPW == 2 ? ((e & 1) ? (w >> 16) : (w & 0xFFFFu)) : w);
          }
        }
      }
    }
  }
  if (!wr_col) return;
  // transposed through shared memory: D[x][p0 + t], as the column chunk was loaded
  __syncthreads();
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < CW; ++c) sm.s[4 * ty + r][tx * CW + c] = acc[r][c];
  __syncthreads();
#pragma unroll
  for (int k = 0; k < SIT; ++k) {
    int x, t;
    col_piece(k, x, t);
    if (x0 + x >= n) continue;
    uint4 v = make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int e = 0; e < E4; ++e) chunk_set<Op>(v, e, elem_bits<Op>(se[(t + e) * SE + x]));
    if (vec && p0 + t + E4 <= n) *reinterpret_cast<uint4 *>(D + L.off(x0 + x, p0 + t)) = v;
    else store_chunk<Op>(D, L, x0 + x, p0 + t, v, col_mask<Op>(p0 + t, n, 0, 0), vec);
  }
}

template <class Op, int XW>
__global__ void __launch_bounds__(PANEL_THREADS)
    fw_panels(typename Op::elem *__restrict__ D, Layout L, int64_t n, int64_t p0, uint32_t *__restrict__ colT,
              int64_t ldT, typename Op::elem *__restrict__ rowP, const DiagBuf *__restrict__ diag, int vec, int sym,
              const int *__restrict__ sym_flag) {
  __shared__ __align__(16) PanelSmem<Op, XW> sm;
  pdl_trigger();
  pdl_wait();
  if (sym_flag) sym = __ldcg(sym_flag) == 0;
  panel_chunk<Op, XW, PANEL_THREADS>(D, L, n, p0, colT, ldT, rowP, diag, vec, sym, blockIdx.x, sm, threadIdx.x);
}

}  // namespace apsp
