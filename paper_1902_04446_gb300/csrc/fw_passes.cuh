// Passes over whole matrices: input (checks, copy, symmetry), output (mirror,
// copy), packing and filling.  All are bound by memory bandwidth, so each
// element is read and written once, 16 bytes a thread where the rows allow it
// and several independent accesses in flight.  Measured, us, one element a thread
// and trip / now: fill of a 12000 x 12000 packed 16-bit matrix 426 / 40, mirror
// of it 190 / under 60, packing a 4096 x 4096 matrix 61 / 15, unpacking 61 / 20.
#pragma once
#include "fw_device.cuh"

namespace apsp {

// A 64 x 64 block on 256 threads: E elements (16 bytes) per access, CPR
// accesses per row, P accesses per thread.
template <class Op>
struct PairTile {
  static constexpr int E = 4 * Op::EPW, CPR = 64 / E, RPP = 256 / CPR, P = 64 / RPP;
  static constexpr int PITCH = 64 + Op::EPW;  // elements per row in shared memory: an odd number of words
};

// Pair p of mirrored 64 x 64 blocks (R, C), R >= C, counted row by row.
__device__ __forceinline__ void pair_of(long long p, int &R, int &C) {
  R = (int)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);
  while ((long long)R * (R + 1) / 2 > p) --R;
  while ((long long)(R + 1) * (R + 2) / 2 <= p) ++R;
  C = (int)(p - (long long)R * (R + 1) / 2);
}
inline long long block_pairs(int64_t n) {
  const long long q = (n + 63) / 64;
  return q * (q + 1) / 2;
}

// The input checks on one access of E elements at (r, c0): diagonal 0, weights
// >= 0, finite weights < INF; bad |= 1 (invalid) or 2 (range).  fp32: -0.0
// becomes +0.0, so that every stored distance is a non-negative float whose bit
// pattern orders like the value under a signed int32 compare -- the Phase-3
// tiles leave by an int32 TMA min-reduction on those bits.  Returns whether v
// was changed.
template <class Op>
__device__ __forceinline__ bool check_input(uint4 &v, int64_t r, int64_t c0, int64_t n, int &bad) {
  constexpr int E = 4 * Op::EPW;
  bool changed = false;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    if (c0 + e >= n) continue;
    const typename Op::elem x = bits_elem<Op>(chunk_get<Op>(v, e));
    if constexpr (Op::DTYPE == 2) {
      if (!(x >= 0.0f)) bad |= 1;  // negative or NaN
      if (__float_as_uint(x) == 0x80000000u) {
        chunk_set<Op>(v, e, 0u);
        changed = true;
      }
    } else {
      if (Op::DTYPE == 0 && x < 0) bad |= 1;
      if (x > Op::inf_elem()) bad |= 2;
    }
    if (r == c0 + e && x != (typename Op::elem)0) bad |= 1;
  }
  return changed;
}

// The elements c0 .. c0 + E-1 of a row that lie in [0, n).
template <class Op>
__device__ __forceinline__ uint32_t row_mask(int64_t c0, int64_t n) {
  constexpr int E = 4 * Op::EPW;
  const int64_t left = n - c0;
  return left >= E ? (1u << E) - 1u : left <= 0 ? 0u : (1u << (int)left) - 1u;
}

// One pair of mirrored blocks of the input W: checks (status nullable: none),
// copies to M (copy; otherwise only fp32 -0.0 is written back) and compares the
// blocks (asym nullable; |= 1 when they differ, bitwise).
template <class Op>
__global__ void __launch_bounds__(256) input_pairs_kernel(const typename Op::elem *W, int64_t ldw, int vw,
                                                          typename Op::elem *M, int64_t ldm, int vm, int copy,
                                                          int64_t n, int *status, int *asym) {
  using T = PairTile<Op>;
  __shared__ typename Op::elem tile[64][T::PITCH];
  int R, C;
  pair_of(blockIdx.x, R, C);
  const int cc = (int)threadIdx.x % T::CPR * T::E, rr = (int)threadIdx.x / T::CPR;
  uint4 a[T::P], b[T::P];
#pragma unroll
  for (int k = 0; k < T::P; ++k) {
    a[k] = load_chunk<Op>(W, ldw, n, n, (int64_t)C * 64 + rr + k * T::RPP, (int64_t)R * 64 + cc, vw != 0);
    if (R != C) b[k] = load_chunk<Op>(W, ldw, n, n, (int64_t)R * 64 + rr + k * T::RPP, (int64_t)C * 64 + cc, vw != 0);
  }
  int bad = 0, diff = 0;
  auto take = [&](uint4 &v, int64_t r, int64_t c0) {
    if (r >= n || c0 >= n) return;
    const bool changed = status && check_input<Op>(v, r, c0, n, bad);
    if (copy || changed) store_chunk<Op>(M, ldm, r, c0, v, row_mask<Op>(c0, n), vm != 0);
  };
#pragma unroll
  for (int k = 0; k < T::P; ++k) {
    take(a[k], (int64_t)C * 64 + rr + k * T::RPP, (int64_t)R * 64 + cc);
    if (R != C) take(b[k], (int64_t)R * 64 + rr + k * T::RPP, (int64_t)C * 64 + cc);
  }
  if (asym) {
#pragma unroll
    for (int k = 0; k < T::P; ++k)
#pragma unroll
      for (int e = 0; e < T::E; ++e) tile[rr + k * T::RPP][cc + e] = bits_elem<Op>(chunk_get<Op>(a[k], e));
    __syncthreads();
#pragma unroll
    for (int k = 0; k < T::P; ++k) {
      const uint4 v = R == C ? a[k] : b[k];
#pragma unroll
      for (int e = 0; e < T::E; ++e)
        diff |= chunk_get<Op>(v, e) != elem_bits<Op>(tile[cc + e][rr + k * T::RPP]);
    }
    if (__syncthreads_or(diff) && threadIdx.x == 0) atomicOr(asym, 1);
  }
  if (bad) atomicOr(status, bad);
}

// One pair of mirrored blocks of the result M (a Layout): into D when D != M,
// and in symmetric mode (sym, or *sym_flag == 0 when given) the elements below
// the diagonal from those above it.
template <class Op>
__global__ void __launch_bounds__(256) output_pairs_kernel(const typename Op::elem *M, Layout LM, int vm,
                                                           typename Op::elem *D, int64_t ldd, int vd, int copy,
                                                           int64_t n, int sym, const int *sym_flag) {
  using T = PairTile<Op>;
  __shared__ typename Op::elem tile[64][T::PITCH];
  if (sym_flag) sym = *sym_flag == 0;
  if (!copy && !sym) return;
  int R, C;
  pair_of(blockIdx.x, R, C);
  const int cc = (int)threadIdx.x % T::CPR * T::E, rr = (int)threadIdx.x / T::CPR;
  const int64_t ru = (int64_t)C * 64 + rr, cu = (int64_t)R * 64 + cc;  // block (C, R)
  const int64_t rl = (int64_t)R * 64 + rr, cl = (int64_t)C * 64 + cc;  // block (R, C)
  uint4 a[T::P];
#pragma unroll
  for (int k = 0; k < T::P; ++k) a[k] = load_chunk<Op>(M, LM, n, n, ru + k * T::RPP, cu, vm != 0);
  if (copy && (R != C || !sym)) {
#pragma unroll
    for (int k = 0; k < T::P; ++k)
      if (ru + k * T::RPP < n) store_chunk<Op>(D, ldd, ru + k * T::RPP, cu, a[k], row_mask<Op>(cu, n), vd != 0);
  }
  if (!sym) {
    if (R == C) return;
#pragma unroll
    for (int k = 0; k < T::P; ++k) a[k] = load_chunk<Op>(M, LM, n, n, rl + k * T::RPP, cl, vm != 0);
#pragma unroll
    for (int k = 0; k < T::P; ++k)
      if (rl + k * T::RPP < n) store_chunk<Op>(D, ldd, rl + k * T::RPP, cl, a[k], row_mask<Op>(cl, n), vd != 0);
    return;
  }
#pragma unroll
  for (int k = 0; k < T::P; ++k)
#pragma unroll
    for (int e = 0; e < T::E; ++e) tile[rr + k * T::RPP][cc + e] = bits_elem<Op>(chunk_get<Op>(a[k], e));
  __syncthreads();
#pragma unroll
  for (int k = 0; k < T::P; ++k) {
    const int row = rr + k * T::RPP;
    if (rl + k * T::RPP >= n) continue;
    uint4 v = a[k];  // the diagonal block keeps its upper elements
#pragma unroll
    for (int e = 0; e < T::E; ++e)
      if (R != C || cc + e < row) chunk_set<Op>(v, e, elem_bits<Op>(tile[cc + e][row]));
    store_chunk<Op>(D, ldd, rl + k * T::RPP, cl, v, row_mask<Op>(cl, n), vd != 0);
  }
}

// dst <- src, rows x cols, 16 bytes a thread and row.
template <class Op>
__global__ void __launch_bounds__(256) copy_rect_kernel(const typename Op::elem *__restrict__ s, int64_t lds, int vs,
                                                        typename Op::elem *__restrict__ d, int64_t ldd, int vd,
                                                        int64_t rows, int64_t cols) {
  const int64_t j = ((int64_t)blockIdx.x * 256 + threadIdx.x) * (4 * Op::EPW);
  if (j >= cols) return;
  for (int64_t i = blockIdx.y; i < rows; i += gridDim.y)
    store_chunk<Op>(d, ldd, i, j, load_chunk<Op>(s, lds, rows, cols, i, j, vs != 0), row_mask<Op>(j, cols), vd != 0);
}

// int32 -> packed 16-bit (saturated to INF16) and back, 8 elements a thread.
static __global__ void __launch_bounds__(256) pack_kernel(const int32_t *__restrict__ s, int64_t lds, int vs,
                                                   uint16_t *__restrict__ d, int64_t ldd, int vd, int64_t n) {
  const int64_t j = ((int64_t)blockIdx.x * 256 + threadIdx.x) * 8;
  if (j >= n) return;
  for (int64_t i = blockIdx.y; i < n; i += gridDim.y) {
    const uint4 x = load_chunk<OpI32>(s, lds, n, n, i, j, vs != 0), y = load_chunk<OpI32>(s, lds, n, n, i, j + 4, vs != 0);
    auto sat = [](uint32_t v) { return (int32_t)v >= 0x7FFF ? 0x7FFFu : v & 0xFFFFu; };
    const uint4 w = make_uint4(sat(x.x) | sat(x.y) << 16, sat(x.z) | sat(x.w) << 16, sat(y.x) | sat(y.y) << 16,
                               sat(y.z) | sat(y.w) << 16);
    store_chunk<OpU16>(d, ldd, i, j, w, row_mask<OpU16>(j, n), vd != 0);
  }
}
static __global__ void __launch_bounds__(256) unpack_kernel(const uint16_t *__restrict__ s, int64_t lds, int vs,
                                                     int32_t *__restrict__ d, int64_t ldd, int vd, int64_t n) {
  const int64_t j = ((int64_t)blockIdx.x * 256 + threadIdx.x) * 8;
  if (j >= n) return;
  for (int64_t i = blockIdx.y; i < n; i += gridDim.y) {
    const uint4 x = load_chunk<OpU16>(s, lds, n, n, i, j, vs != 0);
    auto wide = [](uint32_t v) { return v >= 0x7FFFu ? 1073741823u : v; };
    store_chunk<OpI32>(d, ldd, i, j,
                       make_uint4(wide(x.x & 0xFFFFu), wide(x.x >> 16), wide(x.y & 0xFFFFu), wide(x.y >> 16)),
                       row_mask<OpI32>(j, n), vd != 0);
    store_chunk<OpI32>(d, ldd, i, j + 4,
                       make_uint4(wide(x.z & 0xFFFFu), wide(x.z >> 16), wide(x.w & 0xFFFFu), wide(x.w >> 16)),
                       row_mask<OpI32>(j + 4, n), vd != 0);
  }
}

// Rows [0, rows) of a Layout: 0 on the diagonal below n, INF elsewhere, over
// the stored columns below `cols`.
template <class Op>
__global__ void __launch_bounds__(256) fill_inf_kernel(typename Op::elem *__restrict__ D, Layout L, int64_t rows,
                                                       int64_t cols, int64_t n, int vec) {
  constexpr int E = 4 * Op::EPW;
  const int64_t c0 = ((int64_t)blockIdx.x * 256 + threadIdx.x) * E;
  if (c0 >= cols) return;
  for (int64_t r = blockIdx.y; r < rows; r += gridDim.y) {
    if (!L.stored(r, c0)) continue;
    uint4 v = make_uint4(Op::INF_WORD, Op::INF_WORD, Op::INF_WORD, Op::INF_WORD);
    if (r >= c0 && r < c0 + E && r < n) {
#pragma unroll
      for (int e = 0; e < E; ++e)
        if (c0 + e == r) chunk_set<Op>(v, e, 0u);
    }
    store_chunk<Op>(D, L, r, c0, v, row_mask<Op>(c0, cols), vec != 0);
  }
}

}  // namespace apsp
