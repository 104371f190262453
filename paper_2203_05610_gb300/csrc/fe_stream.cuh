// fe_stream.cuh -- streamed product with the block-CSR tangent: the device
// code shared by the SpMV (fe_krylov.cu), the AMG V-cycle's level-0
// Chebyshev step and its power steps (fe_amg.cu).
//
// The block rows are cut into one contiguous range per warp of a single wave,
// ranges of equal block counts (a partition array of the mesh), so every
// warp streams one region of memory and all end together.  A warp walks its
// range in the 32-block tiles of the value layout (kv_index), one block per
// lane, regardless of where rows start.  While tile i is multiplied, the
// values and the gather of x of tiles i + 1 and i + 2 and the column indices
// of the three tiles after them are in flight.  The three products of every block
// go to the warp's window in shared memory; when the window is full or the
// range ends, four lanes per row (FP32: two) add the rows' products from it
// (every fourth or second place, each in order), 8 or 16 rows at a time, a row
// that runs on into the next window carrying its sum; the rows that end there go through the epilogue
// Epi, lane i on the i-th of them, with operands whose loads are in flight
// during the sums.  Summation order is fixed by the row pointers and the
// partition, so results are deterministic.  A range may hold no rows (a row
// longer than a range) or rows without blocks (vertices that no element uses:
// their sums are zero); the walk goes through it like through any other.
//
// What bounds it, and why this form.  HBM, with the latency of the chain
// column index -> x behind it.  Walking the value tiles where they are aligned
// makes each of the nine value loads one 128-byte line instead of two.  Row sums through shared memory
// take three stores and about three adds per block; a segmented scan across
// the lanes takes five steps of three shuffles and adds, and for FP64 values
// those adds alone (15 per block, at 64 cycles per warp instruction and SM
// quarter) exceed the nine products; four lanes per row take four per block
// where two take eleven (few rows end in a window, so most lanes idled).  The
// three tile buffers take their roles by unrolling a window's nine tiles:
// moved from one set of registers to the next they would wait for the loads
// that were just issued, and only one tile would be in flight.
#pragma once

#include <climits>

#include "fe_internal.h"

template <class V>
__device__ __forceinline__ float ld_val(const V* p);
template <>
__device__ __forceinline__ float ld_val<float>(const float* p) { return __ldg(p); }
template <>
__device__ __forceinline__ float ld_val<__nv_bfloat16>(const __nv_bfloat16* p) {
  return __bfloat162float(*p);
}

constexpr int STREAM_THREADS = 128;
constexpr int STREAM_WARPS = STREAM_THREADS / 32;

// tiles per window (a multiple of the three buffers); resident blocks per SM
// that the SpMV's launch bounds guarantee (80 registers in FP32, 168 in FP64)
constexpr int STREAM_TILES = 9;
constexpr int STREAM_WIN = 32 * STREAM_TILES;
template <class AT>
__host__ __device__ constexpr int stream_blocks_per_sm() { return sizeof(AT) == 8 ? 3 : 6; }

template <class AT>
struct StreamShared {
  AT prod[STREAM_WARPS][3][STREAM_WIN];
};

// asynchronous copy of one value to shared memory
template <class T>
__device__ __forceinline__ void cp_async(T* smem, const T* g) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(g),
               "n"(sizeof(T))
               : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// column index of block k (-1 outside the range)
__device__ __forceinline__ int stream_load_col(const int* __restrict__ col, int k, int kstart, int kend) {
  return k >= kstart && k < kend ? __ldg(col + k) : -1;
}
template <class V, class AT>
__device__ __forceinline__ void stream_load_tile(const V* __restrict__ val, int k, int kstart, int kend, AT (&v)[9]) {
  if (k >= kstart && k < kend) {
    const V* b = val + kv_index(k, 0);
#pragma unroll
    for (int t = 0; t < 9; t++) {
      if constexpr (sizeof(V) == 8) v[t] = __ldg(b + 32 * t);
      else v[t] = (AT)ld_val<V>(b + 32 * t);
    }
  } else {
#pragma unroll
    for (int t = 0; t < 9; t++) v[t] = AT(0);
  }
}

// the three components of node c (0 for c < 0)
template <class XT, class AT>
__device__ __forceinline__ void stream_load_x(const XT* __restrict__ x, int c, AT (&g)[3], int n) {
  const XT* xc = x + 3 * (int64_t)(c >= 0 ? fe_idx(c, n) : 0);
#pragma unroll
  for (int j = 0; j < 3; j++) g[j] = c >= 0 ? (AT)xc[j] : AT(0);
}

// ranges range, range + step, ... (< ranges) of block rows by one warp; prod is
// the warp's window.  Epi: prefetch(r, rb, lane) at a window's start, for the
// rows r .. min(r + 16, rb) - 1 that may end in it; load(r, i0, nd, lane)
// before the sums of the nd rows from r on, the window's i0-th to
// (i0+nd-1)-th row; finish(row, s) in lane i < nd with row r + i's sums.
template <class V, class XT, class AT, class Epi>
__device__ __forceinline__ void stream_rows(int n, int range, int step, int ranges, const int* __restrict__ part,
                                            const int* __restrict__ row_ptr, const int* __restrict__ col,
                                            const V* __restrict__ val, const XT* __restrict__ x,
                                            AT (&prod)[3][STREAM_WIN], Epi& epi) {
  constexpr int L = sizeof(AT) == 8 ? 4 : 2, RP = 32 / L;  // lanes per row in the sums, rows per pass
  if (range >= ranges) return;
  const int lane = threadIdx.x & 31;
  int r = __ldg(part + range), rb = __ldg(part + range + 1);
  int rp = __ldg(row_ptr + min(r + lane, rb));  // starts of rows r .. r + 31 (past rb: the range's end)
  int kstart = __shfl_sync(0xffffffffu, rp, 0), kend = __ldg(row_ptr + rb);
  int kc = kstart & ~31;
  int c[3];
  AT v[3][9], xg[3][3];
#pragma unroll
  for (int t = 0; t < 3; t++) c[t] = stream_load_col(col, kc + 32 * t + lane, kstart, kend);
#pragma unroll
  for (int t = 0; t < 2; t++) stream_load_tile<V, AT>(val, kc + 32 * t + lane, kstart, kend, v[t]);
  for (;;) {
    // the next range's rows, read while this one runs
    range += step;
    int nr = 0, nrb = 0, nrp = 0, nkend = 0;
    if (range < ranges) {
      nr = __ldg(part + range);
      nrb = __ldg(part + range + 1);
      nrp = __ldg(row_ptr + min(nr + lane, nrb));
      nkend = __ldg(row_ptr + nrb);
    }
#pragma unroll
    for (int t = 0; t < 2; t++) {
      stream_load_x<XT, AT>(x, c[t], xg[t], n);
      c[t] = stream_load_col(col, kc + 32 * (t + 3) + lane, kstart, kend);
    }
    AT carry[3] = {AT(0), AT(0), AT(0)};  // row r's sum over the earlier windows
    do {  // (once for a range without blocks: its empty rows' sums, and the next range's loads)
      const int kw = kc;  // the window's first block
      const int kwe = min(kw + STREAM_WIN, kend);
      const int rw = r;
      epi.prefetch(r, rb, lane);
#pragma unroll
      for (int t = 0; t < STREAM_TILES; t++) {
        if (kw + 32 * t < kwe) {
          const int b0 = t % 3, b2 = (t + 2) % 3;
          stream_load_tile<V, AT>(val, kw + 32 * (t + 2) + lane, kstart, kend, v[b2]);
          stream_load_x<XT, AT>(x, c[b2], xg[b2], n);
          c[b2] = stream_load_col(col, kw + 32 * (t + 5) + lane, kstart, kend);
#pragma unroll
          for (int q = 0; q < 3; q++)
            prod[q][32 * t + lane] =
                v[b0][3 * q] * xg[b0][0] + v[b0][3 * q + 1] * xg[b0][1] + v[b0][3 * q + 2] * xg[b0][2];
        }
      }
      kc = kw + STREAM_WIN;  // (past a last, shorter window nothing follows)
      if (kc >= kend && range < ranges) {  // the next range's first tiles, in flight during the sums
        kstart = __shfl_sync(0xffffffffu, nrp, 0);
        const int k0 = kstart & ~31;
#pragma unroll
        for (int t = 0; t < 3; t++) c[t] = stream_load_col(col, k0 + 32 * t + lane, kstart, nkend);
#pragma unroll
        for (int t = 0; t < 2; t++) stream_load_tile<V, AT>(val, k0 + 32 * t + lane, kstart, nkend, v[t]);
      }
      __syncwarp();
      for (int off = 0;;) {  // the next RP rows (one less at the end of the loaded row starts)
        const int i = lane / L, most = off == 32 - RP ? RP - 1 : RP;
        const int rs = __shfl_sync(0xffffffffu, rp, off + i), re = __shfl_sync(0xffffffffu, rp, min(off + i + 1, 31));
        const bool row = i < most && r + i < rb;
        const int nd = __popc(__ballot_sync(0xffffffffu, row && re <= kwe)) / L;  // rows that end in this window
        epi.load(r, r - rw, nd, lane);
        AT s[3], u[3];
#pragma unroll
        for (int q = 0; q < 3; q++) s[q] = lane == 0 ? carry[q] : AT(0);
        const int hi = row ? min(re, kwe) - kw : 0;
#pragma unroll 4
        for (int k = max(rs - kw, 0) + lane % L; k < hi; k += L) {
#pragma unroll
          for (int q = 0; q < 3; q++) s[q] += prod[q][k];
        }
#pragma unroll
        for (int q = 0; q < 3; q++) {
#pragma unroll
          for (int o = 1; o < L; o <<= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
          u[q] = __shfl_sync(0xffffffffu, s[q], (L * lane) & 31);
          carry[q] = nd < most ? __shfl_sync(0xffffffffu, s[q], (L * nd) & 31) : AT(0);
        }
        if (lane < nd) epi.finish(r + lane, u);
        r += nd;
        const bool more = nd == most && r < rb;  // the next row may end in this window, too
        if (r < rb && (!more || off == 32 - RP)) rp = __ldg(row_ptr + min(r + lane, rb));
        if (!more) break;
        off = (off + RP) & 31;
      }
      __syncwarp();
    } while (kc < kend);
    if (range >= ranges) return;
    r = nr;
    rb = nrb;
    rp = nrp;
    kend = nkend;
    kc = kstart & ~31;
  }
}

// Warps of a streamed launch (one wave, at least one tile per warp) and the
// row ranges that they take in turn: about 28 tiles each where a warp has
// more (Cook P2 64x64x8 and 48x48x8: 5 tiles 79 and 49.5 us, 14 tiles 77.5 and
// 48.2, 28 tiles 77.0 and 46.5, one range 77.4 and 46.5; FP64 271, 251, 246,
// 248 us).
constexpr int STREAM_RANGE_TILES = 28;
struct StreamShape {
  int warps, ranges;
};
inline StreamShape stream_shape(int blocks_per_sm, int sm_count, int64_t nnzb) {
  const int64_t wave = (int64_t)blocks_per_sm * sm_count * STREAM_WARPS;
  const int64_t tiles = (nnzb + 31) / 32;
  if (tiles <= wave) return {(int)(tiles < 1 ? 1 : tiles), (int)(tiles < 1 ? 1 : tiles)};
  const int64_t m = (tiles + wave * STREAM_RANGE_TILES / 2) / (wave * STREAM_RANGE_TILES);
  return {(int)wave, (int)(wave * (m < 1 ? 1 : m))};
}
inline unsigned stream_grid(int warps) { return (unsigned)((warps + STREAM_WARPS - 1) / STREAM_WARPS); }
// fe_mesh.cu: row ranges of equal block counts, part [ranges + 1] on the device
int fe_stream_partition(fe_mesh m, int ranges, int* part);
