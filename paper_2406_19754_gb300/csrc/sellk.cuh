// Sliced-ELL row traversal shared by the SpMV, smoother and PCG kernels.
//
// Mapping: one warp per group of R = 32 / TPR consecutive rows (a slice, when
// the slice height C is R).  Lane = t * R + r handles row r of the group and
// the entries k = t, t + TPR, ... of that row, so with C == R every load
// instruction of a warp touches 32 consecutive entries of the column-major
// slice (fully coalesced); with C != R (the autotuner's decoupled layouts) the
// lanes of a row group read C-row runs of one or several slices.  The TPR partial sums of a row are
// combined with xor-shuffles (fixed order).  Matrix values and column indices
// are streamed with evict-first loads; the gathered vectors stay in L2.
#pragma once

#include "common.cuh"

namespace amg {

constexpr int SELL_BLOCK = 256;  // threads per block (8 slices in flight)

// Layout code of a SELL kernel instantiation: threads per row (1, 2, 4, 8,
// or 16 and 32 for wide rows) plus SELL_D16 when the matrix stores
// compressed columns (1..8 threads per row only).
constexpr int SELL_D16 = 64;
// ... or plus SELL_IX (one thread per row, slices of 32 rows) when the matrix
// has packed column indices (Sell::rec): the row's loads are then issued in
// chunks of its exact length, all values and gathers of up to 8 entries
// together.  The plain loop takes four entries at a time and the rest one by
// one, each a column load and the gather that waits for it.
constexpr int SELL_IX = 128;

// Resident blocks per SM the streaming kernels are compiled for: 8 (64 warps,
// full occupancy: at most 32 registers, which they need to keep enough loads in
// flight); packed indices keep twice the loads in flight per thread and need
// the registers for them.
constexpr int sell_blocks(int code) { return (code & SELL_IX) ? 4 : 8; }

template <int TPR>
struct Lanes {
  static constexpr int W = TPR & 63;  // threads per row (1 with SELL_IX)
  static constexpr bool D16 = (TPR & SELL_D16) != 0;
  static constexpr bool IX = (TPR & SELL_IX) != 0;
  static constexpr int C = 32 / W;
  int r, t;
  __device__ __forceinline__ Lanes() {
    int lane = threadIdx.x & 31;
    r = lane % C;
    t = lane / C;
  }
};

// acc (+ or -, NEG) a_k g(col_k) for the N entries k0 .. k0 + N - 1 of this
// lane's row in a slice with packed indices; val and delta point at the lane's
// slot of ELL column 0, head at the slice's index block.
template <int MODE, int N, bool NEG, typename AccT, typename V, typename G>
__device__ __forceinline__ AccT ix_chunk(const V* __restrict__ val,
                                         const int32_t* __restrict__ head,
                                         const uint16_t* __restrict__ delta, int32_t i,
                                         int32_t last, int lane, int k0, AccT acc, G g) {
  V a[N];
  int32_t j[N];
#pragma unroll
  for (int u = 0; u < N; ++u) {
    const int k = k0 + u;
    a[u] = ld_stream(val + k * 32);
    if constexpr (MODE == IX_PLAIN)
      j[u] = ld_stream(head + k * 32 + lane);
    else if constexpr (MODE == IX_DELTA)
      j[u] = __ldg(head + k) + (int)ld_stream(delta + k * 32);
    else if constexpr (MODE == IX_OFFSET)
      j[u] = i + __ldg(head + k);
    else
      j[u] = min(max(i + __ldg(head + k), 0), last);
  }
  AccT x[N];
#pragma unroll
  for (int u = 0; u < N; ++u) x[u] = g(j[u]);
#pragma unroll
  for (int u = 0; u < N; ++u) {
    const AccT e = to_f(a[u], AccT(0));
    acc = fma(NEG ? -e : e, x[u], acc);
  }
  return acc;
}

template <int MODE, bool NEG, typename AccT, typename V, typename G>
__device__ __forceinline__ AccT ix_row(const V* __restrict__ val,
                                       const int32_t* __restrict__ head, int w, int32_t i,
                                       int32_t last, int lane, AccT acc, G g) {
  const uint16_t* delta = (const uint16_t*)(head + ((w + 3) & ~3)) + lane;
#define AMG_IX_CHUNK(N) ix_chunk<MODE, N, NEG>(val, head, delta, i, last, lane, k0, acc, g)
  int k0 = 0;
  for (; k0 + 8 <= w; k0 += 8) acc = AMG_IX_CHUNK(8);
  switch (w - k0) {
    case 1: return AMG_IX_CHUNK(1);
    case 2: return AMG_IX_CHUNK(2);
    case 3: return AMG_IX_CHUNK(3);
    case 4: return AMG_IX_CHUNK(4);
    case 5: return AMG_IX_CHUNK(5);
    case 6: return AMG_IX_CHUNK(6);
    case 7: return AMG_IX_CHUNK(7);
    default: return acc;
  }
#undef AMG_IX_CHUNK
}

// sum_k a_{row,k} * g(col_{row,k}) over the entries of this lane's row in
// warp row-group s (32/TPR rows), accumulated in AccT.  When the slice height
// is 32/TPR (one slice per group, every layout but the autotuner's decoupled
// ones, and every batched one) the group is the slice; otherwise each lane
// finds its row's own slice (row i: slice i / C, slot k at
// sliceptr + k C + i mod C), and the row's entries are visited in the same
// order.  Compressed columns (SELL_D16 in the layout code; A.d16 set) give
// the same j for every slot, so the sum is the same bits either way.
//
// NEG: init - sum_k a_k g(col_k) instead, each entry by an FMA with the
// negated value (no separate subtraction); init is added by the row's first
// lane (t == 0) only.
template <int TPR, typename AccT, bool NEG = false, typename V, typename G>
__device__ __forceinline__ AccT sell_row(const SellView<V>& A, int64_t s, const Lanes<TPR>& ln,
                                         G g, AccT init = AccT(0)) {
  constexpr int C = Lanes<TPR>::C, W = Lanes<TPR>::W;
  if constexpr (Lanes<TPR>::IX) {
    const longlong2 r0 = __ldg((const longlong2*)(A.rec + s));
    const int64_t e = __ldg(&A.rec[s + 1].slot);
    const V* val = A.val + r0.x + ln.r;
    const int32_t* head = (const int32_t*)(A.ix + (r0.y & ~(int64_t)3));
    const int w = (int)((e - r0.x) >> 5);
    const int32_t i = (int32_t)A.rbeg(s, 32) + ln.r, last = A.ncols - 1;
    switch ((int)(r0.y & 3)) {  // warp-uniform
      case IX_OFFSET: return ix_row<IX_OFFSET, NEG>(val, head, w, i, last, ln.r, init, g);
      case IX_CLAMP: return ix_row<IX_CLAMP, NEG>(val, head, w, i, last, ln.r, init, g);
      case IX_DELTA: return ix_row<IX_DELTA, NEG>(val, head, w, i, last, ln.r, init, g);
      default: return ix_row<IX_PLAIN, NEG>(val, head, w, i, last, ln.r, init, g);
    }
  }
  AccT acc = ln.t == 0 ? init : AccT(0);
  if (!A.row0 && A.C != C) {
    const int64_t i = s * C + ln.r;
    if (i < A.n) {
      const int64_t sl = i / A.C;
      const int64_t b0 = __ldg(A.sliceptr + sl);
      const int w = (int)((__ldg(A.sliceptr + sl + 1) - b0) / A.C);
      const int64_t beg = b0 + (i - sl * A.C);
      const V* vp = A.val + beg;
      if constexpr (Lanes<TPR>::D16) {
        const uint16_t* dp = A.d16 + beg;
        const int32_t* bp = A.kbase + b0 / A.C;
#pragma unroll 4
        for (int k = ln.t; k < w; k += W) {
          const int j = __ldg(bp + k) + (int)ld_stream(dp + (int64_t)k * A.C);
          const AccT a = to_f(ld_stream(vp + (int64_t)k * A.C), AccT(0));
          acc = fma(NEG ? -a : a, g(j), acc);
        }
      } else {
        const int32_t* cp = A.col + beg;
#pragma unroll 4
        for (int k = ln.t; k < w; k += W) {
          const int j = ld_stream(cp + (int64_t)k * A.C);
          const AccT a = to_f(ld_stream(vp + (int64_t)k * A.C), AccT(0));
          acc = fma(NEG ? -a : a, g(j), acc);
        }
      }
    }
#pragma unroll
    for (int o = C; o < 32; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc;
  }
  const int64_t beg = __ldg(A.sliceptr + s);
  const int w = (int)((__ldg(A.sliceptr + s + 1) - beg) / C);
  const V* vp = A.val + beg + ln.r;
  if constexpr (Lanes<TPR>::D16) {
    const uint16_t* dp = A.d16 + beg + ln.r;
    const int32_t* bp = A.kbase + beg / C;
#pragma unroll 4
    for (int k = ln.t; k < w; k += W) {
      const int j = __ldg(bp + k) + (int)ld_stream(dp + (int64_t)k * C);
      const AccT a = to_f(ld_stream(vp + (int64_t)k * C), AccT(0));
      acc = fma(NEG ? -a : a, g(j), acc);
    }
  } else {
    const int32_t* cp = A.col + beg + ln.r;
#pragma unroll 4
    for (int k = ln.t; k < w; k += W) {
      const int j = ld_stream(cp + (int64_t)k * C);
      const AccT a = to_f(ld_stream(vp + (int64_t)k * C), AccT(0));
      acc = fma(NEG ? -a : a, g(j), acc);
    }
  }
#pragma unroll
  for (int o = C; o < 32; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return acc;
}

#define AMG_SELL_CASE(code, ...) \
  case code: {                    \
    constexpr int TPR = code;     \
    __VA_ARGS__;                  \
  } break;

// Runs the statement with TPR = the layout code (see Lanes) as a constant.
#define AMG_DISPATCH_TPR(code, ...)        \
  switch (code) {                          \
    AMG_SELL_CASE(1, __VA_ARGS__)          \
    AMG_SELL_CASE(2, __VA_ARGS__)          \
    AMG_SELL_CASE(4, __VA_ARGS__)          \
    AMG_SELL_CASE(8, __VA_ARGS__)          \
    AMG_SELL_CASE(16, __VA_ARGS__)         \
    AMG_SELL_CASE(32, __VA_ARGS__)         \
    AMG_SELL_CASE(65, __VA_ARGS__)         \
    AMG_SELL_CASE(66, __VA_ARGS__)         \
    AMG_SELL_CASE(68, __VA_ARGS__)         \
    AMG_SELL_CASE(72, __VA_ARGS__)         \
    AMG_SELL_CASE(129, __VA_ARGS__)        \
    default:                               \
      return AMG_ERR_ARG;                  \
  }

// vbytes: size of the values the kernel streams.  Packed indices for FP64 values
// only: with FP32 ones twice the warps per SM are worth more than exact chunks
// (batched 12.2M-row pre-smoother 142 us, 169 with them; FP64 product 209, 172
// with them).
inline int sell_code(const Sell& A, size_t vbytes) {
  return A.tpr | (A.rec && vbytes == 8 ? SELL_IX : A.d16 ? SELL_D16 : 0);
}

// Warp row-groups of 32/tpr rows that the one-warp-per-group kernels iterate
// over A (see SellView::ngroups).
inline int64_t sell_groups(const Sell& A) {
  const int R = 32 / A.tpr;
  if (A.row0 || A.C == R) return A.nslices;
  return (A.n + R - 1) / R;
}

template <typename V>
inline SellView<V> view(const Sell& A, const V* val) {
  SellView<V> v;
  v.n = A.n;
  v.nslices = A.nslices;
  v.ngroups = sell_groups(A);
  v.C = A.C;
  v.sliceptr = A.sliceptr;
  v.col = A.col;
  v.val = val;
  v.row0 = A.row0;
  v.sys = A.sys;
  v.d16 = A.d16;
  v.kbase = A.kbase;
  v.rec = A.rec;
  v.ix = A.ix;
  v.ncols = (int32_t)A.ncols;
  v.act = nullptr;
  return v;
}

// Row handled by this lane in warp row-group sl, or -1 (padding lane /
// sub-row lane).
template <int TPR, typename V>
__device__ __forceinline__ int64_t lane_row(const SellView<V>& A, int64_t sl,
                                            const Lanes<TPR>& ln) {
  constexpr int C = Lanes<TPR>::C;
  const int64_t i = A.rbeg(sl, C) + ln.r;
  return (ln.t == 0 && i < A.rend(sl, C)) ? i : -1;
}

// Grid for one-warp-per-group kernels: enough blocks to fill the GPU, capped
// by the group count (grid-stride loop inside).
inline int sell_grid(int64_t ngroups, int num_sms, int blocks_per_sm = 8) {
  return grid_for(ngroups * 32, SELL_BLOCK, num_sms, blocks_per_sm);
}

}  // namespace amg
