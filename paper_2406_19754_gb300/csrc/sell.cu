// CSR -> sliced-ELL conversion and the plain FP64 SpMV (y = alpha A x + beta y).
#include <algorithm>

#include "sellk.cuh"

namespace amg {

// Rows of slice s: [s*C, min(n, s*C + C)), or [row0[s], row0[s+1]) when the
// slices restart at every system boundary.
__device__ __forceinline__ void slice_rows(int64_t s, int C, int64_t n, const int64_t* row0,
                                           int64_t* b, int64_t* e) {
  if (row0) {
    *b = row0[s];
    *e = row0[s + 1];
  } else {
    *b = s * C;
    *e = (s + 1) * C < n ? (s + 1) * C : n;
  }
}

// Slot layout of a slice.  Sorted: slot k of a row holds its k-th entry
// (ascending columns), padding after the last one.  Aligned: the slice's ELL
// columns are the distinct column offsets o = col - row of its rows, in
// ascending order, and a row places each entry in the column of its offset
// (padding where it has none), so a stencil's ELL column k holds one offset
// and its columns differ only by the row.  Aligned is used when the distinct
// offsets are no more than the longest row (no extra padding).  Either way a
// row's entries are visited in ascending column order with zero-valued
// padding in between, so every sum comes out the same.

// Distinct column offsets of rows [rb, re), ascending; writes them to `u`
// (if non-null) and returns their count, or -1 once it exceeds `cap`.
__device__ int slice_offsets(int64_t rb, int64_t re, const int64_t* rowptr, const int32_t* col,
                             int cap, int32_t* u) {
  int pos[64];  // rows of the slice: at most the largest slice height
  const int m = (int)(re - rb);
  for (int r = 0; r < m; ++r) pos[r] = 0;
  int cnt = 0;
  for (;;) {
    int64_t next = INT64_MAX;
    for (int r = 0; r < m; ++r) {
      const int64_t i = rb + r, len = rowptr[i + 1] - rowptr[i];
      if (pos[r] < len) {
        const int64_t o = (int64_t)col[rowptr[i] + pos[r]] - i;
        next = o < next ? o : next;
      }
    }
    if (next == INT64_MAX) return cnt;
    if (cnt == cap) return -1;
    if (u) u[cnt] = (int32_t)next;
    ++cnt;
    for (int r = 0; r < m; ++r) {
      const int64_t i = rb + r, len = rowptr[i + 1] - rowptr[i];
      if (pos[r] < len && (int64_t)col[rowptr[i] + pos[r]] - i == next) ++pos[r];
    }
  }
}

// Slice lengths (width * C) and the aligned flag of every slice.
__global__ void k_sell_widths(int64_t n, int64_t nslices, int C, const int64_t* row0,
                              const int64_t* rowptr, const int32_t* col, int64_t* slen,
                              uint8_t* aligned, int* wmax) {
  int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nslices) return;
  int64_t rb, re, w = 0;
  slice_rows(s, C, n, row0, &rb, &re);
  for (int64_t i = rb; i < re; ++i) {
    int64_t len = rowptr[i + 1] - rowptr[i];
    w = len > w ? len : w;
  }
  aligned[s] = w > 0 && slice_offsets(rb, re, rowptr, col, (int)w, nullptr) >= 0;
  slen[s] = w * C;
  atomicMax(wmax, (int)(w < 0x7fffffff ? w : 0x7fffffff));
}

// Offsets of the aligned slices, stored per ELL column at sliceptr[s]/C + k.
__global__ void k_sell_offsets(int64_t n, int64_t nslices, int C, const int64_t* row0,
                               const int64_t* rowptr, const int32_t* col,
                               const int64_t* sliceptr, const uint8_t* aligned, int32_t* uoff) {
  int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nslices || !aligned[s]) return;
  int64_t rb, re;
  slice_rows(s, C, n, row0, &rb, &re);
  const int w = (int)((sliceptr[s + 1] - sliceptr[s]) / C);
  slice_offsets(rb, re, rowptr, col, w, uoff + sliceptr[s] / C);
}

// One thread per slot row of a slice: place its entries, pad the rest.
__global__ void k_sell_fill(int64_t n, int64_t ncols, int64_t nslices, int C,
                            const int64_t* row0, const int64_t* rowptr, const int32_t* col,
                            const double* val, const int64_t* sliceptr, const uint8_t* aligned,
                            const int32_t* uoff, int32_t* ocol, double* oval) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nslices * C) return;
  const int64_t s = t / C;
  const int r = (int)(t % C);
  int64_t sb, se;
  slice_rows(s, C, n, row0, &sb, &se);
  const int64_t i = sb + r;
  const int64_t beg = sliceptr[s];
  const int w = (int)((sliceptr[s + 1] - beg) / C);
  int64_t rb = 0, len = 0;
  if (i < se) {
    rb = rowptr[i];
    len = rowptr[i + 1] - rowptr[i];
  }
  if (aligned[s]) {
    // ELL column k holds offset u[k]; padding reads column i + u[k] clamped
    // into range (value 0), which keeps the ELL column's columns together
    const int32_t* u = uoff + beg / C;
    const int64_t ir = i < se ? i : se - 1;
    int64_t e = 0;
    for (int k = 0; k < w; ++k) {
      const int64_t dst = beg + (int64_t)k * C + r;
      if (e < len && (int64_t)col[rb + e] - i == u[k]) {
        ocol[dst] = col[rb + e];
        oval[dst] = val[rb + e];
        ++e;
      } else {
        int64_t c = ir + u[k];
        c = c < 0 ? 0 : c >= ncols ? ncols - 1 : c;
        ocol[dst] = (int32_t)c;
        oval[dst] = 0.0;
      }
    }
    return;
  }
  // padding (value 0) reads a valid column: the row's last one (it is in
  // cache, and it keeps the slice's column deltas small), else the row itself
  const int32_t pad_col =
      len > 0 ? col[rb + len - 1] : (int32_t)(i < ncols ? i : ncols - 1);
  for (int k = 0; k < w; ++k) {
    int64_t dst = beg + (int64_t)k * C + r;
    if (k < len) {
      ocol[dst] = col[rb + k];
      oval[dst] = val[rb + k];
    } else {
      ocol[dst] = pad_col;
      oval[dst] = 0.0;
    }
  }
}

// Slices of 32 rows, one warp per slice and one lane per row (the kernels
// above give a whole slice to one thread, whose pointer walk over 32 rows is
// a chain of dependent loads: 0.28 ms a matrix, averaged over a 128^3
// hierarchy; a warp steps all rows at once and finds the smallest offset by
// one reduction).  The merge is slice_offsets' own: at each step the smallest
// col - row among the rows' next entries is one ELL column, and the rows that
// hold it step on.
struct SliceLane {
  int64_t i, beg;
  int len, w;
  bool has;
  __device__ __forceinline__ SliceLane(int64_t s, int64_t n, const int64_t* row0,
                                       const int64_t* rowptr) {
    int64_t sb, se;
    slice_rows(s, 32, n, row0, &sb, &se);
    i = sb + (threadIdx.x & 31);
    has = i < se;
    beg = has ? rowptr[i] : 0;
    len = has ? (int)(rowptr[i + 1] - beg) : 0;
    w = __reduce_max_sync(0xffffffffu, len);
  }
};

// Per slice: packed[s] = (w << 32) | (index block bytes / 16) for one scan of
// both, and the layout: bit 2 = aligned, low bits = the index block's coding
// (ring: aligned slices store one offset per ELL column, others 16-bit deltas
// if every ELL column's columns lie within 65535, else plain columns).
__global__ void k_sell_widths32(int64_t n, int64_t ncols, int64_t nslices, const int64_t* row0,
                                const int64_t* rowptr, const int32_t* col, int ring,
                                int64_t* packed, uint8_t* layout, int* wmax) {
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  __shared__ int wm;
  if (threadIdx.x == 0) wm = 0;
  __syncthreads();
  int wl = 0;
  for (int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < nslices; s += nw) {
    const SliceLane ln(s, n, row0, rowptr);
    bool aligned = ln.w > 0;
    int pos = 0, cnt = 0, umin = 0, umax = 0;
    while (aligned) {
      const int o = pos < ln.len ? col[ln.beg + pos] - (int32_t)ln.i : INT32_MAX;
      const int m = __reduce_min_sync(0xffffffffu, o);
      if (m == INT32_MAX) break;
      aligned = cnt < ln.w;
      umin = cnt ? min(umin, m) : m;
      umax = cnt ? max(umax, m) : m;
      ++cnt;
      if (o == m) ++pos;
    }
    // offsets that leave [0, ncols) from some lane (only padding can) are clamped
    const int64_t i0 = ln.i - (threadIdx.x & 31);
    int mode = i0 + umin < 0 || i0 + 31 + umax >= ncols ? IX_CLAMP : IX_OFFSET;
    if (!aligned) {
      mode = IX_DELTA;
      const int32_t pad = ln.len > 0 ? col[ln.beg + ln.len - 1]
                                     : (int32_t)(ln.i < ncols ? ln.i : ncols - 1);
      for (int k = 0; ring && k < ln.w; ++k) {
        const int32_t c = k < ln.len ? col[ln.beg + k] : pad;
        const int32_t lo = __reduce_min_sync(0xffffffffu, c);
        const int32_t hi = __reduce_max_sync(0xffffffffu, c);
        if (hi - lo > 65535) {
          mode = IX_PLAIN;
          break;
        }
      }
    }
    const int64_t ib = ring ? ix_bytes(mode, ln.w) : 0;
    if ((threadIdx.x & 31) == 0) {
      packed[s] = ((int64_t)ln.w << 32) | (ib >> 4);
      layout[s] = (uint8_t)(mode | (aligned ? 4 : 0));
    }
    wl = max(wl, ln.w);
  }
  if ((threadIdx.x & 31) == 0) atomicMax(&wm, wl);
  __syncthreads();
  if (threadIdx.x == 0 && wm > 0) atomicMax(wmax, wm);
}

// Slots, slice pointers, and (ring) records, index blocks and the largest
// tiles (tmax: ELL columns and index bytes per ring_tile(q)).  pk:
// exclusive scan of `packed`; total: its grand total.
__global__ void k_sell_fill32(int64_t n, int64_t ncols, int64_t nslices, const int64_t* row0,
                              const int64_t* rowptr, const int32_t* col, const double* val,
                              const int64_t* pk, int64_t total, const uint8_t* layout,
                              int64_t* sliceptr, int32_t* ocol, double* oval, SliceRec* rec,
                              unsigned char* ix, int* tmax) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  __shared__ int tm[6];
  if (threadIdx.x < 6) tm[threadIdx.x] = 0;
  __syncthreads();
  for (int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < nslices; s += nw) {
    const SliceLane ln(s, n, row0, rowptr);
    const int64_t beg = (pk[s] >> 32) * 32, ib = (pk[s] & 0xffffffffll) << 4;
    const int mode = layout[s] & 3;
    const bool aligned = layout[s] & 4;
    if (lane == 0) {
      sliceptr[s] = beg;
      if (rec) rec[s] = SliceRec{beg, ib | mode};
      if (s == nslices - 1) {
        sliceptr[nslices] = (total >> 32) * 32;
        if (rec) rec[nslices] = SliceRec{(total >> 32) * 32, (total & 0xffffffffll) << 4};
      }
      for (int q = 0; rec && q < 3; ++q)
        // (batched systems' tiles start at any slice)
        if (row0 || s % ring_tile(q) == 0) {
          const int64_t e = s + ring_tile(q) < nslices ? pk[s + ring_tile(q)] : total;
          atomicMax(&tm[q], (int)((e >> 32) - (pk[s] >> 32)));
          atomicMax(&tm[3 + q], (int)(((e & 0xffffffffll) << 4) - ib));
        }
    }
    int32_t* head = rec ? (int32_t*)(ix + ib) : nullptr;
    if (aligned) {
      // ELL column k holds offset u_k; padding reads column i + u_k clamped
      // into range (value 0; rows past the slice's last use that row)
      const int64_t last = ln.i - lane + __popc(__ballot_sync(0xffffffffu, ln.has)) - 1;
      const int64_t ir = ln.has ? ln.i : last;
      int pos = 0;
      for (int k = 0; k < ln.w; ++k) {
        const int32_t c = pos < ln.len ? col[ln.beg + pos] : 0;
        const int o = pos < ln.len ? c - (int32_t)ln.i : INT32_MAX;
        const int m = __reduce_min_sync(0xffffffffu, o);
        const int64_t dst = beg + (int64_t)k * 32 + lane;
        // a slice with fewer distinct offsets than its longest row cannot be:
        // m is an offset here for every k < w
        if (o == m && pos < ln.len) {
          ocol[dst] = c;
          oval[dst] = val[ln.beg + pos];
          ++pos;
        } else {
          int64_t cc = ir + m;
          cc = cc < 0 ? 0 : cc >= ncols ? ncols - 1 : cc;
          ocol[dst] = (int32_t)cc;
          oval[dst] = 0.0;
        }
        if (rec && lane == 0) head[k] = m;
      }
      continue;
    }
    // sorted: k-th entry in ELL column k; padding (value 0) reads the row's
    // last column, else the row itself
    const int32_t pad = ln.len > 0 ? col[ln.beg + ln.len - 1]
                                   : (int32_t)(ln.i < ncols ? ln.i : ncols - 1);
    uint16_t* d = rec && mode == IX_DELTA ? (uint16_t*)(ix + ib + ((4 * ln.w + 15) & ~15))
                                          : nullptr;
    for (int k = 0; k < ln.w; ++k) {
      const int64_t dst = beg + (int64_t)k * 32 + lane;
      const int32_t c = k < ln.len ? col[ln.beg + k] : pad;
      ocol[dst] = c;
      oval[dst] = k < ln.len ? val[ln.beg + k] : 0.0;
      if (d) {
        const int32_t lo = __reduce_min_sync(0xffffffffu, c);
        if (lane == 0) head[k] = lo;
        d[k * 32 + lane] = (uint16_t)(c - lo);
      } else if (rec) {
        head[k * 32 + lane] = c;
      }
    }
  }
  __syncthreads();
  if (tmax && threadIdx.x < 6 && tm[threadIdx.x] > 0)
    atomicMax(tmax + threadIdx.x, tm[threadIdx.x]);
}

// Column compression, one thread per slice: for each ELL column k the base is
// the smallest column of its C slots and every slot stores its offset from it.
// A slice whose offsets do not fit 16 bits raises *wide (the caller then
// keeps plain columns for the whole matrix).
__global__ void k_sell_compress(int64_t nslices, int C, const int64_t* sliceptr,
                                const int32_t* col, uint16_t* d16, int32_t* kbase, int* wide) {
  int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nslices) return;
  const int64_t beg = sliceptr[s];
  const int w = (int)((sliceptr[s + 1] - beg) / C);
  for (int k = 0; k < w; ++k) {
    const int32_t* c = col + beg + (int64_t)k * C;
    int32_t lo = c[0], hi = c[0];
    for (int r = 1; r < C; ++r) {
      lo = c[r] < lo ? c[r] : lo;
      hi = c[r] > hi ? c[r] : hi;
    }
    if ((int64_t)hi - (int64_t)lo > 65535) *wide = 1;
    kbase[beg / C + k] = lo;
    for (int r = 0; r < C; ++r) d16[beg + (int64_t)k * C + r] = (uint16_t)(c[r] - lo);
  }
}

__global__ void k_to_f32(int64_t n, const double* in, float* out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (float)in[i];
}

__global__ void k_to_bf16(int64_t n, const double* in, __nv_bfloat16* out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = __float2bfloat16_rn((float)in[i]);
}

// Slices of 32 rows (out.n, ncols, nslices, row0 are set): sizes by one warp
// per slice, one scan of slots and index bytes together, one fill.
static int sell_from_csr32(Arena& ar, const int64_t* rowptr, const int32_t* col,
                           const double* val, Sell& out, cudaStream_t s, bool compress,
                           bool ring) {
  int64_t *packed = nullptr, *pk = nullptr;
  uint8_t* layout = nullptr;
  int* mx = nullptr;  // widest slice; then the largest tiles (k_sell_fill32)
  AMG_TRY(ar.alloc_n(&packed, out.nslices));
  AMG_TRY(ar.alloc_n(&pk, out.nslices));
  AMG_TRY(ar.alloc_n(&layout, out.nslices));
  AMG_TRY(ar.alloc_n(&mx, 7));
  AMG_TRY(ar.alloc_n(&out.sliceptr, out.nslices + 1));
  AMG_CUDA_TRY(cudaMemsetAsync(mx, 0, 7 * sizeof(int), s));
  const unsigned g = (unsigned)std::min<int64_t>((out.nslices + 7) / 8, 2048);
  k_sell_widths32<<<g, 256, 0, s>>>(out.n, out.ncols, out.nslices, out.row0, rowptr, col, ring,
                                    packed, layout, mx);
  AMG_LAUNCH_CHECK();
  int mx_h[7] = {};
  AMG_CUDA_TRY(cudaMemcpyAsync(mx_h, mx, sizeof(int), cudaMemcpyDeviceToHost, s));
  int64_t total = 0;
  AMG_TRY(scan_exclusive_i64(ar, packed, pk, out.nslices, &total, s));  // synchronises
  out.wmax = mx_h[0];
  out.nnz_pad = (total >> 32) * 32;
  ring = ring && out.wmax <= RING_MAX_WIDTH;
  AMG_TRY(ar.alloc_n(&out.col, out.nnz_pad));
  AMG_TRY(ar.alloc_n(&out.v64, out.nnz_pad));
  if (ring) {
    out.ix_bytes = (total & 0xffffffffll) << 4;
    int rc = ar.alloc_n(&out.rec, out.nslices + 1);
    if (rc == AMG_OK) rc = ar.alloc_n(&out.ix, out.ix_bytes);
    if (rc == AMG_ERR_OOM) {  // up to 4 bytes an entry beside the plain columns: do without
      ar.release(out.rec);
      out.rec = nullptr;
      out.ix_bytes = 0;
      ring = false;
    } else if (rc < 0) {
      return rc;
    }
  }
  k_sell_fill32<<<g, 256, 0, s>>>(out.n, out.ncols, out.nslices, out.row0, rowptr, col, val, pk,
                                  total, layout, out.sliceptr, out.col, out.v64, out.rec,
                                  out.ix, ring ? mx + 1 : nullptr);
  AMG_LAUNCH_CHECK();
  AMG_CUDA_TRY(cudaMemcpyAsync(mx_h, mx, sizeof(mx_h), cudaMemcpyDeviceToHost, s));
  if (compress && out.tpr <= 8) AMG_TRY(sell_compress(ar, out, s));
  AMG_CUDA_TRY(cudaStreamSynchronize(s));  // the CSR may go when this returns
  for (int q = 0; q < 3; ++q) {
    out.tile_w[q] = mx_h[1 + q];
    out.tile_ix[q] = mx_h[4 + q];
  }
  ar.release(packed);
  ar.release(pk);
  ar.release(layout);
  ar.release(mx);
  return AMG_OK;
}

int sell_from_csr(Arena& ar, int64_t n, int64_t ncols, const int64_t* rowptr, const int32_t* col,
                  const double* val, int C, int tpr, Sell& out, cudaStream_t s,
                  const std::vector<int64_t>* sys_off, bool compress, bool ring) {
  if (n <= 0 || ncols <= 0) return AMG_ERR_ARG;
  // heights 1..64 and 1..32 threads per row, powers of two; batched systems
  // keep one slice per warp (slice height x threads per row = 32)
  if (C < 1 || C > 64 || (C & (C - 1)) || tpr < 1 || tpr > 32 || (tpr & (tpr - 1)))
    return AMG_ERR_ARG;
  if (sys_off && sys_off->size() >= 2 && C * tpr != 32) return AMG_ERR_ARG;
  out.n = n;
  out.ncols = ncols;
  out.C = C;
  out.tpr = tpr;
  out.nslices = (n + C - 1) / C;
  if (sys_off && sys_off->size() >= 2) {  // batched systems: restart slices at each one
    std::vector<int64_t> row0;
    std::vector<int32_t> sys;
    for (size_t k = 0; k + 1 < sys_off->size(); ++k)
      for (int64_t r = (*sys_off)[k]; r < (*sys_off)[k + 1]; r += C) {
        row0.push_back(r);
        sys.push_back((int32_t)k);
      }
    if (sys_off->back() != n) return AMG_ERR_ARG;
    row0.push_back(n);
    out.nslices = (int64_t)sys.size();
    AMG_TRY(ar.alloc_n(&out.row0, out.nslices + 1));
    AMG_TRY(ar.alloc_n(&out.sys, out.nslices));
    AMG_CUDA_TRY(cudaMemcpyAsync(out.row0, row0.data(), sizeof(int64_t) * row0.size(),
                                 cudaMemcpyHostToDevice, s));
    AMG_CUDA_TRY(cudaMemcpyAsync(out.sys, sys.data(), sizeof(int32_t) * sys.size(),
                                 cudaMemcpyHostToDevice, s));
    AMG_CUDA_TRY(cudaStreamSynchronize(s));  // host vectors go out of scope
  }
  if (C == 32)
    return sell_from_csr32(ar, rowptr, col, val, out, s, compress, ring && tpr == 1);
  int64_t* slen = nullptr;
  uint8_t* aligned = nullptr;
  int* wmax = nullptr;
  AMG_TRY(ar.alloc_n(&slen, out.nslices));
  AMG_TRY(ar.alloc_n(&aligned, out.nslices));
  AMG_TRY(ar.alloc_n(&wmax, 1));
  AMG_TRY(ar.alloc_n(&out.sliceptr, out.nslices + 1));
  AMG_CUDA_TRY(cudaMemsetAsync(wmax, 0, sizeof(int), s));
  const unsigned gs = (unsigned)((out.nslices + 127) / 128);
  k_sell_widths<<<gs, 128, 0, s>>>(n, out.nslices, C, out.row0, rowptr, col, slen, aligned,
                                   wmax);
  AMG_LAUNCH_CHECK();
  int wmax_h = 0;
  AMG_CUDA_TRY(cudaMemcpyAsync(&wmax_h, wmax, sizeof(int), cudaMemcpyDeviceToHost, s));
  int64_t total = 0;
  AMG_TRY(scan_exclusive_i64(ar, slen, out.sliceptr, out.nslices, &total, s));
  AMG_CUDA_TRY(cudaMemcpyAsync(out.sliceptr + out.nslices, &total, sizeof(int64_t),
                               cudaMemcpyHostToDevice, s));
  ar.release(slen);
  ar.release(wmax);  // scan_exclusive_i64 synchronised: wmax_h is set
  out.wmax = wmax_h;
  out.nnz_pad = total;
  AMG_TRY(ar.alloc_n(&out.col, total));
  AMG_TRY(ar.alloc_n(&out.v64, total));
  int32_t* uoff = nullptr;
  AMG_TRY(ar.alloc_n(&uoff, total / C));
  k_sell_offsets<<<gs, 128, 0, s>>>(n, out.nslices, C, out.row0, rowptr, col, out.sliceptr,
                                    aligned, uoff);
  AMG_LAUNCH_CHECK();
  int64_t rows = out.nslices * C;
  k_sell_fill<<<(unsigned)((rows + 255) / 256), 256, 0, s>>>(n, ncols, out.nslices, C, out.row0,
                                                             rowptr, col, val, out.sliceptr,
                                                             aligned, uoff, out.col, out.v64);
  AMG_LAUNCH_CHECK();
  if (compress && tpr <= 8) AMG_TRY(sell_compress(ar, out, s));
  AMG_CUDA_TRY(cudaStreamSynchronize(s));
  ar.release(aligned);
  ar.release(uoff);
  AMG_CUDA_TRY(cudaStreamSynchronize(s));  // `total` lives on this stack frame
  return AMG_OK;
}

int sell_compress(Arena& ar, Sell& A, cudaStream_t s) {
  int* wide = nullptr;
  AMG_TRY(ar.alloc_n(&A.d16, A.nnz_pad));
  AMG_TRY(ar.alloc_n(&A.kbase, A.nnz_pad / A.C));
  AMG_TRY(ar.alloc_n(&wide, 1));
  AMG_CUDA_TRY(cudaMemsetAsync(wide, 0, sizeof(int), s));
  k_sell_compress<<<(unsigned)((A.nslices + 127) / 128), 128, 0, s>>>(
      A.nslices, A.C, A.sliceptr, A.col, A.d16, A.kbase, wide);
  AMG_LAUNCH_CHECK();
  int h = 0;
  AMG_CUDA_TRY(cudaMemcpyAsync(&h, wide, sizeof(int), cudaMemcpyDeviceToHost, s));
  AMG_CUDA_TRY(cudaStreamSynchronize(s));
  ar.release(wide);
  if (h) {
    ar.release(A.d16);
    ar.release(A.kbase);
    A.d16 = nullptr;
    A.kbase = nullptr;
  }
  return AMG_OK;
}

int sell_make_copies(Arena& ar, Sell& A, int vstore, cudaStream_t s) {
  if (vstore == VAL_F32 && !A.v32) {
    AMG_TRY(ar.alloc_n(&A.v32, A.nnz_pad));
    k_to_f32<<<1024, 256, 0, s>>>(A.nnz_pad, A.v64, A.v32);
    AMG_LAUNCH_CHECK();
  }
  if (vstore == VAL_BF16 && !A.v16) {
    AMG_TRY(ar.alloc_n(&A.v16, A.nnz_pad));
    k_to_bf16<<<1024, 256, 0, s>>>(A.nnz_pad, A.v64, A.v16);
    AMG_LAUNCH_CHECK();
  }
  return AMG_OK;
}

template <int TPR>
__global__ void __launch_bounds__(SELL_BLOCK, sell_blocks(TPR))
    k_spmv64(SellView<double> A, double alpha, const double* __restrict__ x, double beta,
             double* __restrict__ y) {
  const Lanes<TPR> ln;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < A.ngroups;
       s += nw) {
    double acc = sell_row<TPR, double>(A, s, ln, [&](int j) { return __ldg(x + j); });
    const int64_t i = lane_row(A, s, ln);
    if (i >= 0) y[i] = beta == 0.0 ? alpha * acc : alpha * acc + beta * y[i];
  }
}

int sell_spmv64(const Sell& A, double alpha, const double* x, double beta, double* y,
                int num_sms, cudaStream_t s) {
  const int grid = sell_grid(sell_groups(A), num_sms);
  SellView<double> v = view(A, (const double*)A.v64);
  AMG_DISPATCH_TPR(sell_code(A, 8),
                   (k_spmv64<TPR><<<grid, SELL_BLOCK, 0, s>>>(v, alpha, x, beta, y)));
  AMG_LAUNCH_CHECK();
  return AMG_OK;
}

}  // namespace amg
