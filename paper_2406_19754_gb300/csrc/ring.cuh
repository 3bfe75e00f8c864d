// Sliced-ELL streams through a shared-memory ring filled by bulk copies.
//
// The level operators are HBM streams (Sec. 2.1: sparse kernels move O(1)
// bytes per flop), and a warp that loads its slice entry by entry keeps only
// a few loads in flight, so DRAM latency bounds it.  Here every CTA owns a
// ring of D stages in shared memory.  A producer warp copies whole tiles of
// consecutive slices (values, index blocks, slice records: each one contiguous
// range) with cp.async.bulk, completion counted in bytes on the stage's "full"
// mbarrier; each consumer warp takes one slice of the tile, its lanes read
// their row's entries from shared memory and gather the vector through L2, and
// the warp then arrives on the stage's "empty" mbarrier.  Tiles of a CTA: b,
// b + G, b + 2G, ... (G CTAs in the grid).
//
// The 32 entries per slice of the kernel's per-row vectors (b, s, r, the
// aggregate map, ...) come with the tile, so every DRAM stream of the loop is
// a bulk copy started D - 1 tiles ahead.  Where no bulk copy can be (the ragged
// last tile, whose copy would run past the vectors' end; vectors that start off
// a 16-byte boundary) the producer warp loads and stores the entries itself, so
// the consumers find them in the stage always.
//
// What bounds it: with a ring per warp (every warp refilling its own two
// stages slice by slice) the FP32 level-0 pre-smoother issued 241 warp
// instructions a slice of 7 entries a row, more than half of them to manage
// the ring, and its time did not move when a third of its bytes went.  A tile a
// CTA, operands always staged and 32-bit places take 156 (post-smoother 406 ->
// 224).  What is left is the latency of the gathers in the FP32 pre-smoother and
// sweeps (two slices a warp, SPW = 2) and the FP64 pipe in the FP64 kernels (86%
// busy).  256^3, level 0: FP32 pre-smoother 179 -> 108 us, post-smoother 250 -> 201,
// FP64 pre-smoother 249 -> 223, post-smoother 279 -> 250, product 250 -> 242.
//
// Column indices are a third of an FP64 operator's stream and half of an FP32
// one's, and the columns of 32 consecutive rows say almost the same thing 32
// times.  Each slice's index block takes the smallest coding that holds its
// columns (IX_* in common.cuh): one offset per ELL column where the rows share
// their offsets (every slice of a stencil matrix: 4 bytes instead of 128),
// 16-bit deltas from a base per ELL column where the columns lie close (A P
// and the coarse levels: 68 instead of 128), else plain columns.  In the FP32
// per-lane kernels fewer index bytes did not pay (each load then carries less,
// and their number bounds them: 142 -> 169 us); here the copies are whole blocks,
// so bytes are what counts.
//
// Batched systems (CHUNKED): a CTA takes chunks of consecutive slices of one
// system, leaves out those of systems that have stopped, and cuts each into
// tiles; the producer writes what a tile is (RingTile) into its stage, and a
// last, empty one where the work ends.  A system's rows start anywhere, so the
// per-row copies start at the 16-byte boundary before them.
//
// Requirements (checked on the host by ring_plan): one thread per row and
// slice height 32 (lane = row of the slice), packed indices (Sell::rec), and
// tiles that fit a stage.  Slice s starts at slot
// rec[s].slot, a multiple of 32, and its index block at a multiple of 16 bytes,
// so all copies start on 16-byte boundaries and have sizes that are multiples
// of 16 bytes (32 w values of 2, 4 or 8 bytes; ix_bytes; 16-byte records); the
// per-row copies are 32 tile entries of 4 or 8 bytes at offset 32 tile t
// entries of 256-byte aligned vectors.
//
// Bounded waits: a wait for a stage gives up after RING_WAIT_NS of
// %globaltimer and sets the handle's sticky failure flag; the warp leaves its
// loop, and the producer waits (bounded) for the copies in flight before the
// CTA ends.  Later launches see the flag and return at once, and pcg_solve
// reports AMG_ERR_DEVICE_CHECK.
#pragma once

#include "sellk.cuh"

namespace amg {

constexpr int RING_MAX_STAGES = 4;
constexpr int RING_MAX_TILE = 8;  // slices per tile = consumer warps per CTA
// CTAs per SM that the streaming kernels are compiled for: 36 warps of 56
// registers.  Five or six CTAs leave 40 and 32 registers, too few to keep a
// row's gathers in flight together (256^3 FP32 solve 158.7 -> 175 and 193 ms).
constexpr int RING_CTAS_PER_SM = 4;
constexpr int RING_MAX_THREADS = (RING_MAX_TILE + 1) * 32;
constexpr unsigned long long RING_WAIT_NS = 1000000000ull;  // 1 s
constexpr size_t RING_SMEM_PER_CTA = 112 * 1024;   // at least two CTAs per SM
constexpr size_t RING_SMEM_PER_SM = 227 * 1024;
constexpr size_t RING_ALIGN_SLACK = 128;

constexpr int RING_MAX_ROWS = 5;  // per-row vectors staged with each tile

// Per-row vectors copied into the stage with each tile (the tile's
// consecutive entries of each): base pointers and element sizes.
struct RingRows {
  const void* p[RING_MAX_ROWS] = {};
  int esz[RING_MAX_ROWS] = {};
  int n = 0;
  void add(const void* ptr, int bytes) {
    p[n] = ptr;
    esz[n] = bytes;
    ++n;
  }
};

// Ring geometry of one launch (host-computed).  A stage holds the tile's
// values, its index blocks, its slice records, then its entries of each
// per-row vector.
struct RingGeom {
  int D = 0;            // stages per CTA (0: not eligible)
  int tile = 0;         // slices per tile
  int warps = 0;        // consumer warps (tile, or tile / 2: two slices a warp)
  uint32_t stage = 0;   // bytes per stage
  uint32_t coff = 0;    // offset of the index blocks within a stage
  uint32_t soff = 0;    // offset of the slice records
  uint32_t hoff = 0;    // offset of the tile's description (CHUNKED)
  uint32_t roff[RING_MAX_ROWS] = {};  // offsets of the per-row vectors
  uint32_t direct = 0;  // bit k: row vector k starts off a 16-byte boundary, no bulk copies
  int grid = 0;         // CTAs (ring_prepare)
  size_t smem = 0;      // dynamic shared memory per CTA
  int threads() const { return (warps + 1) * 32; }
};

// Chunks of a batched level: chunk c is slices off[c] .. off[c + 1] - 1, all of
// one system.
struct RingChunks {
  const int64_t* off = nullptr;
  int64_t n = 0;
};
// A chunked tile: ns slices (-1: the end of the work) from slice s0 and row r0,
// `rows` rows; the staged per-row vectors start at row e0.
struct RingTile {
  int64_t s0, r0, e0, chunk;
  int32_t ns, rows, last, pad;  // last: of its chunk
};

// ------------------------------------------------------------------ PTX wrappers

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

// The initialised barriers become visible to the async proxy (bulk copies).
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_test_parity(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ unsigned long long ring_now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Waits until the barrier's phase with this parity has completed; false
// after RING_WAIT_NS.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity) {
  if (mbar_test_parity(bar, parity)) return true;
  const unsigned long long t0 = ring_now_ns();
  for (;;) {
    if (mbar_test_parity(bar, parity)) return true;
    if (ring_now_ns() - t0 > RING_WAIT_NS) return false;
  }
}

// L2 policy for the matrix streams: evict first, so the gathered vectors
// stay in L2.
__device__ __forceinline__ uint64_t l2_evict_first() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

// Global -> shared bulk copy of `bytes` (multiple of 16, both addresses
// 16-byte aligned), completion counted on `bar`.
__device__ __forceinline__ void bulk_copy_g2s(uint32_t dst, const void* src, uint32_t bytes,
                                              uint32_t bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
      "[%0], [%1], %2, [%3], %4;" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar), "l"(pol)
      : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// ------------------------------------------------------------------ the CTA's ring

// Usage (every thread of the CTA):
//   TileRing<V, CHUNKED> ring(A, g, rows, chunks, smem);
//   if (ring.producer()) ring.produce(fail, status);
//   else while (ring.more()) {
//     if (!ring.wait()) { report; break; }
//     if (ring.ended) break;
//     if (ring.slice) { ... ring_row_sum(ring, g, init) of row ring.i ... }
//     ring.release();
//   }
// A consumer warp's slice of the current tile, this lane's row in it.
template <typename V>
struct RingSlot {
  bool slice = false;     // there is a slice
  bool has = false;       // this lane has a row: row i
  uint32_t i = 0, j = 0;  // j: the row's place among the staged entries
  const V* vals = nullptr;  // this lane's values
  const int32_t* ixb = nullptr;
  int wm = 0;  // (ELL width << 2) | IX_* code
  __device__ __forceinline__ V val(int k) const { return vals[k * 32]; }
};

template <typename V, bool CHUNKED = false, int SPW = 1>
struct TileRing {
  const SellView<V>& A;
  const RingGeom& g;
  const RingRows& rows;
  const RingChunks& ch;
  unsigned char* base;  // first stage
  uint32_t bars;        // shared address: full[D], then empty[D]
  int warp, lane;
  // consumer state; rows and slices are counted in 32 bits (columns are int32)
  int stage = 0;
  uint32_t phase = 0;
  uint32_t t, ntiles;    // current tile, tiles (not CHUNKED)
  bool ended = false;    // CHUNKED: no more tiles
  bool last = false;     // CHUNKED: last tile of its chunk
  int64_t chunk = 0;
  const unsigned char* st = nullptr;  // current stage
  RingSlot<V> slot[SPW];              // this warp's slices

  __device__ __forceinline__ TileRing(const SellView<V>& A_, const RingGeom& g_,
                                      const RingRows& rows_, const RingChunks& ch_,
                                      unsigned char* smem_raw)
      : A(A_), g(g_), rows(rows_), ch(ch_) {
    // 128-byte aligned start (the launch adds RING_ALIGN_SLACK bytes)
    base = smem_raw + ((128u - (smem_addr(smem_raw) & 127u)) & 127u);
    bars = smem_addr(base) + (uint32_t)g.D * g.stage;
    warp = threadIdx.x >> 5;
    lane = threadIdx.x & 31;
    ntiles = (uint32_t)((A.nslices + g.tile - 1) / g.tile);
    t = blockIdx.x;
    if (threadIdx.x == 0) {
      for (int d = 0; d < g.D; ++d) {
        mbar_init(full(d), 1);
        mbar_init(empty(d), (uint32_t)g.warps);
      }
      mbar_init_fence();
    }
    __syncthreads();
  }

  __device__ __forceinline__ uint32_t full(int d) const { return bars + 8u * (uint32_t)d; }
  __device__ __forceinline__ uint32_t empty(int d) const {
    return bars + 8u * (uint32_t)(RING_MAX_STAGES + d);
  }
  __device__ __forceinline__ bool producer() const { return warp == g.warps; }
  __device__ __forceinline__ SliceRec load_rec(int64_t s) const {
    const longlong2 r = __ldg((const longlong2*)(A.rec + (s < A.nslices ? s : A.nslices)));
    return SliceRec{r.x, r.y};
  }

  // Producer state: the stage the next copies go to.
  struct Fill {
    int d = 0, issued = 0;
    uint32_t ph = 1;  // the first pass over the stages does not wait
  };
  // Waits until the next stage's consumers have left it; false if that gave up
  // (the whole producer warp, same result in every lane).
  __device__ __forceinline__ bool claim(const Fill& f, int* fail, int* status) const {
    if (f.issued < g.D ||
        __all_sync(0xffffffffu, mbar_wait_bounded(empty(f.d), f.ph)))
      return true;
    if (lane == 0) {
      atomicExch(fail, 1);
      if (status) atomicCAS(status, 0, AMG_ERR_DEVICE_CHECK);
    }
    return false;
  }
  __device__ __forceinline__ void advance(Fill& f) const {
    ++f.issued;
    if (++f.d == g.D) {
      f.d = 0;
      f.ph ^= 1u;
    }
  }
  // Fills the stage (whole producer warp): slices s0 .. s0 + ns - 1 (records b
  // .. e) and nr rows from r0 of the per-row vectors, `bulk` if they may be
  // copied in bulk (they exist, and r0 and nr suit 16-byte boundaries).
  __device__ __forceinline__ void fill(const Fill& f, int64_t s0, uint32_t ns, const SliceRec& b,
                                       const SliceRec& e, bool bulk, int64_t r0, uint32_t nr,
                                       uint64_t pol) const {
    const uint32_t hand = bulk ? g.direct : ~0u;
    if (hand) {
      unsigned char* sp = base + (size_t)f.d * g.stage;
      for (int k = 0; k < rows.n; ++k) {
        if (!((hand >> k) & 1u)) continue;
        if (rows.esz[k] == 8) {
          const long long* p = (const long long*)rows.p[k] + r0;
          for (uint32_t u = lane; u < nr; u += 32) ((long long*)(sp + g.roff[k]))[u] = p[u];
        } else {
          const int* p = (const int*)rows.p[k] + r0;
          for (uint32_t u = lane; u < nr; u += 32) ((int*)(sp + g.roff[k]))[u] = p[u];
        }
      }
      __syncwarp();  // before lane 0's arrival publishes the stage
    }
    if (lane != 0) return;
    const int64_t ib = b.ix & ~(int64_t)3;
    const uint32_t vb = (uint32_t)(e.slot - b.slot) * (uint32_t)sizeof(V);
    const uint32_t cb = (uint32_t)((e.ix & ~(int64_t)3) - ib);
    auto staged = [&](int k) { return k < rows.n && !((hand >> k) & 1u); };
    uint32_t rb = 0;
#pragma unroll
    for (int k = 0; k < RING_MAX_ROWS; ++k)
      if (staged(k)) rb += nr * (uint32_t)rows.esz[k];
    const uint32_t dst = smem_addr(base) + (uint32_t)f.d * g.stage, fb = full(f.d);
    mbar_arrive_expect_tx(fb, vb + cb + 16u * (ns + 1) + rb);
    bulk_copy_g2s(dst + g.soff, A.rec + s0, 16u * (ns + 1), fb, pol);
    if (vb > 0) {
      bulk_copy_g2s(dst, A.val + b.slot, vb, fb, pol);
      bulk_copy_g2s(dst + g.coff, A.ix + ib, cb, fb, pol);
    }
#pragma unroll
    for (int k = 0; k < RING_MAX_ROWS; ++k)
      if (staged(k))
        bulk_copy_g2s(dst + g.roff[k], (const unsigned char*)rows.p[k] + r0 * rows.esz[k],
                      nr * (uint32_t)rows.esz[k], fb, pol);
  }
  // Every copy has landed before the CTA can end (consumers that gave up leave
  // stages unread).
  __device__ __forceinline__ void drain(const Fill& f) const {
    for (int k = f.issued > g.D ? f.issued - g.D : 0; k < f.issued; ++k)
      if (!mbar_wait_bounded(full(k % g.D), (uint32_t)(k / g.D) & 1u)) break;
  }

  // The producer warp: copies every tile of this CTA, a stage as soon as its
  // consumers have left it.
  __device__ __forceinline__ void produce(int* fail, int* status) {
    const uint64_t pol = l2_evict_first();
    Fill f;
    if constexpr (CHUNKED) {
      bool ok = true;
      for (int64_t c = blockIdx.x; ok && c < ch.n; c += gridDim.x) {
        const int64_t c0 = __ldg(ch.off + c), c1 = __ldg(ch.off + c + 1);
        if (!A.live(c0)) continue;  // consumers never see this chunk
        SliceRec b = load_rec(c0);
        int64_t r0 = __ldg(A.row0 + c0);
        for (int64_t s0 = c0; s0 < c1; s0 += g.tile) {
          const int64_t s1 = s0 + g.tile < c1 ? s0 + g.tile : c1;
          const SliceRec e = load_rec(s1);
          const int64_t r1 = __ldg(A.row0 + s1);
          ok = claim(f, fail, status);
          if (!ok) break;
          // whole groups of four rows around the tile's: 16-byte boundaries
          RingTile h;
          h.e0 = r0 & ~(int64_t)3;
          const int64_t e1 = (r1 + 3) & ~(int64_t)3;
          h.s0 = s0;
          h.r0 = r0;
          h.chunk = c;
          h.ns = (int32_t)(s1 - s0);
          h.rows = (int32_t)(r1 - r0);
          h.last = s1 == c1;
          h.pad = 0;
          if (lane == 0) *(RingTile*)(base + (size_t)f.d * g.stage + g.hoff) = h;
          const bool bulk = e1 <= A.n;
          fill(f, s0, (uint32_t)(s1 - s0), b, e, bulk, h.e0,
               (uint32_t)((bulk ? e1 : A.n) - h.e0), pol);
          advance(f);
          b = e;
          r0 = r1;
        }
      }
      if (ok && claim(f, fail, status)) {  // the end: an empty stage
        if (lane == 0) {
          ((RingTile*)(base + (size_t)f.d * g.stage + g.hoff))->ns = -1;
          mbar_arrive(full(f.d));
        }
        advance(f);
      }
    } else {
      int64_t tt = blockIdx.x;
      if (tt >= ntiles) return;
      // the next tile's bounds are loaded a tile ahead
      SliceRec b = load_rec(tt * g.tile), e = load_rec(tt * g.tile + g.tile);
      for (;;) {
        const int64_t nx = tt + gridDim.x;
        SliceRec nb = {0, 0}, ne = {0, 0};
        if (nx < ntiles) {
          nb = load_rec(nx * g.tile);
          ne = load_rec(nx * g.tile + g.tile);
        }
        if (!claim(f, fail, status)) break;
        const int64_t s0 = tt * g.tile, nr = A.n - s0 * 32;
        const uint32_t ns = (uint32_t)(A.nslices - s0 < g.tile ? A.nslices - s0 : g.tile);
        const bool bulk = nr >= 32 * g.tile;
        fill(f, s0, ns, b, e, bulk, s0 * 32, bulk ? 32u * (uint32_t)g.tile : (uint32_t)nr, pol);
        advance(f);
        tt = nx;
        if (tt >= ntiles) break;
        b = nb;
        e = ne;
      }
    }
    drain(f);
  }

  __device__ __forceinline__ bool more() const { return CHUNKED || t < ntiles; }

  // Waits for the next tile; false if the wait gave up.
  __device__ __forceinline__ bool wait() {
    if (!__all_sync(0xffffffffu, mbar_wait_bounded(full(stage), phase))) return false;
    st = base + (uint32_t)stage * g.stage;
    uint32_t ns, r0, rows_, e0 = 0;  // the tile: slices, first row, rows, first staged row
    if constexpr (CHUNKED) {
      const RingTile& h = *(const RingTile*)(st + g.hoff);
      ended = h.ns < 0;
      if (ended) return true;
      ns = (uint32_t)h.ns;
      r0 = (uint32_t)h.r0;
      rows_ = (uint32_t)h.rows;
      e0 = r0 - (uint32_t)h.e0;
      last = h.last != 0;
      chunk = h.chunk;
    } else {
      const uint32_t s0 = t * (uint32_t)g.tile;
      ns = (uint32_t)A.nslices - s0;
      r0 = s0 * 32;
      rows_ = (uint32_t)A.n - r0;
    }
    const int4* r = (const int4*)(st + g.soff);
    const int4 rb = r[0];
#pragma unroll
    for (int m = 0; m < SPW; ++m) {
      RingSlot<V>& o = slot[m];
      const uint32_t k = (uint32_t)warp * SPW + m;
      o.slice = k < ns;
      const uint32_t u = k * 32 + lane;
      o.i = r0 + u;
      o.j = e0 + u;
      o.has = u < rows_;
      if (o.slice) {  // low halves: differences within a tile
        const int4 rw = r[k], rn = r[k + 1];
        o.vals = (const V*)(st + (uint32_t)(rw.x - rb.x) * (uint32_t)sizeof(V)) + lane;
        o.ixb = (const int32_t*)(st + (g.coff + (uint32_t)((rw.z & ~3) - (rb.z & ~3))));
        o.wm = (rn.x - rw.x) >> 5 << 2 | (rw.z & 3);
      }
    }
    return true;
  }

  // this lane's entry (row of slot m) of per-row vector k, of type X
  template <typename X>
  __device__ __forceinline__ X row(int k, int m = 0) const {
    return ((const X*)(st + g.roff[k]))[slot[m].j];
  }

  // every lane is done with the stage
  __device__ __forceinline__ void release() {
    __syncwarp();
    if (lane == 0) mbar_arrive(empty(stage));
    t += gridDim.x;
    if (++stage == g.D) {
      stage = 0;
      phase ^= 1u;
    }
  }
};

// Columns k0 .. k0 + N - 1 of this lane's row in the current stage, by the
// slice's coding, as places from `v` (k0 is a multiple of 4; index blocks start
// at 16 bytes and hold whole groups of four offsets or bases).
template <int N>
__device__ __forceinline__ void ix_heads(const int32_t* c, int k0, int32_t (&o)[N]) {
  const int4* q = (const int4*)(c + k0);
#pragma unroll
  for (int u = 0; u < N; u += 4) {
    const int4 h = q[u / 4];
    o[u] = h.x;
    if (u + 1 < N) o[u + 1 < N ? u + 1 : 0] = h.y;
    if (u + 2 < N) o[u + 2 < N ? u + 2 : 0] = h.z;
    if (u + 3 < N) o[u + 3 < N ? u + 3 : 0] = h.w;
  }
}
template <typename X>
struct IxPlain {
  const X* v;
  const int32_t* c;
  template <int N>
  __device__ __forceinline__ void load(int k0, int32_t (&o)[N]) const {
#pragma unroll
    for (int u = 0; u < N; ++u) o[u] = c[(k0 + u) * 32];
  }
};
template <typename X>
struct IxDelta {
  const X* v;
  const int32_t* base;
  const uint16_t* d;
  template <int N>
  __device__ __forceinline__ void load(int k0, int32_t (&o)[N]) const {
    ix_heads<N>(base, k0, o);
#pragma unroll
    for (int u = 0; u < N; ++u) o[u] += (int)d[(k0 + u) * 32];
  }
};
template <typename X>
struct IxOffset {
  const X* v;  // (at this lane's row)
  const int32_t* off;
  template <int N>
  __device__ __forceinline__ void load(int k0, int32_t (&o)[N]) const {
    ix_heads<N>(off, k0, o);
  }
};
template <typename X>
struct IxClamp {
  const X* v;
  const int32_t* off;
  int32_t i, last;  // the clamp only ever moves padding
  template <int N>
  __device__ __forceinline__ void load(int k0, int32_t (&o)[N]) const {
    ix_heads<N>(off, k0, o);
#pragma unroll
    for (int u = 0; u < N; ++u) o[u] = min(max(i + o[u], 0), last);
  }
};

// acc + sum of a_k v[col_k] (NEG: acc - sum, by FMAs with the negated
// values) for k = k0 .. k0 + N - 1, k ascending, of the rows in NS slices: all
// gathers issue together, then the FMAs follow in order.  Exactly N FMAs a row:
// on GB300's FP64 pipe a predicated-off FMA would still cost its cycles.
template <int N, bool NEG, int NS, typename T, typename S, typename I>
__device__ __forceinline__ void ring_chunk(const S* sl, const I (&ix)[NS], int k0, T* acc) {
  T x[NS][N];
#pragma unroll
  for (int m = 0; m < NS; ++m) {
    int32_t o[N];
    ix[m].load(k0, o);
#pragma unroll
    for (int u = 0; u < N; ++u) x[m][u] = to_f(__ldg(ix[m].v + o[u]), T(0));
  }
#pragma unroll
  for (int m = 0; m < NS; ++m)
#pragma unroll
    for (int u = 0; u < N; ++u) {
      const T a = to_f(sl[m].val(k0 + u), T(0));
      acc[m] = fma(NEG ? -a : a, x[m][u], acc[m]);
    }
}

// Chunks of 8 and one remainder chunk of the exact length (w is
// warp-uniform).
template <bool NEG, int NS, typename T, typename S, typename I>
__device__ __forceinline__ void ring_chunks(const S* sl, const I (&ix)[NS], int w, T* acc) {
  int k0 = 0;
  for (; k0 + 8 <= w; k0 += 8) ring_chunk<8, NEG, NS>(sl, ix, k0, acc);
  switch (w - k0) {
    case 1: ring_chunk<1, NEG, NS>(sl, ix, k0, acc); break;
    case 2: ring_chunk<2, NEG, NS>(sl, ix, k0, acc); break;
    case 3: ring_chunk<3, NEG, NS>(sl, ix, k0, acc); break;
    case 4: ring_chunk<4, NEG, NS>(sl, ix, k0, acc); break;
    case 5: ring_chunk<5, NEG, NS>(sl, ix, k0, acc); break;
    case 6: ring_chunk<6, NEG, NS>(sl, ix, k0, acc); break;
    case 7: ring_chunk<7, NEG, NS>(sl, ix, k0, acc); break;
    default: break;
  }
}

// acc[m] + sum_k a_k v[col_k] (NEG: - sum) over the entries of this lane's row
// in each of NS slices of one width and coding, k ascending (the per-lane
// kernels' order).
template <bool NEG, int NS, typename T, typename S, typename X>
__device__ __forceinline__ void ring_slots_sum(const S* sl, int ncols, int lane, const X* v,
                                               T* acc) {
  const int w = sl[0].wm >> 2;
  switch (sl[0].wm & 3) {
    case IX_OFFSET: {
      IxOffset<X> ix[NS];
#pragma unroll
      for (int m = 0; m < NS; ++m) ix[m] = IxOffset<X>{v + sl[m].i, sl[m].ixb};
      return ring_chunks<NEG, NS>(sl, ix, w, acc);
    }
    case IX_CLAMP: {
      IxClamp<X> ix[NS];
#pragma unroll
      for (int m = 0; m < NS; ++m)
        ix[m] = IxClamp<X>{v, sl[m].ixb, (int32_t)sl[m].i, ncols - 1};
      return ring_chunks<NEG, NS>(sl, ix, w, acc);
    }
    case IX_DELTA: {
      IxDelta<X> ix[NS];
#pragma unroll
      for (int m = 0; m < NS; ++m)
        ix[m] = IxDelta<X>{v, sl[m].ixb,
                           (const uint16_t*)(sl[m].ixb + ((w + 3) & ~3)) + lane};
      return ring_chunks<NEG, NS>(sl, ix, w, acc);
    }
    default: {
      IxPlain<X> ix[NS];
#pragma unroll
      for (int m = 0; m < NS; ++m) ix[m] = IxPlain<X>{v, sl[m].ixb + lane};
      return ring_chunks<NEG, NS>(sl, ix, w, acc);
    }
  }
}

// The same over this warp's slices of the tile (with one slice a warp the caller
// has looked that there is one); two of one width and coding (in
// a stencil matrix nearly always) with all their gathers in flight at once.
template <bool NEG, typename T, typename V, bool CH, int SPW, typename X>
__device__ __forceinline__ void ring_row_sums(const TileRing<V, CH, SPW>& ring, const X* v,
                                              T (&acc)[SPW]) {
  const int nc = ring.A.ncols;
  if constexpr (SPW == 2) {
    if (ring.slot[1].slice && ring.slot[0].wm == ring.slot[1].wm) {
      ring_slots_sum<NEG, 2>(ring.slot, nc, ring.lane, v, acc);
      return;
    }
  }
#pragma unroll
  for (int m = 0; m < SPW; ++m)
    if (SPW == 1 || ring.slot[m].slice)
      ring_slots_sum<NEG, 1>(ring.slot + m, nc, ring.lane, v, acc + m);
}

// A bounded wait gave up: the handle's sticky flag, and the PCG status
// (if given) so a device-side loop stops.
__device__ __forceinline__ void ring_fail(int* fail, int* status) {
  atomicExch(fail, 1);
  if (status) atomicCAS(status, 0, AMG_ERR_DEVICE_CHECK);
}

// Geometry for streaming M (values of `vbytes` bytes) with the ring, or
// D = 0 when M does not qualify.  stages: 2..RING_MAX_STAGES, or 0 for the
// default.  dots: the kernel also sums dot products over its grid.  chunked:
// for batched systems (M.row0), which only chunked kernels take.  The grid is
// left to ring_prepare.  pairs: for kernels with two slices a warp (FP32 values).
// Host code.
RingGeom ring_plan(const Sell& M, int vbytes, int stages, const RingRows& rows,
                   bool dots = false, bool chunked = false, bool pairs = false);

// Prepares kernel `fn` for a launch with geometry g on the current device
// (shared-memory limit, once per device and kernel) and sets g.grid to the
// CTAs that are co-resident (occupancy query), at most `work` (tiles or chunks).
// Host code.
int ring_prepare(const void* fn, RingGeom& g, int64_t work, int num_sms);
inline int64_t ring_tiles(const RingGeom& g, const Sell& M) {
  return (M.nslices + g.tile - 1) / g.tile;
}

}  // namespace amg
