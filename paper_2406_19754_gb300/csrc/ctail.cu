// The small levels of the V-cycle in one thread-block cluster, resident in
// shared memory.
//
// A level of a few thousand rows costs a launch per step whatever its size
// (3 to 8 us), and the one-CTA launch of tail.cu walks its levels through
// dependent L2 round trips, 4 to 6 us a step: 28.6 us of each 75 us iteration
// on 32^3 Poisson, 71 of 190 us of a V-cycle with 664-, 338-, 242- and 214-row
// levels.  Here one cluster of 16 CTAs holds the levels from `lt` down: every
// CTA owns a contiguous power-of-two range of rows of each level, copies its
// part of the operators into its shared memory at the start (one bulk copy a
// level from an image laid out at setup), and keeps the level vectors there.
// A gather reads the owner's shared memory (ld.shared::cluster), and steps are
// separated by the hardware cluster barrier, so no step waits for L2.
//
// Rows run the same operations in the same order as the one-launch-per-step
// kernels (smooth.cuh: pre_slice, restrict_sum, post_slice, sweep_slice,
// coarse_block_solve, coarse_pcg_cta), so results agree bit for bit.
//
// Eligible levels (ct_init): one system, slices of 32 rows with one thread
// per row, at most CT_MAX_ROWS rows (16-bit columns), and together with the
// coarsest solve at most the shared memory of the cluster.
//
// Waits: the image copies complete on one mbarrier a level, waited for with a
// time limit; a wait that gives up sets the handle's failure flag and the
// kernel goes on (its result is then reported as AMG_ERR_DEVICE_CHECK), so
// every CTA reaches every cluster barrier: their number depends on the launch
// parameters alone.
#include <string.h>

#include <algorithm>

#include "cluster.cuh"
#include "ring.cuh"
#include "smooth.cuh"

namespace amg {

namespace {

constexpr int CT_CTAS = 16;
constexpr int CT_THREADS = 512;
constexpr int CT_WARPS = CT_THREADS / 32;
constexpr int CT_MAX_LEVELS = 12;
constexpr int CT_MAX_ROWS = 65534;        // 0xFFFF marks an empty member slot
constexpr int CT_PCG_ROWS = CT_THREADS;   // PCG coarsest solve: one row a thread
constexpr size_t CT_SMEM = 226 * 1024;    // of 227 KB: static arrays take the rest
constexpr uint16_t CT_NONE = 0xFFFF;

// One CTA's image of a level: offsets in bytes, the same for every CTA.
struct CtImage {
  uint32_t spA, spP, valA, colA, valP, colP, s, agg, mem, bytes;
};

struct CtLevel {
  int n, nc, shift, shift_c;  // rows of CTA c: [c << shift, (c + 1) << shift)
  int stride, vstore;
  int nu;
  CtImage im;
  const unsigned char* img;  // CT_CTAS images, im.bytes apart
  // shared-memory offsets: the image, and this CTA's entries of the vectors
  uint32_t o_img, o_b, o_x, o_r, o_r2, o_xp;
};

struct CtParams {
  int nlev;
  int nco, shift_co;
  uint32_t o_cimg, o_cb, o_cx, o_y, o_full, o_bar;
  const unsigned char* cimg;
  uint32_t cbytes, c_second;  // image bytes; offset of L^-T (or of the PCG's parts)
  int pcg, pcg_maxit;
  double pcg_tol;
  uint32_t c_val, c_col, c_sinv;
  // the top level's input: b, or the restriction of the level above's residual
  const void* b;
  const int32_t* members;
  int rstride;
  const void* rfine;
  void* x;
  int* fail;
  int* status;
  CtLevel lv[CT_MAX_LEVELS];
};

// A level vector spread over the cluster: entry j at `base` + (j mod 2^shift)
// in the shared memory of CTA j >> shift.
template <typename T>
struct CtVec {
  uint32_t base;
  int shift;
  __device__ __forceinline__ uint32_t addr(uint32_t j) const {
    return map_rank(base + (j & ((1u << shift) - 1u)) * (uint32_t)sizeof(T), j >> shift);
  }
  __device__ __forceinline__ T operator[](uint32_t j) const {
    return ld_cluster(addr(j), T(0));
  }
};

// init + sum_k a_k v[col_k] (NEG: init - sum) over local row lr, k ascending.
template <typename T, bool NEG, typename V>
__device__ __forceinline__ T ct_row(const int32_t* sp, const V* val, const uint16_t* col, int lr,
                                    const CtVec<T>& v, T init) {
  const int s0 = sp[lr >> 5], w = (sp[(lr >> 5) + 1] - s0) >> 5;
  const V* a = val + s0 + (lr & 31);
  const uint16_t* c = col + s0 + (lr & 31);
  T acc = init;
  int k = 0;
  for (; k + 4 <= w; k += 4) {
    uint32_t j[4];
    T x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) j[u] = c[(k + u) * 32];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = v[j[u]];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const T e = to_f(a[(k + u) * 32], T(0));
      acc = fma(NEG ? -e : e, x[u], acc);
    }
  }
  T x[3];
#pragma unroll
  for (int u = 0; u < 3; ++u)
    if (k + u < w) x[u] = v[c[(k + u) * 32]];
#pragma unroll
  for (int u = 0; u < 3; ++u)
    if (k + u < w) {
      const T e = to_f(a[(k + u) * 32], T(0));
      acc = fma(NEG ? -e : e, x[u], acc);
    }
  return acc;
}

// This CTA's rows of one level.
template <typename T>
struct CtRows {
  const CtLevel& L;
  unsigned char* sm;
  uint32_t smb;  // shared address of sm
  int r0, rows;  // first row and number of rows here
  __device__ __forceinline__ CtRows(const CtLevel& L_, unsigned char* sm_, int rank)
      : L(L_), sm(sm_), smb(smem_addr(sm_)) {
    r0 = rank << L.shift;
    rows = min(max(L.n - r0, 0), 1 << L.shift);
  }
  template <typename X>
  __device__ __forceinline__ X* at(uint32_t off) const {
    return (X*)(sm + off);
  }
  template <typename X>
  __device__ __forceinline__ const X* im(uint32_t off) const {
    return (const X*)(sm + L.o_img + off);
  }
  __device__ __forceinline__ CtVec<T> vec(uint32_t off) const { return {smb + off, L.shift}; }

  template <typename V>
  __device__ __forceinline__ void pre() const {
    const T* b = at<T>(L.o_b);
    T* r = at<T>(L.o_r);
    const CtVec<T> bv = vec(L.o_b);
    for (int lr = threadIdx.x; lr < rows; lr += CT_THREADS)
      r[lr] = ct_row<T, true>(im<int32_t>(L.im.spA), im<V>(L.im.valA), im<uint16_t>(L.im.colA),
                              lr, bv, b[lr]);
  }
  template <typename V>
  __device__ __forceinline__ void sweep(bool pre, uint32_t o_in, uint32_t o_out, bool first) const {
    const T* r = at<T>(o_in);
    T* ro = at<T>(o_out);
    T* x = at<T>(pre ? L.o_xp : L.o_x);
    const T* s = im<T>(L.im.s);
    const T* b = at<T>(L.o_b);
    const CtVec<T> rv = vec(o_in);
    for (int lr = threadIdx.x; lr < rows; lr += CT_THREADS) {
      const T acc = ct_row<T, false>(im<int32_t>(L.im.spA), im<V>(L.im.valA),
                                     im<uint16_t>(L.im.colA), lr, rv, T(0));
      const T ri = r[lr], rn = ri - acc, si = s[lr];
      ro[lr] = rn;
      if (pre) {
        const T xi = first ? si * b[lr] : x[lr];
        x[lr] = sweep_pre_x(xi, si, ri);
      } else {
        x[lr] = sweep_post_y(x[lr], si, rn);
      }
    }
  }
  // o_xc: the next level's x; xg: the level's global x (top level), or null
  template <typename V>
  __device__ __forceinline__ void post(uint32_t o_r, uint32_t o_e, uint32_t o_xc, T* xg) const {
    const T* b = at<T>(L.o_b);
    const T* r = at<T>(o_r);
    T* x = at<T>(L.o_x);
    const T* s = im<T>(L.im.s);
    const uint16_t* agg = im<uint16_t>(L.im.agg);
    const CtVec<T> xc{smb + o_xc, L.shift_c};
    const bool ms = L.nu > 1;
    for (int lr = threadIdx.x; lr < rows; lr += CT_THREADS) {
      const T xci = xc[agg[lr]], si = s[lr];
      T z;
      if (!ms) {
        const T acc = ct_row<T, true>(im<int32_t>(L.im.spP), im<V>(L.im.valP),
                                      im<uint16_t>(L.im.colP), lr, xc, b[lr] + r[lr]);
        z = fma(si, acc, xci);
      } else {
        const T acc = ct_row<T, false>(im<int32_t>(L.im.spP), im<V>(L.im.valP),
                                       im<uint16_t>(L.im.colP), lr, xc, T(0));
        const T yi = at<T>(L.o_xp)[lr] + xci;
        const T ei = r[lr] - acc;
        z = fma(si, ei, yi);
        at<T>(o_e)[lr] = ei;
      }
      x[lr] = z;
      if (xg) xg[r0 + lr] = z;
    }
  }
  // b_{l+1} on this CTA's rows of the next level
  __device__ __forceinline__ void restrict_to(uint32_t o_r, uint32_t o_bc, int rank) const {
    const int c0 = rank << L.shift_c, rc = min(max(L.nc - c0, 0), 1 << L.shift_c);
    const uint16_t* mem = im<uint16_t>(L.im.mem);
    const CtVec<T> rv = vec(o_r);
    T* bc = at<T>(o_bc);
    for (int I = threadIdx.x; I < rc; I += CT_THREADS) {
      const uint16_t* m = mem + I * L.stride;
      T acc = rv[m[0]];
      for (int k = 1; k < L.stride; ++k) {
        if (m[k] == CT_NONE) break;
        acc = acc + rv[m[k]];
      }
      bc[I] = acc;
    }
  }
};

#define CT_BY_VALUE(L, ...)                                       \
  do if constexpr (sizeof(T) == 8) {                              \
    using V = double;                                             \
    __VA_ARGS__;                                                  \
  } else if ((L).vstore == VAL_BF16) {                            \
    using V = __nv_bfloat16;                                      \
    __VA_ARGS__;                                                  \
  } else {                                                        \
    using V = float;                                              \
    __VA_ARGS__;                                                  \
  } while (0)

// x = L^-T (L^-1 b): row i of both factors sits in CTA i mod 16 (rows of all
// lengths everywhere), one warp per row, summed as coarse_block_solve does.  Runs
// after a wait that gave up too: its places come from P alone, and it holds a
// cluster barrier.
template <typename T>
__device__ void ct_cholesky(const CtParams& P, unsigned char* sm, int rank) {
  const uint32_t smb = smem_addr(sm);
  const int n = P.nco, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double* full = (double*)(sm + P.o_full);
  double* y = (double*)(sm + P.o_y);
  const double* Li = (const double*)(sm + P.o_cimg);
  const double* LT = (const double*)(sm + P.o_cimg + P.c_second);
  const CtVec<T> bv{smb + P.o_cb, P.shift_co};
  for (int i = threadIdx.x; i < n; i += CT_THREADS) full[i] = (double)bv[i];
  __syncthreads();
  for (int q = warp; rank + CT_CTAS * q < n; q += CT_WARPS) {
    const int i = rank + CT_CTAS * q;
    const double* row = Li + q * (rank + 1) + CT_CTAS * (q * (q - 1) / 2);
    double acc = 0.0;
    for (int k = lane; k <= i; k += 32) acc = fma(row[k], full[k], acc);
    acc = warp_sum(acc);
    if (lane == 0) y[q] = acc;
  }
  cluster_barrier();
  for (int i = threadIdx.x; i < n; i += CT_THREADS)
    full[i] = ld_cluster(map_rank(smb + P.o_y + 8u * (uint32_t)(i / CT_CTAS), i % CT_CTAS), 0.0);
  __syncthreads();
  const CtVec<T> xv{smb + P.o_cx, P.shift_co};
  for (int q = warp; rank + CT_CTAS * q < n; q += CT_WARPS) {
    const int k = rank + CT_CTAS * q;
    const double* row = LT + q * (n - rank) - CT_CTAS * (q * (q - 1) / 2) - k;
    double acc = 0.0;
    for (int i = k + lane; i < n; i += 32) acc = fma(row[i], full[i], acc);
    acc = warp_sum(acc);
    if (lane == 0) st_cluster(xv.addr(k), (T)acc);
  }
}

// Sums over the block's n rows (one per thread) by coarse_pcg_cta's tree: the
// lanes of each warp, then the warps; f turns the sums into what every thread
// reads back from `out`.  Warps without rows would only add zeros and leave
// their part out, and one thread divides: sixteen warps' shuffled additions
// and divisions took the SM's FP64 pipe (16 clocks a warp instruction) longer
// than the rest of an iteration on 33 rows.
template <int NV, typename F>
__device__ __forceinline__ void ct_sum(double (&t)[NV], int n, double (*part)[CT_WARPS],
                                       double* out, F f) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (32 * warp < n) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      t[v] = warp_sum(t[v]);
      if (lane == 0) part[v][warp] = t[v];
    }
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int v = 0; v < NV; ++v) t[v] = warp_sum(32 * lane < n ? part[v][lane] : 0.0);
    if (lane == 0) f(t, out);
  }
  __syncthreads();
}

// PCG with the l1-Jacobi preconditioner on the coarsest level, by CTA 0 with
// one row per thread (coarse_pcg_cta's arithmetic; rows <= CT_PCG_ROWS).
template <typename T>
__device__ void ct_pcg(const CtParams& P, unsigned char* sm) {
  // two sets: a set is rewritten only after the other's sums were read
  __shared__ double part[2][2][CT_WARPS], out[2][3];
  const uint32_t smb = smem_addr(sm);
  const int n = P.nco, i = threadIdx.x;
  const bool has = i < n;
  double* p = (double*)(sm + P.o_full);
  const int32_t* sp = (const int32_t*)(sm + P.o_cimg);
  const double* val = (const double*)(sm + P.o_cimg + P.c_val);
  const uint16_t* col = (const uint16_t*)(sm + P.o_cimg + P.c_col);
  const double si = has ? ((const double*)(sm + P.o_cimg + P.c_sinv))[i] : 0.0;
  const CtVec<T> bv{smb + P.o_cb, P.shift_co};
  double x = 0.0, r = has ? (double)bv[i] : 0.0, z = 0.0;
  double t[1] = {has ? r * r : 0.0};
  ct_sum<1>(t, n, part[0], out[0], [](const double* v, double* o) { o[0] = sqrt(v[0]); });
  const double bnorm = out[0][0];
  if (bnorm > 0.0) {
    z = si * r;
    if (has) p[i] = z;
    t[0] = has ? r * z : 0.0;
    ct_sum<1>(t, n, part[1], out[1], [](const double* v, double* o) { o[0] = v[0]; });
    double rz = out[1][0];
    for (int k = 0; k < P.pcg_maxit; ++k) {
      double q = 0.0;
      if (has) {
        const int s0 = sp[i >> 5], w = (sp[(i >> 5) + 1] - s0) >> 5;
        const double* a = val + s0 + (i & 31);
        const uint16_t* c = col + s0 + (i & 31);
#pragma unroll 4
        for (int e = 0; e < w; ++e) q = fma(a[e * 32], p[c[e * 32]], q);
      }
      t[0] = has ? p[i] * q : 0.0;
      ct_sum<1>(t, n, part[0], out[0], [rz](const double* v, double* o) {
        o[0] = v[0];
        o[1] = rz / v[0];
      });
      if (!(out[0][0] > 0.0)) break;
      const double alpha = out[0][1];
      double d[2] = {0.0, 0.0};
      if (has) {
        x = x + alpha * p[i];
        r = r - alpha * q;
        z = si * r;
        d[0] += r * r;
        d[1] += r * z;
      }
      ct_sum<2>(d, n, part[1], out[1],
                [rz, tol = P.pcg_tol, bnorm](const double* v, double* o) {
                  o[0] = v[1];
                  o[1] = v[1] / rz;
                  o[2] = sqrt(v[0]) <= tol * bnorm ? 1.0 : 0.0;
                });
      if (out[1][2] != 0.0) break;
      rz = out[1][0];
      const double beta = out[1][1];
      if (has) p[i] = z + beta * p[i];
      __syncthreads();
    }
  }
  if (has) st_cluster(CtVec<T>{smb + P.o_cx, P.shift_co}.addr(i), bnorm > 0.0 ? (T)x : T(0));
}

template <typename T>
__global__ void __launch_bounds__(CT_THREADS, 1)
    k_cluster_tail(const __grid_constant__ CtParams P) {
  extern __shared__ __align__(128) unsigned char sm[];
  const int rank = (int)cluster_rank();
  const uint32_t bar = smem_addr(sm) + P.o_bar;
  if (threadIdx.x == 0) {
    for (int l = 0; l <= P.nlev; ++l) mbar_init(bar + 8u * l, 1);
    mbar_init_fence();
    uint64_t pol;  // read once per V-cycle, from L2 or DRAM
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    for (int l = 0; l < P.nlev; ++l) {
      const CtLevel& L = P.lv[l];
      mbar_arrive_expect_tx(bar + 8u * l, L.im.bytes);
      bulk_copy_g2s(smem_addr(sm) + L.o_img, L.img + (size_t)rank * L.im.bytes, L.im.bytes,
                    bar + 8u * l, pol);
    }
    if (P.pcg == 0 || rank == 0) {
      mbar_arrive_expect_tx(bar + 8u * P.nlev, P.cbytes);
      bulk_copy_g2s(smem_addr(sm) + P.o_cimg, P.cimg + (size_t)rank * P.cbytes, P.cbytes,
                    bar + 8u * P.nlev, pol);
    }
  }
  // this CTA's part of the top level's b
  {
    const CtLevel& L = P.lv[0];
    const int r0 = rank << L.shift, rows = min(max(L.n - r0, 0), 1 << L.shift);
    T* b = (T*)(sm + L.o_b);
    for (int i = threadIdx.x; i < rows; i += CT_THREADS)
      b[i] = P.rfine ? restrict_sum<LdRO>(P.members + (int64_t)(r0 + i) * P.rstride, P.rstride,
                                          (const T*)P.rfine)
                     : __ldg((const T*)P.b + r0 + i);
  }
  bool ok = true;
  unsigned cur = 0;  // bit l: the residual of level l is in r2
  cluster_barrier();
  for (int l = 0; l < P.nlev; ++l) {
    const CtLevel& L = P.lv[l];
    const CtRows<T> R(L, sm, rank);
    ok = __syncthreads_and(mbar_wait_bounded(bar + 8u * l, 0) && ok);
    if (ok) CT_BY_VALUE(L, R.template pre<V>());
    cluster_barrier();
    bool c = false;
    for (int k = 2; k <= L.nu; ++k) {
      const uint32_t from = c ? L.o_r2 : L.o_r, to = c ? L.o_r : L.o_r2;
      if (ok) CT_BY_VALUE(L, R.template sweep<V>(true, from, to, k == 2));
      cluster_barrier();
      c = !c;
    }
    if (c) cur |= 1u << l;
    if (ok) R.restrict_to(c ? L.o_r2 : L.o_r, l + 1 < P.nlev ? P.lv[l + 1].o_b : P.o_cb, rank);
    cluster_barrier();
  }
  if (P.pcg == 0 || rank == 0)
    ok = __syncthreads_and(mbar_wait_bounded(bar + 8u * P.nlev, 0) && ok);
  if (P.pcg == 0)
    ct_cholesky<T>(P, sm, rank);
  else if (rank == 0 && ok)
    ct_pcg<T>(P, sm);
  cluster_barrier();
  for (int l = P.nlev - 1; l >= 0; --l) {
    const CtLevel& L = P.lv[l];
    const CtRows<T> R(L, sm, rank);
    bool c = (cur >> l) & 1u;
    const uint32_t o_xc = l + 1 < P.nlev ? P.lv[l + 1].o_x : P.o_cx;
    T* xg = l == 0 && L.nu == 1 ? (T*)P.x : nullptr;
    if (ok) CT_BY_VALUE(L, R.template post<V>(c ? L.o_r2 : L.o_r, c ? L.o_r : L.o_r2, o_xc, xg));
    if (L.nu > 1) {
      c = !c;
      for (int k = 2; k <= L.nu; ++k) {
        cluster_barrier();
        const uint32_t from = c ? L.o_r2 : L.o_r, to = c ? L.o_r : L.o_r2;
        if (ok) CT_BY_VALUE(L, R.template sweep<V>(false, from, to, false));
        c = !c;
      }
      if (l == 0) {
        const T* x = (const T*)(sm + L.o_x);
        for (int i = threadIdx.x; i < R.rows; i += CT_THREADS) ((T*)P.x)[R.r0 + i] = x[i];
      }
    }
    cluster_barrier();  // also: no CTA ends while another reads its memory
  }
  if (!ok && threadIdx.x == 0) {
    ring_fail(P.fail, P.status);
    for (int l = 0; l < P.nlev; ++l) mbar_wait_bounded(bar + 8u * l, 0);
    if (P.pcg == 0 || rank == 0) mbar_wait_bounded(bar + 8u * P.nlev, 0);
  }
}

// ------------------------------------------------------------------ images

// Slots of the largest CTA's rows: out[0] of A, out[1] of AP.
__global__ void k_ct_slots(const int64_t* spA, int64_t nslA, const int64_t* spP, int64_t nslP,
                           int slices, int* out) {
  const int c = threadIdx.x;
  if (c >= CT_CTAS) return;
  auto at = [](const int64_t* sp, int64_t nsl, int64_t s) { return sp[s < nsl ? s : nsl]; };
  const int64_t s0 = (int64_t)c * slices, s1 = s0 + slices;
  atomicMax(out, (int)(at(spA, nslA, s1) - at(spA, nslA, s0)));
  if (spP) atomicMax(out + 1, (int)(at(spP, nslP, s1) - at(spP, nslP, s0)));
}

struct CtSrc {
  const int64_t* sp;
  int64_t nsl;
  const int32_t* col;
  const void* val;
};

template <typename X>
__device__ void ct_copy_rows(unsigned char* im, uint32_t o_sp, uint32_t o_val, uint32_t o_col,
                             const CtSrc& S, int64_t s0, int slices) {
  int32_t* sp = (int32_t*)(im + o_sp);
  const int64_t base = S.sp[s0 < S.nsl ? s0 : S.nsl];
  for (int q = threadIdx.x; q <= slices; q += blockDim.x)
    sp[q] = (int32_t)(S.sp[s0 + q < S.nsl ? s0 + q : S.nsl] - base);
  const int64_t end = S.sp[s0 + slices < S.nsl ? s0 + slices : S.nsl];
  X* val = (X*)(im + o_val);
  uint16_t* col = (uint16_t*)(im + o_col);
  for (int64_t e = base + threadIdx.x; e < end; e += blockDim.x) {
    val[e - base] = ((const X*)S.val)[e];
    col[e - base] = (uint16_t)S.col[e];
  }
}

__device__ void ct_copy_any(int vbytes, unsigned char* im, uint32_t o_sp, uint32_t o_val,
                            uint32_t o_col, const CtSrc& S, int64_t s0, int slices) {
  if (vbytes == 8)
    ct_copy_rows<double>(im, o_sp, o_val, o_col, S, s0, slices);
  else if (vbytes == 4)
    ct_copy_rows<float>(im, o_sp, o_val, o_col, S, s0, slices);
  else
    ct_copy_rows<uint16_t>(im, o_sp, o_val, o_col, S, s0, slices);
}

// CTA c writes image c of a level.
__global__ void k_ct_image(unsigned char* img, CtImage I, CtSrc A, CtSrc AP, int vbytes, int n,
                           int nc, int shift, int shift_c, int stride, const double* s64,
                           const float* s32, const int32_t* agg, const int32_t* members) {
  const int c = blockIdx.x, slices = (1 << shift) >> 5;
  unsigned char* im = img + (size_t)c * I.bytes;
  ct_copy_any(vbytes, im, I.spA, I.valA, I.colA, A, (int64_t)c * slices, slices);
  ct_copy_any(vbytes, im, I.spP, I.valP, I.colP, AP, (int64_t)c * slices, slices);
  const int r0 = c << shift;
  for (int q = threadIdx.x; q < (1 << shift) && r0 + q < n; q += blockDim.x) {
    if (s32)
      ((float*)(im + I.s))[q] = s32[r0 + q];
    else
      ((double*)(im + I.s))[q] = s64[r0 + q];
    ((uint16_t*)(im + I.agg))[q] = (uint16_t)agg[r0 + q];
  }
  const int64_t c0 = (int64_t)c << shift_c, m = (int64_t)stride << shift_c;
  for (int64_t q = threadIdx.x; q < m && c0 * stride + q < (int64_t)nc * stride; q += blockDim.x) {
    const int32_t v = members[c0 * stride + q];
    ((uint16_t*)(im + I.mem))[q] = v < 0 ? CT_NONE : (uint16_t)v;
  }
}

// CTA c writes image c of the coarsest level's factors.
__global__ void k_ct_factor(unsigned char* img, uint32_t bytes, uint32_t second, int n,
                            const double* Li, const double* LT) {
  const int c = blockIdx.x;
  double* a = (double*)(img + (size_t)c * bytes);
  double* b = (double*)(img + (size_t)c * bytes + second);
  for (int q = 0; c + CT_CTAS * q < n; ++q) {
    const int i = c + CT_CTAS * q;
    double* ra = a + q * (c + 1) + CT_CTAS * (q * (q - 1) / 2);
    double* rb = b + q * (n - c) - CT_CTAS * (q * (q - 1) / 2) - i;
    for (int k = threadIdx.x; k <= i; k += blockDim.x) ra[k] = Li[(int64_t)i * n + k];
    for (int k = i + threadIdx.x; k < n; k += blockDim.x) rb[k] = LT[(int64_t)i * n + k];
  }
}

__global__ void k_ct_pcg_image(unsigned char* im, uint32_t o_val, uint32_t o_col, uint32_t o_sinv,
                               CtSrc A, int slices, int n, const double* sinv) {
  ct_copy_rows<double>(im, 0, o_val, o_col, A, 0, slices);
  for (int q = threadIdx.x; q < n; q += blockDim.x) ((double*)(im + o_sinv))[q] = sinv[q];
}

int row_shift(int64_t n) {
  int sh = 5;  // at least one slice a CTA
  while (((int64_t)CT_CTAS << sh) < n) ++sh;
  return sh;
}

size_t up16(size_t v) { return (v + 15) & ~(size_t)15; }

}  // namespace

// Images of the levels that fit, from the coarsest up; H->ct_start is the
// first level, or -1.
struct CtState {
  int start = -1, nl = 0;
  CtLevel lv[CT_MAX_LEVELS + 1];  // by distance from the coarsest level, nearest first
  CtParams base;                  // the coarsest level's part
  int count = 0;
};

template <typename T>
static const void* ct_fn() {
  return (const void*)k_cluster_tail<T>;
}

// Shared-memory offsets of a launch with the `m` levels nearest the coarsest;
// returns the bytes.
static size_t ct_layout(const CtState& S, int m, size_t vb, CtParams* P) {
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o = up16(o + bytes);
    return (uint32_t)at;
  };
  *P = S.base;
  P->nlev = m;
  P->o_bar = take(8 * (size_t)(m + 1));
  const size_t crow = (size_t)1 << S.base.shift_co;
  P->o_cb = take(vb * crow);
  P->o_cx = take(vb * crow);
  P->o_y = take(8 * (size_t)((S.base.nco + CT_CTAS - 1) / CT_CTAS));
  P->o_full = take(8 * (size_t)S.base.nco);
  P->o_cimg = take(S.base.cbytes);
  for (int k = 0; k < m; ++k) {
    CtLevel& L = P->lv[k];
    L = S.lv[m - 1 - k];
    const size_t rows = (size_t)1 << L.shift;
    L.o_b = take(vb * rows);
    L.o_x = take(vb * rows);
    L.o_r = take(vb * rows);
    if (L.nu > 1) {
      L.o_r2 = take(vb * rows);
      L.o_xp = take(vb * rows);
    }
    L.o_img = take(L.im.bytes);
  }
  return o;
}

int ct_init(amg_handle* H, cudaStream_t s) {
  ct_free(H);
  const int nl = (int)H->L.size();
  if (H->batched || H->opt.tail_rows <= 0 || H->opt.smooth_prolongator || nl < 3) return AMG_OK;
  const bool f32 = H->opt.precision == AMG_PREC_F32;
  const size_t vb = f32 ? 4 : 8;
  const Level& Lc = H->L[nl - 1];
  if (Lc.n > 1024 || H->nblk != 1) return AMG_OK;
  const bool pcg = H->opt.coarse_solver == 1;
  if (pcg && (Lc.n > CT_PCG_ROWS || Lc.A.C != 32 || Lc.A.tpr != 1)) return AMG_OK;
  auto fits_layout = [](const Sell& M) { return M.C == 32 && M.tpr == 1 && !M.row0; };
  int m = 0;  // candidate levels, nearest the coarsest first
  while (m < CT_MAX_LEVELS && nl - 2 - m >= 1) {
    const Level& L = H->L[nl - 2 - m];
    if (L.n > CT_MAX_ROWS || !fits_layout(L.A) || !fits_layout(L.AP) || L.nu > (1 << 28)) break;
    ++m;
  }
  if (m == 0) return AMG_OK;
  // a cluster of this size must be schedulable with the largest launch
  const void* fn = f32 ? ct_fn<float>() : ct_fn<double>();
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
          cudaSuccess ||
      cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CT_SMEM) !=
          cudaSuccess) {
    cudaGetLastError();
    return AMG_OK;
  }
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CT_CTAS;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(CT_CTAS);
  cfg.blockDim = dim3(CT_THREADS);
  cfg.dynamicSmemBytes = CT_SMEM;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) != cudaSuccess || clusters < 1) {
    cudaGetLastError();
    return AMG_OK;
  }
  Arena& ar = H->arena;
  int* d_slots = nullptr;
  AMG_TRY(ar.alloc_n(&d_slots, 2 * (CT_MAX_LEVELS + 1)));
  AMG_CUDA_TRY(cudaMemsetAsync(d_slots, 0, sizeof(int) * 2 * (CT_MAX_LEVELS + 1), s));
  for (int k = 0; k < m; ++k) {
    const Level& L = H->L[nl - 2 - k];
    k_ct_slots<<<1, 32, 0, s>>>(L.A.sliceptr, L.A.nslices, L.AP.sliceptr, L.AP.nslices,
                                (1 << row_shift(L.n)) >> 5, d_slots + 2 * k);
    AMG_LAUNCH_CHECK();
  }
  int slots[2 * (CT_MAX_LEVELS + 1)];
  AMG_CUDA_TRY(cudaMemcpyAsync(slots, d_slots, sizeof(slots), cudaMemcpyDeviceToHost, s));
  AMG_CUDA_TRY(cudaStreamSynchronize(s));
  ar.release(d_slots);
  CtState* S = new CtState();
  H->ct = S;
  CtParams& B = S->base;
  memset(&B, 0, sizeof(B));
  B.nco = (int)Lc.n;
  B.shift_co = row_shift(Lc.n);
  const int64_t n = Lc.n, cnt = (n + CT_CTAS - 1) / CT_CTAS;
  if (pcg) {
    size_t o = up16(4 * (size_t)(Lc.A.nslices + 1));
    B.c_val = (uint32_t)o;
    o = up16(o + 8 * (size_t)Lc.A.nnz_pad);
    B.c_col = (uint32_t)o;
    o = up16(o + 2 * (size_t)Lc.A.nnz_pad);
    B.c_sinv = (uint32_t)o;
    o = up16(o + 8 * (size_t)n);
    B.cbytes = (uint32_t)std::min<size_t>(o, 1u << 30);
    B.pcg = 1;
    B.pcg_maxit = H->opt.coarse_maxit;
    B.pcg_tol = H->opt.coarse_tol;
  } else {
    const size_t first = (size_t)(cnt * CT_CTAS + CT_CTAS * (cnt * (cnt - 1) / 2));
    const size_t second = (size_t)(cnt * n - CT_CTAS * (cnt * (cnt - 1) / 2));
    B.c_second = (uint32_t)up16(8 * first);
    B.cbytes = (uint32_t)(B.c_second + up16(8 * second));
  }
  for (int k = 0; k < m; ++k) {
    const int l = nl - 2 - k;
    const Level& L = H->L[l];
    CtLevel& D = S->lv[k];
    memset(&D, 0, sizeof(D));
    D.n = (int)L.n;
    D.nc = (int)L.nc;
    D.shift = row_shift(L.n);
    D.shift_c = row_shift(L.nc);
    D.stride = L.stride;
    D.vstore = L.vstore;
    D.nu = (int)L.nu;
    const size_t vs = L.vstore == VAL_F64 ? 8 : L.vstore == VAL_F32 ? 4 : 2;
    const size_t rows = (size_t)1 << D.shift;
    size_t o = 0;
    auto take = [&](size_t bytes) {
      const size_t at0 = o;
      o = up16(o + bytes);
      return (uint32_t)at0;
    };
    D.im.spA = take(4 * (rows / 32 + 1));
    D.im.spP = take(4 * (rows / 32 + 1));
    D.im.valA = take(vs * (size_t)slots[2 * k]);
    D.im.colA = take(2 * (size_t)slots[2 * k]);
    D.im.valP = take(vs * (size_t)slots[2 * k + 1]);
    D.im.colP = take(2 * (size_t)slots[2 * k + 1]);
    D.im.s = take(vb * rows);
    D.im.agg = take(2 * rows);
    D.im.mem = take(2 * (size_t)L.stride << D.shift_c);
    D.im.bytes = (uint32_t)std::min<size_t>(o, 1u << 30);
    CtParams P;
    if (ct_layout(*S, k + 1, vb, &P) > CT_SMEM) break;
    S->count = k + 1;
  }
  if (S->count == 0) {
    ct_free(H);
    return AMG_OK;
  }
  S->start = nl - 1 - S->count;
  unsigned char* cimg = nullptr;
  AMG_TRY(ar.alloc_n(&cimg, (int64_t)B.cbytes * CT_CTAS));
  B.cimg = cimg;
  AMG_CUDA_TRY(cudaMemsetAsync(cimg, 0, (size_t)B.cbytes * CT_CTAS, s));
  if (pcg)
    k_ct_pcg_image<<<1, 256, 0, s>>>(cimg, B.c_val, B.c_col, B.c_sinv,
                                     CtSrc{Lc.A.sliceptr, Lc.A.nslices, Lc.A.col, Lc.A.v64},
                                     (int)Lc.A.nslices, (int)n, Lc.s64);
  else
    k_ct_factor<<<CT_CTAS, 256, 0, s>>>(cimg, B.cbytes, B.c_second, (int)n, H->Linv, H->LinvT);
  AMG_LAUNCH_CHECK();
  for (int k = 0; k < S->count; ++k) {
    const Level& L = H->L[nl - 2 - k];
    CtLevel& D = S->lv[k];
    unsigned char* img = nullptr;
    AMG_TRY(ar.alloc_n(&img, (int64_t)D.im.bytes * CT_CTAS));
    AMG_CUDA_TRY(cudaMemsetAsync(img, 0, (size_t)D.im.bytes * CT_CTAS, s));
    D.img = img;
    const bool f64 = L.vstore == VAL_F64, b16 = L.vstore == VAL_BF16;
    const CtSrc A{L.A.sliceptr, L.A.nslices, L.A.col,
                  f64 ? (const void*)L.ah64 : b16 ? (const void*)L.ah16 : (const void*)L.ah32};
    const CtSrc AP{L.AP.sliceptr, L.AP.nslices, L.AP.col,
                   f64 ? (const void*)L.AP.v64
                       : b16 ? (const void*)L.AP.v16 : (const void*)L.AP.v32};
    k_ct_image<<<CT_CTAS, 512, 0, s>>>(img, D.im, A, AP, f64 ? 8 : b16 ? 2 : 4, D.n, D.nc,
                                       D.shift, D.shift_c, D.stride, f32 ? nullptr : L.s64,
                                       f32 ? L.s32 : nullptr, L.agg, L.members);
    AMG_LAUNCH_CHECK();
  }
  return AMG_OK;
}

void ct_free(amg_handle* H) {
  delete (CtState*)H->ct;  // the images belong to the arena
  H->ct = nullptr;
}

int ct_start(const amg_handle* H) {
  const CtState* S = (const CtState*)H->ct;
  return S ? S->start : -1;
}

template <typename T>
int ct_launch(const amg_handle* H, int lt, const T* rfine, cudaStream_t s) {
  const CtState* S = (const CtState*)H->ct;
  const int nl = (int)H->L.size();
  if (!S || lt < S->start || lt > nl - 2) return AMG_ERR_ARG;
  CtParams P;
  const size_t smem = ct_layout(*S, nl - 1 - lt, sizeof(T), &P);
  const Level& F = H->L[lt - 1];
  P.b = H->L[lt].b;
  P.x = H->L[lt].x;
  P.members = F.members;
  P.rstride = F.stride;
  P.rfine = rfine;
  P.fail = H->wait_fail;
  P.status = &H->sc->status;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CT_CTAS;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(CT_CTAS);
  cfg.blockDim = dim3(CT_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  AMG_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_cluster_tail<T>, P));
  return AMG_OK;
}

template int ct_launch<float>(const amg_handle*, int, const float*, cudaStream_t);
template int ct_launch<double>(const amg_handle*, int, const double*, cudaStream_t);

}  // namespace amg
