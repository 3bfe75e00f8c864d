// Two-grid error-reduction loss of the level-0 smoother weights and its
// gradient, the training signal for the learned smoother.
//
//   L = mean_j log(||E^K e0_j||_A / ||e0_j||_A) / K,
//   E = S (I - P A_c^-1 P^T A) S,   S = I - diag(s) A,  s_i = omega_i / d_i,
//
// with P the level-0 aggregate map and A_c the level-1 matrix (Sec. 2.3:
// Eq. amg with two levels, l1-Jacobi smoother).  A_c^-1 is applied by PCG
// preconditioned with the hierarchy of levels >= 1 (a second handle) to a
// relative residual of 1e-12, or exactly by Cholesky when level 1 is the
// coarsest.  The gradient comes from the adjoint pass: S and the coarse
// correction are linear, S^T = I - A diag(s) and
// (I - P A_c^-1 P^T A)^T = I - A P A_c^-1 P^T, run in reverse order over the
// stored forward states, with d(S x)_i / d s_i = -(A x)_i.  All FP64.
//
// Samples run in lockstep, up to TG_GROUP at a time (tg_group), so each coarse
// solve is one blocked PCG over the group's right-hand sides (columns): the inner
// hierarchy's levels are small (27,648 rows below a 48^3 problem) and an
// iteration is bound by its launches, whatever the number of columns.  One
// sample at a time, a 48^3 training step of 4 samples and 2 cycles ran 540
// inner iterations of 0.15 ms, 82 of its 98 ms.
#include <math.h>

#include <type_traits>
#include <vector>

#include "sellk.cuh"

namespace amg {

template <int TPR>
__global__ void __launch_bounds__(SELL_BLOCK, sell_blocks(TPR))
    k_tg_smooth(SellView<double> A, const double* __restrict__ s, const double* __restrict__ x,
                double* __restrict__ out, double* __restrict__ Ax) {
  const Lanes<TPR> ln;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t sl = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; sl < A.ngroups;
       sl += nw) {
    const double acc = sell_row<TPR, double>(A, sl, ln, [&](int j) { return __ldg(x + j); });
    const int64_t i = lane_row(A, sl, ln);
    if (i >= 0) {
      Ax[i] = acc;
      out[i] = x[i] - s[i] * acc;
    }
  }
}

enum { TG_PROLONG_SUB = 0, TG_PROLONG = 1, TG_SCALE_S = 2, TG_SUB = 3, TG_SBAR = 4,
       TG_SCALE = 5, TG_DOMEGA = 6 };

// Elementwise steps of the forward and adjoint passes.  The coarse vector of
// the prolongations is one column of a row-major block of `ld` columns.
template <int OP>
__global__ void k_tg_vec(int64_t n, const double* __restrict__ x, const double* __restrict__ w,
                         const int32_t* __restrict__ agg, const double* __restrict__ s,
                         double c, double* __restrict__ out, float* __restrict__ outf,
                         int64_t ld) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (OP == TG_PROLONG_SUB) out[i] = x[i] - w[agg[i] * ld];  // x - P y
    if (OP == TG_PROLONG) out[i] = w[agg[i] * ld];              // P y
    if (OP == TG_SCALE_S) out[i] = s[i] * x[i];            // diag(s) x
    if (OP == TG_SUB) out[i] = x[i] - w[i];
    if (OP == TG_SBAR) out[i] = out[i] - x[i] * w[i];      // sbar -= u o w
    if (OP == TG_SCALE) out[i] = c * x[i];
    if (OP == TG_DOMEGA) outf[i] = (float)(x[i] / w[i]);   // d L / d omega = sbar / d
  }
}

// g = P^T x: sum over each aggregate's members (ascending); g is one column
// of a row-major block of `ld` columns.
__global__ void k_tg_restrict(int64_t nc, int stride, const int32_t* __restrict__ members,
                              const double* __restrict__ x, double* __restrict__ g, int64_t ld) {
  for (int64_t I = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; I < nc;
       I += (int64_t)gridDim.x * blockDim.x) {
    const int32_t* m = members + I * stride;
    double acc = x[m[0]];
    for (int k = 1; k < stride && m[k] >= 0; ++k) acc = acc + x[m[k]];
    g[I * ld] = acc;
  }
}

struct DotEpi {
  double* dst;
  __device__ void operator()(double (&t)[1]) const { *dst = t[0]; }
};

__global__ void k_tg_dot(int64_t n, const double* __restrict__ x, const double* __restrict__ y,
                         Reduce red, double* dst) {
  double d[1] = {0.0};
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    d[0] += x[i] * y[i];
  grid_reduce<1>(d, red, DotEpi{dst});
}

constexpr int TG_GROUP = 8;

// Samples of the next group when `left` are left: an even number from four to
// TG_GROUP, else one, solved by itself.  The blocked solve of an odd number of
// columns takes its per-column kernels, and two columns cost it nearly as much as
// eight, while the single solve runs its loop on the device.  Two cycles of 24^3
// and 80^3 diffusion problems: one sample 5.6 and 22 ms; blocked 2 samples 18 and
// 77, 3 samples 65 and 373, 4 samples 16 and 80, 8 samples 16 and 95.
static int tg_group(int left, int most) {
  const int m = (left < most ? left : most) & ~1;
  return m >= 4 ? m : 1;
}

// Work vectors of a group of G samples: each entry of e .. ab, Ae[k], Ac[k]
// holds G fine vectors one after the other; g and y are nc x G row-major.
struct TgWs {
  int64_t n = 0, nc = 0;
  int K = 0, G = 0;
  double *e = nullptr, *a = nullptr, *c = nullptr, *t = nullptr, *t2 = nullptr, *sbar = nullptr;
  double *eb = nullptr, *cb = nullptr, *ab = nullptr;
  double *g = nullptr, *y = nullptr, *dots = nullptr;
  std::vector<double*> Ae, Ac;
  double* dots_host = nullptr;  // pinned
};

}  // namespace amg

struct amg_tg {
  amg_handle* inner = nullptr;  // PCG-AMG on level 1
  amg::TgWs w;
};

namespace amg {

void tg_free(amg_handle* H) {
  amg_tg* T = (amg_tg*)H->tg;
  if (!T) return;
  if (T->inner) amg_destroy(T->inner);
  if (T->w.dots_host) cudaFreeHost(T->w.dots_host);
  delete T;
  H->tg = nullptr;
}

// The inner solver and the vectors that do not depend on the group.
static int tg_create(amg_handle* H, cudaStream_t s) {
  Arena& ar = H->arena;
  amg_tg* T = new amg_tg();
  H->tg = T;
  TgWs& w = T->w;
  const Level& L1 = H->L[1];
  amg_csr A1{L1.n, L1.nnz, L1.rowptr, L1.col, L1.val};
  amg_options o = H->opt;
  o.precision = AMG_PREC_F64;
  o.autotune = 0;
  AMG_TRY(amg_setup(&A1, &o, (amg_stream_t)s, &T->inner));
  w.n = H->L[0].n;
  w.nc = L1.n;
  AMG_TRY(ar.alloc_n(&w.sbar, w.n));
  AMG_TRY(ar.alloc_n(&w.dots, 2 * TG_GROUP));
  AMG_CUDA_TRY(cudaMallocHost((void**)&w.dots_host, 2 * TG_GROUP * sizeof(double)));
  return AMG_OK;
}

// Releases the group's vectors (no group is then prepared).
static void tg_drop_group(Arena& ar, TgWs& w) {
  w.G = w.K = 0;
  for (double** p : {&w.e, &w.a, &w.c, &w.t, &w.t2, &w.eb, &w.cb, &w.ab, &w.g, &w.y}) {
    ar.release(*p);
    *p = nullptr;
  }
  for (auto* v : {&w.Ae, &w.Ac}) {
    for (double* p : *v) ar.release(p);
    v->clear();
  }
}

// Vectors for groups of G samples and K cycles; G and K are stored once every
// allocation has succeeded.
static int tg_alloc_group(Arena& ar, TgWs& w, int G, int K) {
  for (double** p : {&w.e, &w.a, &w.c, &w.t, &w.t2, &w.eb, &w.cb, &w.ab})
    AMG_TRY(ar.alloc_n(p, w.n * G));
  for (double** p : {&w.g, &w.y}) AMG_TRY(ar.alloc_n(p, w.nc * G));
  for (auto* v : {&w.Ae, &w.Ac}) {
    v->assign(K, nullptr);
    for (double*& p : *v) AMG_TRY(ar.alloc_n(&p, w.n * G));
  }
  w.G = G;
  w.K = K;
  return AMG_OK;
}

static int tg_prepare(amg_handle* H, int K, int nsamples, cudaStream_t s, amg_tg** out) {
  Arena& ar = H->arena;
  if (!H->tg) {
    const int rc = tg_create(H, s);
    if (rc < 0) {  // a later call starts over
      TgWs& w = ((amg_tg*)H->tg)->w;
      ar.release(w.sbar);
      ar.release(w.dots);
      tg_free(H);
      return rc;
    }
  }
  amg_tg* T = (amg_tg*)H->tg;
  TgWs& w = T->w;
  // the blocked PCG needs two levels and the dense coarsest factor; a one-level
  // inner hierarchy solves exactly, and one with the PCG coarsest solve by its
  // own V-cycle, one column at a time
  const bool blocked = T->inner->L.size() > 1 && T->inner->opt.coarse_solver == 0;
  const int G = blocked ? tg_group(nsamples, TG_GROUP) : 1;
  if (w.G < G || w.K < K) {
    // a group of G holds up to eight times one sample's vectors: where they do
    // not fit, smaller groups do
    const int k = K > w.K ? K : w.K;
    int rc = AMG_ERR_OOM;
    for (int q = G > w.G ? G : w.G; q >= 1 && rc == AMG_ERR_OOM;
         q = q > 1 ? tg_group(q / 2, TG_GROUP) : 0) {
      tg_drop_group(ar, w);
      rc = tg_alloc_group(ar, w, q, k);
      if (rc == AMG_OK && q > 1) rc = multi_reserve(T->inner, q);
    }
    if (rc < 0) {
      tg_drop_group(ar, w);
      return rc;
    }
  }
  *out = T;
  return AMG_OK;
}

int twogrid_loss(amg_handle* H, int nsamples, int K, const double* e0, double* loss,
                 float* domega, cudaStream_t s) {
  if (H->L.size() < 2 || H->batched) return AMG_ERR_UNSUPPORTED;
  amg_tg* T = nullptr;
  AMG_TRY(tg_prepare(H, K, nsamples, s, &T));
  TgWs& w = T->w;
  const Level& L0 = H->L[0];
  const int64_t n = w.n;
  const SellView<double> A = view<double>(L0.A, L0.A.v64);
  const int gs = sell_grid(sell_groups(L0.A), H->num_sms);
  const int gv = grid_for(n, 256, H->num_sms, 8);
  const double* sv = L0.s64;
  pcg_options po;
  pcg_default_options(&po);
  po.tol = 1e-12;
  po.maxit = 1000;
  po.beta_form = PCG_BETA_FR;
  int m = 0;  // samples of the current group
  auto spmv = [&](const double* x, double* y) {
    return sell_spmv64(L0.A, 1.0, x, 0.0, y, H->num_sms, s);
  };
  auto smooth = [&](const double* x, double* o, double* Ax) -> int {
    AMG_DISPATCH_TPR(sell_code(L0.A, 8),
                     (k_tg_smooth<TPR><<<gs, SELL_BLOCK, 0, s>>>(A, sv, x, o, Ax)));
    AMG_LAUNCH_CHECK();
    return AMG_OK;
  };
  auto csolve = [&]() -> int {  // y = A_c^-1 g, every column
    AMG_CUDA_TRY(cudaMemsetAsync(w.y, 0, sizeof(double) * w.nc * m, s));
    const int rc =
        m == 1 ? pcg_solve(T->inner, w.g, w.y, &po, nullptr, (amg_stream_t)s)
               : pcg_solve_multi(T->inner, m, w.g, w.y, &po, nullptr, (amg_stream_t)s);
    return rc == AMG_NOT_CONVERGED ? AMG_OK : rc;  // 1e-12 is a target, not a requirement
  };
  auto restrict_ = [&](const double* x, int q) -> int {  // column q of g = P^T x
    k_tg_restrict<<<grid_for(L0.nc, 256, H->num_sms, 8), 256, 0, s>>>(
        L0.nc, L0.stride, L0.members, x, w.g + q, m);
    AMG_LAUNCH_CHECK();
    return AMG_OK;
  };
  auto vec = [&](auto op, const double* x, const double* y2, double c, double* o) -> int {
    k_tg_vec<decltype(op)::value><<<gv, 256, 0, s>>>(n, x, y2, L0.agg, sv, c, o, nullptr, m);
    AMG_LAUNCH_CHECK();
    return AMG_OK;
  };
  auto dot = [&](const double* x, const double* y2, int slot) -> int {
    k_tg_dot<<<gv, 256, 0, s>>>(n, x, y2, H->red, w.dots + slot);
    AMG_LAUNCH_CHECK();
    return AMG_OK;
  };
  using PS = std::integral_constant<int, TG_PROLONG_SUB>;
  using PR = std::integral_constant<int, TG_PROLONG>;
  using SS = std::integral_constant<int, TG_SCALE_S>;
  using SB = std::integral_constant<int, TG_SUB>;
  using SR = std::integral_constant<int, TG_SBAR>;
  using SC = std::integral_constant<int, TG_SCALE>;
  AMG_CUDA_TRY(cudaMemsetAsync(w.sbar, 0, sizeof(double) * n, s));
  double total = 0.0;
  for (int j0 = 0; j0 < nsamples; j0 += m) {
    m = tg_group(nsamples - j0, w.G);
    AMG_CUDA_TRY(cudaMemcpyAsync(w.e, e0 + (int64_t)j0 * n, sizeof(double) * n * m,
                                 cudaMemcpyDeviceToDevice, s));
    for (int q = 0; q < m; ++q) {
      const int64_t o = (int64_t)q * n;
      AMG_TRY(spmv(w.e + o, w.t + o));
      AMG_TRY(dot(w.e + o, w.t + o, 2 * q));
    }
    for (int k = 0; k < K; ++k) {
      for (int q = 0; q < m; ++q) {
        const int64_t o = (int64_t)q * n;
        AMG_TRY(smooth(w.e + o, w.a + o, w.Ae[k] + o));  // a = S e
        AMG_TRY(spmv(w.a + o, w.t + o));                 // c = a - P A_c^-1 P^T A a
        AMG_TRY(restrict_(w.t + o, q));
      }
      AMG_TRY(csolve());
      for (int q = 0; q < m; ++q) {
        const int64_t o = (int64_t)q * n;
        AMG_TRY(vec(PS(), w.a + o, w.y + q, 0.0, w.c + o));
        AMG_TRY(smooth(w.c + o, w.e + o, w.Ac[k] + o));  // e = S c
      }
    }
    for (int q = 0; q < m; ++q) {
      const int64_t o = (int64_t)q * n;
      AMG_TRY(spmv(w.e + o, w.t + o));
      AMG_TRY(dot(w.e + o, w.t + o, 2 * q + 1));
    }
    AMG_CUDA_TRY(cudaMemcpyAsync(w.dots_host, w.dots, 2 * m * sizeof(double),
                                 cudaMemcpyDeviceToHost, s));
    AMG_CUDA_TRY(cudaStreamSynchronize(s));
    for (int q = 0; q < m; ++q) {
      const double n0 = w.dots_host[2 * q], nK = w.dots_host[2 * q + 1];
      if (!(n0 > 0.0) || !(nK > 0.0)) return AMG_ERR_NAN;
      total += 0.5 * log(nK / n0) / K;
    }
    if (!domega) continue;
    // reverse pass; seed d/de_K = A e_K / (e_K^T A e_K) / (K nsamples)
    for (int q = 0; q < m; ++q) {
      const int64_t o = (int64_t)q * n;
      AMG_TRY(vec(SC(), w.t + o, nullptr, 1.0 / (w.dots_host[2 * q + 1] * K * nsamples),
                  w.eb + o));
    }
    for (int k = K - 1; k >= 0; --k) {
      for (int q = 0; q < m; ++q) {
        const int64_t o = (int64_t)q * n;
        AMG_TRY(vec(SR(), w.eb + o, w.Ac[k] + o, 0.0, w.sbar));   // sbar -= eb o (A c_k)
        AMG_TRY(vec(SS(), w.eb + o, nullptr, 0.0, w.t2 + o));     // cb = S^T eb = eb - A (s o eb)
        AMG_TRY(spmv(w.t2 + o, w.t + o));
        AMG_TRY(vec(SB(), w.eb + o, w.t + o, 0.0, w.cb + o));
        AMG_TRY(restrict_(w.cb + o, q));                          // ab = cb - A P A_c^-1 P^T cb
      }
      AMG_TRY(csolve());
      for (int q = 0; q < m; ++q) {
        const int64_t o = (int64_t)q * n;
        AMG_TRY(vec(PR(), nullptr, w.y + q, 0.0, w.t2 + o));
        AMG_TRY(spmv(w.t2 + o, w.t + o));
        AMG_TRY(vec(SB(), w.cb + o, w.t + o, 0.0, w.ab + o));
        AMG_TRY(vec(SR(), w.ab + o, w.Ae[k] + o, 0.0, w.sbar));   // sbar -= ab o (A e_k)
        AMG_TRY(vec(SS(), w.ab + o, nullptr, 0.0, w.t2 + o));     // eb = S^T ab
        AMG_TRY(spmv(w.t2 + o, w.t + o));
        AMG_TRY(vec(SB(), w.ab + o, w.t + o, 0.0, w.eb + o));
      }
    }
  }
  *loss = total / nsamples;
  if (domega) {
    k_tg_vec<TG_DOMEGA><<<gv, 256, 0, s>>>(n, w.sbar, L0.d, nullptr, nullptr, 0.0, nullptr,
                                           domega, 1);
    AMG_LAUNCH_CHECK();
  }
  AMG_CUDA_TRY(cudaStreamSynchronize(s));
  return AMG_OK;
}

}  // namespace amg
