// Dense Cholesky of the coarsest level's diagonal blocks and the inverse of
// the factor, by panels of 32 columns over the whole GPU.
//
// What it replaces: one CUDA block per diagonal block (up to 1024 rows) that
// updated the trailing matrix in global memory after every column and formed
// L^-1 with one thread per column.  GB300 issues two FP64 lane operations per
// SM clock, so a block on one SM is bound by that SM: 20.4 ms for the coarsest
// level of a 128^3 diffusion problem, a quarter of the setup.
//
// Here every panel takes two launches over all diagonal blocks:
//   k_chol_panel   factors the 32 x 32 diagonal tile (every CTA for itself, in
//                  one warp's registers: 32 dependent square roots and
//                  divisions), then solves the rows below it (L_ik) and the
//                  tile's rows of L^-1, one thread per row or column;
//   k_chol_update  subtracts the panel's 32 rank-1 terms from the trailing
//                  matrix and from the rows of L^-1 still to come, one 32 x 32
//                  tile per CTA, operands in shared memory.
// L^-1 is formed by the same right-looking order: it starts as the identity
// and row k, once final, is subtracted a_ik times from every later row.
//
// A panel takes 189 us in the set-up of a 128^3 diffusion problem.  The FP64
// operations of one warp's chain account for about a quarter of that; what it
// waits for besides is not known (254 registers, no spills).
//
// Every entry receives the same explicitly rounded operations in the same
// order (k ascending, product and difference rounded separately) as the
// textbook loops of a sequential factorisation, so the factor is reproducible
// bit for bit.
#include "common.cuh"

namespace amg {

namespace {

constexpr int NB = 32;          // panel width
// A warp per CTA: a 128^3 diffusion set-up takes 36.0 and 35.9 ms, with 128
// threads 36.7 and 36.0 (in turn).
constexpr int PANEL_THREADS = 32;
constexpr int TILE_THREADS = 256;

// Block b: rows n, dense row-major a (below the diagonal tiles it becomes L; the
// tiles' own factors stay in the panel kernel), L^-1, L^-T.
struct Blk {
  int64_t n;
  double *a, *inv, *invT;
};

__device__ __forceinline__ Blk blk_of(const int64_t* brow, const int64_t* bmat, double* dense,
                                      double* inv, double* invT, int b) {
  return Blk{brow[b + 1] - brow[b], dense + bmat[b], inv + bmat[b], invT + bmat[b]};
}

// L^-1 starts as the identity, L^-T as zero (its lower triangle stays zero).
__global__ void k_inverse_init(const int64_t* brow, const int64_t* bmat, double* inv_all,
                               double* invT_all) {
  const Blk B = blk_of(brow, bmat, inv_all, inv_all, invT_all, blockIdx.y);
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < B.n * B.n;
       t += (int64_t)gridDim.x * blockDim.x) {
    B.inv[t] = t / B.n == t % B.n ? 1.0 : 0.0;
    B.invT[t] = 0.0;
  }
}

__global__ void __launch_bounds__(PANEL_THREADS)
    k_chol_panel(const int64_t* brow, const int64_t* bmat, double* dense, double* inv_all,
                 double* invT_all, int64_t kb, int* status) {
  const Blk B = blk_of(brow, bmat, dense, inv_all, invT_all, blockIdx.y);
  const int64_t n = B.n;
  if (kb >= n) return;
  const int nb = (int)(n - kb < NB ? n - kb : NB);
  // work items: rows kb+nb .. n-1 of the panel, then columns 0 .. kb+nb-1 of
  // the tile's rows of L^-1
  const int64_t below = n - kb - nb, items = below + kb + nb;
  if ((int64_t)blockIdx.x * PANEL_THREADS >= items) return;
  __shared__ double t[NB][NB + 1];
  for (int e = threadIdx.x; e < nb * nb; e += PANEL_THREADS)
    t[e / nb][e % nb] = B.a[(kb + e / nb) * n + kb + e % nb];
  __syncthreads();
  if (threadIdx.x < 32) {
    // the tile in registers, lane = row: r[j] = entry (lane, j)
    const int lane = threadIdx.x;
    double r[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j) r[j] = lane < nb && j < nb ? t[lane][j] : (lane == j ? 1.0 : 0.0);
    bool bad = false;
#pragma unroll
    for (int k = 0; k < NB; ++k) {
      if (k >= nb) break;  // (a 2-row block takes 2 steps, not 32)
      const double piv = __shfl_sync(0xffffffffu, r[k], k);
      if (!(piv > 0.0)) bad = true;
      const double lkk = sqrt(piv);
      const double l = lane == k ? lkk : __ddiv_rn(r[k], lkk);
      r[k] = l;
#pragma unroll
      for (int j = k + 1; j < NB; ++j) {
        const double lj = __shfl_sync(0xffffffffu, l, j);
        if (lane >= j) r[j] = __dsub_rn(r[j], __dmul_rn(l, lj));
      }
    }
    if (bad && lane == 0) atomicExch(status, AMG_ERR_NOT_SPD);
#pragma unroll
    for (int j = 0; j < NB; ++j)
      if (lane < nb && j < nb && j <= lane) t[lane][j] = r[j];
  }
  __syncthreads();
  const int64_t it = (int64_t)blockIdx.x * PANEL_THREADS + threadIdx.x;
  if (it < below) {
    // row i below the tile: columns in order, each divided by its pivot and
    // subtracted from the later ones
    double* row = B.a + (kb + nb + it) * n + kb;
    double v[NB];
#pragma unroll
    for (int k = 0; k < NB; ++k) v[k] = k < nb ? row[k] : 0.0;
#pragma unroll
    for (int k = 0; k < NB; ++k) {
      if (k >= nb) break;
      v[k] = __ddiv_rn(v[k], t[k][k]);
#pragma unroll
      for (int j = k + 1; j < NB; ++j)
        if (j < nb) v[j] = __dsub_rn(v[j], __dmul_rn(v[k], t[j][k]));
    }
#pragma unroll
    for (int k = 0; k < NB; ++k)
      if (k < nb) row[k] = v[k];
  } else if (it < items) {
    // column c of the tile's rows of L^-1, forward substitution in row order
    const int64_t c = it - below;
    double v[NB];
#pragma unroll
    for (int k = 0; k < NB; ++k) v[k] = k < nb ? B.inv[(kb + k) * n + c] : 0.0;
#pragma unroll
    for (int k = 0; k < NB; ++k) {
      if (k >= nb) break;
      if (c <= kb + k) v[k] = __ddiv_rn(v[k], t[k][k]);
#pragma unroll
      for (int j = k + 1; j < NB; ++j)
        if (j < nb && c <= kb + k) v[j] = __dsub_rn(v[j], __dmul_rn(t[j][k], v[k]));
    }
#pragma unroll
    for (int k = 0; k < NB; ++k)
      if (k < nb) {
        B.inv[(kb + k) * n + c] = v[k];
        B.invT[c * n + kb + k] = v[k];
      }
  }
}

// Tile (ti, tj) of the rows below panel kb: tj < tiles(c < kb + nb) are tiles
// of L^-1, the others tiles of the trailing matrix (lower triangle).
__global__ void __launch_bounds__(TILE_THREADS)
    k_chol_update(const int64_t* brow, const int64_t* bmat, double* dense, double* inv_all,
                  double* invT_all, int64_t kb) {
  const Blk B = blk_of(brow, bmat, dense, inv_all, invT_all, blockIdx.y);
  const int64_t n = B.n;
  const int64_t t0 = kb + NB;  // a panel with rows below it is full
  if (t0 >= n) return;
  const int64_t rt = (n - t0 + NB - 1) / NB;     // row tiles
  const int64_t ct = t0 / NB;                    // column tiles of L^-1
  const int64_t ninv = rt * ct, ntot = ninv + rt * (rt + 1) / 2;
  __shared__ double li[NB][NB + 1], lj[NB][NB + 1];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int64_t id = blockIdx.x; id < ntot; id += gridDim.x) {
    int64_t i0, c0;
    const bool inv = id < ninv;
    if (inv) {
      i0 = t0 + (id / ct) * NB;
      c0 = (id % ct) * NB;
    } else {
      const int64_t q = id - ninv;
      int64_t r = (int64_t)((sqrt(8.0 * (double)q + 1.0) - 1.0) * 0.5);
      while (r * (r + 1) / 2 > q) --r;
      while ((r + 1) * (r + 2) / 2 <= q) ++r;
      i0 = t0 + r * NB;
      c0 = t0 + (q - r * (r + 1) / 2) * NB;
    }
    // li[r][k] = L(i0 + r, kb + k); lj[k][c]: L^-1(kb + k, c0 + c), or
    // L(c0 + c, kb + k)
    for (int r = ty; r < NB; r += TILE_THREADS / 32) {
      li[r][tx] = i0 + r < n ? B.a[(i0 + r) * n + kb + tx] : 0.0;
      if (inv)
        lj[r][tx] = B.inv[(kb + r) * n + c0 + tx];
      else
        lj[tx][r] = c0 + r < n ? B.a[(c0 + r) * n + kb + tx] : 0.0;
    }
    __syncthreads();
    double* out = inv ? B.inv : B.a;
    for (int r = ty; r < NB; r += TILE_THREADS / 32) {
      const int64_t i = i0 + r, c = c0 + tx;
      if (i >= n || c >= n || (!inv && c > i)) continue;
      double v = out[i * n + c];
#pragma unroll 8
      for (int k = 0; k < NB; ++k) {
        // a column of L^-1 starts at its own row: earlier terms are not there
        if (inv && c > kb + k) continue;
        v = __dsub_rn(v, __dmul_rn(li[r][k], lj[k][tx]));
      }
      out[i * n + c] = v;
    }
    __syncthreads();
  }
}

}  // namespace

// Launches of up to this many diagonal blocks: gridDim.y ends there.
constexpr int CHOL_GRID_BLOCKS = 65535;

// Factors nblk diagonal blocks (block b: rows brow[b] .. brow[b+1], matrices
// at bmat[b]; device arrays), the largest of `largest` rows.  Asynchronous;
// a pivot <= 0 puts AMG_ERR_NOT_SPD into *status.
int chol_blocks(int nblk, int64_t largest, const int64_t* brow, const int64_t* bmat,
                double* dense, double* Linv, double* LinvT, int* status, int num_sms,
                cudaStream_t s) {
  const unsigned pg = (unsigned)((largest + PANEL_THREADS - 1) / PANEL_THREADS);
  for (; nblk > 0; nblk -= CHOL_GRID_BLOCKS, brow += CHOL_GRID_BLOCKS, bmat += CHOL_GRID_BLOCKS) {
    const unsigned nb = (unsigned)(nblk < CHOL_GRID_BLOCKS ? nblk : CHOL_GRID_BLOCKS);
    k_inverse_init<<<dim3(grid_for(largest * largest, 256, num_sms, 8), nb), 256, 0, s>>>(
        brow, bmat, Linv, LinvT);
    AMG_LAUNCH_CHECK();
    for (int64_t kb = 0; kb < largest; kb += NB) {
      k_chol_panel<<<dim3(pg, nb), PANEL_THREADS, 0, s>>>(brow, bmat, dense, Linv, LinvT, kb,
                                                          status);
      AMG_LAUNCH_CHECK();
      if (kb + NB >= largest) break;
      const int64_t rt = (largest - kb - 1) / NB;  // row tiles of the largest block
      const int64_t tiles = rt * ((kb + NB) / NB) + rt * (rt + 1) / 2;
      k_chol_update<<<dim3(grid_for(tiles, 1, num_sms, 8), nb), TILE_THREADS, 0, s>>>(
          brow, bmat, dense, Linv, LinvT, kb);
      AMG_LAUNCH_CHECK();
    }
  }
  return AMG_OK;
}

}  // namespace amg
