// Host side of the shared-memory ring streams (ring.cuh): which matrices
// qualify, the ring's geometry, and the kernels' shared-memory limit.
#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

#include "ring.cuh"

namespace amg {

// Stages and tile: the largest tile (8, 4 or 2 slices, one consumer warp
// each) that leaves room for the warps of RING_CTAS_PER_SM CTAs of 8 slices
// per SM, else of three, else of two.  Three stages while the SM's rings then stay
// within half of its unified memory, so that the rest caches the gathered
// vector, else two: measured at 256^3 (FP32), the level-0 pre-smoother (9 KB
// stages) took 0.136 ms with three against 0.143 with two, the level-1 one of
// a diffusion matrix (18 KB stages) 0.092 against 0.080.
//
// Pairs (two slices a warp, tiles of 16): where two CTAs on each of 152 SMs have a
// tile and four rings fit an SM.  256^3 FP32, level-0 pre-smoother: 137 us with one
// slice a warp, 108 with two; four warps of two slices in six or seven CTAs an SM
// 118 and 114.
constexpr size_t RING_L1_SPLIT = 128 * 1024;

RingGeom ring_plan(const Sell& M, int vbytes, int stages, const RingRows& rows, bool dots,
                   bool chunked, bool pairs) {
  RingGeom none;
  if (M.C != 32 || M.tpr != 1 || (M.row0 != nullptr) != chunked || !M.rec || M.wmax <= 0 ||
      M.nslices <= 0)
    return none;
  if (vbytes != 2 && vbytes != 4 && vbytes != 8) return none;
  if (stages == 1 || stages > RING_MAX_STAGES || rows.n > RING_MAX_ROWS) return none;
  uint32_t direct = 0;
  for (int k = 0; k < rows.n; ++k) {
    if (rows.esz[k] != 4 && rows.esz[k] != 8) return none;
    if (((uintptr_t)rows.p[k] & 15u) != 0) direct |= 1u << k;  // no bulk copy from there
  }
  auto up = [](size_t v) { return (v + 127) & ~(size_t)127; };
  // values, index blocks, records, per-row vectors; every part starts on 128 bytes
  auto plan = [&](int q, int D) {
    RingGeom g;
    const int f = pairs ? 2 : 1;  // (tile_w and tile_ix bound two tiles together)
    g.tile = ring_tile(q) * f;
    g.warps = pairs ? g.tile / 2 : g.tile;
    size_t off = up((size_t)M.tile_w[q] * f * 32 * (size_t)vbytes);
    g.coff = (uint32_t)off;
    off = up(off + (size_t)M.tile_ix[q] * f);
    g.soff = (uint32_t)off;
    off = up(off + 16 * (size_t)(g.tile + 1));
    if (chunked) {
      g.hoff = (uint32_t)off;
      off = up(off + sizeof(RingTile));
    }
    for (int k = 0; k < rows.n; ++k) {
      g.roff[k] = (uint32_t)off;
      // (chunked: up to three rows more on either side of the tile's)
      off = up(off + (size_t)(32 * g.tile + (chunked ? 8 : 0)) * rows.esz[k]);
    }
    g.D = D;
    g.direct = direct;
    g.stage = (uint32_t)off;
    g.smem = (size_t)D * off + 2 * RING_MAX_STAGES * 8 + RING_ALIGN_SLACK;
    return g;
  };
  // smaller tiles where 8 slices a CTA would leave SMs without work (two
  // CTAs on each of 152); with dot products 8 slices, the blocks of the
  // per-lane kernels, so that both sum small levels alike
  const int q0 = dots || chunked || M.nslices >= 304 * ring_tile(0) ? 0
                 : M.nslices >= 304 * ring_tile(1)       ? 1
                                                         : 2;
  if (pairs) {
    const int c = RING_CTAS_PER_SM;
    if (M.nslices < 304 * 2 * ring_tile(0)) return none;
    const size_t smem = c * (plan(0, 3).smem + 1024);
    const RingGeom g = plan(0, stages ? stages : smem <= RING_L1_SPLIT ? 3 : 2);
    const bool fits = g.smem <= RING_SMEM_PER_CTA && c * (g.smem + 1024) <= RING_SMEM_PER_SM;
    return fits ? g : none;
  }
  for (int ctas : {RING_CTAS_PER_SM, RING_CTAS_PER_SM - 1, 2})
    for (int q = q0; q < (chunked ? 1 : 3); ++q) {
      const int c = ctas * ring_tile(0) / ring_tile(q);  // the same number of warps
      const size_t smem = c * (plan(q, 3).smem + 1024);
      const RingGeom g = plan(q, stages ? stages : smem <= RING_L1_SPLIT ? 3 : 2);
      if (g.smem <= RING_SMEM_PER_CTA && (size_t)c * (g.smem + 1024) <= RING_SMEM_PER_SM)
        return g;
    }
  return none;
}

int ring_prepare(const void* fn, RingGeom& g, int64_t work, int num_sms) {
  static std::mutex mu;
  static std::map<std::pair<const void*, int>, bool> attr;
  static std::map<std::pair<const void*, std::pair<size_t, int>>, int> occ;
  int dev = 0;
  AMG_CUDA_TRY(cudaGetDevice(&dev));
  int per_sm = 0;
  {
    std::lock_guard<std::mutex> lock(mu);
    bool& done = attr[{fn, dev}];
    if (!done) {
      AMG_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)RING_SMEM_PER_CTA));
      // the unified L1 / shared array mostly as shared memory: several rings per SM
      AMG_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout,
                                        (int)cudaSharedmemCarveoutMaxShared));
      done = true;
    }
    int& nb = occ[{fn, {g.smem, g.tile}}];  // the same on every device of one kind
    if (!nb) {
      AMG_CUDA_TRY(
          cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, g.threads(), g.smem));
      if (nb < 1) nb = -1;
    }
    per_sm = nb;
  }
  if (per_sm < 1) return AMG_ERR_UNSUPPORTED;
  const int64_t full = (int64_t)num_sms * std::min(per_sm, 16);  // grid reductions hold 16 per SM
  g.grid = (int)(work < full ? work : full);
  return AMG_OK;
}

}  // namespace amg
