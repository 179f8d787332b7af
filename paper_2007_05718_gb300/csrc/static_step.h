// The static step (kernels_static.cuh): one call per launch or occupancy
// query, dispatched to the translation unit of its storage and tile plan.
#pragma once

#include "lb_rt_internal.h"

namespace lbrt {

// On a 2D grid no direction leaves the plane: tiles march along y instead of z
// (and need no seed plane).
inline bool marches_in_y(const Grid& g) { return g.dims == 2; }
inline int march_rows(const Grid& g) { return marches_in_y(g) ? 1 : g.ny; }
inline int march_length(const Grid& g) { return marches_in_y(g) ? g.ny : g.nz; }
inline int static_tiles(const Grid& g, int nchunks) { return (g.nx + 63) / 64 * march_rows(g) * nchunks; }
// the collision depends on the flux only with kappa_1 scattering (lambda != 0)
inline bool has_flux(const StaticCoef& c) { return c.lam || c.lam_s != 0.f; }

constexpr size_t kStaticSmemMax = 226 * 1024;

struct StaticCall {
  int mode = 0;              // 0 one problem, 1 batch, 2 one problem with the E, F epilogue
  bool budget = false;       // modes 0 and 2: with the energy budget
  bool flux = false;         // some problem has lambda != 0 (or the epilogue needs F)
  bool alt = false;          // batch: the alternative kernel of the plan
  int dpt = 0, zc = 0, N = 0;  // directions per warp, planes per batch, internal directions
  const CUtensorMap* tmap = nullptr;   // one problem: maps of the populations and of E
  const CUtensorMap* emap = nullptr;
  const ProblemDesc* one = nullptr;
  const ProblemDesc* table = nullptr;  // batch: device array
  int nprob = 0, ntiles = 0, ctas = 0;
  unsigned* err = nullptr;
  unsigned* sched = nullptr; // tile counter and CTAs done (zero between launches)
  const DirTable* dirs = nullptr;
  cudaStream_t stream = nullptr;
  int* per_sm = nullptr;     // set: only query the resident CTAs per SM
};

struct StaticPairCall {
  bool flux = false;
  BatchLaunch a{}, b{};
  const DirTable *dirs_a = nullptr, *dirs_b = nullptr;
  int ctas_a = 0, ctas = 0;
  cudaStream_t stream = nullptr;
  int* per_sm = nullptr;
};

cudaError_t static_f32_d5(const StaticCall& c);
cudaError_t static_f32_d11(const StaticCall& c);
cudaError_t static_f32_d10(const StaticCall& c);
cudaError_t static_f32_d84(const StaticCall& c);
cudaError_t static_f32_pair(const StaticPairCall& c);
cudaError_t static_f16_d5(const StaticCall& c);
cudaError_t static_f16_d11(const StaticCall& c);
cudaError_t static_f16_d10(const StaticCall& c);
cudaError_t static_f16_d84(const StaticCall& c);
cudaError_t static_f16_pair(const StaticPairCall& c);
cudaError_t static_bf16_d5(const StaticCall& c);
cudaError_t static_bf16_d11(const StaticCall& c);
cudaError_t static_bf16_d10(const StaticCall& c);
cudaError_t static_bf16_d84(const StaticCall& c);
cudaError_t static_bf16_pair(const StaticPairCall& c);

}  // namespace lbrt
