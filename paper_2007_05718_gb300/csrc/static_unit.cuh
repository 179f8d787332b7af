// Launch and occupancy of one static tile plan, instantiated by the
// static_<storage>_<plan>.cu files (one translation unit per storage and
// directions per warp, compiled in parallel).
#pragma once

#include "kernels_static.cuh"
#include "static_step.h"

namespace lbrt {
namespace {

// opt-in shared memory is a per-device function attribute
template <class F>
cudaError_t allow_smem(F* kernel, unsigned long long& done) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 64 && (done >> dev & 1ull)) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kStaticSmemMax);
  if (e == cudaSuccess && dev < 64) done |= 1ull << dev;
  return e;
}

template <class ST, int MODE, bool FLUX, int DPT, int ZC, int HU, int H, int MAXT, int REGS>
cudaError_t static_kernel(const StaticCall& c) {
  auto* k = k_static<ST, MODE, FLUX, DPT, ZC, HU, H, MAXT, REGS>;
  static unsigned long long done = 0;
  const int G = c.N / DPT;
  if (G < 1 || G * DPT != c.N || 32 * G > MAXT) return cudaErrorInvalidValue;
  const size_t smem = StLayout<ST, MODE == 1, FLUX, DPT, ZC, MAXT / 32>::bytes(G);
  if (smem > kStaticSmemMax) return cudaErrorInvalidValue;
  const cudaError_t e = allow_smem(k, done);
  if (e != cudaSuccess) return e;
  if (c.per_sm) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(c.per_sm, k, 32 * G, smem);
  if (c.ctas < 1 || c.ntiles < 1) return cudaErrorInvalidValue;
  k<<<c.ctas, dim3(32, G), smem, c.stream>>>(*c.tmap, *c.emap, *c.one, c.table, c.nprob, c.ntiles, c.err,
                                             c.sched, *c.dirs);
  return cudaGetLastError();
}

// kernels of a plan with the flux terms
template <class ST, int DPT, int ZC, int HU, int H, int MAXT, int REGS>
cudaError_t static_flux(const StaticCall& c) {
  if (c.mode == 1) return static_kernel<ST, 1, true, DPT, ZC, HU, H, MAXT, REGS>(c);
  if constexpr (SV<ST>::F32) {
    if (c.mode == 2)
      return c.budget ? static_kernel<ST, 2 + 4, true, DPT, ZC, HU, H, MAXT, REGS>(c)
                      : static_kernel<ST, 2, true, DPT, ZC, HU, H, MAXT, REGS>(c);
  }
  return c.budget ? static_kernel<ST, 4, true, DPT, ZC, HU, H, MAXT, REGS>(c)
                  : static_kernel<ST, 0, true, DPT, ZC, HU, H, MAXT, REGS>(c);
}

// and without them
template <class ST, int DPT, int ZC, int HU, int H, int MAXT, int REGS>
cudaError_t static_plain(const StaticCall& c) {
  if (c.mode == 1) return static_kernel<ST, 1, false, DPT, ZC, HU, H, MAXT, REGS>(c);
  return c.budget ? static_kernel<ST, 4, false, DPT, ZC, HU, H, MAXT, REGS>(c)
                  : static_kernel<ST, 0, false, DPT, ZC, HU, H, MAXT, REGS>(c);
}

template <class ST, int DPT, int ZC, int HU, int H, int MAXT, int REGS>
cudaError_t static_plan(const StaticCall& c) {
  return c.flux || c.mode == 2 ? static_flux<ST, DPT, ZC, HU, H, MAXT, REGS>(c)
                               : static_plain<ST, DPT, ZC, HU, H, MAXT, REGS>(c);
}

template <class ST, bool FLUX, int DA, int ZA, int UA, int HA, int DB, int ZB, int UB, int HB, int MAXT, int REGS>
cudaError_t pair_kernel(const StaticPairCall& c) {
  auto* k = k_static_pair<ST, FLUX, DA, ZA, UA, HA, DB, ZB, UB, HB, MAXT, REGS>;
  static unsigned long long done = 0;
  const int ga = c.a.N / DA, gb = c.b.N / DB, gm = std::max(ga, gb);
  if (ga < 1 || ga * DA != c.a.N || gb < 1 || gb * DB != c.b.N || 32 * gm > MAXT) return cudaErrorInvalidValue;
  const size_t smem = std::max(StLayout<ST, true, FLUX, DA, ZA, MAXT / 32>::bytes(ga),
                               StLayout<ST, true, FLUX, DB, ZB, MAXT / 32>::bytes(gb));
  if (smem > kStaticSmemMax) return cudaErrorInvalidValue;
  const cudaError_t e = allow_smem(k, done);
  if (e != cudaSuccess) return e;
  if (c.per_sm) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(c.per_sm, k, 32 * gm, smem);
  if (c.ctas_a < 1 || c.ctas_a >= c.ctas || !c.a.table || !c.b.table || c.a.nprob < 1 || c.b.nprob < 1 ||
      c.a.ntiles < 1 || c.b.ntiles < 1)
    return cudaErrorInvalidValue;
  CUtensorMap unused{};
  ProblemDesc none{};
  k<<<c.ctas, dim3(32, gm), smem, c.stream>>>(unused, none, c.a.table, c.a.nprob, c.a.ntiles, ga, c.ctas_a,
                                              c.b.table, c.b.nprob, c.b.ntiles, gb, c.b.err, c.b.sched,
                                              *c.dirs_a, *c.dirs_b);
  return cudaGetLastError();
}

}  // namespace
}  // namespace lbrt
