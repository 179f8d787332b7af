// float32 storage, 5 directions per warp (the 42-direction icosahedral set),
// and its launch shared with the 162-direction set.  Two planes a batch; one
// plane with the flux terms, on a 2D grid and in the alternative batched kernel
// (static_zc).  Directions streamed ahead of the collision scalars, 128^3 x 42
// sphere, 40 steps: 2: 6.55, 4: 6.21, 5: 6.18 ms.
//
// The flux kernel takes 72 registers, three CTAs of nine warps an SM: its batches
// wait for one another's chain more than for anything else.  us a step with
// kappa_1, 64^3 / 128^3 x 42 / 256^3 x 42: two CTAs of 96 registers 64 / 266 /
// 1719, two planes a batch 62 / 329 / 2136; 72 registers with no direction
// streamed ahead 48 / 238 / 1570, two of them 46 / 228 / 1511.
#include "static_unit.cuh"

namespace lbrt {

cudaError_t static_f32_d5(const StaticCall& c) {
  if (c.flux || c.mode == 2) return static_flux<float, 5, 1, 0, 2, 320, 72>(c);
  if (c.alt) return static_kernel<float, 1, false, 5, 1, 1, 2, 320, 72>(c);
  return c.zc == 1 ? static_plain<float, 5, 1, 2, 5, 320, 96>(c) : static_plain<float, 5, 2, 1, 5, 320, 96>(c);
}

cudaError_t static_f32_pair(const StaticPairCall& c) {
  return c.flux ? pair_kernel<float, true, 5, 1, 2, 5, 11, 1, 3, 7, 512, 128>(c)
                : pair_kernel<float, false, 5, 2, 1, 5, 11, 1, 3, 7, 512, 128>(c);
}

}  // namespace lbrt
