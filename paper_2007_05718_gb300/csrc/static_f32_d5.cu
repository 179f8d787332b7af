// float32 storage, 5 directions per warp (the 42-direction icosahedral set),
// and its launch shared with the 162-direction set.  Two planes a batch; one
// plane with the flux terms, on a 2D grid and in the alternative batched kernel
// (static_zc).  Directions streamed ahead of the collision scalars, 128^3 x 42
// sphere, 40 steps: 2: 6.56, 4: 6.22, 5: 6.19 ms.
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
