// 16-bit storage, 5 directions per warp (the 42-direction icosahedral set), and
// its launch shared with the 162-direction set.  Two planes a batch; one plane
// with the flux terms, on a 2D grid and in the alternative batched kernel
// (static_zc).  Directions streamed ahead of the collision scalars, 128^3 x 42
// sphere, float16, 40 steps: 2: 7.36, 3: 7.44, 4: 8.04 ms.
#include "static_unit.cuh"

namespace lbrt {

cudaError_t static_f16_d5(const StaticCall& c) {
  if (c.flux || c.alt || c.zc == 1) return static_plan<__half, 5, 1, 2, 5, 320, 96>(c);
  return static_plain<__half, 5, 2, 1, 2, 320, 96>(c);
}

cudaError_t static_f16_pair(const StaticPairCall& c) {
  return c.flux ? pair_kernel<__half, true, 5, 1, 2, 5, 11, 1, 3, 11, 512, 128>(c)
                : pair_kernel<__half, false, 5, 2, 1, 2, 11, 1, 3, 11, 512, 128>(c);
}

}  // namespace lbrt
