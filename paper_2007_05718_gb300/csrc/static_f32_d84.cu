// float32 storage, 8 and 4 directions per warp (small direction sets)
#include "static_unit.cuh"

namespace lbrt {

cudaError_t static_f32_d84(const StaticCall& c) {
  // The launch bound sizes the partial sums in shared memory, so that few warps
  // want a small one: 512^2 x 4 with the flux terms, float32 20.6 -> 16.4 us a
  // step, float16 23.9 -> 18.5; 512^2 x 12 float32 22.6 -> 20.6 (within 1 % of
  // each other without the flux terms).
  if (c.dpt == 8)
    return c.N <= 32 ? static_plan<float, 8, 1, 2, 4, 128, 128>(c) : static_plan<float, 8, 1, 2, 4, 512, 128>(c);
  return c.N <= 20 ? static_plan<float, 4, 1, 2, 4, 160, 96>(c) : static_plan<float, 4, 1, 2, 4, 640, 96>(c);
}

}  // namespace lbrt
