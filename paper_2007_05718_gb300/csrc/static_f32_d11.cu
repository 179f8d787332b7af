// float32 storage, 11 directions per warp (the 162-direction icosahedral set).
// The directions streamed ahead of the collision scalars (7 of 11) measured at
// 256^3 x 162, eight steps and the moments: 3: 44.1, 5: 41.4, 7: 39.6, 9: 44.9 ms.
#include "static_unit.cuh"

namespace lbrt {

cudaError_t static_f32_d11(const StaticCall& c) { return static_plan<float, 11, 1, 3, 7, 512, 128>(c); }

}  // namespace lbrt
