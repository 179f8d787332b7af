// 16-bit storage, 11 directions per warp (the 162-direction icosahedral set).
// All directions are streamed ahead of the collision scalars: 256^3 x 162,
// eight steps and the moments (float16), 3: 41.1, 5: 38.9, 7: 36.8, 9: 35.8,
// 11: 35.3 ms.
#include "static_unit.cuh"

namespace lbrt {

cudaError_t static_bf16_d11(const StaticCall& c) { return static_plan<__nv_bfloat16, 11, 1, 3, 11, 512, 128>(c); }

}  // namespace lbrt
