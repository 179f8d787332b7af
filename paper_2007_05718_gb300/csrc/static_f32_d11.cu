// float32 storage, 11 directions per warp (the 162-direction icosahedral set)
#include "static_unit.cuh"

namespace lbrt {

cudaError_t static_f32_d11(const StaticCall& c) { return static_plan<float, 11, 1, 3, 5, 512, 128>(c); }

}  // namespace lbrt
