// 16-bit storage, 11 directions per warp (the 162-direction icosahedral set)
#include "static_unit.cuh"

namespace lbrt {

cudaError_t static_bf16_d11(const StaticCall& c) { return static_plan<__nv_bfloat16, 11, 1, 3, 5, 512, 128>(c); }

}  // namespace lbrt
