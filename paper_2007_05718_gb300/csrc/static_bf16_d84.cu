// 16-bit storage, 8 and 4 directions per warp (small direction sets)
#include "static_unit.cuh"

namespace lbrt {

cudaError_t static_bf16_d84(const StaticCall& c) {
  // 8 directions: up to 4 warps (32 directions), or 12 to 16; 4: up to 5, or 20
  if (c.dpt == 8)
    return c.N <= 32 ? static_plan<__nv_bfloat16, 8, 1, 2, 4, 128, 128>(c) : static_plan<__nv_bfloat16, 8, 1, 2, 4, 512, 128>(c);
  return c.N <= 20 ? static_plan<__nv_bfloat16, 4, 1, 2, 4, 160, 96>(c) : static_plan<__nv_bfloat16, 4, 1, 2, 4, 640, 96>(c);
}

}  // namespace lbrt
