// 16-bit storage, 10 directions per warp.  Up to 8 warps (80 directions) two CTAs
// fit an SM at 128 registers; 17 warps leave 96 registers a thread (resident
// warps are counted in fours).
#include "static_unit.cuh"

namespace lbrt {

cudaError_t static_bf16_d10(const StaticCall& c) {
  if (c.N <= 80) return static_plan<__nv_bfloat16, 10, 1, 3, 5, 256, 128>(c);
  return c.N <= 160 ? static_plan<__nv_bfloat16, 10, 1, 3, 5, 512, 128>(c) : static_plan<__nv_bfloat16, 10, 1, 1, 3, 544, 96>(c);
}

}  // namespace lbrt
