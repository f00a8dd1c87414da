// Instantiations of the FP64 fixed-point stage kernels: DCT-I / DST-I lines with a contiguous output.
#include "p3_fix64.cuh"

namespace p3 {
namespace fx {

void* fn_ecs(int cap)
{
    return cap == 8 ? (void*)kernel<K_ECS, 8> : cap == 10 ? (void*)kernel<K_ECS, 10> : (void*)kernel<K_ECS, 16>;
}
void* fn_ess(int cap)
{
    return cap == 8 ? (void*)kernel<K_ESS, 8> : cap == 10 ? (void*)kernel<K_ESS, 10> : (void*)kernel<K_ESS, 16>;
}

}  // namespace fx
}  // namespace p3
