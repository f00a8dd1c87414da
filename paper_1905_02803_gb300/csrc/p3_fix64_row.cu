// Instantiations of the FP64 fixed-point stage kernels: even real rows.
#include "p3_fix64.cuh"

namespace p3 {
namespace fx {

void* fn_r2c(int cap)
{
    return cap == 8 ? (void*)kernel<K_R2C, 8> : cap == 10 ? (void*)kernel<K_R2C, 10> : (void*)kernel<K_R2C, 16>;
}
void* fn_c2r(int cap)
{
    return cap == 8 ? (void*)kernel<K_C2R, 8> : cap == 10 ? (void*)kernel<K_C2R, 10> : (void*)kernel<K_C2R, 16>;
}

}  // namespace fx
}  // namespace p3
