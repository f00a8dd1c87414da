// Instantiations of the FP64 fixed-point stage kernels: odd real rows in pairs.
#include "p3_fix64.cuh"

namespace p3 {
namespace fx {

void* fn_rp(int cap)
{
    return cap == 8 ? (void*)kernel<K_RP, 8> : cap == 10 ? (void*)kernel<K_RP, 10> : (void*)kernel<K_RP, 16>;
}
void* fn_cp(int cap)
{
    return cap == 8 ? (void*)kernel<K_CP, 8> : cap == 10 ? (void*)kernel<K_CP, 10> : (void*)kernel<K_CP, 16>;
}

}  // namespace fx
}  // namespace p3
