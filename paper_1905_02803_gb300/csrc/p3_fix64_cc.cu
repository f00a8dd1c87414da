// Instantiations of the FP64 fixed-point stage kernels: complex lines with a strided output.
#include "p3_fix64.cuh"

namespace p3 {
namespace fx {

void* fn_cc(int cap)
{
    return cap == 8 ? (void*)kernel<K_CC, 8> : cap == 10 ? (void*)kernel<K_CC, 10> : (void*)kernel<K_CC, 16>;
}
void* fn_sc(int cap)
{
    return cap == 8 ? (void*)kernel<K_SC, 8> : cap == 10 ? (void*)kernel<K_SC, 10> : (void*)kernel<K_SC, 16>;
}

}  // namespace fx
}  // namespace p3
