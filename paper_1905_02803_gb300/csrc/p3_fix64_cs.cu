// Instantiations of the FP64 fixed-point stage kernels: complex lines with a contiguous output.
#include "p3_fix64.cuh"

namespace p3 {
namespace fx {

void* fn_cs(int cap)
{
    return cap == 8 ? (void*)kernel<K_CS, 8> : cap == 10 ? (void*)kernel<K_CS, 10> : (void*)kernel<K_CS, 16>;
}
void* fn_ss(int cap)
{
    return cap == 8 ? (void*)kernel<K_SS, 8> : cap == 10 ? (void*)kernel<K_SS, 10> : (void*)kernel<K_SS, 16>;
}

}  // namespace fx
}  // namespace p3
