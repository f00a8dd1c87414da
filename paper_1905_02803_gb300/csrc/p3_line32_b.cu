// Instantiations of the FP32 line kernels: contiguous outputs and rows.
#include "p3_line32.cuh"

namespace p3 {
namespace l32 {

void* fn_b(int k)
{
    switch (k) {
    case K_CS: return (void*)kernel<K_CS>;
    case K_ECS: return (void*)kernel<K_ECS>;
    case K_R2C: return (void*)row_kernel<K_R2C>;
    case K_C2R: return (void*)row_kernel<K_C2R>;
    case K_RP: return (void*)row_kernel<K_RP>;
    case K_CP: return (void*)row_kernel<K_CP>;
    default: return nullptr;
    }
}

}  // namespace l32
}  // namespace p3
