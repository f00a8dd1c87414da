// Instantiations of the FP32 line kernels: strided outputs.
#include "p3_line32.cuh"

namespace p3 {
namespace l32 {

void* fn_a(int k, int tma)
{
    switch (k) {
    case K_CC: return (void*)kernel<K_CC>;
    case K_CCI: return (void*)kernel<K_CCI>;
    case K_SCI: return tma ? (void*)kernel<K_SCI, true> : (void*)kernel<K_SCI>;
    case K_ECC: return (void*)kernel<K_ECC>;
    case K_ESC: return (void*)kernel<K_ESC>;
    default: return nullptr;
    }
}

}  // namespace l32
}  // namespace p3
