// Instantiations of the FP64 fixed-point stage kernels: DCT-I / DST-I lines with a strided output.
#include "p3_fix64.cuh"

namespace p3 {
namespace fx {

void* fn_ecc(int cap)
{
    return cap == 8 ? (void*)kernel<K_ECC, 8> : cap == 10 ? (void*)kernel<K_ECC, 10> : (void*)kernel<K_ECC, 16>;
}
void* fn_esc(int cap)
{
    return cap == 8 ? (void*)kernel<K_ESC, 8> : cap == 10 ? (void*)kernel<K_ESC, 10> : (void*)kernel<K_ESC, 16>;
}

}  // namespace fx
}  // namespace p3
