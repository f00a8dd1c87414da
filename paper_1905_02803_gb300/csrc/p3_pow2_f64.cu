// Instantiations of the power-of-two stage kernels for double data: the forward
// transform of volumes of more than kFix64MaxPoints points (other stages of
// these lengths run in fixed point: p3_fix64.cuh).
#include "p3_pow2.cuh"

namespace p3 {

namespace {
using namespace pw;

// sym: 0 plain, 1 Chebyshev (DCT-I), 2 sine (DST-I)
template <int N, int MODE> void* col_fn(int sym)
{
    constexpr int E = col_E<double>(N, MODE), B = col_B<double>(N);
    return sym == 2 ? (void*)col_kernel<double, N, E, B, MODE, false, 2>
           : sym    ? (void*)col_kernel<double, N, E, B, MODE, false, 1>
                    : (void*)col_kernel<double, N, E, B, MODE, false, 0>;
}
template <int N> void* pick_n(int kind, int sym)
{
    switch (kind) {
    case KIND_COL_DD: return col_fn<N, 0>(sym);
    case KIND_COL_DS: return col_fn<N, 1>(sym);
    case KIND_ROW_R2C: return (void*)row_kernel<double, N, row_E<double>(N), row_B<double>(N), 0>;
    default: return nullptr;
    }
}
}  // namespace

void* pow2_pick_f64(int kind, int N, bool inv, int sym)
{
    if (inv) return nullptr;
    switch (N) {
    case 64: return pick_n<64>(kind, sym);
    case 128: return pick_n<128>(kind, sym);
    case 256: return pick_n<256>(kind, sym);
    case 512: return pick_n<512>(kind, sym);
    case 1024: return pick_n<1024>(kind, sym);
    case 2048: return pick_n<2048>(kind, sym);
    case 4096: return pick_n<4096>(kind, sym);
    default: return nullptr;
    }
}

void pow2_shape_f64(int kind, int N, int* B, int* tpl, size_t* smem)
{
    using namespace pw;
    if (kind == KIND_ROW_R2C) {
        const int E = row_E<double>(N);
        *B = row_B<double>(N);
        *tpl = N / E;
        *smem = (size_t)(*B) * (size_t)(N + N / E + 1) * sizeof(double) * 2;
    } else {
        *B = col_B<double>(N);
        *tpl = N / col_E<double>(N, kind == KIND_COL_DS ? 1 : 0);
        *smem = (size_t)(cpad_c(N - 1) + 1) * (size_t)(*B) * sizeof(double) * 2;
    }
}

}  // namespace p3
