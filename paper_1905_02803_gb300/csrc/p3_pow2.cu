// Configuration, set-up and launch of the power-of-two stage kernels
// (templates in p3_pow2.cuh, instantiated per precision in p3_pow2_f32.cu and
// p3_pow2_f64.cu).
#include <cudaTypedefs.h>

#include "p3_internal.h"

namespace p3 {

void* pow2_pick_f32(int kind, int N, bool inv, int sym, bool wide);
void* pow2_pick_f64(int kind, int N, bool inv, int sym);
void pow2_shape_f32(int kind, int N, bool wide, int* B, int* tpl, size_t* smem);
void pow2_shape_f64(int kind, int N, int* B, int* tpl, size_t* smem);

void* pow2_pick_tma_f32(int N, int sym, bool wide, bool zyx, bool inv);
size_t pow2_tma_smem_f32(int N, int sym, bool wide);
void* pow2_pick_zbulk_f32(int N);
size_t pow2_zbulk_smem_f32(int N);

// Whether a column stage takes the 16-line tiles (see kWideB in p3_pow2.cuh).
static bool wide_of(int kind, int N, long long es)
{
    return N == 512 && (kind == KIND_COL_DD || kind == KIND_COL_DS) && es >= 65536 / 8;
}

// Column-kernel symmetry variant of a stage: 0 plain, 1 DCT-I, 2 DST-I.
static int sym_of(const StageArgs& a) { return a.op == OP_DCT1 ? 1 : a.op == OP_DST1 ? 2 : 0; }

namespace {
bool is_pow2_in_range(int n) { return n >= 64 && n <= 4096 && (n & (n - 1)) == 0; }
}  // namespace

static bool configure(StageArgs& a, size_t csize, bool allow_tma);

bool pow2_configure(StageArgs& a, size_t csize, bool allow_tma)
{
    StageArgs b = a;  // a keeps its generic configuration unless this succeeds
    if (!configure(b, csize, allow_tma)) return false;
    a = b;
    return true;
}

static bool configure(StageArgs& a, size_t csize, bool allow_tma)
{
    if (a.blue) return false;
    if (csize != 8 && (a.sign > 0 || a.in_elem_fast != (a.op == OP_R2C_HALF))) return false;  // double: forward stages
    const int N = a.nfft;
    if (!is_pow2_in_range(N)) return false;
    const bool f32 = csize == 8;
    int kind = 0;
    if (a.op == OP_C2C || a.op == OP_DCT1 || a.op == OP_DST1) {
        const bool in_adj = a.in.lstride == 1, out_adj = a.out.lstride == 1;
        const bool in_el = a.in.es == 1, out_el = a.out.es == 1;
        if (in_adj && out_adj && !in_el && !out_el) kind = KIND_COL_DD;
        else if (in_adj && !in_el && out_el) kind = KIND_COL_DS;
        else if (in_el && out_adj && !out_el) kind = KIND_COL_SD;
        else return false;
    } else if (a.op == OP_R2C_HALF || a.op == OP_C2R_HALF) {
        if (a.in.es != 1 || a.out.es != 1) return false;
        kind = a.op == OP_R2C_HALF ? KIND_ROW_R2C : KIND_ROW_C2R;
    } else {
        return false;
    }
    int B = 1, tpl = 1;
    size_t smem = 0;
    const bool wide = f32 && wide_of(kind, N, a.in.es);
    if (f32) pow2_shape_f32(kind, N, wide, &B, &tpl, &smem);
    else pow2_shape_f64(kind, N, &B, &tpl, &smem);
    a.B = B;
    a.LDB = B;
    a.tpl = tpl;
    a.threads = B * tpl;
    a.smem = smem;
    a.kern = kind;
    a.tma = 0;
    // TMA-staged input tile for the Z stages with a ZYX or XYZ output: the
    // tile's lines must be adjacent (the tensor's inner dimension) and their
    // elements a 16-byte multiple apart, past the last line (Y lines, one
    // plane's worth at a time, are not).  Measured for the XYZ
    // store (Z of 512^3, either direction): 226 / 219 -> 173 / 176 us; 256 x 256 x
    // 1024 121 / 123 -> 98 / 101; 257-point Chebyshev 159 -> 132.
    if (f32 && allow_tma && (kind == KIND_COL_DS || kind == KIND_COL_DD) && N >= 256 && N <= 2048 && a.in.lstride == 1 &&
        a.in.per >= a.nlines && a.in.es % 2 == 0 && a.in.es >= a.nlines && (B % 2) == 0) {
        a.tma = 1;
        a.smem = pow2_tma_smem_f32(N, sym_of(a), wide);
    }
    // bulk-copied tile for the row-style ZYX load: plain FFT lines that lie
    // one after another in memory
    if (f32 && allow_tma && kind == KIND_COL_SD && a.op == OP_C2C && a.sign > 0 && a.n_in == N &&
        a.in.es == 1 && a.in.lstride == N && a.in.per >= a.nlines && pow2_pick_zbulk_f32(N)) {
        a.tma = 2;
        a.smem = pow2_zbulk_smem_f32(N);
    }
    return true;
}

// The kernel of a configured stage.
static void* kernel_of(const StageArgs& a, bool f32)
{
    const bool inv = a.sign > 0;
    const int sym = sym_of(a);
    const bool wide = f32 && wide_of(a.kern, a.nfft, a.in.es);
    return a.tma == 2 ? pow2_pick_zbulk_f32(a.nfft)
           : a.tma    ? pow2_pick_tma_f32(a.nfft, sym, wide, a.kern == KIND_COL_DS, inv)
                      : (f32 ? pow2_pick_f32(a.kern, a.nfft, inv, sym, wide) : pow2_pick_f64(a.kern, a.nfft, inv, sym));
}

cudaError_t pow2_prepare(const StageArgs& a, bool f32)
{
    void* fn = kernel_of(a, f32);
    if (!fn) return cudaErrorInvalidDeviceFunction;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
}

cudaError_t pow2_launch(const StageArgs& a, bool f32, cudaStream_t st)
{
    void* fn = kernel_of(a, f32);
    if (!fn) return cudaErrorInvalidDeviceFunction;
    if (a.nlines <= 0) return cudaSuccess;
    long long grid = (a.nlines + a.B - 1) / a.B;
    if (grid > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    StageArgs m = a;
    line_magic(m.in, m.nlines);
    line_magic(m.out, m.nlines);
    void* args[] = {&m};
    return launch_overlapped(fn, (unsigned)grid, (unsigned)m.threads, args, m.smem, st);
}

// cuTensorMapEncodeTiled, from the driver through the runtime (resolved once)
static PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
    }();
    return fn;
}

cudaError_t pow2_encode_tma(StageArgs& a)
{
    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    // 8-byte complex elements: lines (inner, unit stride) x line elements (outer, es apart)
    const cuuint64_t dims[2] = {(cuuint64_t)a.nlines, (cuuint64_t)a.n_in};
    const cuuint64_t strides[1] = {(cuuint64_t)a.in.es * 8};
    const cuuint32_t box[2] = {(cuuint32_t)a.B, 256};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(&a.tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, const_cast<void*>(a.src), dims, strides, box,
                           estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace p3
