// Configuration, set-up and launch of the FP64 fixed-point stage kernels
// (templates in p3_fix64.cuh, instantiated in p3_fix64_*.cu).
#include "p3_fix64.cuh"

namespace p3 {

namespace fx {
void* fn_cc(int cap);
void* fn_cs(int cap);
void* fn_sc(int cap);
void* fn_ss(int cap);
void* fn_ecc(int cap);
void* fn_ecs(int cap);
void* fn_esc(int cap);
void* fn_ess(int cap);
void* fn_r2c(int cap);
void* fn_c2r(int cap);
void* fn_rp(int cap);
void* fn_cp(int cap);
}  // namespace fx

namespace {

void* pick(int k, int cap)
{
    switch (k) {
    case fx::K_CC: return fx::fn_cc(cap);
    case fx::K_CS: return fx::fn_cs(cap);
    case fx::K_SC: return fx::fn_sc(cap);
    case fx::K_SS: return fx::fn_ss(cap);
    case fx::K_ECC: return fx::fn_ecc(cap);
    case fx::K_ECS: return fx::fn_ecs(cap);
    case fx::K_ESC: return fx::fn_esc(cap);
    case fx::K_ESS: return fx::fn_ess(cap);
    case fx::K_R2C: return fx::fn_r2c(cap);
    case fx::K_C2R: return fx::fn_c2r(cap);
    case fx::K_RP: return fx::fn_rp(cap);
    case fx::K_CP: return fx::fn_cp(cap);
    default: return nullptr;
    }
}

int butterflies(int R, int cap)
{
    if (cap <= 10) return 1;
    return R == 2 ? fx::bfly<2, 16>() : R == 3 ? fx::bfly<3, 16>() : R == 4 ? fx::bfly<4, 16>()
           : R == 5 ? fx::bfly<5, 16>() : R <= 8 ? fx::bfly<8, 16>() : 1;
}

}  // namespace

int fix64_threads(int n, int npass, const int* rad, int cap)
{
    int tpl = 1;
    for (int p = 0; p < npass; ++p) {
        const int nb = n / rad[p], bm = butterflies(rad[p], cap);
        const int need = (nb + bm - 1) / bm;
        if (need > tpl) tpl = need;
    }
    return tpl <= fx::kThreads ? tpl : 0;
}

bool fix64_configure(StageArgs& a, int shrink)
{
    const int n = a.nfft;
    int k;
    switch (a.op) {
    case OP_R2C_HALF: k = fx::K_R2C; break;
    case OP_C2R_HALF: k = fx::K_C2R; break;
    case OP_R2C_PAIR: k = fx::K_RP; break;
    case OP_C2R_PAIR: k = fx::K_CP; break;
    default:
        k = a.in_elem_fast ? (a.out_elem_fast ? fx::K_SS : fx::K_SC) : (a.out_elem_fast ? fx::K_CS : fx::K_CC);
        if (a.op != OP_C2C) k += fx::K_ECC - fx::K_CC;
        break;
    }
    const int cap = a.fix & 31;
    const int tpl = fix64_threads(n, a.npass, a.rad, cap);
    if (tpl < 1) return false;
    const bool staged = k != fx::K_CC && k != fx::K_ECC;
    const int slots = (k == fx::K_C2R || k == fx::K_CP) ? n + 1 : n;
    // tiles of at most 110 KB, so that two CTAs fit an SM
    constexpr size_t most = 110 * 1024;
    auto pitch = [&](int B) { return staged && B % 2 == 0 ? B + 1 : B; };
    int B = 1;
    while (2 * B * tpl <= fx::kThreads && 2 * B <= fx::kMaxB && (size_t)slots * pitch(2 * B) * 16 <= most) B *= 2;
    // small volumes: narrower tiles while they leave SMs without a CTA
    while (B > 4 && (a.nlines + B - 1) / B < 304) B /= 2;
    B >>= shrink;
    if (B < 1) return false;
    a.tpl = tpl;
    a.B = B;
    a.LDB = pitch(B);
    a.threads = (B * tpl + 31) / 32 * 32;
    a.smem = (size_t)slots * a.LDB * 16;
    a.kern = KIND_FIX64;
    a.fix = 32 * k + cap;
    a.tc = 0;
    a.tma = 0;
    return true;
}

const char* fix64_name(const StageArgs& a)
{
    // in the order of fx::Kind; forms 8, 10, 16
#define P3_FX_NAMES(k) {"fix64_" k "_8", "fix64_" k "_10", "fix64_" k "_16"}
    static const char* const names[][3] = {P3_FX_NAMES("cc"),  P3_FX_NAMES("cs"),  P3_FX_NAMES("sc"),  P3_FX_NAMES("ss"),
                                           P3_FX_NAMES("ecc"), P3_FX_NAMES("ecs"), P3_FX_NAMES("esc"), P3_FX_NAMES("ess"),
                                           P3_FX_NAMES("r2c"), P3_FX_NAMES("c2r"), P3_FX_NAMES("rp"),  P3_FX_NAMES("cp")};
#undef P3_FX_NAMES
    static_assert(sizeof(names) / sizeof(names[0]) == fx::K_CP + 1, "one row per kind");
    const int cap = a.fix & 31;
    return names[a.fix >> 5][cap == 8 ? 0 : cap == 10 ? 1 : 2];
}

cudaError_t fix64_prepare(const StageArgs& a)
{
    return cudaFuncSetAttribute(pick(a.fix >> 5, a.fix & 31), cudaFuncAttributeMaxDynamicSharedMemorySize, 110 * 1024);
}

cudaError_t fix64_launch(const StageArgs& a0, cudaStream_t st)
{
    if (a0.nlines <= 0) return cudaSuccess;
    const long long grid = (a0.nlines + a0.B - 1) / a0.B;
    if (grid > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    StageArgs a = a0;
    const long long nl = a.nrows > a.nlines ? a.nrows : a.nlines;  // pair ops index rows
    line_magic(a.in, nl);
    line_magic(a.out, nl);
    generic_consts(a);
    void* args[] = {&a};
    return launch_overlapped(pick(a.fix >> 5, a.fix & 31), (unsigned)grid, (unsigned)a.threads, args, a.smem, st);
}

}  // namespace p3
