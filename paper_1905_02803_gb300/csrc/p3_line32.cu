// Configuration, set-up and launch of the FP32 line kernels (templates in
// p3_line32.cuh, instantiated in p3_line32_a.cu and p3_line32_b.cu).
#include "p3_line32.cuh"

namespace p3 {

namespace l32 {
void* fn_a(int k);
void* fn_b(int k);
}  // namespace l32

namespace {

void* pick(int k)
{
    void* f = l32::fn_a(k);
    return f ? f : l32::fn_b(k);
}

int butterflies(int R)
{
    return R == 2 ? l32::bfly<2>() : R == 3 ? l32::bfly<3>() : R == 4 ? l32::bfly<4>() : R == 5 ? l32::bfly<5>()
           : R <= 8 ? l32::bfly<8>() : 1;
}

constexpr size_t kSmemMost = 110 * 1024;  // two CTAs per SM

// Pad shift of the row kernels' shared-memory lines (a slot after every 2^ps
// values; 31: none) with the fewest wavefronts over the exchanges of a CTA's
// first 64 threads.  A first pass of radix R writes R apart: R = 16 without a
// pad puts 16 lanes on one bank, and so does R = 15 with a pad every 16
// values (X stage of 375 x 360 x 343: 176 us with that pad, 125 without).  One
// 8-byte access of 16 lanes takes as many wavefronts as the most slots of one
// bank pair that they touch.
int row_pad(int n, int npass, const int* rad, int tpl, int B)
{
    static const int cand[] = {31, 4, 3, 2};
    int best = 31;
    long long least = -1;
    for (int ps : cand) {
        const int pitch = l32::rpitch(n, ps);
        long long waves = 0;
        long long Ns = 1;
        for (int p = 0; p < npass; ++p) {
            const int R = rad[p], nb = n / R;
            for (int rw = p == 0 ? 1 : 0; rw < 2; ++rw)  // 0: reads, 1: writes
                for (int h = 0; h < B * tpl && h < 64; h += 16)
                    for (int r = 0; r < R; ++r) {
                        int slot[16], most = 1;
                        int m = 0;
                        for (int i = h; i < h + 16 && i < B * tpl; ++i) {
                            const int l = i / tpl, j = i % tpl;
                            if (j >= nb) continue;
                            const int e = rw ? (int)((j / Ns) * Ns * R + j % Ns + r * Ns) : j + r * nb;
                            slot[m++] = l * pitch + l32::rslot(e, ps);
                        }
                        int cnt[16] = {0};
                        for (int i = 0; i < m; ++i) most = ++cnt[slot[i] & 15] > most ? cnt[slot[i] & 15] : most;
                        waves += most;
                    }
            Ns *= R;
        }
        if (least < 0 || waves < least) {
            least = waves;
            best = ps;
        }
    }
    return best;
}

}  // namespace

bool line32_configure(StageArgs& a, int shrink)
{
    if (a.blue || a.op == OP_COPY || a.npass < 1 || a.nfft < 2) return false;
    const bool si = a.in_elem_fast, so = a.out_elem_fast;
    int k = -1;
    switch (a.op) {
    case OP_R2C_HALF: k = l32::K_R2C; break;
    case OP_C2R_HALF: k = l32::K_C2R; break;
    case OP_R2C_PAIR: k = l32::K_RP; break;
    case OP_C2R_PAIR: k = l32::K_CP; break;
    case OP_C2C:
        if (a.sign < 0 && !si) k = so ? l32::K_CS : l32::K_CC;
        if (a.sign > 0 && !so) k = si ? l32::K_SCI : l32::K_CCI;
        break;
    default:
        if (!si || !so) k = si ? l32::K_ESC : so ? l32::K_ECS : l32::K_ECC;
        break;
    }
    if (k < 0) return false;
    const int n = a.nfft;
    int tpl = 1;
    for (int p = 0; p < a.npass; ++p) {
        const int R = a.rad[p], nb = n / R, bm = butterflies(R);
        if (R > 16 || R == 11 || R == 13) return false;
        tpl = tpl > (nb + bm - 1) / bm ? tpl : (nb + bm - 1) / bm;
    }
    if (tpl > l32::kThreads) return false;
    if (k >= l32::K_R2C) {
        // rows: any number of lines per CTA
        int B = l32::kThreads / tpl;
        const int ps = row_pad(n, a.npass, a.rad, tpl, B);
        const size_t row = (size_t)l32::rpitch(n, ps) * 8;
        while (B > 1 && B * row > kSmemMost) --B;
        while (B > 1 && (a.nlines + B - 1) / B < 304 && B * tpl > 32) B = (B + 1) / 2;
        B >>= shrink;
        if (B < 1) return false;
        a.B = B;
        a.LDB = ps;
        a.smem = B * row;
    } else {
        auto pitch = [&](int B) { return l32::staged_kind(k) && B % 2 == 0 ? B + 1 : B; };
        int B = 1;
        while (2 * B * tpl <= l32::kThreads && 2 * B <= l32::kMaxB && (size_t)n * pitch(2 * B) * 8 <= kSmemMost) B *= 2;
        // small volumes: narrower tiles while they leave SMs without a CTA
        while (B > 8 && (a.nlines + B - 1) / B < 304) B /= 2;
        B >>= shrink;
        if (B < 1) return false;
        a.B = B;
        a.LDB = pitch(B);
        a.smem = (size_t)n * a.LDB * 8;
    }
    if (a.smem > kSmemMost) return false;
    a.tpl = tpl;
    a.threads = (a.B * tpl + 31) / 32 * 32;
    a.kern = KIND_LINE32;
    a.fix = k;
    a.tc = 0;
    a.tma = 0;
    return true;
}

cudaError_t line32_prepare(const StageArgs& a)
{
    return cudaFuncSetAttribute(pick(a.fix), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMost);
}

cudaError_t line32_launch(const StageArgs& a0, cudaStream_t st)
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
    return launch_overlapped(pick(a.fix), (unsigned)grid, (unsigned)a.threads, args, a.smem, st);
}

}  // namespace p3
