// Configuration, set-up and launch of the FP32 line kernels (templates in
// p3_line32.cuh, instantiated in p3_line32_a.cu and p3_line32_b.cu).
#include "p3_line32.cuh"

namespace p3 {

namespace l32 {
void* fn_a(int k, int tma);
void* fn_b(int k);
}  // namespace l32

namespace {

void* pick(const StageArgs& a)
{
    void* f = l32::fn_a(a.fix, a.tma);
    return f ? f : l32::fn_b(a.fix);
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

bool line32_configure(StageArgs& a, int shrink, bool allow_tma)
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
    if (tpl > l32::kThreadsMost) return false;
    if (k >= l32::K_R2C) {
        // rows: any number of lines per CTA
        // Short even rows stay with the generic kernel, whose threads walk a tile's
        // rows as one run: a row's one to three threads here read its values
        // apart.  32 x 256 x 512: 58 us against 76; 60-point rows 53 against 57;
        // 48 the same; 80-point rows 64 against 62.  Volumes below 2^20 values are
        // bound by latency and run faster here (48 x 40 x 36: 25 us against 31).
        if ((k == l32::K_R2C || k == l32::K_C2R) && n < 32 && a.nlines * n >= (1LL << 20)) return false;
        int B = tpl < l32::kThreads ? l32::kThreads / tpl : 1;
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
        // up to 8 lines; 16 for the ZYX store, whose odd pitch then has no bank
        // conflicts (343 points: 117 -> 107 us; the other kinds lose 3 - 15 %)
        const int wide = k == l32::K_CS || k == l32::K_ECS ? 16 : 8;
        int B = 1;
        while (2 * B * tpl <= (B < wide ? l32::kThreadsMost : l32::kThreads) && 2 * B <= l32::kMaxB &&
               (size_t)n * pitch(2 * B) * 8 <= kSmemMost)
            B *= 2;
        // small volumes: narrower tiles while they leave SMs without a CTA
        while (B > 8 && (a.nlines + B - 1) / B < 304) B /= 2;
        B >>= shrink;
        if (B < 1) return false;
        a.B = B;
        a.LDB = pitch(B);
        a.smem = (size_t)n * a.LDB * 8;
    }
    if (a.smem > kSmemMost) return false;
    a.tma = 0;
    a.box = 0;
    const size_t plain = a.smem;
    if (allow_tma && k == l32::K_SCI && n % 2 == 0 && a.in.lstride % 2 == 0 && a.in.gstride % 2 == 0 &&
        a.nlines * n >= (1LL << 22)) {
        // line copies: lines of whole 16 bytes; the pitch puts a half-warp's
        // lines on distinct banks.  384^3: 137 -> 121 us, 300 x 324 x 270 80 -> 75;
        // volumes of a few MB lie in L2, where the barrier costs more than the
        // loads' latency (24 mixed grids: 1 % slower with it everywhere)
        a.box = n + 2;
        while (a.box % 4 != 2) a.box += 2;
        const size_t tile = (size_t)a.B * a.box * 8;
        a.smem = ((plain > tile ? plain : tile) + 15) / 16 * 16 + 144;
        a.tma = 2;
    }
    if (a.smem > kSmemMost + 1024) {
        a.tma = 0;
        a.box = 0;
        a.smem = plain;
    }
    a.tpl = tpl;
    a.threads = (a.B * tpl + 31) / 32 * 32;
    a.kern = KIND_LINE32;
    a.fix = k;
    a.tc = 0;
    return true;
}

cudaError_t line32_prepare(const StageArgs& a)
{
    return cudaFuncSetAttribute(pick(a), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMost + 1024);
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
    return launch_overlapped(pick(a), (unsigned)grid, (unsigned)a.threads, args, a.smem, st);
}

}  // namespace p3
