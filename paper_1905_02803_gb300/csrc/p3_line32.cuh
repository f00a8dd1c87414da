// FP32 stage kernels for smooth line lengths that have no power-of-two kernel.
//
// The tile-in-shared-memory kernel (p3_kernels.cu) moved every value through
// shared memory once per pass and once more on the way in and out, from one
// buffer to another.  Here a thread takes up to 16 values of a line into
// registers for each pass and writes them back in place, so a tile needs one
// buffer; the first pass of a strided line reads HBM and the last pass
// writes HBM, and only contiguous sides (rows, the ZYX layout) are staged.
// A three-pass strided stage then touches shared memory 4 times per value
// instead of 8, and a tile takes half the bytes:
// four CTAs of 256 threads fit an SM.  Rows run with the lanes along the line
// and read HBM straight into the first pass.  The arithmetic is the same
// operation for operation, so the results are too.
//
// Pass twiddles come from tables in the order that consecutive butterflies read
// them (one sector per warp and value instead of up to one per lane).
//
// Measured (forward + inverse): 384^3 907 -> 671 us, 375 x 360 x 343 885 ->
// 645 us, 24 mixed grids 2.49 -> 1.75 ms, 48 x 40 x 36 37 -> 24 us (replayed
// graph).  Per complex point a strided stage of 384 issues 80 instructions
// (112 before), a row stage about 80 (125).  What bounds them now: no single
// unit (L1 data pipe 41 - 64 % busy, issue about 50 %); the rest waits for the
// tile's loads and the block barriers.  85 registers (three CTAs) were 5 - 10 %
// slower, 512-thread CTAs throughout 7 %.
#pragma once

#include "p3_copy.cuh"
#include "p3_dft.cuh"
#include "p3_internal.h"
#include "p3_launch.cuh"

namespace p3 {
namespace l32 {

typedef float2 C;
typedef long long ll;

enum Kind : int {
    K_CC = 0,   // complex lines, strided in and out, forward
    K_CCI = 1,  // the same, inverse
    K_CS = 2,   // strided in, contiguous out, forward (ZYX store)
    K_SCI = 3,  // contiguous in, strided out, inverse (ZYX load)
    K_ECC = 4,  // even and odd extensions (DCT-I, DST-I): strided in and out
    K_ECS = 5,  // strided in, contiguous out
    K_ESC = 6,  // contiguous in, strided out
    K_R2C = 7,  // even real rows -> half spectra
    K_C2R = 8,  // half spectra -> even real rows
    K_RP = 9,   // odd real rows in pairs -> half spectra
    K_CP = 10,  // half spectra in pairs -> odd real rows
    K_COUNT = 11,
};
template <int K> __host__ __device__ constexpr bool extended() { return K >= K_ECC && K <= K_ESC; }
template <int K> __host__ __device__ constexpr bool in_staged() { return K == K_SCI || K == K_ESC; }
template <int K> __host__ __device__ constexpr bool out_staged() { return K == K_CS || K == K_ECS; }
__host__ __device__ constexpr bool staged_kind(int k) { return k != K_CC && k != K_CCI && k != K_ECC; }
// the inverse-sign DFT as swp(DFT(swp(x)))
template <int K> __host__ __device__ constexpr bool inverse() { return K == K_CCI || K == K_SCI; }

constexpr int kMaxB = 32;
constexpr int kThreads = 256;  // threads of a CTA, four CTAs per SM (64 registers) ...
constexpr int kThreadsMost = 512;  // ... and for long lines, to keep tiles of up to 8 lines

// Butterflies a thread holds per pass (at most 16 values)
template <int R> __host__ __device__ constexpr int bfly()
{
    return R == 2 ? 8 : R == 3 ? 5 : R == 4 ? 4 : R == 5 ? 3 : R <= 8 ? 2 : 1;
}

struct Shared {
    ll bin[kMaxB], bout[kMaxB];  // line bases (elements)
};

// Butterflies past the end (and threads and lines past theirs) read the last
// one's values, which exist, and write nothing.
__device__ __forceinline__ int clamp(int j, int nb) { return j < nb ? j : nb - 1; }

struct Thread {
    int l, t;    // line of the tile, thread of the line
    bool act;    // takes part in the passes
    bool valid;  // ... and its line exists
};

// One Stockham pass of radix R over the tile, FIRST from the input (HBM or the
// staged tile).  Butterfly j reads elements j + r n/R, multiplies by
// exp(-2 pi i (j mod Ns) r / (Ns R)) and writes (j / Ns) Ns R + j mod Ns + r Ns.
// BULK: the input tile came line by line by bulk copies, element e of line l at
// l * a.box + e.
template <int K, bool BULK, int R, bool FIRST>
__device__ __forceinline__ void pass(const StageArgs& a, C* s, const Shared& sh, const Thread& th, int p, int Ns, int toff)
{
    constexpr int BM = bfly<R>();
    const int n = a.nfft, nb = n / R, tpl = a.tpl, LDB = a.LDB;
    const int l = th.l, t = th.t;
    const PassConsts& c = a.pc[p];
    const bool last = p + 1 == a.npass;
    const int q0 = FIRST ? t : (int)(((unsigned long long)(unsigned)t * c.pm) >> c.ps);
    const int r0 = FIRST ? 0 : t - q0 * Ns;
    const C zero = mk<C>(0.f, 0.f);
    C v[BM * R];

    if constexpr (FIRST && !in_staged<K>()) {
        const ll es = a.in.es;
        const int M = n >> 1;
        const C* g = static_cast<const C*>(a.src) + sh.bin[l];
#pragma unroll
        for (int b = 0; b < BM; ++b) {
            const int j = clamp(t + b * tpl, nb);
            const C* gp = g + j * es;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                C x = zero;
                if constexpr (!extended<K>()) {
                    x = *gp;
                    gp += nb * es;
                } else {
                    const int e = j + r * nb;
                    if (a.op == OP_DCT1) {
                        x = g[(e <= M ? e : n - e) * es];
                    } else if (e != 0 && e != M) {  // OP_DST1: 0, x[0..M-2], 0, -x[M-2..0]
                        x = g[(e < M ? e - 1 : n - 1 - e) * es];
                        if (e > M) x = mk<C>(-x.x, -x.y);
                    }
                }
                v[b * R + r] = inverse<K>() ? swp(x) : x;
            }
        }
    } else {
        const C* tw = static_cast<const C*>(a.twr) + toff;
        int rr = r0;
#pragma unroll
        for (int b = 0; b < BM; ++b) {
            const int j = clamp(t + b * tpl, nb);
            const int es = FIRST && BULK ? 1 : LDB;
            const C* si = FIRST && BULK ? s + l * a.box : s + l;
            const C* sp = si + j * es;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                C x = zero;
                if constexpr (FIRST && extended<K>()) {
                    const int e = j + r * nb, M = n >> 1;
                    if (a.op == OP_DCT1) {
                        x = si[(e <= M ? e : n - e) * es];
                    } else if (e != 0 && e != M) {
                        x = si[(e < M ? e - 1 : n - 1 - e) * es];
                        if (e > M) x = mk<C>(-x.x, -x.y);
                    }
                } else {
                    x = sp[r * nb * es];
                }
                v[b * R + r] = FIRST && inverse<K>() ? swp(x) : x;
            }
            if constexpr (!FIRST) {
                if (rr) {
                    const C* tp = tw + rr;
#pragma unroll
                    for (int r = 1; r < R; ++r) {
                        v[b * R + r] = mul(v[b * R + r], ldg(tp));
                        tp += Ns;
                    }
                }
                if (b + 1 < BM) {
                    rr += c.dr;
                    if (rr >= Ns) rr -= Ns;
                }
            }
        }
    }

#pragma unroll
    for (int b = 0; b < BM; ++b) Dft<C, float, R>::run(v + b * R);

    if constexpr (!out_staged<K>()) {
        if (last) {
            const ll es = a.out.es;
            const int M = n >> 1;
            C* g = static_cast<C*>(a.dst) + sh.bout[l];
            int qq = q0, rr = r0;
#pragma unroll
            for (int b = 0; b < BM; ++b) {
                const int j = t + b * tpl;
                const int o = FIRST ? j * R : qq * Ns * R + rr;
                if (th.valid && j < nb) {
                    C* gp = g + o * es;
                    const ll step = Ns * es;
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const C x = v[b * R + r];
                        if constexpr (!extended<K>()) {
                            *gp = inverse<K>() ? swp(x) : x;
                            gp += step;
                        } else {
                            const int e = o + r * Ns;
                            if (a.op == OP_DCT1) {
                                if (e <= M) g[e * es] = x;
                            } else if (e >= 1 && e < M) {  // i times bin e
                                g[(e - 1) * es] = mk<C>(-x.y, x.x);
                            }
                        }
                    }
                }
                if (!FIRST && b + 1 < BM) {
                    rr += c.dr;
                    qq += c.dq;
                    if (rr >= Ns) {
                        rr -= Ns;
                        ++qq;
                    }
                }
            }
            return;
        }
    }
    __syncthreads();  // every thread has read its inputs
    {
        int qq = q0, rr = r0;
#pragma unroll
        for (int b = 0; b < BM; ++b) {
            const int j = t + b * tpl;
            const int o = FIRST ? j * R : qq * Ns * R + rr;
            C* dp = s + o * LDB + l;
            if (th.act && j < nb) {
#pragma unroll
                for (int r = 0; r < R; ++r) dp[r * Ns * LDB] = v[b * R + r];
            }
            if (!FIRST && b + 1 < BM) {
                rr += c.dr;
                qq += c.dq;
                if (rr >= Ns) {
                    rr -= Ns;
                    ++qq;
                }
            }
        }
    }
    __syncthreads();
}

template <int K, bool BULK, bool FIRST>
__device__ __forceinline__ void pass_any(const StageArgs& a, C* s, const Shared& sh, const Thread& th, int p, int Ns,
                                         int toff)
{
    switch (a.rad[p]) {
#define P3_L32_PASS(R) \
    case R: pass<K, BULK, R, FIRST>(a, s, sh, th, p, Ns, toff); break;
        P3_L32_PASS(2) P3_L32_PASS(3) P3_L32_PASS(4) P3_L32_PASS(5) P3_L32_PASS(6) P3_L32_PASS(7) P3_L32_PASS(8)
        P3_L32_PASS(9) P3_L32_PASS(10) P3_L32_PASS(12) P3_L32_PASS(14) P3_L32_PASS(15) P3_L32_PASS(16)
#undef P3_L32_PASS
    default: break;
    }
}

template <int K, bool BULK = false>
__global__ void __launch_bounds__(kThreadsMost, 2) kernel(const __grid_constant__ StageArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Shared sh;
    // a bulk-copied tile is 128-byte aligned (144 bytes more are requested), with
    // its barrier after it
    unsigned char* base = BULK ? smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u) : smem_raw;
    C* s = reinterpret_cast<C*>(base);
    const int tid = threadIdx.x, B = a.B, LDB = a.LDB, n = a.nfft;
    const unsigned bar = BULK ? smem_u32(base + a.smem - 144) : 0u;
    if (BULK && tid == 0) copy_bar_init(bar, a.wait_extra);
    const int lb = __ffs(B) - 1;
    const ll L0 = (ll)blockIdx.x * B;
    const int rows = (int)(a.nlines - L0 < B ? a.nlines - L0 : B);
    if (tid < B) {
        const ll L = tid < rows ? L0 + tid : L0;  // lines past the end read the tile's first
        sh.bin[tid] = line_base(a.in, L);
        sh.bout[tid] = line_base(a.out, L);
    }
    __syncthreads();
    stage_begin();

    if constexpr (BULK) {
        if (tid == 0) {
            copy_bar_expect(bar, (unsigned)(rows * a.n_in * 8));
            for (int k = 0; k < rows; ++k)
                copy_bulk(smem_u32(s + k * a.box), static_cast<const C*>(a.src) + sh.bin[k], (unsigned)(a.n_in * 8), bar);
        }
        if (!copy_bar_wait(a, bar)) return;
    } else if constexpr (in_staged<K>()) {
        const C* F = static_cast<const C*>(a.src);
        walk<4>(rows, a.n_in, [&](int l, int e) { cp_async8(smem_u32(s + e * LDB + l), F + sh.bin[l] + e); });
        cp_async_wait();
        __syncthreads();
    }

    Thread th;
    th.l = tid & (B - 1);
    th.t = tid >> lb;
    th.act = th.t < a.tpl;
    th.valid = th.act && th.l < rows;
    pass_any<K, BULK, true>(a, s, sh, th, 0, 1, 0);
    int Ns = a.rad[0], toff = 0;  // toff: the pass's place in the table of pass twiddles
    for (int p = 1; p < a.npass; ++p) {
        pass_any<K, BULK, false>(a, s, sh, th, p, Ns, toff);
        toff += (a.rad[p] - 1) * Ns;
        Ns *= a.rad[p];
    }

    if constexpr (K == K_CS) {
        C* F = static_cast<C*>(a.dst);
        if (n % 2 == 0 && a.out.lstride % 2 == 0 && a.out.gstride % 2 == 0) {
            // lines start on 16 bytes: two values per store
            walk<4>(rows, n / 2, [&](int l, int h) {
                const C x = s[2 * h * LDB + l], y = s[(2 * h + 1) * LDB + l];
                *reinterpret_cast<float4*>(F + sh.bout[l] + 2 * h) = make_float4(x.x, x.y, y.x, y.y);
            });
        } else {
            walk<4>(rows, n, [&](int l, int e) { F[sh.bout[l] + e] = s[e * LDB + l]; });
        }
    } else if constexpr (K == K_ECS) {
        C* F = static_cast<C*>(a.dst);
        const bool dst1 = a.op == OP_DST1;  // i times bin e + 1
        walk<4>(rows, a.n_out, [&](int l, int e) {
            const C x = s[(e + (dst1 ? 1 : 0)) * LDB + l];
            F[sh.bout[l] + e] = dst1 ? mk<C>(-x.y, x.x) : x;
        });
    }
}

// ---------------------------------------------------------------------------
// Rows (X stage).  Lanes run along the line here: thread tid works on line
// tid / tpl, whose values sit in shared memory one after another, with a pad
// slot after every 2^LDB of them (the shift that leaves the fewest bank
// conflicts over all passes, found by the host: row_pad).  The first pass reads
// the rows from HBM with the real-to-complex packing or the inverse
// pre-twiddle on the way; the inverse's last pass writes HBM, and the
// forward's result crosses shared memory once more for the real split, which
// needs Z[k] and Z[n-k] together.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int rslot(int e, int ps) { return e + (e >> ps); }
__host__ __device__ constexpr int rpitch(int n, int ps) { return (rslot(n - 1, ps) + 1) | 1; }

struct Row {
    int t;               // thread of the line
    bool valid;          // the line exists and the thread takes part
    bool two;            // pairs: the second row exists
    ll bi, bo, bi2, bo2; // row bases (elements)
};

template <int K, int R, bool FIRST>
__device__ __forceinline__ void row_pass(const StageArgs& a, C* s, const Row& th, int p, int Ns, int toff)
{
    constexpr int BM = bfly<R>();
    const int n = a.nfft, nb = n / R, tpl = a.tpl, t = th.t, ps = a.LDB;
    const PassConsts& c = a.pc[p];
    const bool last = p + 1 == a.npass;
    const int q0 = FIRST ? t : (int)(((unsigned long long)(unsigned)t * c.pm) >> c.ps);
    const int r0 = FIRST ? 0 : t - q0 * Ns;
    C v[BM * R];

    if constexpr (FIRST) {
#pragma unroll
        for (int b = 0; b < BM; ++b) {
            const int j = clamp(t + b * tpl, nb);
            if constexpr (K == K_R2C) {
                const C* g = reinterpret_cast<const C*>(static_cast<const float*>(a.src) + th.bi) + j;
#pragma unroll
                for (int r = 0; r < R; ++r) v[b * R + r] = g[r * nb];
            } else if constexpr (K == K_RP) {
                const float* f1 = static_cast<const float*>(a.src) + th.bi + j;
                const float* f2 = static_cast<const float*>(a.src) + th.bi2 + j;
#pragma unroll
                for (int r = 0; r < R; ++r) v[b * R + r] = mk<C>(f1[r * nb], th.two ? f2[r * nb] : 0.f);
            } else if constexpr (K == K_C2R) {
                // Z[k] = (F[k] + conj F[n-k]) + i (F[k] - conj F[n-k]) exp(+2 pi i k / 2n),
                // imaginary parts of F[0] and F[n] dropped; swapped for the inverse
                const C* F = static_cast<const C*>(a.src) + th.bi;
                const C* tw2 = static_cast<const C*>(a.tw2);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int k = j + r * nb;
                    C Fk = F[k], Fm = F[n - k];
                    if (r == 0 && k == 0) {
                        Fk.y = 0.f;
                        Fm.y = 0.f;
                    }
                    const C B_ = cnj(Fm);
                    const C ze = add(Fk, B_);
                    const C zo = mul(sub(Fk, B_), cnj(ldg(tw2 + k)));
                    v[b * R + r] = swp(mk<C>(ze.x - zo.y, ze.y + zo.x));
                }
            } else {
                // Z[k] = X1[k] + i X2[k], Z[n-k] = conj X1[k] + i conj X2[k] (k >= 1);
                // imaginary parts of X1[0], X2[0] dropped; swapped for the inverse
                const C* F1 = static_cast<const C*>(a.src) + th.bi;
                const C* F2 = static_cast<const C*>(a.src) + th.bi2;
                const int H = a.n_in;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int e = j + r * nb;
                    const bool low = e < H;
                    const int k = low ? e : n - e;
                    C A = F1[k], Bv = mk<C>(0.f, 0.f);
                    if (th.two) Bv = F2[k];
                    if (r == 0 && k == 0) {
                        A.y = 0.f;
                        Bv.y = 0.f;
                    }
                    v[b * R + r] = low ? swp(mk<C>(A.x - Bv.y, A.y + Bv.x)) : swp(mk<C>(A.x + Bv.y, Bv.x - A.y));
                }
            }
        }
    } else {
        const C* tw = static_cast<const C*>(a.twr) + toff;
        int rr = r0;
#pragma unroll
        for (int b = 0; b < BM; ++b) {
            const int j = clamp(t + b * tpl, nb);
#pragma unroll
            for (int r = 0; r < R; ++r) v[b * R + r] = s[rslot(j + r * nb, ps)];
            if (rr) {
                const C* tp = tw + rr;
#pragma unroll
                for (int r = 1; r < R; ++r) {
                    v[b * R + r] = mul(v[b * R + r], ldg(tp));
                    tp += Ns;
                }
            }
            if (b + 1 < BM) {
                rr += c.dr;
                if (rr >= Ns) rr -= Ns;
            }
        }
    }

#pragma unroll
    for (int b = 0; b < BM; ++b) Dft<C, float, R>::run(v + b * R);

    const bool direct = last && (K == K_C2R || K == K_CP);
    if (!direct) __syncthreads();  // every thread has read its inputs
    int qq = q0, rr = r0;
#pragma unroll
    for (int b = 0; b < BM; ++b) {
        const int j = t + b * tpl;
        const int o = FIRST ? j * R : qq * Ns * R + rr;
        if (th.valid && j < nb) {
            if (!direct) {
#pragma unroll
                for (int r = 0; r < R; ++r) s[rslot(o + r * Ns, ps)] = v[b * R + r];
            } else if constexpr (K == K_C2R) {
                C* f = reinterpret_cast<C*>(static_cast<float*>(a.dst) + th.bo) + o;
#pragma unroll
                for (int r = 0; r < R; ++r) f[r * Ns] = swp(v[b * R + r]);
            } else if constexpr (K == K_CP) {
                float* f1 = static_cast<float*>(a.dst) + th.bo + o;
                float* f2 = static_cast<float*>(a.dst) + th.bo2 + o;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    f1[r * Ns] = v[b * R + r].y;
                    if (th.two) f2[r * Ns] = v[b * R + r].x;
                }
            }
        }
        if (!FIRST && b + 1 < BM) {
            rr += c.dr;
            qq += c.dq;
            if (rr >= Ns) {
                rr -= Ns;
                ++qq;
            }
        }
    }
    if (!direct) __syncthreads();
}

template <int K, bool FIRST> __device__ __forceinline__ void row_any(const StageArgs& a, C* s, const Row& th, int p, int Ns, int toff)
{
    switch (a.rad[p]) {
#define P3_L32_PASS(R) \
    case R: row_pass<K, R, FIRST>(a, s, th, p, Ns, toff); break;
        P3_L32_PASS(2) P3_L32_PASS(3) P3_L32_PASS(4) P3_L32_PASS(5) P3_L32_PASS(6) P3_L32_PASS(7) P3_L32_PASS(8)
        P3_L32_PASS(9) P3_L32_PASS(10) P3_L32_PASS(12) P3_L32_PASS(14) P3_L32_PASS(15) P3_L32_PASS(16)
#undef P3_L32_PASS
    default: break;
    }
}

template <int K> __global__ void __launch_bounds__(kThreadsMost, 2) row_kernel(const __grid_constant__ StageArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* s = reinterpret_cast<C*>(smem_raw);
    constexpr bool PAIR = K == K_RP || K == K_CP;
    const int tid = threadIdx.x, B = a.B, n = a.nfft, tpl = a.tpl;
    int l = tid / tpl;
    const bool in = l < B;
    if (!in) l = B - 1;  // threads past the last line follow it and write nothing
    Row th;
    th.t = in ? tid - l * tpl : 0;
    ll L = (ll)blockIdx.x * B + l;
    th.valid = in && L < a.nlines;
    if (L >= a.nlines) L = a.nlines - 1;
    th.bi = line_base(a.in, PAIR ? 2 * L : L);
    th.bo = line_base(a.out, PAIR ? 2 * L : L);
    th.bi2 = th.bi;
    th.bo2 = th.bo;
    th.two = PAIR && 2 * L + 1 < a.nrows;
    if (th.two) {
        th.bi2 = line_base(a.in, 2 * L + 1);
        th.bo2 = line_base(a.out, 2 * L + 1);
    }
    const int ps = a.LDB;
    C* sl = s + l * rpitch(n, ps);
    stage_begin();
    row_any<K, true>(a, sl, th, 0, 1, 0);
    int Ns = a.rad[0], toff = 0;
    for (int p = 1; p < a.npass; ++p) {
        row_any<K, false>(a, sl, th, p, Ns, toff);
        toff += (a.rad[p] - 1) * Ns;
        Ns *= a.rad[p];
    }
    if constexpr (K == K_R2C) {
        // F[k] = (Z[k] + conj Z[n-k]) / 2 - i W (Z[k] - conj Z[n-k]) / 2, W = exp(-2 pi i k / 2n);
        // F[n-k] the same with W (Z[k] - conj Z[n-k]) conjugated
        if (th.valid) {
            const C* tw2 = static_cast<const C*>(a.tw2);
            C* F = static_cast<C*>(a.dst) + th.bo;
            for (int k = th.t; 2 * k <= n; k += tpl) {
                const C zk = sl[rslot(k, ps)], zn = sl[rslot(k == 0 ? 0 : n - k, ps)];
                const C q = mul(ldg(tw2 + k), sub(zk, cnj(zn)));
                F[k] = mk<C>(0.5f * (zk.x + zn.x + q.y), 0.5f * (zk.y - zn.y - q.x));
                if (2 * k < n) F[n - k] = mk<C>(0.5f * (zn.x + zk.x - q.y), 0.5f * (zn.y - zk.y - q.x));
            }
        }
    } else if constexpr (K == K_RP) {
        // X1[k] = (Z[k] + conj Z[n-k]) / 2, X2[k] = -i (Z[k] - conj Z[n-k]) / 2
        if (th.valid) {
            C* F1 = static_cast<C*>(a.dst) + th.bo;
            C* F2 = static_cast<C*>(a.dst) + th.bo2;
            for (int k = th.t; k < a.n_out; k += tpl) {
                const C zk = sl[rslot(k, ps)], zm = sl[rslot(k == 0 ? 0 : n - k, ps)];
                F1[k] = mk<C>(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
                if (th.two) F2[k] = mk<C>(0.5f * (zk.y + zm.y), 0.5f * (zm.x - zk.x));
            }
        }
    }
}

}  // namespace l32
}  // namespace p3
