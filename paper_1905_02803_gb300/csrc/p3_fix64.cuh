// FP64 line transforms in 64-bit block fixed point.
//
// The FP64 pipe of this part issues 2 lanes per clock and SM; its 32-bit
// integer pipe adds 128 and multiplies (32 x 32 + 64) 64.  A double-precision
// FFT in double arithmetic is therefore bound by the FP64 pipe at more than
// ten times its memory time (512^3 pair 22.6 ms against 1.9 ms of HBM
// traffic).  These kernels keep the values of one line as 64-bit integers
// with one exponent per line (block floating point): a butterfly addition is
// two 32-bit additions, a multiplication by a 64-bit twiddle part three
// 32 x 32 -> 64 multiply-adds.  Doubles appear only in HBM.  Measured against
// the double kernels: 32^3 forward + inverse 145 -> 30 us, 243 x 250 x 180 2450 ->
// 767 us; inverse of 512^3 11.2 -> 3.1 ms (stages 3.45 / 3.45 / 4.27 -> 0.89 /
// 0.87 / 1.33 ms), of the 480 x 360 x 257 channel grid 5.3 -> 1.4 ms.  What bounds
// them now: issue slots 40-50 % busy, the rest waits for instruction fetch (long
// unrolled passes), the double conversions and the dependent chains of 16 to 32
// warps per SM.
//
// Precision.  A line is aligned to its largest component: |v| < 2^58, so the
// quantum is at least 2^-58 of that component, 2^5 finer than the last bit of
// a double of its size.  Between passes the line is shifted up by its actual
// headroom (an OR over all magnitudes), so a pass loses only the bits that
// the data really grew; twiddles carry 60 fractional bits and the butterfly
// constants 64 (a double: 53).  The result is rounded once, to nearest, when
// it becomes a double again.  Components below 2^-5 of the line's largest keep
// fewer bits than a double, those below 2^-58 none; as every output sums over
// the whole line (over both rows of an odd pair), errors are relative to the
// line's largest component, as they are in double arithmetic.  Relative errors of a forward + inverse pair
// against a 64-bit reference: 3.5e-16 -> 2.7e-16 (32^3) and 6.0e-16 -> 3.7e-16
// (243 x 250 x 180) from the double kernels to these.
//
// Bounds.  Components of |v| < 2^58 make complex moduli below 2^58.5; a
// radix-R butterfly (R <= 16) and all its partial sums stay below
// R 2^58.5 <= 2^62.5, inside a signed 64-bit integer.  The twiddle product
// multiplies by w 2^60 and keeps the high 64 bits, a scale of 2^-4, which
// returns every modulus below 2^62.5 to below 2^58.5.
//
// Lines with an infinity or a NaN give NaN throughout (every output of such
// a line is undefined in double arithmetic too); lines whose largest value
// is below 2^-959 are scaled up before and down after, and results beyond
// the double range overflow to infinity or round to denormals.
#pragma once

#include <cuda_runtime.h>

#include "p3_copy.cuh"
#include "p3_internal.h"
#include "p3_launch.cuh"

// the arithmetic below also builds for the host, where the tests pin it
#define P3_FX_HD __host__ __device__ __forceinline__

namespace p3 {
namespace fx {

typedef long long ll;

// complex value of a line: v * 2^(line exponent)
struct __align__(16) Q {
    ll x, y;
};

P3_FX_HD Q add(Q a, Q b) { return Q{a.x + b.x, a.y + b.y}; }
P3_FX_HD Q sub(Q a, Q b) { return Q{a.x - b.x, a.y - b.y}; }
P3_FX_HD Q swp(Q a) { return Q{a.y, a.x}; }
P3_FX_HD Q add_mmi(Q a, Q t) { return Q{a.x + t.y, a.y - t.x}; }  // a + (-i) t
P3_FX_HD Q sub_mmi(Q a, Q t) { return Q{a.x - t.y, a.y + t.x}; }  // a - (-i) t

// v = h 2^32 + l with a signed low half
struct Half {
    int h, l;
};
P3_FX_HD Half split(ll v)
{
    const int l = (int)v;
    return Half{(int)(v >> 32) + (int)((unsigned)l >> 31), l};
}
__host__ __device__ constexpr int lo_of(ll f) { return (int)(unsigned)(unsigned long long)f; }
__host__ __device__ constexpr int hi_of(ll f) { return (int)((f - (ll)lo_of(f)) >> 32); }

// Compile-time constant c = B + F / 2^64, |F| < 2^63 (B the nearest integer).
// floor(v F / 2^64), short of the product of the low halves (below 1 unit)
template <ll F> P3_FX_HD ll mulf(Half v)
{
    ll c = (ll)v.l * hi_of(F);
    c += (ll)v.h * lo_of(F);
    return (c >> 32) + (ll)v.h * hi_of(F);
}
template <int B> P3_FX_HD ll times(ll v) { return B == 0 ? 0 : B > 0 ? v : -v; }

// a (c + i s) with constant parts; |fractions of c| + |s| < 0.75, moduli below
// 2^61, so the sum of the four cross products stays below 2^63
template <int CB, ll CF, int SB, ll SF> P3_FX_HD Q rot(Q a)
{
    const Half x = split(a.x), y = split(a.y);
    ll r = (ll)x.l * hi_of(CF);
    r += (ll)y.l * hi_of(-SF);
    r += (ll)x.h * lo_of(CF);
    r += (ll)y.h * lo_of(-SF);
    r = (r >> 32) + (ll)x.h * hi_of(CF);
    r += (ll)y.h * hi_of(-SF);
    ll i = (ll)x.l * hi_of(SF);
    i += (ll)y.l * hi_of(CF);
    i += (ll)x.h * lo_of(SF);
    i += (ll)y.h * lo_of(CF);
    i = (i >> 32) + (ll)x.h * hi_of(SF);
    i += (ll)y.h * hi_of(CF);
    return Q{r + times<CB>(a.x) - times<SB>(a.y), i + times<SB>(a.x) + times<CB>(a.y)};
}

// Twiddle w 2^60 as {re high, re low, im high, im low}, low halves signed.
// a w / 2^4 (moduli of a below 2^62.5)
P3_FX_HD Q mulw(Q a, int4 w)
{
    const Half x = split(a.x), y = split(a.y);
    const int nh = -w.z, nl = -w.w;
    ll r = (ll)x.l * w.x;
    r += (ll)y.l * nh;
    r += (ll)x.h * w.y;
    r += (ll)y.h * nl;
    r = (r >> 32) + (ll)x.h * w.x;
    r += (ll)y.h * nh;
    ll i = (ll)x.l * w.z;
    i += (ll)y.l * w.x;
    i += (ll)x.h * w.w;
    i += (ll)y.h * w.y;
    i = (i >> 32) + (ll)x.h * w.z;
    i += (ll)y.h * w.x;
    return Q{r, i};
}

// ---------------------------------------------------------------------------
// Forward DFT butterflies exp(-2 pi i n m / R) on v[0..R), in place.
// Constants: fractional parts times 2^64, rounded (from 60-digit values).
// ---------------------------------------------------------------------------
constexpr ll kC1 = -1404174782535421627LL;  // cos(pi/8) = 1 + F
constexpr ll kS1 = 7059263338087549767LL;   // sin(pi/8) = F
constexpr ll kH = -5402926248376769404LL;   // sqrt(1/2) = 1 + F
constexpr ll kR3 = -2471395088767036514LL;  // sqrt(3)/2 = 1 + F
constexpr ll kR5 = -8134700645620564469LL;  // sqrt(5)/4 = 1 + F
constexpr ll kS51 = -902847917979075853LL;  // sin(2 pi/5) = 1 + F
constexpr ll kS52 = -7604019954369499282LL; // sin(4 pi/5) = 1 + F

P3_FX_HD ll mulh(ll v) { return v + mulf<kH>(split(v)); }  // v sqrt(1/2)
P3_FX_HD Q rot45(Q a) { return Q{mulh(a.x + a.y), mulh(a.y - a.x)}; }    // exp(-i pi/4)
P3_FX_HD Q rot135(Q a) { return Q{mulh(a.y - a.x), -mulh(a.x + a.y)}; }  // exp(-3i pi/4)

template <bool R2 = false> P3_FX_HD void dft4(Q& a0, Q& a1, Q& a2, Q& a3)
{
    const Q s02 = R2 ? add_mmi(a0, a2) : add(a0, a2), d02 = R2 ? sub_mmi(a0, a2) : sub(a0, a2);
    const Q s13 = add(a1, a3), t = sub(a1, a3);
    a0 = add(s02, s13);
    a2 = sub(s02, s13);
    a1 = add_mmi(d02, t);
    a3 = sub_mmi(d02, t);
}

template <int R> struct D;

template <> struct D<2> {
    static P3_FX_HD void run(Q* v)
    {
        const Q a = v[0];
        v[0] = add(a, v[1]);
        v[1] = sub(a, v[1]);
    }
};
template <> struct D<3> {
    static P3_FX_HD void run(Q* v)
    {
        const Q t = add(v[1], v[2]), d = sub(v[1], v[2]);
        const Q m = Q{v[0].x - (t.x >> 1), v[0].y - (t.y >> 1)};
        const Q e = Q{d.x + mulf<kR3>(split(d.x)), d.y + mulf<kR3>(split(d.y))};
        v[0] = add(v[0], t);
        v[1] = add_mmi(m, e);
        v[2] = sub_mmi(m, e);
    }
};
template <> struct D<4> {
    static P3_FX_HD void run(Q* v) { dft4(v[0], v[1], v[2], v[3]); }
};
template <> struct D<5> {
    // cos(2 pi/5) = -1/4 + sqrt(5)/4, cos(4 pi/5) = -1/4 - sqrt(5)/4
    static P3_FX_HD void part(ll v0, ll t1, ll t2, ll t3, ll t4, ll& m0, ll& p, ll& q, ll& r1, ll& r2)
    {
        const ll t5 = t1 + t2, u = t1 - t2;
        const ll a = v0 - (t5 >> 2), b = u + mulf<kR5>(split(u));
        m0 = v0 + t5;
        p = a + b;
        q = a - b;
        const Half h3 = split(t3), h4 = split(t4);
        r1 = t3 + mulf<kS51>(h3) + t4 + mulf<kS52>(h4);
        r2 = t3 + mulf<kS52>(h3) - t4 - mulf<kS51>(h4);
    }
    static P3_FX_HD void run(Q* v)
    {
        const Q t1 = add(v[1], v[4]), t2 = add(v[2], v[3]), t3 = sub(v[1], v[4]), t4 = sub(v[2], v[3]);
        Q m0, p, q, r1, r2;
        part(v[0].x, t1.x, t2.x, t3.x, t4.x, m0.x, p.x, q.x, r1.x, r2.x);
        part(v[0].y, t1.y, t2.y, t3.y, t4.y, m0.y, p.y, q.y, r1.y, r2.y);
        v[0] = m0;
        v[1] = add_mmi(p, r1);
        v[4] = sub_mmi(p, r1);
        v[2] = add_mmi(q, r2);
        v[3] = sub_mmi(q, r2);
    }
};
template <> struct D<7> {
    // cos / sin of 2 pi k / 7, k = 1, 2, 3, as B + F / 2^64
    static P3_FX_HD ll c1(ll v, Half h) { return v + mulf<-6945387266253616282LL>(h); }
    static P3_FX_HD ll c2(ll, Half h) { return mulf<-4104786719734957267LL>(h); }
    static P3_FX_HD ll c3(ll v, Half h) { return mulf<1826801949133797741LL>(h) - v; }
    static P3_FX_HD ll s1(ll v, Half h) { return v + mulf<-4024498807852869538LL>(h); }
    static P3_FX_HD ll s2(ll v, Half h) { return v + mulf<-462498387375470819LL>(h); }
    static P3_FX_HD ll s3(ll, Half h) { return mulf<8003742293245756417LL>(h); }
    static P3_FX_HD void part(ll a, ll p1, ll p2, ll p3, ll q1, ll q2, ll q3, ll (&re)[4], ll (&im)[4])
    {
        const Half P1 = split(p1), P2 = split(p2), P3 = split(p3);
        const Half Q1 = split(q1), Q2 = split(q2), Q3 = split(q3);
        re[0] = a + p1 + p2 + p3;
        re[1] = a + c1(p1, P1) + c2(p2, P2) + c3(p3, P3);
        re[2] = a + c2(p1, P1) + c3(p2, P2) + c1(p3, P3);  // multiples 2, 4 = -3, 6 = -1
        re[3] = a + c3(p1, P1) + c1(p2, P2) + c2(p3, P3);  // multiples 3, 6 = -1, 9 = 2
        im[1] = s1(q1, Q1) + s2(q2, Q2) + s3(q3, Q3);
        im[2] = s2(q1, Q1) - s3(q2, Q2) - s1(q3, Q3);
        im[3] = s3(q1, Q1) - s1(q2, Q2) + s2(q3, Q3);
    }
    static P3_FX_HD void run(Q* v)
    {
        const Q p1 = add(v[1], v[6]), p2 = add(v[2], v[5]), p3 = add(v[3], v[4]);
        const Q q1 = sub(v[1], v[6]), q2 = sub(v[2], v[5]), q3 = sub(v[3], v[4]);
        ll rx[4], ry[4], ix[4], iy[4];
        part(v[0].x, p1.x, p2.x, p3.x, q1.x, q2.x, q3.x, rx, ix);
        part(v[0].y, p1.y, p2.y, p3.y, q1.y, q2.y, q3.y, ry, iy);
        v[0] = Q{rx[0], ry[0]};
#pragma unroll
        for (int m = 1; m < 4; ++m) {
            v[m] = add_mmi(Q{rx[m], ry[m]}, Q{ix[m], iy[m]});
            v[7 - m] = sub_mmi(Q{rx[m], ry[m]}, Q{ix[m], iy[m]});
        }
    }
};
template <> struct D<8> {
    static P3_FX_HD void run(Q* v)
    {
        Q u0 = add(v[0], v[4]), u1 = add(v[1], v[5]), u2 = add(v[2], v[6]), u3 = add(v[3], v[7]);
        Q w0 = sub(v[0], v[4]), w1 = sub(v[1], v[5]), w2 = sub(v[2], v[6]), w3 = sub(v[3], v[7]);
        w1 = rot45(w1);
        w3 = rot135(w3);
        dft4(u0, u1, u2, u3);
        dft4<true>(w0, w1, w2, w3);
        v[0] = u0; v[2] = u1; v[4] = u2; v[6] = u3;
        v[1] = w0; v[3] = w1; v[5] = w2; v[7] = w3;
    }
};
template <> struct D<9> {
    // 3 x 3: DFT3 over n1 of x[3 n1 + n2], exp(-2 pi i n2 k1 / 9), DFT3 over n2
    static P3_FX_HD void run(Q* v)
    {
        Q y[9];
#pragma unroll
        for (int n2 = 0; n2 < 3; ++n2) {
            Q a[3] = {v[n2], v[n2 + 3], v[n2 + 6]};
            D<3>::run(a);
            y[n2] = a[0];
            y[3 + n2] = a[1];
            y[6 + n2] = a[2];
        }
        constexpr ll c1 = -4315718282406409839LL, s1 = -6589405544070453923LL;  // 40 degrees: 1 + F, 1 + F
        constexpr ll c2 = 3203243492287910726LL, s2 = -280247492088382768LL;    // 80: F, 1 + F
        constexpr ll c4 = 1112474790118499113LL, s4 = 6309158051982071155LL;    // 160: -1 + F, F
        y[4] = rot<1, c1, -1, -s1>(y[4]);  // k1 = 1, n2 = 1
        y[5] = rot<0, c2, -1, -s2>(y[5]);  // k1 = 1, n2 = 2
        y[7] = rot<0, c2, -1, -s2>(y[7]);  // k1 = 2, n2 = 1
        y[8] = rot<-1, c4, 0, -s4>(y[8]);  // k1 = 2, n2 = 2
#pragma unroll
        for (int k1 = 0; k1 < 3; ++k1) {
            D<3>::run(y + 3 * k1);
            v[k1] = y[3 * k1];
            v[k1 + 3] = y[3 * k1 + 1];
            v[k1 + 6] = y[3 * k1 + 2];
        }
    }
};
template <> struct D<16> {
    // 4 x 4, as the double kernels' radix 16
    static P3_FX_HD void run(Q* v)
    {
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2) dft4(v[n2], v[n2 + 4], v[n2 + 8], v[n2 + 12]);
        v[5] = rot<1, kC1, 0, -kS1>(v[5]);
        v[9] = rot45(v[9]);
        v[13] = rot<0, kS1, -1, -kC1>(v[13]);
        v[6] = rot45(v[6]);
        v[14] = rot135(v[14]);
        v[7] = rot<0, kS1, -1, -kC1>(v[7]);
        v[11] = rot135(v[11]);
        v[15] = rot<-1, -kC1, 0, kS1>(v[15]);
        Q o[16];
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            Q a0 = v[4 * k1], a1 = v[4 * k1 + 1], a2 = v[4 * k1 + 2], a3 = v[4 * k1 + 3];
            if (k1 == 2) dft4<true>(a0, a1, a2, a3);
            else dft4<false>(a0, a1, a2, a3);
            o[k1] = a0; o[k1 + 4] = a1; o[k1 + 8] = a2; o[k1 + 12] = a3;
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = o[i];
    }
};
// Coprime products R1 R2 (Good-Thomas prime-factor map, no twiddles):
// input n = (R2 n1 + R1 n2) mod R; output k = (c1 k1 + c2 k2) mod R with
// c1 = 1 mod R1, 0 mod R2 and c2 = 0 mod R1, 1 mod R2.
template <int R1, int R2> struct Pfa {
    static constexpr int R = R1 * R2;
    __host__ __device__ static constexpr int crt(int m, int q)  // multiple of q that is 1 mod m
    {
        int c = 0;
        for (int i = 0; i < m; ++i)
            if ((q * i) % m == 1) c = q * i;
        return c;
    }
    static P3_FX_HD void run(Q* v)
    {
        constexpr int c1 = crt(R1, R2), c2 = crt(R2, R1);
        Q y[R];
#pragma unroll
        for (int n2 = 0; n2 < R2; ++n2) {
            Q a[R1];
#pragma unroll
            for (int n1 = 0; n1 < R1; ++n1) a[n1] = v[(R2 * n1 + R1 * n2) % R];
            D<R1>::run(a);
#pragma unroll
            for (int k1 = 0; k1 < R1; ++k1) y[k1 * R2 + n2] = a[k1];
        }
#pragma unroll
        for (int k1 = 0; k1 < R1; ++k1) {
            D<R2>::run(y + k1 * R2);
#pragma unroll
            for (int k2 = 0; k2 < R2; ++k2) v[(c1 * k1 + c2 * k2) % R] = y[k1 * R2 + k2];
        }
    }
};
template <> struct D<6> : Pfa<2, 3> {};
template <> struct D<10> : Pfa<2, 5> {};
template <> struct D<12> : Pfa<4, 3> {};
template <> struct D<14> : Pfa<2, 7> {};
template <> struct D<15> : Pfa<3, 5> {};

// ---------------------------------------------------------------------------
// Doubles <-> fixed point
// ---------------------------------------------------------------------------
P3_FX_HD unsigned hi_abs(ll raw) { return (unsigned)((unsigned long long)raw >> 32) & 0x7fffffffu; }
P3_FX_HD unsigned long long shr64(unsigned long long v, unsigned s)
{
    // shift counts of 64 and more give 0
#ifdef __CUDA_ARCH__
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
#else
    return s < 64 ? v >> s : 0;
#endif
}

// double bits -> trunc(x 2^(AL - (emax - 1022))): |result| < 2^AL for
// exponent fields up to emax.  emax >= 64, so that values whose implicit bit
// is absent (zeros, denormals) shift out entirely.
template <int AL> P3_FX_HD ll to_fix(ll raw, unsigned emax)
{
    const unsigned hi = (unsigned)((unsigned long long)raw >> 32), lo = (unsigned)raw;
    const unsigned s = emax - ((hi >> 20) & 0x7ffu);
    const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
    const ll g = (ll)((int)hi >> 31);
    return ((ll)shr64(m << (AL - 53), s) ^ g) - g;
}

// v 2^sexp as a double, rounded to nearest; -1021 <= sexp <= 960
__device__ __forceinline__ double to_f64(ll v, int sexp)
{
    const double d = (double)v;
    int hi = __double2hiint(d);
    if (hi != 0) hi += sexp << 20;
    return __hiloint2double(hi, __double2loint(d));
}
__device__ __forceinline__ double2 to_f64(Q v, int sexp) { return make_double2(to_f64(v.x, sexp), to_f64(v.y, sexp)); }

// Exponent of a line at its store: values are v 2^sexp f, f = 1 unless the
// exponent leaves the range of to_f64 (f a power of two) or the line held an
// infinity or a NaN (f a NaN).
struct LineExp {
    int sexp;
    double f;
};
__device__ __forceinline__ LineExp line_exp(int sexp, bool bad)
{
    LineExp e{sexp, 1.0};
    if (sexp < -1021 || sexp > 960) {
        e.sexp = sexp < 0 ? -1021 : 960;
        e.f = scalbn(1.0, sexp - e.sexp);
    }
    if (bad) e.f = __longlong_as_double(0x7ff8000000000000LL);
    return e;
}

// ---------------------------------------------------------------------------
// Stage kernels.  A CTA owns B lines; thread tid works on line tid mod B, with
// tpl threads per line.  Every pass reads a thread's butterflies (at most
// kVals values) into registers and writes them back in place, so one copy of
// the tile sits in shared memory: element e of line l at s[e * LDB + l].
// Strided sides (lines adjacent in memory) go straight between HBM and
// registers; contiguous sides are staged through the tile with lanes walking
// the elements.
// ---------------------------------------------------------------------------
enum Kind : int {
    K_CC = 0,   // complex lines: strided in, strided out
    K_CS = 1,   // strided in, contiguous out (ZYX store)
    K_SC = 2,   // contiguous in (ZYX load), strided out
    K_SS = 3,   // contiguous both sides
    K_ECC = 4,  // the same for the even and odd extensions (DCT-I, DST-I)
    K_ECS = 5,
    K_ESC = 6,
    K_ESS = 7,
    K_R2C = 8,  // even real rows -> half spectra
    K_C2R = 9,  // half spectra -> even real rows
    K_RP = 10,  // odd real rows in pairs -> half spectra
    K_CP = 11,  // half spectra in pairs -> odd real rows
};
template <int K> __host__ __device__ constexpr bool extended() { return K >= K_ECC && K <= K_ESS; }
template <int K> __host__ __device__ constexpr bool in_staged() { return K != K_CC && K != K_CS && K != K_ECC && K != K_ECS; }
template <int K> __host__ __device__ constexpr bool out_staged() { return K != K_CC && K != K_SC && K != K_ECC && K != K_ESC; }

constexpr int kMaxB = 32;
constexpr int kThreads = 256;

// Three forms of each kernel, by the largest radix: CAP 8 and 10 hold one
// butterfly per thread (64 registers, four CTAs per SM), CAP 16 as many as
// fill 16 values (128 registers, two CTAs).
template <int R, int CAP> __host__ __device__ constexpr int bfly()
{
    return CAP <= 10 ? 1 : R == 2 ? 8 : R == 3 ? 5 : R == 4 ? 4 : R == 5 ? 3 : R <= 8 ? 2 : 1;
}

struct Shared {
    unsigned word[(kMaxPasses + 1) * kMaxB];  // [0]: largest magnitude word; [p]: OR of the magnitudes after pass p - 1
    ll bin[kMaxB], bout[kMaxB];               // line bases (elements)
    ll bin2[kMaxB], bout2[kMaxB];             // second row of a pair
    int has[kMaxB];                           // rows present: 0, 1 or (pairs) 2
    int sexp[kMaxB];
    double f[kMaxB];                          // as LineExp
    int odd[kMaxB];                           // f is not 1
};

// Combines a per-thread word over the lanes of a warp that share a line and
// posts it to the line's word (B a power of two; every lane takes part).
template <bool MAXOP> __device__ __forceinline__ void post(unsigned m, unsigned* w, int B, int l)
{
    for (int o = 16; o >= B; o >>= 1) {
        const unsigned q = __shfl_xor_sync(0xffffffffu, m, o);
        m = MAXOP ? (m > q ? m : q) : (m | q);
    }
    if ((int)(threadIdx.x & 31) < B || B >= 32) {
        if (MAXOP) atomicMax(w + l, m);
        else atomicOr(w + l, m);
    }
}

struct Thread {
    int l, t;        // line of the tile, thread of the line
    bool act;        // takes part in the passes
    bool valid;      // ... and its line exists
    int sexp;        // exponent of the line's values
    bool bad;        // the line holds an infinity or a NaN
};

// One pass.  FIRST: from the input (HBM or the staged tile); otherwise from
// the tile of fixed-point values.
template <int K, int CAP, int R, bool FIRST>
__device__ __forceinline__ void pass(const StageArgs& a, Q* s, Shared& sh, Thread& th, int p, int Ns)
{
    constexpr int BM = bfly<R, CAP>();
    const int n = a.nfft, nb = n / R, tpl = a.tpl, LDB = a.LDB, B = a.B;
    const int l = th.l, t = th.t;
    const PassConsts& c = a.pc[p];
    const bool last = p + 1 == a.npass;
    const int q0 = FIRST ? t : (int)(((unsigned long long)(unsigned)t * c.pm) >> c.ps);
    const int r0 = FIRST ? 0 : t - q0 * Ns;
    Q v[BM * R];

    if constexpr (FIRST) {
        // largest high word of the line's magnitudes; the low words only count as
        // zero or not, so that a line of denormals below 2^-1042, whose high
        // words are all 0, is told from a line of zeros
        unsigned m = 0, low = 0;
        if constexpr (K != K_C2R && K != K_CP) {
            const ll es = a.in.es;
            const int M = n >> 1;
            const Q* g = in_staged<K>() ? s + l : static_cast<const Q*>(a.src) + sh.bin[l];
            const ll gs = in_staged<K>() ? (ll)LDB : es;
#pragma unroll
            for (int b = 0; b < BM; ++b) {
                const int j = t + b * tpl;
                const bool ok = th.valid && j < nb;
                const Q* gp = g + j * gs;  // plain lines: stepping through elements nb apart
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    Q x = Q{0, 0};
                    if (!extended<K>()) {
                        if (ok) x = *gp;
                        gp += nb * gs;
                        v[b * R + r] = x;
                        continue;
                    }
                    const int e = j + r * nb;
                    if (a.op == OP_DCT1) {
                        if (ok) x = g[(e <= M ? e : n - e) * gs];
                    } else {  // OP_DST1: 0, x[0..M-2], 0, -x[M-2..0]
                        if (ok && e != 0 && e != M) {
                            x = g[(e < M ? e - 1 : n - 1 - e) * gs];
                            if (e > M) {
                                x.x ^= (ll)0x8000000000000000ULL;
                                x.y ^= (ll)0x8000000000000000ULL;
                            }
                        }
                    }
                    v[b * R + r] = x;
                }
            }
#pragma unroll
            for (int b = 0; b < BM; ++b) {
#pragma unroll
                for (int i = b * R; i < b * R + R; ++i) {
                    m = max(m, hi_abs(v[i].x));
                    m = max(m, hi_abs(v[i].y));
                    low |= (unsigned)v[i].x | (unsigned)v[i].y;
                }
            }
        } else {
            // half spectra: the staged slots of the line (n + 1 of them); the
            // imaginary parts of F[0] and F[n] (X1[0], X2[0]) do not count
            const int d1 = K == K_C2R ? n : a.n_in;
            for (int e = t; e <= n && th.valid; e += tpl) {
                const Q x = s[e * LDB + l];
                m = max(m, hi_abs(x.x));
                low |= (unsigned)x.x;
                if (e != 0 && e != d1) {
                    m = max(m, hi_abs(x.y));
                    low |= (unsigned)x.y;
                }
            }
        }
        if (low) m |= 1u;
        post<true>(m, sh.word, B, l);
        __syncthreads();
        const unsigned mw = sh.word[l];
        unsigned emax = mw >> 20;
        const bool bad = emax == 0x7ffu, tiny = emax < 64u;
        double up = 1.0;
        int back = 0;
        if (mw == 0) {
            emax = 1023u;  // a line of zeros
        } else if (tiny) {  // scaled by 2^200 so that no denormal is left
            emax = (emax ? emax : 1u) + 200u;
            up = 1.6069380442589903e60;
            back = 200;
        }
        auto scaled = [&](ll raw) -> ll { return __double_as_longlong(__longlong_as_double(raw) * up); };
        constexpr int AL = K == K_C2R ? 60 : K == K_CP ? 57 : 58;
        int sexp = (int)emax - back - 1022 - AL;
        if constexpr (K != K_C2R && K != K_CP) {
            const bool half = K == K_R2C && last;  // room for the sums of the real split
            if (half) sexp += 1;
#pragma unroll
            for (int b = 0; b < BM; ++b) {
                if (tiny && mw) {
#pragma unroll
                    for (int i = b * R; i < b * R + R; ++i) v[i] = Q{scaled(v[i].x), scaled(v[i].y)};
                }
#pragma unroll
                for (int i = b * R; i < b * R + R; ++i) {
                    v[i] = Q{to_fix<AL>(v[i].x, emax), to_fix<AL>(v[i].y, emax)};
                    if (half) v[i] = Q{v[i].x >> 1, v[i].y >> 1};
                }
            }
        } else if constexpr (K == K_C2R) {
            // Z[k] = E + i O, Z[n-k] = conj E + i conj O with E = F[k] + conj F[n-k],
            // O = (F[k] - conj F[n-k]) exp(+2 pi i k / 2n), the imaginary parts of
            // F[0] and F[n] dropped; one thread per pair of bins, in place.
            // Scaled by 2^-4 (the twiddle product's scale) and swapped for the
            // inverse.
            const int4* w2 = static_cast<const int4*>(a.tw2);
            if (th.valid) {
                for (int k = t; 2 * k <= n; k += tpl) {
                    Q f = s[k * LDB + l], h = s[(n - k) * LDB + l];
                    if (tiny && mw) {
                        f = Q{scaled(f.x), scaled(f.y)};
                        h = Q{scaled(h.x), scaled(h.y)};
                    }
                    Q A = Q{to_fix<AL>(f.x, emax), to_fix<AL>(f.y, emax)};
                    Q Bc = Q{to_fix<AL>(h.x, emax), -to_fix<AL>(h.y, emax)};
                    if (k == 0) {
                        A.y = 0;
                        Bc.y = 0;
                    }
                    int4 w = __ldg(w2 + k);
                    w.z = -w.z;
                    w.w = -w.w;
                    const Q E = add(A, Bc), O = mulw(sub(A, Bc), w);
                    s[k * LDB + l] = Q{(E.y >> 4) + O.x, (E.x >> 4) - O.y};
                    if (k > 0 && 2 * k < n) s[(n - k) * LDB + l] = Q{O.x - (E.y >> 4), (E.x >> 4) + O.y};
                }
            }
            sexp += 4;
            __syncthreads();
#pragma unroll
            for (int b = 0; b < BM; ++b) {
                const int j = t + b * tpl;
                const bool ok = th.valid && j < nb;
                const Q* sp = s + j * LDB + l;
#pragma unroll
                for (int r = 0; r < R; ++r) v[b * R + r] = ok ? sp[r * nb * LDB] : Q{0, 0};
            }
        } else {
            // Z[k] = X1[k] + i X2[k], Z[n-k] = conj X1[k] + i conj X2[k]
            // (k >= 1); imaginary parts of X1[0], X2[0] dropped; swapped.  One
            // thread per pair of bins, in place: X1[k] sits at slot k and X2[k] at
            // H + k, where Z[k] and Z[n-k] take their places.
            const int H = a.n_in;
            if (th.valid) {
                for (int k = t; k < H; k += tpl) {
                    Q f = s[k * LDB + l], h = s[(H + k) * LDB + l];
                    if (tiny && mw) {
                        f = Q{scaled(f.x), scaled(f.y)};
                        h = Q{scaled(h.x), scaled(h.y)};
                    }
                    Q A = Q{to_fix<AL>(f.x, emax), to_fix<AL>(f.y, emax)};
                    Q C = Q{to_fix<AL>(h.x, emax), to_fix<AL>(h.y, emax)};
                    if (k == 0) {
                        A.y = 0;
                        C.y = 0;
                    }
                    s[k * LDB + l] = Q{A.y + C.x, A.x - C.y};
                    s[(H + k) * LDB + l] = Q{C.x - A.y, A.x + C.y};
                }
            }
            __syncthreads();
#pragma unroll
            for (int b = 0; b < BM; ++b) {
                const int j = t + b * tpl;
                const bool ok = th.valid && j < nb;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int e = j + r * nb;
                    v[b * R + r] = ok ? s[(e < H ? e : H + n - e) * LDB + l] : Q{0, 0};
                }
            }
        }
        if constexpr (K == K_C2R || K == K_CP) __syncthreads();  // every thread has read its values
        th.sexp = sexp;
        th.bad = bad;
    } else {
        // shift the line up by its headroom, multiply by the twiddles (2^-4)
        const unsigned w = sh.word[p * kMaxB + l];
        int k = __clz(w) - 2;
        k = k < 0 ? 0 : k;
        th.sexp += 4 - k;
        const bool drop = K == K_R2C && last;  // room for the sums of the real split
        if (drop) th.sexp += 1;
        const int4* tw = static_cast<const int4*>(a.tw);
        int rr = r0;
#pragma unroll
        for (int b = 0; b < BM; ++b) {
            const int j = t + b * tpl;
            const bool ok = th.act && j < nb;
            const int step = rr * c.tstep;
            int idx = 0;
            const Q* sp = s + j * LDB + l;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                Q x = Q{0, 0};
                if (ok) x = sp[r * nb * LDB];
                if (K == K_R2C && drop) x = Q{x.x >> 1, x.y >> 1};
                x = Q{(ll)((unsigned long long)x.x << k), (ll)((unsigned long long)x.y << k)};
                if (r == 0) {
                    v[b * R] = Q{x.x >> 4, x.y >> 4};
                } else {
                    idx += step;
                    v[b * R + r] = mulw(x, ok ? __ldg(tw + idx) : make_int4(0, 0, 0, 0));
                }
            }
            if (b + 1 < BM) {
                rr += c.dr;
                if (rr >= Ns) rr -= Ns;
            }
        }
    }

#pragma unroll
    for (int b = 0; b < BM; ++b) {
        D<R>::run(v + b * R);
    }

    // positions (j / Ns) Ns R + j mod Ns + r Ns
    if constexpr (!out_staged<K>()) {
        if (last) {
            const LineExp le = line_exp(th.sexp, th.bad);
            double2* g = static_cast<double2*>(a.dst) + sh.bout[l];
            const ll es = a.out.es;
            const int M = n >> 1;
            const bool inv = a.sign > 0;  // plain lines: the inverse-sign bin k is the forward bin -k
            int qq = q0, rr = r0;
#pragma unroll
            for (int b = 0; b < BM; ++b) {
                const int j = t + b * tpl;
                const int o = FIRST ? j * R : qq * Ns * R + rr;
                if (th.valid && j < nb) {
                    // inverse: bin e goes to n - e (0 to 0)
                    double2* gp = g + (inv && o > 0 ? n - o : o) * es;
                    const ll step = inv ? -Ns * es : Ns * es;
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const double2 d = to_f64(v[b * R + r], le.sexp);
                        if (!extended<K>()) {
                            *gp = d;
                            if (r == 0 && inv && o == 0) gp += n * es;
                            gp += step;
                            continue;
                        }
                        const int e = o + r * Ns;
                        if (a.op == OP_DCT1) {
                            if (e <= M) g[e * es] = d;
                        } else {  // i times bin e, 1 <= e < M
                            if (e >= 1 && e < M) g[(e - 1) * es] = make_double2(-d.y, d.x);
                        }
                    }
                    if (le.f != 1.0) {
#pragma unroll 1
                        for (int r = 0; r < R; ++r) {
                            const int e = o + r * Ns;
                            const int k = !extended<K>() ? (inv && e > 0 ? n - e : e) : a.op == OP_DCT1 ? e : e - 1;
                            if (!extended<K>() || (a.op == OP_DCT1 ? e <= M : e >= 1 && e < M)) {
                                const double2 d = g[k * es];
                                g[k * es] = make_double2(d.x * le.f, d.y * le.f);
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
    if (!last) {
        unsigned m = 0;
#pragma unroll
        for (int b = 0; b < BM; ++b) {
#pragma unroll
            for (int i = b * R; i < b * R + R; ++i) {
                const int hx = (int)(v[i].x >> 32), hy = (int)(v[i].y >> 32);
                m |= (unsigned)(hx ^ (hx >> 31)) | (unsigned)(hy ^ (hy >> 31));
            }
        }
        post<false>(m, sh.word + (p + 1) * kMaxB, B, l);
    } else if (t == 0) {
        // the real split of even rows scales by 2^3
        const LineExp le = line_exp(th.sexp + (K == K_R2C ? 3 : 0), th.bad);
        sh.sexp[l] = le.sexp;
        sh.f[l] = le.f;
        sh.odd[l] = le.f != 1.0;
    }
    if (!FIRST || !in_staged<K>()) __syncthreads();  // every thread has read its inputs
    {
        int qq = q0, rr = r0;
#pragma unroll
        for (int b = 0; b < BM; ++b) {
            const int j = t + b * tpl;
            const int o = FIRST ? j * R : qq * Ns * R + rr;
            Q* dp = s + o * LDB + l;
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

template <int K, int CAP, bool FIRST>
__device__ __forceinline__ void pass_any(const StageArgs& a, Q* s, Shared& sh, Thread& th, int p, int Ns)
{
    switch (a.rad[p]) {
#define P3_FX_PASS(R) \
    case R: \
        if constexpr (R <= CAP) pass<K, CAP, R, FIRST>(a, s, sh, th, p, Ns); \
        break;
        P3_FX_PASS(2) P3_FX_PASS(3) P3_FX_PASS(4) P3_FX_PASS(5) P3_FX_PASS(6) P3_FX_PASS(7) P3_FX_PASS(8)
        P3_FX_PASS(9) P3_FX_PASS(10) P3_FX_PASS(12) P3_FX_PASS(14) P3_FX_PASS(15) P3_FX_PASS(16)
#undef P3_FX_PASS
    default: break;
    }
}

template <int K, int CAP>
__global__ void __launch_bounds__(kThreads, CAP <= 10 ? 4 : 2) kernel(const __grid_constant__ StageArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Shared sh;
    Q* s = reinterpret_cast<Q*>(smem_raw);
    const int tid = threadIdx.x, B = a.B, LDB = a.LDB, n = a.nfft;
    const int lb = __ffs(B) - 1;
    const ll L0 = (ll)blockIdx.x * B;
    const int rows = (int)(a.nlines - L0 < B ? a.nlines - L0 : B);
    for (int i = tid; i < a.npass * kMaxB; i += blockDim.x) sh.word[i] = 0;
    if (tid < B) {
        const ll L = L0 + tid;
        int has = 0;
        ll bi = 0, bo = 0, bi2 = 0, bo2 = 0;
        if (tid < rows) {
            has = 1;
            if (K == K_RP || K == K_CP) {
                bi = line_base(a.in, 2 * L);
                bo = line_base(a.out, 2 * L);
                if (2 * L + 1 < a.nrows) {
                    has = 2;
                    bi2 = line_base(a.in, 2 * L + 1);
                    bo2 = line_base(a.out, 2 * L + 1);
                }
            } else {
                bi = line_base(a.in, L);
                bo = line_base(a.out, L);
            }
        }
        sh.has[tid] = has;
        sh.bin[tid] = bi;
        sh.bout[tid] = bo;
        sh.bin2[tid] = bi2;
        sh.bout2[tid] = bo2;
    }
    __syncthreads();
    stage_begin();

    if constexpr (in_staged<K>()) {
        if constexpr (K == K_RP) {
            const double* f = static_cast<const double*>(a.src);
            walk<1>(rows, n, [&](int l, int e) {
                double* d = reinterpret_cast<double*>(s + e * LDB + l);
                cp_async8(smem_u32(d), f + sh.bin[l] + e);
                if (sh.has[l] == 2) cp_async8(smem_u32(d + 1), f + sh.bin2[l] + e);
                else d[1] = 0.0;
            });
        } else if constexpr (K == K_CP) {
            const double2* F = static_cast<const double2*>(a.src);
            const int H = a.n_in;
            walk<1>(rows, H, [&](int l, int e) {
                cp_async16(smem_u32(s + e * LDB + l), F + sh.bin[l] + e);
                Q* d = s + (H + e) * LDB + l;
                if (sh.has[l] == 2) cp_async16(smem_u32(d), F + sh.bin2[l] + e);
                else *d = Q{0, 0};
            });
        } else if constexpr (K == K_R2C) {
            const double* f = static_cast<const double*>(a.src);
            walk<1>(rows, n, [&](int l, int e) { cp_async16(smem_u32(s + e * LDB + l), f + sh.bin[l] + 2 * e); });
        } else {  // contiguous complex lines; C2R: n + 1 bins
            const double2* F = static_cast<const double2*>(a.src);
            walk<1>(rows, K == K_C2R ? n + 1 : a.n_in, [&](int l, int e) { cp_async16(smem_u32(s + e * LDB + l), F + sh.bin[l] + e); });
        }
        cp_async_wait();
        __syncthreads();
    }

    Thread th;
    th.l = tid & (B - 1);
    th.t = tid >> lb;
    th.act = th.t < a.tpl;
    th.valid = th.act && th.l < rows;
    th.sexp = 0;
    th.bad = false;
    pass_any<K, CAP, true>(a, s, sh, th, 0, 1);
    int Ns = a.rad[0];
    for (int p = 1; p < a.npass; ++p) {
        pass_any<K, CAP, false>(a, s, sh, th, p, Ns);
        Ns *= a.rad[p];
    }

    if constexpr (out_staged<K>()) {
        // value of a slot as doubles
        auto out = [&](Q v, int l) -> double2 {
            double2 d = to_f64(v, sh.sexp[l]);
            if (sh.odd[l]) d = make_double2(d.x * sh.f[l], d.y * sh.f[l]);
            return d;
        };
        if constexpr (K == K_CS || K == K_SS) {
            double2* F = static_cast<double2*>(a.dst);
            const bool inv = a.sign > 0;  // the inverse-sign bin k is the forward bin -k
            walk<1>(rows, n, [&](int l, int e) { F[sh.bout[l] + e] = out(s[(inv && e > 0 ? n - e : e) * LDB + l], l); });
        } else if constexpr (K == K_ECS || K == K_ESS) {
            double2* F = static_cast<double2*>(a.dst);
            const bool dst1 = a.op == OP_DST1;  // i times bin e + 1
            walk<1>(rows, a.n_out, [&](int l, int e) {
                const double2 d = out(s[(e + (dst1 ? 1 : 0)) * LDB + l], l);
                F[sh.bout[l] + e] = dst1 ? make_double2(-d.y, d.x) : d;
            });
        } else if constexpr (K == K_C2R) {
            double* f = static_cast<double*>(a.dst);
            walk<1>(rows, n, [&](int l, int e) {
                const double2 d = out(s[e * LDB + l], l);
                *reinterpret_cast<double2*>(f + sh.bout[l] + 2 * e) = make_double2(d.y, d.x);
            });
        } else if constexpr (K == K_R2C) {
            // F[k] = (E - i P) / 2, F[n-k] = conj(E + i P) / 2 with
            // E = Z[k] + conj Z[n-k], P = exp(-2 pi i k / 2n) (Z[k] - conj Z[n-k]); the
            // sums stay below 2^62.5 (the last pass left room for them)
            double2* F = static_cast<double2*>(a.dst);
            const int4* w2 = static_cast<const int4*>(a.tw2);
            walk<1>(rows, n / 2 + 1, [&](int l, int k) {
                const Q zk = s[k * LDB + l];
                Q zm = s[(k == 0 ? 0 : n - k) * LDB + l];
                zm.y = -zm.y;
                const Q p = mulw(sub(zk, zm), __ldg(w2 + k));
                const Q z = add(zk, zm);
                double2* g = F + sh.bout[l];
                g[k] = out(Q{(z.x >> 4) + p.y, (z.y >> 4) - p.x}, l);
                if (2 * k < n) g[n - k] = out(Q{(z.x >> 4) - p.y, -(z.y >> 4) - p.x}, l);
            });
        } else if constexpr (K == K_RP) {
            // X1[k] = (Z[k] + conj Z[n-k]) / 2, X2[k] = -i (Z[k] - conj Z[n-k]) / 2
            double2* F = static_cast<double2*>(a.dst);
            walk<1>(rows, a.n_out, [&](int l, int k) {
                Q zk = s[k * LDB + l], zm = s[(k == 0 ? 0 : n - k) * LDB + l];
                zk = Q{zk.x >> 1, zk.y >> 1};
                zm = Q{zm.x >> 1, zm.y >> 1};
                F[sh.bout[l] + k] = out(Q{zk.x + zm.x, zk.y - zm.y}, l);
                if (sh.has[l] == 2) F[sh.bout2[l] + k] = out(Q{zk.y + zm.y, zm.x - zk.x}, l);
            });
        } else {  // K_CP: real rows from the (swapped) result
            double* f = static_cast<double*>(a.dst);
            walk<1>(rows, a.n_out, [&](int l, int e) {
                const double2 d = out(s[e * LDB + l], l);
                f[sh.bout[l] + e] = d.y;
                if (sh.has[l] == 2) f[sh.bout2[l] + e] = d.x;
            });
        }
    }
}

}  // namespace fx
}  // namespace p3
