"""Host build of the FP64 fixed-point arithmetic (p3_fix64.cuh): every register
butterfly at the edge of its declared range, the twiddle product and the
double -> fixed conversion, against long-double arithmetic, with signed
overflow trapped.  No GPU needed (nvcc compiles the header for the host)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1905_02803_gb300", "csrc")

HARNESS = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "p3_fix64.cuh"
using namespace p3::fx;
typedef long double ld;
static const ld kTwoPi = 6.283185307179586476925286766559005768L;
static unsigned long long state = 88172645463325252ULL;
static unsigned long long rnd() { state ^= state << 13; state ^= state >> 7; state ^= state << 17; return state; }
// |v| < 2^58: random, or one of the corners
static ll val(int mode)
{
    const ll top = (1LL << 58) - 1;
    if (mode == 0) return (ll)(rnd() >> 6) - (1LL << 57);
    if (mode == 1) return rnd() & 1 ? top : -top;
    return rnd() % 3 == 0 ? 0 : rnd() & 1 ? top : (ll)(rnd() >> 40);
}
template <int R> static void check()
{
    double worst = 0;
    for (int it = 0; it < 6000; ++it) {
        Q v[R], in[R];
        // every eighth: inputs aligned with a bin's conjugate twiddles, which
        // drives that bin to its largest modulus
        for (int i = 0; i < R; ++i) {
            v[i] = Q{val(it % 3), val(it % 3)};
            if (it % 8 == 7) {
                const ld a = kTwoPi * ((ld)(i * (it / 8 % R) % R) / R + 0.125L), m = 407631148868860968.0L;  // < 2^58.5
                v[i] = Q{llrintl(m * cosl(a)), llrintl(m * sinl(a))};
            }
            in[i] = v[i];
        }
        D<R>::run(v);
        for (int k = 0; k < R; ++k) {
            ld re = 0, im = 0;
            for (int n = 0; n < R; ++n) {
                const ld a = kTwoPi * (ld)(n * k % R) / R, c = cosl(a), s = -sinl(a);
                re += (ld)in[n].x * c - (ld)in[n].y * s;
                im += (ld)in[n].x * s + (ld)in[n].y * c;
            }
            worst = fmax(worst, fmax(fabs((double)((ld)v[k].x - re)), fabs((double)((ld)v[k].y - im))));
        }
    }
    printf("D%d %.3f\n", R, worst);
}
int main()
{
    check<2>(); check<3>(); check<4>(); check<5>(); check<6>(); check<7>(); check<8>(); check<9>(); check<10>();
    check<12>(); check<14>(); check<15>(); check<16>();
    // twiddle product: a w / 16 for moduli up to 2^62.5
    double worst = 0;
    for (int it = 0; it < 200000; ++it) {
        const ld m = 6521908912666391106.0L * (it & 1 ? 1.0L : (ld)(rnd() >> 11) / 9007199254740992.0L);  // 2^62.5
        const ld p = kTwoPi * (ld)(rnd() >> 11) / 9007199254740992.0L, q = kTwoPi * (ld)(rnd() % 4096) / 4096;
        const Q a = Q{llrintl(m * cosl(p)), llrintl(m * sinl(p))};
        const ll wr = llrintl(cosl(q) * 1152921504606846976.0L), wi = llrintl(-sinl(q) * 1152921504606846976.0L);
        const int4 w = make_int4(hi_of(wr), lo_of(wr), hi_of(wi), lo_of(wi));
        const Q z = mulw(a, w);
        const ld re = ((ld)a.x * wr - (ld)a.y * wi) / 18446744073709551616.0L;
        const ld im = ((ld)a.x * wi + (ld)a.y * wr) / 18446744073709551616.0L;
        worst = fmax(worst, fmax(fabs((double)((ld)z.x - re)), fabs((double)((ld)z.y - im))));
    }
    printf("mulw %.3f\n", worst);
    // double -> fixed: exact when the bits fit, truncated otherwise; zeros
    // and denormals vanish
    int bad = 0;
    for (int it = 0; it < 200000; ++it) {
        const unsigned emax = 64 + rnd() % 1983, below = rnd() % 90;
        if (emax <= below) continue;
        ll raw = (ll)((rnd() & 0x800fffffffffffffULL) | ((unsigned long long)(emax - below) << 52));
        double x;
        memcpy(&x, &raw, 8);
        const double e = trunc(ldexp(x, 58 - ((int)emax - 1022)));
        if ((double)to_fix<58>(raw, emax) != e || to_fix<58>(raw & 0x800fffffffffffffLL, emax) != 0) ++bad;
        if (llabs(to_fix<60>(raw, emax)) >= (1LL << 60)) ++bad;
    }
    printf("to_fix %d\n", bad);
    return 0;
}
"""


@pytest.fixture(scope="module")
def result(tmp_path_factory):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if not nvcc:
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("fix64")
    src = d / "fix64.cu"
    src.write_text(HARNESS)
    exe = d / "fix64"
    san = "-fsanitize=signed-integer-overflow,-fno-sanitize-recover=all".replace(",-f", " -f").split()
    r = subprocess.run([nvcc, "-O1", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)]
                       + [x for f in san for x in ("-Xcompiler", f)], capture_output=True, text=True)
    if r.returncode != 0:
        pytest.fail("harness build failed:\n" + r.stderr)
    p = subprocess.run([str(exe)], capture_output=True, text=True)
    assert p.returncode == 0, p.stdout + p.stderr
    return dict(line.split() for line in p.stdout.splitlines())


@pytest.mark.parametrize("radix", [2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 14, 15, 16])
def test_butterfly_error_in_units(result, radix):
    # each constant product is low by less than 2 units (its floor, and the
    # dropped product of the low halves), each shift by less than 1, and up
    # to R + 8 of them meet in one output; the long-double reference adds
    # R 2^-1 units of its own at 2^62.5
    assert float(result["D%d" % radix]) <= (0.5 if radix in (2, 4) else 2 * (radix + 8))


def test_twiddle_product_error_in_units(result):
    # one floor (below 1), two dropped low products (below 1/2 each in units
    # of 2^64), and half a unit of the long-double reference
    assert float(result["mulw"]) <= 2.5


def test_conversion_to_fixed_point(result):
    assert int(result["to_fix"]) == 0


# Stage lengths in X (rows), Y and Z: every radix of every form of the kernels
# (largest radix 8, 10, 16), one pass only, ragged tiles and single lines
GRIDS = [(2, 3, 5), (4, 7, 9), (14, 16, 12), (15, 6, 10), (9, 14, 15), (40, 49, 64), (36, 30, 25), (27, 125, 21),
         (512, 33, 18), (250, 243, 10), (128, 256, 100), (300, 196, 90), (243, 112, 75), (33, 1, 2048), (2, 4096, 1),
         (1536, 5, 512), (1, 225, 8), (8192, 1, 3)]


@pytest.mark.gpu
@pytest.mark.parametrize("shape", GRIDS)
@pytest.mark.parametrize("layout", ["zyx", "xyz"])
def test_forms_against_oracle(shape, layout):
    from _gpu_helpers import check_case
    ef, eb, plan = check_case(*shape, "f64", layout=layout, seed=sum(shape))
    if shape != (33, 1, 2048) and shape[0] != 1:
        assert "fix64" in plan.describe(), plan.describe()
    # a stage adds at most about 1.2e-16 (the double it is rounded to, and the
    # fixed-point passes); the oracle's own error is 1e-16 per stage
    assert ef <= 6e-16 and eb <= 6e-16, (ef, eb)


# grid, Z transform, layout, then the kinds of the six stages in order
NAMED = [((64, 128, 256), "fft", "zyx", "r2c cc cs sc cc c2r"), ((64, 54, 225), "fft", "xyz", "r2c cc cc cc cc c2r"),
         ((15, 60, 90), "fft", "zyx", "rp cc cs sc cc cp"), ((30, 9, 65), "cheb", "zyx", "r2c cc ecs esc cc c2r"),
         ((12, 36, 31), "sine", "xyz", "r2c cc ecc ecc cc c2r")]


@pytest.mark.gpu
@pytest.mark.parametrize("shape,z,layout,kinds", NAMED)
def test_description_names_what_runs(shape, z, layout, kinds):
    """The description gives each stage's own kernel and its passes: one radix
    per pass (composite ones whole, none above the form's largest), whose
    product is the line's length."""
    from math import prod

    from paper_1905_02803_gb300.p3dfft import Plan
    desc = Plan(*shape, precision="f64", ttypes=("fft", "fft", z), layout=layout).describe()
    lines = [dict(w.split("=", 1) for w in l.split() if "=" in w) for l in desc.splitlines() if "kernel=" in l]
    assert len(lines) == 6
    for f, kind in zip(lines, kinds.split()):
        fix, got, form = f["kernel"].split("_")
        assert (fix, got) == ("fix64", kind), f
        rad = [int(r) for r in f["radices"].split("x")]
        assert prod(rad) == int(f["nfft"]) and max(rad) <= int(form), f
        if form != "16":  # one butterfly per thread: the narrowest pass sets the threads
            assert int(f["tpl"]) == int(f["nfft"]) // min(rad), f


@pytest.mark.gpu
@pytest.mark.parametrize("shape,ttypes", [((24, 20, 18), ("fft", "fft", "fft")), ((15, 9, 33), ("fft", "fft", "cheb")),
                                          ((64, 50, 31), ("fft", "fft", "sine"))])
@pytest.mark.parametrize("layout", ["zyx", "xyz"])
def test_scales_zeros_and_non_finite_lines(shape, ttypes, layout):
    """Powers of two scale exactly, down to lines whose values are denormal;
    zeros stay zeros; a NaN or an infinity makes every output of a forward
    transform non-finite, as it does in double arithmetic."""
    import torch
    from paper_1905_02803_gb300.p3dfft import Plan
    nx, ny, nz = shape
    plan = Plan(nx, ny, nz, precision="f64", ttypes=ttypes, layout=layout)
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    x = torch.rand(plan.real_shape, generator=g, device="cuda", dtype=torch.float64) - 0.5
    X, y = plan.forward(x), None
    y = plan.backward(X)
    for e in (-900, -500, 300, 900):
        s = 2.0 ** e
        Xs = plan.forward(x * s)
        assert torch.equal(torch.view_as_real(Xs), torch.view_as_real(X) * s), e
        assert torch.equal(plan.backward(Xs), y * s), e
    # values near and below the smallest normal double: each intermediate
    # array is rounded to multiples of 2^-1074
    tiny = plan.forward(x * 2.0 ** -1030)
    err = (torch.view_as_real(tiny) * 2.0 ** 500 * 2.0 ** 530 - torch.view_as_real(X)).abs().max().item()
    assert err <= 2.0 ** -44 * nx * ny * nz
    # overflow to infinity, not wrap
    big = plan.forward(torch.full_like(x, 1.5e308))
    assert not torch.isfinite(torch.view_as_real(big)).all()
    assert torch.count_nonzero(torch.view_as_real(plan.forward(torch.zeros_like(x)))).item() == 0
    # zero lines beside others
    z = x.clone()
    z[:, ::2] = 0
    assert torch.isfinite(torch.view_as_real(plan.forward(z))).all()
    for bad in (float("nan"), float("inf"), -float("inf")):
        xb = x.clone()
        xb[nz // 2, ny // 2, nx // 2] = bad
        assert not torch.isfinite(torch.view_as_real(plan.forward(xb))).any()
        Xb = X.clone()
        Xb.view(-1)[Xb.numel() // 2] = complex(bad, 0.0)
        assert not torch.isfinite(plan.backward(Xb)).any()
    # the dropped imaginary parts of the inverse (bins 0 and Nx / 2) do not
    # matter, whatever they hold
    if ttypes == ("fft", "fft", "fft") and layout == "xyz" and nx % 2 == 0:
        p1 = Plan(nx, 1, 1, precision="f64", layout="xyz")
        L = torch.view_as_complex(torch.rand((1, 1, nx // 2 + 1, 2), generator=g, device="cuda", dtype=torch.float64))
        ref = p1.backward(L)
        M = L.clone()
        M[0, 0, 0] = complex(M[0, 0, 0].real.item(), float("nan"))
        M[0, 0, nx // 2] = complex(M[0, 0, nx // 2].real.item(), 1e300)
        assert torch.equal(p1.backward(M), ref)


@pytest.mark.gpu
@pytest.mark.parametrize("shape,z", [((24, 20, 18), "fft"), ((15, 12, 9), "fft"), ((15, 9, 17), "cheb"), ((32, 10, 15), "sine")])
@pytest.mark.parametrize("layout", ["zyx", "xyz"])
def test_lines_of_the_smallest_denormals(shape, z, layout):
    """Values of a few units of 2^-1074: every stage's lines, sums included, lie
    below 2^-1042, where a double's high word is zero.  Forward and inverse
    equal the transform of the same whole numbers, times 2^-1074, but for the
    rounding of each stage's results to whole units."""
    import torch
    from paper_1905_02803_gb300.p3dfft import Plan
    nx, ny, nz = shape
    plan = Plan(nx, ny, nz, precision="f64", ttypes=("fft", "fft", z), layout=layout)
    g = torch.Generator(device="cuda")
    g.manual_seed(nx)
    unit = 2.0 ** -537  # 2^-1074 in two steps, each exact
    n = torch.randint(0, 16, plan.real_shape, generator=g, device="cuda").double()
    m = torch.randint(0, 16, plan.complex_shape + (2,), generator=g, device="cuda").double()
    got = torch.view_as_real(plan.forward(n * unit * unit)) / unit / unit
    back = plan.backward(torch.view_as_complex(m * unit * unit)) / unit / unit
    # a unit per stage (half by rounding to whole units, less by the rounding to
    # 53 bits before it), in each part of a value; the transforms after it add up
    # as many of them as their lines have points
    zl = {"fft": nz, "cheb": 2 * (nz - 1), "sine": 2 * (nz + 1)}[z]
    bound = 1.5 * (1 + zl + ny * zl)
    boundb = 1.5 * (1 + nx + nx * ny)
    want, wantb = torch.view_as_real(plan.forward(n)), plan.backward(torch.view_as_complex(m))
    assert (got - want).abs().max().item() <= bound < 0.2 * want.abs().max().item()
    assert (back - wantb).abs().max().item() <= boundb < 0.2 * wantb.abs().max().item()


# a line whose passes need more threads than a block has (radix 9 of 2430: 270)
# has no fixed-point form: double arithmetic in both directions
@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(4860, 2, 3), (2835, 3, 5), (6, 3645, 4), (3, 4, 2916), (5, 2430, 2), (2, 3, 4050)])
@pytest.mark.parametrize("layout", ["zyx", "xyz"])
def test_lengths_without_a_form(shape, layout):
    from _gpu_helpers import check_case
    ef, eb, plan = check_case(*shape, "f64", layout=layout, seed=sum(shape))
    long = [l for l in plan.describe().splitlines() if "kernel=" in l and int(l.split("nfft=")[1].split()[0]) > 2304]
    assert len(long) == 2 and all("kernel=generic" in l for l in long), long
    # half a unit of the last place per butterfly level (12 of them here, and 4
    # in the short lines)
    assert ef <= 18e-16 and eb <= 18e-16, (ef, eb)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(96, 64, 60), (75, 50, 81)])
@pytest.mark.parametrize("layout", ["zyx", "xyz"])
def test_steep_spectrum(shape, layout):
    """Amplitudes that fall by 30 orders of magnitude over the bins.  A line has
    one exponent, so its error is relative to its largest value, as a sum over
    the line in double arithmetic is to the largest term: both directions
    are as near to the oracle as for a flat spectrum, and no single bin is
    further off than that error would be if it all fell on one of them."""
    import numpy as np
    import torch

    import oracle as O
    from _gpu_helpers import random_complex, rel_l2
    from paper_1905_02803_gb300.p3dfft import Plan
    nx, ny, nz = shape
    kz, ky, kx = (np.minimum(np.arange(n), n - np.arange(n)) / (n / 2) for n in (nz, ny, nx))
    k = kz[:, None, None] + ky[None, :, None] + kx[None, None, :nx // 2 + 1]
    F = random_complex(k.shape, 5) * 10.0 ** (-10 * k)
    plan = Plan(nx, ny, nz, precision="f64", layout=layout)
    y = plan.backward(torch.from_numpy(O.to_zyx(F) if layout == "zyx" else F).cuda()).cpu().numpy()
    ref = O.backward(F, nx)
    assert rel_l2(y, ref) <= 6e-16
    X = plan.forward(torch.from_numpy(ref).cuda()).cpu().numpy()
    X = O.from_zyx(X) if layout == "zyx" else X
    Xr = O.forward(ref)
    assert rel_l2(X, Xr) <= 6e-16
    assert np.abs(X - Xr).max() <= 6e-16 * np.linalg.norm(Xr.ravel())


@pytest.mark.gpu
@pytest.mark.parametrize("nx", [96, 75])
@pytest.mark.parametrize("layout", ["zyx", "xyz"])
def test_rows_of_unlike_size(nx, layout):
    """Rows alone (no Y or Z transform), every other one 1e-9 of its
    neighbour.  Even rows are as accurate each for itself; odd ones run two to a
    complex line, in double arithmetic as here, so their errors are relative to
    the pair."""
    import numpy as np
    import torch

    import oracle as O
    from _gpu_helpers import random_complex
    from paper_1905_02803_gb300 import inputs
    from paper_1905_02803_gb300.p3dfft import Plan
    ny, nz = 8, 6
    tt = (O.FFT, O.EMPTY, O.EMPTY)
    size = np.where(np.arange(ny) % 2 == 0, 1.0, 1e-9)[None, :, None]
    f = inputs.uniform_field((nz, ny, nx), 9) * size
    F = random_complex((nz, ny, nx // 2 + 1), 4) * size
    plan = Plan(nx, ny, nz, precision="f64", ttypes=("fft", "empty", "empty"), layout=layout)
    X = plan.forward(torch.from_numpy(f).cuda()).cpu().numpy()
    X = O.from_zyx(X) if layout == "zyx" else X
    y = plan.backward(torch.from_numpy(O.to_zyx(F) if layout == "zyx" else F).cuda()).cpu().numpy()
    for got, ref in ((X, O.forward(f, tt)), (y, O.backward(F, nx, tt))):
        err, norm = np.linalg.norm(got - ref, axis=2), np.linalg.norm(ref, axis=2)
        if nx % 2:
            norm[:, 1::2] = norm[:, ::2]
        assert (err <= 6e-16 * norm).all(), (err / norm).max()


@pytest.mark.gpu
def test_volume_limit_keeps_double_kernels():
    """Forward transforms of more than 12,582,912 points keep the double
    kernels (test_gpu_double.py runs them); every inverse of a length with a form
    runs in fixed point."""
    from paper_1905_02803_gb300.p3dfft import Plan
    for nz, fixed in ((192, True), (196, False)):
        lines = [w for w in Plan(256, 256, nz, precision="f64").describe().splitlines() if "kernel=" in w]
        assert len(lines) == 6
        for w in lines:
            assert ("fix64" in w) == (fixed or w.startswith("bwd")), w
