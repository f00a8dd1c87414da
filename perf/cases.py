"""The work a program has this library do, as cases that can be timed and checked.

A case is one pass of a spectral code's inner loop through the public Python
entry points: the forward transform of a real field into a kept spectrum
buffer and the inverse transform back (`Plan.forward`, `Plan.backward`,
`Batch.forward`, `Batch.backward`), with the plan, the buffers and the
workspace that such a program keeps between passes.

Fields of a case:
  nx, ny, nz   grid
  precision    "f32" | "f64"
  z            third dimension: "fft" | "cheb" | "sine"
  layout       "zyx" (STRIDE1 output) | "xyz"
  mode         "pair": forward, then inverse into a second real buffer
               "inplace": padded rows; the inverse runs in place on the spectrum
               "batch": `grids` independent 7-smooth grids (sizes drawn from
               `sizes_seed` between `lo` and `hi`) over `nstreams` streams (0:
               one persistent launch per direction)
"""
import math
import random

import torch

from paper_1905_02803_gb300 import p3dfft as P


def case(name, nx, ny, nz, precision="f32", z="fft", layout="zyx", mode="pair"):
    return {"name": name, "nx": nx, "ny": ny, "nz": nz, "precision": precision, "z": z, "layout": layout,
            "mode": mode}


def batch_case(name, grids, lo, hi, sizes_seed, nstreams):
    return {"name": name, "mode": "batch", "precision": "f32", "z": "fft", "layout": "zyx", "grids": grids, "lo": lo,
            "hi": hi, "sizes_seed": sizes_seed, "nstreams": nstreams}


def unnamed(c):
    return {k: v for k, v in c.items() if k != "name"}


def listed():
    return [
        # the smallest calls: a unit-test or boundary-layer sized grid, where
        # launches and host time count
        case("f64_32cubed", 32, 32, 32, "f64"),
        case("f32_64cubed_xyz", 64, 64, 64, layout="xyz"),
        # ordinary simulation grids of a power of two
        case("f32_256cubed", 256, 256, 256),
        # memory-lean code: padded rows, the inverse in place
        case("f32_512cubed_inplace", 512, 512, 512, layout="xyz", mode="inplace"),
        # the headline grid: a production turbulence field
        case("f32_1024cubed", 1024, 1024, 1024),
        # double precision, as most production codes run
        case("f64_512cubed", 512, 512, 512, "f64"),
        # channel flow: Fourier in X and Y, Chebyshev between the walls
        case("f64_channel_480x360x257", 480, 360, 257, "f64", z="cheb"),
        # double precision on dealiased (3/2-rule) and odd grids, plain layout
        case("f64_243x250x180_xyz", 243, 250, 180, "f64", layout="xyz"),
        # dealiased single precision grid
        case("f32_384cubed", 384, 384, 384),
        # odd sizes in every dimension
        case("f32_375x360x343", 375, 360, 343),
        # Dirichlet walls: sine transform in Z
        case("f32_sine_512x512x255", 512, 512, 255, z="sine"),
        # many small independent fields (particles, scalars, ensembles)
        batch_case("f32_batch_24_grids", 24, 48, 384, 0, 16),
    ]


def smooth7(lo, hi):
    def is_smooth(n):
        for p in (2, 3, 5, 7):
            while n % p == 0:
                n //= p
        return n == 1
    return [n for n in range(lo, hi + 1) if is_smooth(n)]


def log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: any transform kind, precision,
    layout and mode, sizes spread over their logarithm, odd, prime and ragged
    ones among them."""
    kind = rng.choice(["pow2", "smooth", "any", "cheb", "sine", "inplace", "batch", "f64", "f64_any"])
    if kind == "batch":
        lo = rng.randint(24, 64)
        return unnamed(batch_case("", rng.randint(6, 24), lo, rng.randint(lo + 40, 384), rng.randint(1, 10**6),
                                  rng.choice([0, 8, 16])))
    precision = "f64" if kind.startswith("f64") or (kind == "cheb" and rng.random() < 0.7) else "f32"
    most = 1 << (26 if precision == "f64" else 29)
    layout = rng.choice(["zyx", "zyx", "xyz"])
    z, mode = "fft", "pair"
    while True:
        if kind == "pow2":
            d = [1 << rng.randint(5, 11) for _ in range(3)]
        elif kind in ("any", "f64_any"):
            # no structure at all: primes and large factors (chirp lines)
            d = [log_int(rng, 17, 400) for _ in range(3)]
        else:
            sizes = smooth7(24, 1024 if precision == "f32" else 600)
            d = [min(sizes, key=lambda s, v=log_int(rng, 24, sizes[-1]): abs(s - v)) for _ in range(3)]
        if kind == "cheb":
            z, d[2] = "cheb", rng.choice([33, 65, 97, 121, 129, 193, 257, 301])
        elif kind == "sine":
            z, d[2] = "sine", rng.choice([31, 63, 95, 127, 149, 255, 319, 511])
        elif kind == "inplace":
            mode, layout = "inplace", "xyz"
        if d[0] * d[1] * d[2] <= (most >> 5 if kind in ("any", "f64_any") else most):
            break
    return unnamed(case("", d[0], d[1], d[2], precision, z, layout, mode))


def grids_of(c):
    """(nx, ny, nz) of every grid of a case."""
    if c["mode"] != "batch":
        return [(c["nx"], c["ny"], c["nz"])]
    r = random.Random(c["sizes_seed"])
    sizes = smooth7(c["lo"], c["hi"])
    return [tuple(r.choice(sizes) for _ in range(3)) for _ in range(c["grids"])]


def field(nx, ny, nz, precision, z, seed):
    """A real field [nz][ny][nx] of unit size: waves of falling amplitude in
    X and Y and the Z basis of the transform (Fourier, Chebyshev or sine), and
    noise, which every spectrum has at its small scales."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    dt = torch.float32 if precision == "f32" else torch.float64
    waves = 12
    u = torch.rand((4, waves), generator=g, device="cuda", dtype=torch.float64)
    # wavenumbers log-uniform up to the Nyquist bin, amplitude k^(-1/3)
    kx = torch.floor(torch.exp(u[0] * math.log(max(2, nx // 2))))
    ky = torch.floor(torch.exp(u[1] * math.log(max(2, ny // 2))))
    kz = torch.floor(torch.exp(u[2] * math.log(max(2, nz // 2))))
    amp = 0.4 * (kx * kx + ky * ky + kz * kz) ** (-1.0 / 6.0)
    phase = 2 * math.pi * u[3]
    X, Y, Z = (torch.arange(n, device="cuda", dtype=torch.float64) for n in (nx, ny, nz))
    ax = 2 * math.pi / nx * X[:, None] * kx
    ay = 2 * math.pi / ny * Y[:, None] * ky + phase
    if z == "fft":
        th = ay[None, :, :] + (2 * math.pi / nz * Z[:, None] * kz)[:, None, :]
        cz = None
    else:
        th = ay[None, :, :].expand(nz, ny, waves)
        if z == "cheb":  # T_n on the Gauss-Lobatto points
            cz = torch.cos(math.pi / (nz - 1) * Z[:, None] * kz)[:, None, :]
        else:
            cz = torch.sin(math.pi / (nz + 1) * (Z[:, None] + 1) * kz)[:, None, :]
    c, s = torch.cos(th) * amp, torch.sin(th) * amp
    if cz is not None:
        c, s = c * cz, s * cz
    a = torch.cat([c, -s], dim=2).reshape(nz * ny, 2 * waves).to(dt)
    b = torch.cat([torch.cos(ax), torch.sin(ax)], dim=1).t().to(dt)
    f = torch.randn((nz * ny, nx), generator=g, device="cuda", dtype=torch.float32).mul_(0.05).to(dt)
    f.addmm_(a, b)
    return f.view(nz, ny, nx)


def fields(c, seed):
    return [field(nx, ny, nz, c["precision"], c["z"], 1000 * seed + i) for i, (nx, ny, nz) in enumerate(grids_of(c))]


def prepare(c, seed):
    flags = P.P3_FLAG_PADDED_REAL if c["mode"] == "inplace" else 0
    plans = [P.Plan(nx, ny, nz, precision=c["precision"], ttypes=("fft", "fft", c["z"]), layout=c["layout"],
                    flags=flags) for nx, ny, nz in grids_of(c)]
    state = {"mode": c["mode"], "plans": plans, "X": [p.empty_complex() for p in plans]}
    xs = fields(c, seed)
    if c["mode"] == "inplace":
        p, x = plans[0], xs[0]
        padded = torch.zeros(p.real_shape, dtype=p.real_dtype, device="cuda")
        padded[:, :, :p.nx] = x
        state["x"] = [padded]
    else:
        state["x"] = xs
        state["y"] = [p.empty_real() for p in plans]
    for p in plans:
        p.workspace()
    if c["mode"] == "batch":
        state["batch"] = P.Batch(plans, nstreams=c["nstreams"])
    return state


def run(state):
    if state["mode"] == "batch":
        X = state["batch"].forward(state["x"], state["X"])
        y = state["batch"].backward(X, state["y"])
        return {"spectra": X, "fields": y}
    plan = state["plans"][0]
    X = plan.forward(state["x"][0], out=state["X"][0])
    if state["mode"] == "inplace":
        # the spectrum becomes the field in its own storage; the padding of
        # each row holds nothing
        return {"field": plan.backward(X, out=plan.real_view(X))[:, :, :plan.nx]}
    return {"spectrum": X, "field": plan.backward(X, out=state["y"][0])}


def work(c):
    """The real and the complex array once per direction; 2.5 N log2 N flops
    per direction."""
    e = 4 if c["precision"] == "f32" else 8
    b = f = 0.0
    for nx, ny, nz in grids_of(c):
        b += 2 * (e * nx * ny * nz + 2 * e * (nx // 2 + 1) * ny * nz)
        f += 2 * 2.5 * nx * ny * nz * math.log2(max(2, nx * ny * nz))
    return {"bytes": b, "flops": f}


def tolerance(c):
    # about four times the error of a whole forward + inverse pass against 64
    # bits, over samples of the outputs that may miss a spectrum's few strong
    # bins: up to 7e-7 in single and 2.7e-15 in double precision; chirp lines
    # (lengths with a prime factor above 7) are three longer transforms
    smooth = all(lines_smooth(n, c["z"]) for n in grids_of(c))
    if c["precision"] == "f32":
        return {"rel": 2.8e-6 if smooth else 4e-6}
    return {"rel": 1.1e-14 if smooth else 1.6e-14}


def lines_smooth(grid, z):
    nx, ny, nz = grid
    lines = [nx // 2 if nx % 2 == 0 else nx, ny, {"fft": nz, "cheb": 2 * (nz - 1), "sine": 2 * (nz + 1)}[z]]
    for n in lines:
        for p in (2, 3, 5, 7):
            while n % p == 0:
                n //= p
        if n != 1:
            return False
    return True


def spectrum64(x, z, layout):
    """The unnormalised transform of a real field in double precision: real
    FFT in X, complex FFT in Y, and the Z transform (DCT-I and DST-I by the
    FFT of their even and odd extensions)."""
    X = torch.fft.fft(torch.fft.rfft(x.double(), dim=2), dim=1)
    nz = X.shape[0]
    if z == "fft":
        X = torch.fft.fft(X, dim=0)
    elif z == "cheb":
        X = torch.fft.fft(torch.cat([X, X[1:-1].flip(0)], dim=0), dim=0)[:nz]
    else:
        o = torch.zeros_like(X[:1])
        X = 1j * torch.fft.fft(torch.cat([o, X, o, -X.flip(0)], dim=0), dim=0)[1:nz + 1]
    return X.permute(2, 1, 0).contiguous() if layout == "zyx" else X.contiguous()


def exact(c, seed):
    xs = fields(c, seed)
    Xs, ys = [], []
    for (nx, ny, nz), x in zip(grids_of(c), xs):
        # both directions unnormalised: the round trip is this factor
        scale = nx * ny * {"fft": nz, "cheb": 2 * (nz - 1), "sine": 2 * (nz + 1)}[c["z"]]
        ys.append(x.double() * scale)
        if c["mode"] != "inplace":
            Xs.append(spectrum64(x, c["z"], c["layout"]))
    if c["mode"] == "batch":
        return {"spectra": Xs, "fields": ys}
    if c["mode"] == "inplace":
        return {"field": ys[0]}
    return {"spectrum": Xs[0], "field": ys[0]}
