"""Forward transforms in double arithmetic: FP64 volumes of more than
12,582,912 points, against the oracle.  Every line length and form of the
double power-of-two kernels (rows of 64 to 4096 complex points, Y and Z lines
of 64 to 4096 points, plain, Chebyshev and sine, both layouts), and the generic
kernel's radices, odd rows in pairs and extensions."""
import math

import numpy as np
import pytest

import oracle as O
from paper_1905_02803_gb300 import inputs

from _gpu_helpers import TT, rel_l2

pytestmark = pytest.mark.gpu

# grid, Z transform, lengths that the power-of-two kernels run (X as half lengths)
VOLUMES = [((128, 4096, 25), "fft", {64, 4096}), ((8192, 64, 25), "fft", {4096, 64}), ((256, 2048, 25), "fft", {128, 2048}),
           ((4096, 128, 25), "fft", {2048, 128}), ((512, 192, 129), "cheb", {256, 256}),
           ((1024, 100, 128), "fft", {512, 128}), ((2048, 25, 256), "fft", {1024, 256}),
           ((50, 512, 512), "fft", {512}), ((25, 512, 1024), "fft", {512, 1024}), ((96, 64, 2049), "cheb", {64, 4096}),
           ((200, 1024, 64), "fft", {1024, 64}), ((50, 256, 1024), "fft", {256, 1024}), ((50, 64, 4096), "fft", {64, 4096}),
           ((50, 128, 2048), "fft", {128, 2048}), ((600, 700, 33), "cheb", {64}), ((512, 400, 65), "cheb", {256, 128}),
           ((256, 200, 257), "cheb", {128, 512}), ((128, 200, 513), "cheb", {64, 1024}), ((64, 200, 1025), "cheb", {2048}),
           ((700, 600, 31), "sine", {64}), ((512, 400, 63), "sine", {256, 128}), ((256, 400, 127), "sine", {128, 256}),
           ((200, 256, 255), "sine", {256, 512}), ((200, 128, 511), "sine", {128, 1024}), ((100, 128, 1023), "sine", {128, 2048}),
           ((64, 100, 2047), "sine", {4096}),
           # the generic kernel: odd rows in pairs, radices 3, 5 and 7, a long line
           ((375, 343, 100), "fft", set()), ((245, 252, 210), "fft", set()), ((300, 210, 200), "fft", set()),
           ((375, 360, 101), "cheb", set()), ((405, 225, 139), "sine", set()), ((12, 3645, 300), "fft", set())]


@pytest.mark.parametrize("shape,z,lengths", VOLUMES)
def test_double_forward_against_oracle(shape, z, lengths):
    import torch
    from paper_1905_02803_gb300.p3dfft import Plan
    nx, ny, nz = shape
    assert nx * ny * nz > 12582912
    field = inputs.uniform_field((nz, ny, nx), nx)
    ref = O.forward(field, (O.FFT, O.FFT, TT[z]))
    x = torch.from_numpy(field).cuda()
    for layout in ("zyx", "xyz"):
        plan = Plan(nx, ny, nz, precision="f64", ttypes=("fft", "fft", z), layout=layout)
        fwd = [dict(w.split("=", 1) for w in l.split() if "=" in w) for l in plan.describe().splitlines()
               if l.startswith("fwd") and "kernel=" in l]
        assert all("fix64" not in f["kernel"] for f in fwd), fwd
        assert lengths <= {int(f["nfft"]) for f in fwd if f["kernel"].startswith("pow2_")}, fwd
        X = plan.forward(x)
        if layout == "zyx":
            X = X.permute(2, 1, 0)
        # half a unit of the last place per butterfly level, added up
        levels = math.log2(nx * ny * {"fft": nz, "cheb": 2 * nz - 2, "sine": 2 * nz + 2}[z])
        err = rel_l2(X.cpu().numpy(), ref)
        assert err <= 1.1e-16 * levels, (layout, err)
