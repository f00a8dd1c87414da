"""FP32 line kernels (p3_line32.cuh) against the tile-in-shared-memory kernel
that the persistent batch runs: the same operations in the same order, so the
results agree bit for bit."""
import pytest

from paper_1905_02803_gb300 import inputs

pytestmark = pytest.mark.gpu

# (nx, ny, nz): every radix (2 .. 10, 12, 14, 15, 16), single-pass lines, odd
# rows in pairs with a last single row, ragged tiles, long and short lines
GRIDS = [(4, 3, 2), (14, 6, 9), (12, 15, 10), (9, 5, 7), (15, 3, 11 * 3 + 2), (20, 14, 12), (28, 18, 24), (30, 49, 63),
         (98, 40, 36), (135, 27, 25), (243, 7, 20), (192, 96, 84), (300, 36, 150), (750, 12, 375), (1500, 4, 486),
         (6, 2016, 3), (2, 3000, 2), (3645, 3, 3)]


def both(plan, Batch):
    import torch
    nx, ny, nz = plan.nx, plan.ny, plan.nz
    x = torch.from_numpy(inputs.uniform_field((nz, ny, nx), nx + 7 * ny + nz)).to("cuda", torch.float32)
    g = torch.Generator(device="cuda")
    g.manual_seed(ny)
    G = torch.view_as_complex(torch.randn(plan.complex_shape + (2,), generator=g, device="cuda"))
    batch = Batch([plan], nstreams=0)
    return ((plan.forward(x), batch.forward([x])[0]), (plan.backward(G), batch.backward([G])[0]))


@pytest.mark.parametrize("shape", GRIDS)
@pytest.mark.parametrize("layout", ["zyx", "xyz"])
def test_same_bits_as_tile_kernel(shape, layout):
    import torch
    from paper_1905_02803_gb300.p3dfft import Batch, Plan
    plan = Plan(*shape, precision="f32", layout=layout)
    if max(shape) > 2:
        assert "line32" in plan.describe(), plan.describe()
    for a, b in both(plan, Batch):
        assert torch.equal(a, b)


@pytest.mark.parametrize("z,nz", [("cheb", 2), ("cheb", 19), ("cheb", 121), ("sine", 1), ("sine", 20), ("sine", 149)])
@pytest.mark.parametrize("layout", ["zyx", "xyz"])
def test_same_bits_extensions(z, nz, layout):
    import torch
    from paper_1905_02803_gb300.p3dfft import Batch, Plan
    plan = Plan(22, 9, nz, precision="f32", ttypes=("fft", "fft", z), layout=layout)
    for a, b in both(plan, Batch):
        assert torch.equal(a, b)


@pytest.mark.parametrize("shape", [(24, 10, 9), (15, 6, 7), (150, 21, 40)])
def test_in_place_rows(shape):
    import torch
    from paper_1905_02803_gb300 import p3dfft as P
    nx, ny, nz = shape
    plan = P.Plan(nx, ny, nz, precision="f32", layout="xyz", flags=P.P3_FLAG_PADDED_REAL)
    ref = P.Plan(nx, ny, nz, precision="f32", layout="xyz")
    x = torch.from_numpy(inputs.uniform_field((nz, ny, nx), 3)).to("cuda", torch.float32)
    buf = torch.zeros(plan.real_shape, device="cuda")
    buf[:, :, :nx] = x
    X = plan.forward(buf, out=plan.complex_view(buf))
    Xr = ref.forward(x)
    assert torch.equal(X, Xr)
    y = plan.backward(X, out=plan.real_view(X))[:, :, :nx]
    assert torch.equal(y, ref.backward(Xr))


@pytest.mark.parametrize("shape", [(384, 60, 384), (190, 93, 486), (4094, 91, 24), (102, 41, 2000)])
def test_bulk_copied_lines(shape):
    """Inverse Z stage of the ZYX layout whose tile arrives line by line by bulk
    copies: bit for bit the plan with P3_FLAG_NO_TMA; a wait that runs out is
    reported."""
    import torch
    from paper_1905_02803_gb300 import p3dfft as P
    pt = P.Plan(*shape, precision="f32")
    pn = P.Plan(*shape, precision="f32", flags=P.P3_FLAG_NO_TMA)
    assert "line32_bulk" in pt.describe() and "line32_bulk" not in pn.describe(), pt.describe()
    g = torch.Generator(device="cuda")
    g.manual_seed(shape[0])
    G = torch.view_as_complex(torch.randn(pt.complex_shape + (2,), generator=g, device="cuda"))
    y = pt.backward(G)
    assert torch.equal(y, pn.backward(G))
    assert P.p3_plan_wait_status(pt.handle) == P.P3_OK
    P.p3_plan_set_wait_limits(pt.handle, 2000, 1)
    pt.backward(G)
    assert P.p3_plan_wait_flags(pt.handle) == P.P3_WAIT_COPY
    P.p3_plan_set_wait_limits(pt.handle, 1 << 23, 0)
    assert torch.equal(y, pt.backward(G))
    assert P.p3_plan_wait_status(pt.handle) == P.P3_OK
