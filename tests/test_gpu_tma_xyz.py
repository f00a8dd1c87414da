"""Z stages of the XYZ layout whose input tile arrives by tensor copies (strided
store, both directions, in place too): bit for bit the plan with
P3_FLAG_NO_TMA, with ragged last tiles and volumes narrower than one tile."""
import pytest

from paper_1905_02803_gb300 import inputs

pytestmark = pytest.mark.gpu

CASES = [((64, 32, 256), "fft", 0), ((48, 20, 512), "fft", 0), ((30, 26, 512), "fft", 0), ((2, 3, 1024), "fft", 0),
         ((18, 9, 2048), "fft", 0), ((256, 256, 512), "fft", 0), ((512, 512, 512), "fft", 2), ((40, 12, 257), "cheb", 0),
         ((512, 260, 257), "cheb", 0), ((36, 10, 511), "sine", 0), ((130, 32, 255), "sine", 2), ((512, 256, 256), "fft", 0)]


@pytest.mark.parametrize("shape,z,flags", CASES)
def test_strided_store_matches(shape, z, flags):
    import torch
    from paper_1905_02803_gb300 import p3dfft as P
    nx, ny, nz = shape
    tt = ("fft", "fft", z)
    pt = P.Plan(nx, ny, nz, precision="f32", ttypes=tt, layout="xyz", flags=flags)
    pn = P.Plan(nx, ny, nz, precision="f32", ttypes=tt, layout="xyz", flags=flags | P.P3_FLAG_NO_TMA)
    assert "pow2_col_tma" in pt.describe() and "col_tma" not in pn.describe(), pt.describe()
    f = torch.from_numpy(inputs.uniform_field((nz, ny, nx), nz)).to("cuda", torch.float32)
    x = torch.zeros(pt.real_shape, device="cuda")
    x[:, :, :nx] = f
    g = torch.Generator(device="cuda")
    g.manual_seed(nx)
    G = torch.view_as_complex(torch.randn(pt.complex_shape + (2,), generator=g, device="cuda"))
    if flags & P.P3_FLAG_PADDED_REAL:
        got = []
        for p in (pt, pn):
            a, b = x.clone(), G.clone()
            got.append((p.forward(a, out=p.complex_view(a)), p.backward(b, out=p.real_view(b))[:, :, :nx]))
        (Xt, yt), (Xn, yn) = got
    else:
        Xt, Xn, yt, yn = pt.forward(x), pn.forward(x), pt.backward(G), pn.backward(G)
    assert torch.equal(Xt, Xn) and torch.equal(yt, yn)
    assert P.p3_plan_wait_status(pt.handle) == P.P3_OK


def test_copy_wait_gives_up_and_reports():
    """The bounded wait of the strided-store form: an arrival that never comes
    ends the wait, the plan reports it, and the next call works."""
    import torch
    from paper_1905_02803_gb300 import p3dfft as P
    plan = P.Plan(32, 16, 256, precision="f32", layout="xyz")
    assert "pow2_col_tma" in plan.describe()
    x = torch.from_numpy(inputs.uniform_field((256, 16, 32), 4)).to("cuda", torch.float32)
    ref = plan.forward(x).clone()
    P.p3_plan_set_wait_limits(plan.handle, 2000, 1)
    plan.forward(x)
    assert P.p3_plan_wait_flags(plan.handle) == P.P3_WAIT_COPY
    P.p3_plan_set_wait_limits(plan.handle, 1 << 23, 0)
    assert torch.equal(plan.forward(x), ref)
    assert P.p3_plan_wait_status(plan.handle) == P.P3_OK
