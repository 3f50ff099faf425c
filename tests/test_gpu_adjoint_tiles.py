"""The FP32 record-based reverse kernels on tiles of 64 x 4 cells: lattices that end
in part of a tile both ways, against the FP64 reverse mode of the same lattice."""
import numpy as np
import pytest

from paper_1712_06079_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(64, 54), (68, 57), (124, 59), (132, 66)])
@pytest.mark.parametrize("force,tau", [("sc", 1.0), ("zc", 0.9)])
def test_fp32_gradient_follows_fp64(nx, ny, force, tau):
    torch = pytest.importorskip("torch")
    t = inputs.EOS_TABLE["cs"]
    xi = inputs.uniform01(nx + 5 * ny, 2 * nx * ny).reshape(2, ny, nx)
    out = {}
    for prec, dt in (("f64", torch.float64), ("f32", torch.float32)):
        p = lbm.Params(nx=nx, ny=ny, eos="cs", a=t["a"], b=t["b"], Tr=0.85, k=t["k"], tau=tau, force=force, prec=prec,
                       stream=torch.cuda.current_stream().cuda_stream)
        g, l = lbm.maxwell(p)
        x = torch.tensor(inputs.droplet(nx, ny, ny / 4, g, l, 3.0) * (1 + 0.01 * (xi[0] - 0.5)), dtype=dt, device="cuda")
        v = torch.tensor(xi[1] - 0.5, dtype=dt, device="cuda")
        rT, g0 = torch.empty_like(x), torch.empty_like(x)
        torch.cuda.synchronize()
        with lbm.Lattice(p) as lat:
            assert (lat.segment_rows() > 0) == (prec == "f32")   # the single-pass kernel's record
            lat.adjoint_forward(x.data_ptr(), 12, 4, rT.data_ptr())
            _, gtr, _ = lat.adjoint_backward(v.data_ptr(), g0.data_ptr())
        out[prec] = (gtr, g0.double().cpu().numpy())
    # twelve steps of FP32 rounding, a few ulp each way and step: 1e-4 of the largest
    # entry, and of the sum's size for the scalar
    (ga, fa), (gb, fb) = out["f64"], out["f32"]
    assert np.max(np.abs(fb - fa)) < 1e-4 * np.max(np.abs(fa))
    assert abs(gb - ga) < 2e-3 * abs(ga) + 1e-3


@pytest.mark.parametrize("nx,ny", [(128, 152), (132, 152), (512, 608), (516, 608)])
def test_overlapping_launches_change_nothing(nx, ny):
    # 76 | 114 tiles and 1216 | 1368: both sides of the lines at which the launches are
    # spread over the SMs.  A tape with every state and one of short segments, whose first
    # launches do not overlap, take the same steps: bit for bit the same gradient
    torch = pytest.importorskip("torch")
    t = inputs.EOS_TABLE["cs"]
    xi = inputs.uniform01(nx + 5 * ny, 2 * nx * ny).reshape(2, ny, nx)
    p = lbm.Params(nx=nx, ny=ny, eos="cs", a=t["a"], b=t["b"], Tr=0.85, k=t["k"], prec="f32",
                   stream=torch.cuda.current_stream().cuda_stream)
    g, l = lbm.maxwell(p)
    x = torch.tensor(inputs.droplet(nx, ny, ny / 4, g, l, 3.0) * (1 + 0.01 * (xi[0] - 0.5)), dtype=torch.float32, device="cuda")
    v = torch.tensor(xi[1] - 0.5, dtype=torch.float32, device="cuda")
    out = []
    for chunk in (1, 9):
        rT, g0 = torch.empty_like(x), torch.empty_like(x)
        torch.cuda.synchronize()
        with lbm.Lattice(p) as lat:
            lat.adjoint_forward(x.data_ptr(), 9, chunk, rT.data_ptr())
            lat.adjoint_backward(v.data_ptr(), g0.data_ptr())
            out.append(g0.cpu().numpy())
    assert np.isfinite(out[0]).all() and np.array_equal(out[0], out[1])
