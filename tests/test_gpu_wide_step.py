"""The FP64-arithmetic two-pass step with the HDM by block sums (wide_step.cu)
against the oracle, whose operator is the cyclic tridiagonal solve: lines
shorter and longer than a block of 8 cells and than the 40 cells that are
joined, ends in a block of every length, mirrored columns between walls."""
import numpy as np
import pytest

import oracle
from paper_1712_06079_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu


def make(nx, ny, prec, force="sc", grad="hdm", tau=1.0, walls=False, radius=0):
    t = inputs.EOS_TABLE["cs"]
    gp = lbm.Params(nx=nx, ny=ny, eos="cs", a=t["a"], b=t["b"], Tr=0.8, k=t["k"], tau=tau, force=force, grad=grad,
                    prec=prec, walls=walls, hdm_radius=radius, two_pass=True)
    op = oracle.params_at(nx, ny, "cs", t["a"], t["b"], 0.8, k=t["k"], tau=tau, force=force, grad=grad, walls=walls)
    g, l, _ = oracle.maxwell(op)
    xi = inputs.uniform01(nx * 131 + ny, 12 * nx * ny).reshape(12, ny, nx)
    f = oracle.init(op, g + (l - g) * xi[11], 0.1 * (xi[0] - 0.5), 0.1 * (xi[1] - 0.5))
    return gp, op, f * (1.0 + 1e-3 * (xi[2:11] - 0.5))


SIZES = [(2, 2), (3, 9), (7, 40), (8, 8), (9, 17), (16, 5), (15, 41), (39, 81), (23, 64), (121, 10), (130, 133)]


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("force,grad,tau,walls", [("sc", "hdm", 1.0, False), ("zc", "hdm", 0.8, False),
                                                  ("sc", "hdm", 1.2, True), ("zc", "hdm", 1.0, True),
                                                  ("sc", "cdm", 0.9, True), ("zc", "cdm", 1.0, False)])
def test_one_step_is_the_oracles(nx, ny, force, grad, tau, walls):
    # FP64: the per-step bar of 1e-12 on every population (a random density
    # field, so the derivative is as rough as the lattice carries)
    gp, op, f0 = make(nx, ny, "f64", force, grad, tau, walls)
    with lbm.Lattice(gp) as lat:
        lat.set_f(f0)
        r, vx, vy = lat.moments()   # (of the given state: a step of so rough a field may leave the stable range)
        lat.step(1)
        fg = lat.get_f()
    fo = oracle.step(op, f0)
    scale = np.abs(fo).max(axis=0)   # (a small population of a cell can cancel: relative to the cell's largest)
    assert np.max(np.abs(fg - fo) / scale) < 1e-12
    ro, vxo, vyo = oracle.moments(op, f0)
    assert np.max(np.abs(r / ro - 1)) < 1e-12
    assert max(np.abs(vx - vxo).max(), np.abs(vy - vyo).max()) < 1e-12 * max(1.0, np.abs(vxo).max())


@pytest.mark.parametrize("nx,ny", [(9, 17), (39, 81), (130, 133)])
def test_fp32_storage_adds_one_rounding(nx, ny):
    # FP32 distributions, FP64 arithmetic: the oracle's step of the stored
    # state, rounded once (half an ulp, 6e-8 relative to each population)
    gp, op, f0 = make(nx, ny, "f32")
    f0 = f0.astype(np.float32).astype(np.float64)
    with lbm.Lattice(gp) as lat:
        lat.set_f(f0)
        lat.step(1)
        fg = lat.get_f()
    fo = oracle.step(op, f0)
    assert np.max(np.abs(fg - fo) / np.abs(fo).max(axis=0)) < 6.0e-8


def test_a_requested_radius_keeps_its_truncation():
    # hdm_radius is part of the result: 8 and the automatic radius differ by
    # about r^9 = 2e-4 of the derivative on a rough field, and 40 equals it
    out = {}
    for radius in (0, 8, 40):
        gp, op, f0 = make(64, 48, "f64", radius=radius)
        with lbm.Lattice(gp) as lat:
            lat.set_f(f0)
            lat.step(1)
            out[radius] = lat.get_f()
    scale = np.abs(out[0]).max()
    assert np.abs(out[40] - out[0]).max() < 1e-14 * scale * 100
    assert np.abs(out[8] - out[0]).max() > 1e-9 * scale


@pytest.mark.parametrize("nx,ny", [(17, 9), (8, 33), (23, 41), (6, 100)])
@pytest.mark.parametrize("eos,force,grad,tau", [("pr", "sc", "hdm", 1.0), ("rk", "zc", "hdm", 0.9), ("vdw", "sc", "cdm", 1.1),
                                                ("cs", "zc", "cdm", 1.0)])
def test_reverse_step_is_the_complex_step_derivative(nx, ny, eos, force, grad, tau):
    # the FP64 reverse kernels on short and ragged lines, 5 steps with a
    # checkpoint every 2 (a recomputed segment among them): 1e-11, the bar of the
    # oracle's derivative on the larger lattices
    torch = pytest.importorskip("torch")
    t = inputs.EOS_TABLE[eos]
    p = lbm.Params(nx=nx, ny=ny, eos=eos, a=t["a"], b=t["b"], omega=t["omega"], Tr=0.9, k=t["k"], tau=tau, force=force,
                   grad=grad, prec="f64", stream=torch.cuda.current_stream().cuda_stream)
    op = oracle.params_at(nx, ny, eos, t["a"], t["b"], 0.9, omega=t["omega"], k=t["k"], tau=tau, force=force, grad=grad)
    g, l, _ = oracle.maxwell(op)
    xi = inputs.uniform01(nx + 3 * ny, 3 * nx * ny).reshape(3, ny, nx)
    rho0 = 0.5 * (g + l) * (1 + 0.1 * (xi[0] - 0.5))
    v = xi[1] - 0.5                                # dL/drho_T
    with lbm.Lattice(p) as lat:
        x = torch.tensor(rho0, device="cuda")
        rT, g0 = torch.empty_like(x), torch.empty_like(x)
        gr = torch.tensor(v, device="cuda")
        torch.cuda.synchronize()
        lat.adjoint_forward(x.data_ptr(), 5, 2, rT.data_ptr())
        _, gtr, _ = lat.adjoint_backward(gr.data_ptr(), g0.data_ptr())
        out, grad0 = rT.cpu().numpy(), g0.cpu().numpy()
    r, dT = oracle.tangent(op, rho0, 5, dTr=1.0)
    assert np.max(np.abs(out / r - 1)) < 1e-12
    assert abs(gtr - (v * dT).sum()) < 1e-11 * np.abs(v * dT).sum()
    d = xi[2] - 0.5
    _, dd = oracle.tangent(op, rho0, 5, drho0=d)
    assert abs((grad0 * d).sum() - (v * dd).sum()) < 1e-11 * np.abs(v * dd).sum()


@pytest.mark.parametrize("nx,ny", [(608, 16), (616, 16), (304, 256), (304, 264)])
@pytest.mark.parametrize("prec,tau", [("f64", 1.0), ("f32", 0.9)])
def test_overlapping_launches_change_nothing(nx, ny, prec, tau):
    # 76 | 78 tiles and 608 | 627: both sides of the two lines at which the
    # launches change between spreading over the SMs and not.  Steps whose
    # launches overlap are bit for bit the steps that are waited for one by one
    gp, op, _ = make(nx, ny, prec, tau=tau)
    g, l, _ = oracle.maxwell(op)
    y, x = np.mgrid[0:ny, 0:nx]
    wave = np.sin(2 * np.pi * x / nx) * np.cos(2 * np.pi * y / ny)
    f0 = oracle.init(op, 0.5 * (g + l) + 0.1 * (l - g) * wave, 0.01 * wave, -0.01 * wave)
    out = []
    for chunks in ([1] * 8, [8]):
        with lbm.Lattice(gp) as lat:
            lat.set_f(f0)
            for n in chunks:
                lat.step(n)
                last = lat.get_f()
            out.append(last)
    assert np.isfinite(out[0]).all() and np.array_equal(out[0], out[1])
