"""Fields of equal values have no derivative, bit for bit, in the FP64-arithmetic step:
a uniform lattice at rest stays at rest, and a state that is uniform along one direction
stays so (lines longer and shorter than a block of 8 cells, and ending in part of one)."""
import numpy as np
import pytest

from paper_1712_06079_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu

SIZES = [(2, 2), (5, 9), (37, 19), (40, 24), (129, 66), (200, 12)]


def make(nx, ny, prec, force, tau, walls):
    t = inputs.EOS_TABLE["cs"]
    return lbm.Params(nx=nx, ny=ny, eos="cs", a=t["a"], b=t["b"], Tr=0.8, k=t["k"], tau=tau, force=force, prec=prec,
                      walls=walls, two_pass=True)


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("prec,force,tau,walls", [("f64", "sc", 1.0, False), ("f64", "zc", 0.8, True),
                                                  ("f32", "sc", 1.2, True), ("f32", "zc", 1.0, False)])
def test_a_uniform_lattice_at_rest_stays_at_rest(nx, ny, prec, force, tau, walls):
    with lbm.Lattice(make(nx, ny, prec, force, tau, walls)) as lat:
        lat.init_density(np.full((ny, nx), 0.3))
        for _ in range(3):
            lat.step(2)
            rho, vx, vy = lat.moments()
            assert (vx == 0).all() and (vy == 0).all()
            assert (rho == rho[0, 0]).all()


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("prec,force,tau,along", [("f64", "sc", 1.0, "y"), ("f64", "zc", 0.8, "x"),
                                                  ("f64", "sc", 1.1, "x"), ("f32", "zc", 1.0, "y")])
def test_a_state_uniform_along_a_direction_stays_so(nx, ny, prec, force, tau, along):
    p = make(nx, ny, prec, force, tau, False)
    g, l = lbm.maxwell(p)
    n = nx if along == "y" else ny
    line = 0.5 * (g + l) + 0.3 * (l - g) * np.sin(2 * np.pi * np.arange(n) / n + 0.3)
    rho = np.broadcast_to(line if along == "y" else line[:, None], (ny, nx)).copy()
    with lbm.Lattice(p) as lat:
        lat.init_density(rho)
        lat.step(20)
        f = lat.get_f()
    assert np.isfinite(f).all()
    first = f[:, :1, :] if along == "y" else f[:, :, :1]
    assert np.array_equal(f, np.broadcast_to(first, f.shape))
