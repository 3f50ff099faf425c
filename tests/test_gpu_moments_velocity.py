"""The velocities of single-pass lattices carry no rounding but their own: on a state of
equal densities, where the force is zero, and populations whose sums are exact, v is the
FP32 quotient j / rho; and a light gas shows the rounding of its own field, not that of a
liquid film's some way off, whichever row the segments of the sweep begin at."""
import numpy as np
import pytest

import oracle
from paper_1712_06079_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu


def make(nx, ny, grad="hdm", walls=False):
    t = inputs.EOS_TABLE["cs"]
    return lbm.Params(nx=nx, ny=ny, eos="cs", a=t["a"], b=t["b"], Tr=0.85, k=t["k"], grad=grad, prec="f32", walls=walls)


@pytest.mark.parametrize("nx,ny,grad,walls", [(128, 70, "hdm", False), (124, 55, "cdm", False), (64, 54, "hdm", True)])
def test_velocity_is_the_rounded_quotient(nx, ny, grad, walls):
    unit = 2.0 ** -20    # every population and every sum of some of them a multiple of it, below 1: exact in FP32
    xi = np.round(inputs.uniform01(nx + ny, 8 * nx * ny).reshape(8, ny, nx) * 2 ** 14)
    f = np.empty((9, ny, nx))
    f[1:] = unit * (2 ** 15 + xi)
    total = unit * 699051                          # the density of every cell
    f[0] = total - f[1:].sum(0)
    assert (f > 0).all()
    ex = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1.0])
    ey = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1.0])
    jx, jy = (np.tensordot(e, f, 1).astype(np.float32) for e in (ex, ey))
    with lbm.Lattice(make(nx, ny, grad, walls)) as lat:
        assert lat.segment_rows() > 0              # the single-pass kernel
        lat.set_f(f)
        r, vx, vy = lat.moments()
    assert (r == total).all()
    rho = np.float32(total)
    assert np.array_equal(vx, (jx / rho).astype(np.float64)) and np.array_equal(vy, (jy / rho).astype(np.float64))


@pytest.mark.parametrize("walls", [False, True])
def test_a_light_gas_shows_the_rounding_of_its_own_field_only(walls):
    # Peng-Robinson at 0.7 T_c: a film 145 times as dense as the gas; segments of 62 rows,
    # the second beginning in the film; rows 40 and more from it.  With u = 2^-24: the field
    # U = k p - rho / 3 of a gas cell is off by at most 8 u (the density's sum) + 6 u (the
    # equation of state) of its terms, which are below 0.37 rho; D sums 2.74 times that (the
    # weights' magnitudes) and adds 6 u of it by its own operations; v takes D / (2 rho), and
    # j and the quotient add a few u of the largest |v| and of the populations over rho
    nx, ny = 128, 186
    t = inputs.EOS_TABLE["pr"]
    gp = lbm.Params(nx=nx, ny=ny, eos="pr", a=t["a"], b=t["b"], omega=t["omega"], Tr=0.7, k=t["k"], force="zc", prec="f32",
                    walls=walls)
    op = oracle.params_at(nx, ny, "pr", t["a"], t["b"], 0.7, omega=t["omega"], k=t["k"], force="zc", walls=walls)
    g, l = lbm.maxwell(gp)
    rho = g * (1 + 1e-3 * (inputs.uniform01(5, nx * ny).reshape(ny, nx) - 0.5))
    rho[55:65] = l
    with lbm.Lattice(gp) as lat:
        lat.set_segment_rows(62)
        lat.set_f(oracle.init(op, rho))
        _, vx, vy = lat.moments()
        f = lat.get_f()
    _, vxo, vyo = oracle.moments(op, f)
    far, u = np.arange(105, 150), 2.0 ** -24
    tol = 2.74 * (8 + 6 + 6) * u * 0.37 * 1.001 / (2 * 0.999) + 8 * u
    assert np.abs(vy[far] - vyo[far]).max() < tol and np.abs(vx[far] - vxo[far]).max() < tol
