"""Moments of single-pass lattices do not need the step's segment height to be one that
a launch can take."""
import numpy as np
import pytest

from paper_1712_06079_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu


def test_moments_of_a_lattice_whose_segments_no_launch_takes():
    # 70,000 segments of one row are more than a grid has rows (65,535): the step is
    # refused with them, the moments are not
    nx, ny = 64, 70000
    t = inputs.EOS_TABLE["cs"]
    p = lbm.Params(nx=nx, ny=ny, eos="cs", a=t["a"], b=t["b"], Tr=0.85, k=t["k"], prec="f32")
    g, l = lbm.maxwell(p)
    rho0 = np.broadcast_to(g + (l - g) * inputs.uniform01(3, nx), (ny, nx)).astype(np.float32).astype(np.float64)
    with lbm.Lattice(p) as lat:
        lat.init_density(rho0)
        lat.set_segment_rows(1)
        rho, _, _ = lat.moments()
    assert np.max(np.abs(rho / rho0 - 1)) < 1e-6   # nine products w_i rho and their sum: a few ulp
