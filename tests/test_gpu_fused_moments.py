"""The moments variant of the single-pass kernel against the oracle's moments of
the same FP32 state: ragged strips and segments, the smallest lattice, walls,
CDM, output arrays off the 16-byte grid, before the first step (the field is
formed from f) and after one (the field the step left)."""
import numpy as np
import pytest

import oracle
from paper_1712_06079_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu

CASES = [(64, 54, "sc", "hdm", 1.0, False, 0), (124, 55, "zc", "hdm", 0.8, False, 1), (132, 129, "sc", "hdm", 1.0, True, 3),
         (236, 60, "sc", "cdm", 1.2, False, 2), (128, 70, "zc", "cdm", 1.0, True, 1)]


@pytest.mark.parametrize("nx,ny,force,grad,tau,walls,shift", CASES)
def test_moments_are_the_oracles(nx, ny, force, grad, tau, walls, shift):
    torch = pytest.importorskip("torch")
    t = inputs.EOS_TABLE["cs"]
    gp = lbm.Params(nx=nx, ny=ny, eos="cs", a=t["a"], b=t["b"], Tr=0.85, k=t["k"], tau=tau, force=force, grad=grad,
                    prec="f32", walls=walls, stream=torch.cuda.current_stream().cuda_stream)
    op = oracle.params_at(nx, ny, "cs", t["a"], t["b"], 0.85, k=t["k"], tau=tau, force=force, grad=grad, walls=walls)
    g, l, _ = oracle.maxwell(op)
    xi = inputs.uniform01(nx + 7 * ny, 2 * nx * ny).reshape(2, ny, nx)
    f0 = oracle.init(op, inputs.droplet(nx, ny, ny / 4, g, l, 3.0), 0.05 * (xi[0] - 0.5), 0.05 * (xi[1] - 0.5))
    n = nx * ny
    buf = torch.full((3 * (n + 4) + 4,), -1.0, dtype=torch.float32, device="cuda")
    at = [shift + k * (n + 4) for k in range(3)]   # shift 0: 16-byte aligned starts, else not
    with lbm.Lattice(gp) as lat:
        assert lat.segment_rows() > 0              # the single-pass kernel
        lat.set_f(f0)
        for _ in range(2):
            lat.moments_device(*(buf.data_ptr() + 4 * a for a in at))
            out = buf.double().cpu().numpy()
            r, vx, vy = (out[a:a + n].reshape(ny, nx) for a in at)
            keep = np.ones(out.size, bool)
            for a in at:
                keep[a:a + n] = False
            assert (out[keep] == -1).all()         # nothing written beside the three arrays
            ro, vxo, vyo = oracle.moments(op, lat.get_f())
            assert np.max(np.abs(r / ro - 1)) < 1e-6
            # rho v = j + F/2: j to a few ulp of rho (the largest 0.35), F = 2 Phi D to a few ulp
            # of its factors (Phi below 0.4, the stencil's weights summing below 3): under 1e-6
            assert np.max(np.abs(vx - vxo) * ro) < 1e-6 and np.max(np.abs(vy - vyo) * ro) < 1e-6
            lat.step(1)
