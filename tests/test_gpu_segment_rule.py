"""The segment height the library picks for the single-pass kernel on a GPU of
152 SMs: whole slabs (8k - 2 rows) and, for the HDM, the fewest waves x slabs."""
import numpy as np
import pytest

from paper_1712_06079_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,grad,rows", [(64, 54, "hdm", 6), (512, 512, "hdm", 14), (768, 768, "hdm", 22),
                                             (1024, 1024, "hdm", 38), (1024, 1024, "cdm", 38), (256, 4096, "hdm", 46),
                                             (2048, 2048, "hdm", 134), (2048, 2048, "cdm", 62)])
def test_picked_height(nx, ny, grad, rows):
    torch = pytest.importorskip("torch")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the heights are those of 152 SMs")
    with lbm.Lattice(lbm.Params(nx=nx, ny=ny, eos="cs", Tr=0.8, k=0.04, grad=grad)) as lat:
        assert lat.segment_rows() == rows
        lat.set_segment_rows(54 if ny >= 54 else ny)
        lat.set_segment_rows(0)               # back to the library's choice
        assert lat.segment_rows() == rows


@pytest.mark.parametrize("nx,ny", [(128, 228), (128, 234), (256, 300), (256, 306)])
@pytest.mark.parametrize("grad", ["hdm", "cdm"])
def test_overlapping_launches_change_nothing(nx, ny, grad):
    # 76 | 78 and 150 | 153 segments of six rows: both sides of the lines between which
    # a CTA gets an SM to itself.  Steps whose launches overlap are bit for bit the steps
    # that are waited for one by one
    rho = 0.2 + 0.02 * (inputs.uniform01(nx + ny, nx * ny).reshape(ny, nx) - 0.5)
    out = []
    for chunks in ([1] * 8, [8]):
        with lbm.Lattice(lbm.Params(nx=nx, ny=ny, eos="cs", Tr=0.8, k=0.04, grad=grad)) as lat:
            lat.set_segment_rows(6)
            lat.init_density(rho)
            for n in chunks:
                lat.step(n)
                last = lat.get_f()
            out.append(last)
    assert np.isfinite(out[0]).all() and np.array_equal(out[0], out[1])
