"""The segment height the library picks for the single-pass kernel on a GPU of
152 SMs: whole slabs (8k - 2 rows) and, for the HDM, the fewest waves x slabs."""
import pytest

from paper_1712_06079_gb300 import lbm

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
