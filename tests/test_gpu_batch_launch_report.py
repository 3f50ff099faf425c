"""What a batch reports of its launch is what it launches."""
import pytest

from paper_1712_06079_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu


def make(nx, ny):
    t = inputs.EOS_TABLE["cs"]
    return lbm.Params(nx=nx, ny=ny, eos="cs", a=t["a"], b=t["b"], Tr=0.85, k=t["k"], prec="f32")


def test_the_reported_grid_is_the_launched_one():
    torch = pytest.importorskip("torch")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with lbm.Batch([make(96, 64), make(200, 200)]) as b:
        threads, blocks = b.launch()   # the default: 256 threads, every block that is resident at once
        assert threads == 256 and blocks % sms == 0
        b.set_launch(256, 1)
        assert b.launch() == (256, sms)
        b.set_launch(256, 5)           # accepted; more than the tiles leave room for
        assert b.launch() == (256, blocks)
