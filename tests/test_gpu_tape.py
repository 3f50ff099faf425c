"""The reverse mode's kept records: a sweep from the records of the forward and a
second one, which recomputes them, give the same gradient bit for bit, for
checkpoint intervals that keep all, some and none of the segments."""
import numpy as np
import pytest

from paper_1712_06079_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("nsteps,C", [(25, 5), (26, 5), (13, 2), (7, 7), (5, 9), (9, 1)])
def test_kept_and_recomputed_records_agree(prec, nsteps, C):
    torch = pytest.importorskip("torch")
    t = inputs.EOS_TABLE["cs"]
    p = lbm.Params(nx=96, ny=64, eos="cs", a=t["a"], b=t["b"], Tr=0.85, k=t["k"], prec=prec,
                   stream=torch.cuda.current_stream().cuda_stream)
    g, l = lbm.maxwell(p)
    dt = torch.float64 if prec == "f64" else torch.float32
    x = torch.tensor(inputs.droplet(96, 64, 18, g, l, 3.0), dtype=dt, device="cuda")
    v = torch.tensor(inputs.uniform01(3, 96 * 64).reshape(64, 96) - 0.5, dtype=dt, device="cuda")
    rT = torch.empty_like(x)
    grads = []
    with lbm.Lattice(p) as lat:
        for _ in range(2):                      # the second forward reuses the tape
            lat.adjoint_forward(x.data_ptr(), nsteps, C, rT.data_ptr())
            for _ in range(2):                  # kept records, then recomputed ones
                g0 = torch.empty_like(x)
                torch.cuda.synchronize()
                grads.append((lat.adjoint_backward(v.data_ptr(), g0.data_ptr())[0], g0.cpu().numpy()))
    for gt, g0 in grads[1:]:
        assert gt == grads[0][0] and np.array_equal(g0, grads[0][1])
