"""The reverse mode's further records: at most half of the free device memory (made
small by LBM_DEBUG_FREE_BYTES) is taken for them, and the gradient is the same bit for bit
with all, some and none of the segments kept, with the allocation refused, on a tape
reused for another step count, and with every state in one segment."""
import os

import numpy as np
import pytest

from paper_1712_06079_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu
FREE, FAIL = "LBM_DEBUG_FREE_BYTES", "LBM_DEBUG_FAIL_ALLOC"
NX = NY = 256
C = 4


@pytest.fixture(autouse=True)
def no_hooks():
    yield
    os.environ.pop(FREE, None)
    os.environ.pop(FAIL, None)


def make(prec, tau=1.0):
    torch = pytest.importorskip("torch")
    t = inputs.EOS_TABLE["cs"]
    p = lbm.Params(nx=NX, ny=NY, eos="cs", a=t["a"], b=t["b"], Tr=0.85, k=t["k"], tau=tau, prec=prec,
                   stream=torch.cuda.current_stream().cuda_stream)
    g, l = lbm.maxwell(p)
    dt = torch.float64 if prec == "f64" else torch.float32
    x = torch.tensor(inputs.droplet(NX, NY, 70, g, l, 3.0), dtype=dt, device="cuda")
    v = torch.tensor(inputs.uniform01(3, NX * NY).reshape(NY, NX) - 0.5, dtype=dt, device="cuda")
    with lbm.Lattice(p) as lat:   # (the kernels are loaded before memory is counted)
        sweep(torch, lat, x, v, 24, C)
    return torch, p, x, v


def sweep(torch, lat, x, v, nsteps, interval):
    """(bytes the forward took, gradients of two sweeps)"""
    rT, g0 = torch.empty_like(x), torch.empty_like(x)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    lat.adjoint_forward(x.data_ptr(), nsteps, interval, rT.data_ptr())
    torch.cuda.synchronize()
    took = free - torch.cuda.mem_get_info()[0]
    out = []
    for _ in range(2):   # kept records, then recomputed ones
        out.append((lat.adjoint_backward(v.data_ptr(), g0.data_ptr())[0], g0.cpu().numpy()))
    return took, out


def same(a, b):
    return all(x[0] == y[0] and np.array_equal(x[1], y[1]) for x in a for y in b)


@pytest.mark.parametrize("prec,tau", [("f32", 1.0), ("f64", 1.0), ("f64", 0.9)])
def test_half_of_the_free_memory_is_the_limit(prec, tau):
    torch, p, x, v = make(prec, tau)
    esz = 8 if prec == "f64" else 4
    # a segment: C records of five planes and C fields (padded by 64 columns in the FP32 layout)
    per = C * esz * NY * (5 * NX + NX + (64 if prec == "f32" else 0))
    took, grads = {}, {}
    for kept in (0, 1, 2, 4):                    # of the four segments before the last two
        os.environ[FREE] = str(2 * kept * per + per)
        with lbm.Lattice(p) as lat:
            took[kept], grads[kept] = sweep(torch, lat, x, v, 24, C)
    for kept in (1, 2, 4):
        # memory is mapped in pieces of 2 MiB: one more or less on either side
        assert abs(took[kept] - took[0] - kept * per) <= 2 * (2 << 20), (kept, took, per)
    os.environ.pop(FREE)
    with lbm.Lattice(p) as lat:
        _, one = sweep(torch, lat, x, v, 24, 24)   # every state in one segment
    for g in grads.values():
        assert same(g, one)


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_a_refused_allocation_leaves_the_tape_without(prec):
    torch, p, x, v = make(prec)
    with lbm.Lattice(p) as lat:
        full, want = sweep(torch, lat, x, v, 24, C)
    for n in range(200):
        with lbm.Lattice(p) as lat:
            os.environ[FAIL] = str(n)
            try:
                took, got = sweep(torch, lat, x, v, 24, C)
            except lbm.LBMError as e:
                assert e.status == lbm.E_NOMEM
                continue
            finally:
                os.environ.pop(FAIL)
        break
    assert took < full and same(got, want)


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("first,then", [(11, 8), (8, 11), (23, 21)])
def test_a_tape_reused_for_another_step_count(prec, first, then):
    torch, p, x, v = make(prec)
    with lbm.Lattice(p) as lat:
        _, want = sweep(torch, lat, x, v, then, C)
    with lbm.Lattice(p) as lat:
        sweep(torch, lat, x, v, first, C)
        took, got = sweep(torch, lat, x, v, then, C)
    assert took == 0 and same(got, want)   # (the same number of checkpoints: nothing is allocated)
