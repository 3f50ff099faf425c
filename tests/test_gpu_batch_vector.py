"""The batch's vector path (FP32 HDM lattices on rows of at least 53 cells): every
form against the oracle's step and against each other, on rows of every length
modulo four, the shortest, tiles and slices that end in part of one, columns with
folded weights and with windows."""
import numpy as np
import pytest

import oracle
from paper_1712_06079_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu


def make(nx, ny, eos, force, tau):
    t = inputs.EOS_TABLE[eos]
    gp = lbm.Params(nx=nx, ny=ny, eos=eos, a=t["a"], b=t["b"], omega=t["omega"], Tr=0.85, k=t["k"], tau=tau, force=force,
                    prec="f32")
    op = oracle.params_at(nx, ny, eos, t["a"], t["b"], 0.85, omega=t["omega"], k=t["k"], tau=tau, force=force)
    g, l, _ = oracle.maxwell(op)
    xi = inputs.uniform01(nx * 17 + ny, 12 * nx * ny).reshape(12, ny, nx)
    f = oracle.init(op, inputs.slab(nx, ny, g, l, 4.0) * (1 + 0.01 * (xi[11] - 0.5)), 0.02 * (xi[0] - 0.5), 0.02 * (xi[1] - 0.5))
    f = f * (1.0 + 1e-3 * (xi[2:11] - 0.5))
    return gp, op, f.astype(np.float32).astype(np.float64)


MIXES = [
    [(53, 8, "cs", "sc", 1.0), (54, 3, "vdw", "zc", 0.9), (55, 1, "pr", "sc", 1.0), (57, 8, "rk", "zc", 1.2)],
    [(256, 8, "cs", "sc", 0.9), (257, 8, "pr", "zc", 1.0), (330, 7, "rk", "sc", 1.1), (515, 5, "vdw", "sc", 0.8)],
    [(63, 9, "cs", "zc", 1.0), (65, 17, "pr", "sc", 0.9), (70, 52, "vdw", "sc", 1.0), (98, 33, "rk", "zc", 1.0)],
    [(64, 53, "cs", "sc", 1.0), (53, 70, "vdw", "zc", 0.9), (201, 129, "vdw", "sc", 1.0), (96, 64, "rk", "sc", 1.1)],
]


@pytest.mark.parametrize("mix", range(len(MIXES)))
def test_forms_are_the_oracles_step_and_each_other(mix):
    made = [make(*m) for m in MIXES[mix]]
    f0 = [f for _, _, f in made]
    first = None
    forms = [lambda b: b.set_launch(128, 1), lambda b: b.set_launch(512, 1), lambda b: b.set_cluster(2, 128),
             lambda b: b.set_cluster(8, 512), lambda b: b.set_groups(0, 256), lambda b: b.set_groups(lbm.GROUPS_BALANCED, 1024)]
    ran = 0
    for choose in forms:
        with lbm.Batch([gp for gp, _, _ in made]) as b:
            try:
                choose(b)
            except lbm.LBMError as e:
                assert e.status == lbm.E_INVALID   # a slice narrower than the HDM radius, or too large
                continue
            ran += 1
            b.set_f(f0)
            b.step(1)
            f1 = b.get_f()
            b.step(3)
            f4 = b.get_f()
            rho, vx, vy = b.moments()
        if first is None:
            first = (f1, f4, rho, vx, vy)
            for (gp, op, a), got, r, u, v, g4 in zip(made, f1, rho, vx, vy, f4):
                fo = oracle.step(op, a)
                # one FP32 step: a few ulp per population, more where U = k p - rho/3 cancels
                assert np.max(np.abs(got - fo) / np.abs(fo)) < 1e-5, (gp.nx, gp.ny)
                ro, vxo, vyo = oracle.moments(op, g4)
                assert np.max(np.abs(r / ro - 1)) < 1e-6
                assert max(np.max(np.abs(u - vxo) * ro), np.max(np.abs(v - vyo) * ro)) < 1e-6   # as rho v = j + F/2
        for x, y in zip(first, (f1, f4, rho, vx, vy)):
            for p, q in zip(x, y):
                assert np.array_equal(p, q)
    assert ran >= 2


def test_every_grid_shape_is_taken_and_survives_other_batches():
    # 1280 threads per SM are accepted, whatever fits at once is launched, and the bits
    # are the default shape's; a batch of smaller tiles made in between changes nothing
    tall, thin = [make(*m) for m in MIXES[3]], [make(*m) for m in MIXES[0]]
    out = []
    for shape in (None, (128, 10), (256, 5), (512, 2)):
        with lbm.Batch([gp for gp, _, _ in tall]) as b:
            if shape:
                b.set_launch(*shape)
                with pytest.raises(lbm.LBMError):
                    b.set_launch(shape[0], shape[1] + 1)
            with lbm.Batch([gp for gp, _, _ in thin]) as other:
                other.set_f([f for _, _, f in thin])
                other.step(1)
                other.sync()
            b.set_f([f for _, _, f in tall])
            b.step(2)
            b.sync()
            out.append(np.concatenate([f.ravel() for f in b.get_f()]))
    for o in out[1:]:
        assert np.array_equal(o, out[0])


@pytest.mark.parametrize("nx,ny", [(512, 8), (520, 8), (756, 8), (58, 96)])
def test_cluster_of_each_thread_count_is_the_grid_form(nx, ny):
    # two CTAs of 512 | 520 threads, where the kernel changes, 760 and 768, the most that
    # a slice can have
    gp, _, f = make(nx, ny, "cs", "sc", 0.9)
    out = []
    for choose in (lambda b: b.set_launch(256, 1), lambda b: b.set_cluster(2, 512)):
        with lbm.Batch([gp, gp]) as b:
            choose(b)
            b.set_f([f, f])
            b.step(3)
            b.sync()
            out.append(np.stack(b.get_f()))
    assert np.array_equal(out[0], out[1])
