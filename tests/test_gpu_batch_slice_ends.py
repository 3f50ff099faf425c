"""The batch's cluster and grouped forms read no shared memory that they have not
written: with what a diverged batch left on the SMs (NaN everywhere) they give the grid
form's bits, on rows whose last group of four holds one, two, three and four cells."""
import numpy as np
import pytest

from paper_1712_06079_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu


def params(nx, ny, eos="cs", tau=1.0):
    t = inputs.EOS_TABLE[eos]
    return lbm.Params(nx=nx, ny=ny, eos=eos, a=t["a"], b=t["b"], omega=t["omega"], Tr=0.85, k=t["k"], tau=tau, prec="f32")


def leave_nan():
    """Steps a batch of densities past the equation of state's range, whose
    populations become NaN, in CTAs that together cover every SM's shared memory."""
    ps = [params(512, 8) for _ in range(160)]
    with lbm.Batch(ps) as b:
        b.set_cluster(2, 512)
        b.init_density([np.full((8, 512), 1e30) for _ in ps])
        b.step(4)
        with pytest.raises(lbm.LBMError) as e:
            b.sync()
        assert e.value.status == lbm.E_UNSTABLE


MIXES = [([(53, 8, "cs", 1.0), (57, 5, "pr", 0.9), (54, 8, "vdw", 1.0)], (2,)),
         ([(257, 8, "cs", 0.9), (258, 8, "rk", 1.0), (259, 8, "pr", 1.0), (509, 8, "vdw", 1.1)], (2, 4, 8)),
         ([(65, 17, "pr", 1.0), (57, 64, "cs", 1.0), (58, 96, "rk", 0.9)], (2,))]


@pytest.mark.parametrize("mix", range(len(MIXES)))
def test_forms_agree_on_whatever_shared_memory_holds(mix):
    cases, sizes = MIXES[mix]
    ps = [params(*c) for c in cases]
    rho = []
    for p in ps:
        g, l = lbm.maxwell(p)
        xi = inputs.uniform01(p.nx + 31 * p.ny, p.nx * p.ny).reshape(p.ny, p.nx)
        rho.append(0.5 * (g + l) * (1 + 0.05 * (xi - 0.5)))
    ref = None
    forms = [lambda b: b.set_launch(256, 1)] + [lambda b, c=c: b.set_cluster(c, 256) for c in sizes]
    forms += [lambda b: b.set_groups(0, 256), lambda b: b.set_groups(lbm.GROUPS_BALANCED, 256)]
    for choose in forms:
        for _ in range(3):
            with lbm.Batch(ps) as b:
                choose(b)
                b.init_density(rho)
                leave_nan()
                b.step(5)
                b.sync()
                f = np.concatenate([a.ravel() for a in b.get_f()])
            ref = f if ref is None else ref
            assert np.isfinite(f).all() and np.array_equal(f, ref)
