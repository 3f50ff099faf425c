"""The bounds-checked build (see test_gpu_checked.py) on the batch's vector path, whose
kernels check their shared-memory accesses too: rows that end in part of a group, the
shortest and narrowest slices, columns with folded weights and with windows, in the
grid, cluster and grouped forms.  No bounds report, the forms' bits equal, every canary
intact."""
import os
import subprocess
import sys
import textwrap

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = textwrap.dedent('''
    import numpy as np
    from paper_1712_06079_gb300 import inputs, lbm
    lbm.load()
    assert lbm.damaged_canaries() == 0                 # the checked library is loaded
    MIXES = [([(53, 8), (54, 3), (55, 1), (57, 8)], (2,)), ([(256, 8), (257, 7), (330, 8), (515, 5)], (2, 4, 8)),
             ([(53, 70), (58, 96), (65, 17), (98, 33)], (2,))]
    for cases, sizes in MIXES:
        ps = []
        for k, (nx, ny) in enumerate(cases):
            t = inputs.EOS_TABLE[("cs", "pr", "vdw", "rk")[k]]
            ps.append(lbm.Params(nx=nx, ny=ny, eos=("cs", "pr", "vdw", "rk")[k], a=t["a"], b=t["b"], omega=t["omega"],
                                 Tr=0.85, k=t["k"], tau=(1.0, 0.9)[k % 2], force=("sc", "zc")[k // 2], prec="f32"))
        rho = []
        for p in ps:
            g, l = lbm.maxwell(p)
            xi = inputs.uniform01(p.nx + p.ny, p.nx * p.ny).reshape(p.ny, p.nx)
            rho.append(0.5 * (g + l) * (1 + 0.02 * (xi - 0.5)))
        outs = []
        for choose in [lambda b: b.set_launch(128, 1)] + [lambda b, c=c: b.set_cluster(c, 128) for c in sizes] + [
                lambda b: b.set_groups(0, 256)]:
            with lbm.Batch(ps) as b:
                choose(b)
                b.init_density(rho)
                b.step(4)
                outs.append(np.concatenate([m.ravel() for field in b.moments() for m in field]))   # (a bounds report raises)
        assert np.isfinite(outs[0]).all()
        for other in outs[1:]:
            assert np.array_equal(outs[0], other)
    assert lbm.damaged_canaries() == 0
    print("checked batch ok")
''')


def test_checked_build_runs_clean_on_the_vector_path():
    from paper_1712_06079_gb300 import build
    build.build(checked=True)
    env = dict(os.environ, LBM_CHECKED="1", PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "checked batch ok" in r.stdout
