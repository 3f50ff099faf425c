"""Batches of different slices stepped by several threads do not disturb one another's
launches."""
import threading

import numpy as np
import pytest

from paper_1712_06079_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu


def make(nx, ny, prec="f32"):
    t = inputs.EOS_TABLE["cs"]
    return lbm.Params(nx=nx, ny=ny, eos="cs", a=t["a"], b=t["b"], Tr=0.85, k=t["k"], prec=prec)


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_threads_with_different_slices(prec):
    # every step count is new, so every call prepares a launch of its own
    shapes = [(320, 16), (176, 4)] if prec == "f32" else [(320, 8), (176, 4)]
    failures = []

    def run(nx, ny):
        try:
            with lbm.Batch([make(nx, ny, prec)] * 2) as b:
                b.set_cluster(2, 256)
                b.init_density([np.full((ny, nx), 0.3)] * 2)
                for n in range(1, 301):
                    b.step(n % 2 + 2 * n)
                b.sync()
        except Exception as e:   # (reported by the main thread)
            failures.append(repr(e))

    threads = [threading.Thread(target=run, args=s) for s in shapes for _ in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures
