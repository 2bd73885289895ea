"""Solvers on general meshes stepped by several host threads at once, each on its own stream: the launches of
the kinetic kernel take shared memory by the solver's own number of colours and the limit on it belongs to the
kernel, so solvers of different meshes must not lower it for each other between setting and launching.  Every thread's state equals that of the same steps alone, bit for bit."""
import threading

import numpy as np
import pytest

from paper_2310_18916_gb300 import gsis
from paper_2310_18916_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _solver(k):
    import torch

    sizes = [(4, 6), (24, 48), (8, 12), (16, 96)]
    n_r, n_th = sizes[k % len(sizes)]
    p = wl.cylinder(n_r=n_r, n_theta=n_th, nv=8, R=0.5, R_out=3.0, Ma=0.3, Kn=0.2)
    with torch.cuda.stream(torch.cuda.Stream()):
        return gsis.Solver(p, precision="f32", mode="dvm", kinetic_presteps=0, n_sweeps=1,
                           init_W=wl.perturbed_state(p, seed=k, amp=0.01))


def test_threads_with_meshes_of_different_colour_counts():
    steps, out, errors = 150, {}, []

    def work(k, to):
        s = _solver(k)
        for _ in range(steps):
            s.step()
        to[k] = s.W()
        s.close()

    alone = {}
    for k in range(4):
        work(k, alone)

    def guarded(k):
        try:
            work(k, out)
        except Exception as e:  # noqa: BLE001 - reported by the main thread
            errors.append(f"thread {k}: {e}")

    ts = [threading.Thread(target=guarded, args=(k,)) for k in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors
    for k in range(4):
        assert np.array_equal(out[k], alone[k]), f"thread {k}"
