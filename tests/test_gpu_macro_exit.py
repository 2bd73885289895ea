"""The early exit of the synthetic solve on rectilinear blocks, whose test of an inner step runs beside the next
one: the same number of inner steps as the oracle in every outer step, some stopped early, on one, two and all
SMs, and the same state."""
import pytest

from gpu_common import scaled_close
from oracle.oracle import Oracle
from paper_2310_18916_gb300 import gsis
from paper_2310_18916_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

PROBLEMS = {
    "couette": (lambda: wl.couette(n_cells=37, nv=10), 1e-4),
    "cavity": (lambda: wl.cavity(n=17, ny=14, nv=10), 1e-5),
    "box": (lambda: wl.box3d(7, 6, 5, nv=10), 1e-5),
    "cavity_rykov": (lambda: wl.as_rykov(wl.cavity(n=11, ny=13, nv=10)), 1e-4),
}


@pytest.mark.parametrize("kind", sorted(PROBLEMS))
@pytest.mark.parametrize("sms", [1, 2, 0])
def test_early_exit_takes_the_same_inner_steps(kind, sms):
    make, tol = PROBLEMS[kind]
    p = make()
    kw = dict(macro_steps=300, macro_tol=tol)
    g = gsis.Solver(p, precision="f64", mode="gsis", kinetic_presteps=0, macro_sms=sms, **kw)
    o = Oracle(p, mode=0, **kw)
    taken = []
    for _ in range(4):
        g.step()
        o.step()
        taken.append(o.macro_iters)
        assert g.stats()[1] == o.macro_iters
    assert min(taken) < 300, taken
    scaled_close(g.W(), o.W(), 1e-10, f"{kind} on {sms or 'all'} SMs")
    g.close()
