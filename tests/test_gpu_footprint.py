"""gsis_footprint_bytes is what a solver allocates, byte for byte: every storage, gas, mode, kind of mesh and
velocity grid."""
import numpy as np
import pytest

from paper_2310_18916_gb300 import gsis
from paper_2310_18916_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

PROBLEMS = {
    "couette": lambda: wl.couette(n_cells=37, nv=24),
    "cavity": lambda: wl.cavity(n=33, ny=20, nv=12),
    "box": lambda: wl.box3d(9, 8, 7, nv=11),
    "cylinder": lambda: wl.cylinder(n_r=8, n_theta=16, nv=12, R=0.5, R_out=3.0, Ma=0.5, Kn=0.2),
    "hybrid": lambda: wl.unstructured_cavity(n=6, nv=12, Kn=0.2, hybrid=0.5),
}


@pytest.mark.parametrize("kind", sorted(PROBLEMS))
@pytest.mark.parametrize("precision", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("mode,rykov", [("gsis", False), ("dvm", False), ("gsis", True)])
def test_footprint_is_what_is_allocated(kind, precision, mode, rykov):
    import torch

    p = PROBLEMS[kind]()
    if rykov:
        p = wl.as_rykov(p)
    want = gsis.footprint_bytes(p, precision, mode=gsis.MODE_GSIS if mode == "gsis" else gsis.MODE_DVM)
    key = "requested_bytes.all.current"
    torch.zeros(1, device="cuda")
    before = torch.cuda.memory_stats()[key]
    g = gsis.Solver(p, precision=precision, mode=mode, kinetic_presteps=0)
    held = torch.cuda.memory_stats()[key] - before
    assert held == want
    g.step()
    assert np.isfinite(g.W()).all()
    g.close()
    assert torch.cuda.memory_stats()[key] == before
