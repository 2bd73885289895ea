"""The general meshes' kinetic kernel in the forms that the number of passes, the storage, the face values and
the orientation of the mesh select, against the oracle: one, two and three passes (first, middle and last are
compiled apart), BF16 storage and positive face values with two velocities per lane (29^3: 765 velocity blocks,
an odd number in some octants) and with one, and meshes turned so that many velocities run along faces, where
every phase has to take the same decision on the side they leave.

BF16 storage is held to the bounds of the other BF16 tests on general meshes: 2e-3 of their scale for the state
and the wall fluxes of a kinetic step."""
import numpy as np
import pytest

from gpu_common import scaled_close
from oracle.oracle import Oracle
from paper_2310_18916_gb300 import gsis
from paper_2310_18916_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _problem(kind, nv):
    if kind.startswith("cylinder"):
        p = wl.cylinder(n_r=4, n_theta=8, nv=nv, R=0.5, R_out=2.0, Ma=0.5, Kn=0.2)
    elif kind.startswith("sphere"):
        p = wl.sphere(n_r=4, n_pol=3, n_az=4, nv=nv, R=0.5, R_out=2.0, Ma=0.5, Kn=0.2)
    else:
        p = wl.unstructured_cavity(n=4, nv=nv, Kn=0.2)
        if kind == "turned":
            # by the angle of the velocities (3, 1), (9, 3), ...: they run along the faces up to rounding
            c, s = 3.0 / np.sqrt(10.0), 1.0 / np.sqrt(10.0)
            p.unodes = np.ascontiguousarray(p.unodes @ np.array([[c, s, 0.0], [-s, c, 0.0], [0.0, 0.0, 1.0]]))
    return wl.as_rykov(p) if kind.endswith("rykov") else p


@pytest.mark.parametrize("kind,precision,nv,sweeps,positive", [
    ("cylinder", "f32", 29, 1, 0), ("cylinder", "f32", 29, 3, 0), ("sphere", "f32", 29, 1, 0), ("sphere", "f32", 29, 3, 0),
    ("hybrid", "f32", 29, 1, 0), ("hybrid", "f32", 29, 3, 0), ("cylinder", "f32", 12, 1, 0), ("cylinder", "f32", 12, 3, 0),
    ("cylinder", "f32", 29, 2, 1), ("sphere", "f32", 12, 2, 1), ("hybrid", "f64", 12, 2, 1),
    ("cylinder_rykov", "f32", 12, 1, 0), ("sphere_rykov", "f32", 12, 3, 0),
    ("turned", "f32", 29, 2, 0), ("turned", "f32", 12, 2, 0), ("turned", "f64", 12, 2, 0),
])
def test_forms_against_the_oracle(kind, precision, nv, sweeps, positive):
    p = _problem(kind, nv)
    W0 = wl.perturbed_state(p, seed=13, amp=0.02)
    rel = {"f64": 1e-11, "f32": 2e-5}[precision]
    kw = dict(n_sweeps=sweeps, positive_faces=positive)
    g = gsis.Solver(p, precision=precision, mode="dvm", kinetic_presteps=0, init_W=W0, **kw)
    o = Oracle(p, W0=W0, mode=1, **kw)
    g.step()
    o.step()
    rykov = p.model == wl.RYKOV
    for q, (fg, fo) in enumerate(zip(g.get_f(both=True) if rykov else (g.get_f(),), o.get_f())):
        scale = np.maximum(np.abs(fo).max(axis=0), 1e-3 * np.abs(fo).max())
        err = (np.abs(fg - fo) / scale).max()
        assert err < rel, f"f{q} differs by {err:.3e} of its scale"
    wg, wo = g.wall(), o.wall()
    assert np.array_equal(wg[0], wo[0]) and np.array_equal(wg[1], wo[1])
    scaled_close(wg[3], wo[3], 10 * rel, "wall fluxes", vector=True)
    g.close()
    kw.update(macro_steps=5, macro_tol=0.0)
    g = gsis.Solver(p, precision=precision, mode="gsis", kinetic_presteps=0, init_W=W0, **kw)
    o = Oracle(p, W0=W0, mode=0, **kw)
    g.step()
    o.step()
    scaled_close(g.W(), o.W(), 10 * rel, "W after one GSIS step")
    g.close()


@pytest.mark.parametrize("kind,nv,sweeps", [("cylinder", 29, 2), ("sphere", 29, 1), ("hybrid", 29, 3), ("sphere", 12, 3),
                                             ("sphere_rykov", 20, 2)])
def test_bf16_forms_against_the_oracle(kind, nv, sweeps):
    p = _problem(kind, nv)
    W0 = wl.perturbed_state(p, seed=13, amp=0.02)
    g = gsis.Solver(p, precision="bf16", mode="dvm", kinetic_presteps=0, init_W=W0, n_sweeps=sweeps)
    o = Oracle(p, W0=W0, mode=1, n_sweeps=sweeps)
    for _ in range(2):
        g.step()
        o.step()
    Wg, Wo = g.W(), o.W()
    scaled_close(Wg[:, [0, 4, 5]], Wo[:, [0, 4, 5]], 2e-3, "rho, T after two kinetic steps")
    scaled_close(Wg[:, 1:4], Wo[:, 1:4], 2e-3, "u after two kinetic steps", vector=True)
    scaled_close(g.wall()[3], o.wall()[3], 2e-3, "wall fluxes", vector=True)
    g.close()
