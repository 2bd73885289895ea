"""Moments of the two-VDF gas in FP64 at high speed: the heat fluxes of a flow at |u| = 40 thermal speeds
against quadruple or extended precision sums over the solver's own f.

Tolerance: the state velocity and the mean velocity are rounded at |u|, 40 x 1.1e-16 = 4.4e-15 each, and the
heat flux changes by (5/2) rho T per unit of it: 2.2e-14 for the two; sums about that velocity add at most 40
roundings (32 plain terms, then compensated) of sum w f |c|^3 ~ 2: 1e-14.  2e-13 leaves a factor of six.
Sums about the origin shifted afterwards cancel terms of |u|^3 = 64000: 7e-12 per rounding."""
import numpy as np
import pytest

from paper_2310_18916_gb300 import gsis
from paper_2310_18916_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _exact(p, f0, f1):
    vx, vy, vz = np.meshgrid(p.vx, p.vy, p.vz, indexing="ij")
    w = (np.asarray(p.wx)[:, None, None] * np.asarray(p.wy)[None, :, None] * np.asarray(p.wz)).astype(np.longdouble)
    # canonical velocity order: x fastest
    xi = np.stack([a.transpose(2, 1, 0).reshape(-1) for a in (vx, vy, vz)], -1).astype(np.longdouble)
    w = w.transpose(2, 1, 0).reshape(-1)
    a, b = f0.astype(np.longdouble) * w, f1.astype(np.longdouble) * w
    rho = a.sum(1)
    u = (a[:, :, None] * xi).sum(1) / rho[:, None]
    c = xi[None] - u[:, None]
    q = 0.5 * (a[:, :, None] * (c * c).sum(-1)[:, :, None] * c).sum(1)
    qr = (b[:, :, None] * c).sum(1)
    return rho, u, q, qr


@pytest.mark.parametrize("kind", ["couette", "cylinder"])
@pytest.mark.parametrize("nv", [12, 9])  # tiled and untiled velocity grids
def test_heat_fluxes_at_high_speed(kind, nv):
    U = 40.0
    if kind == "couette":
        p = wl.as_rykov(wl.couette(n_cells=5, nv=nv))
    else:
        p = wl.as_rykov(wl.cylinder(n_r=4, n_theta=6, nv=nv, R=0.5, R_out=2.0, Ma=0.3, Kn=0.2))
    # along z, to which every face of both meshes is parallel
    (p.vx, p.wx), (p.vy, p.wy), (p.vz, p.wz) = (wl.midpoint_grid(nv, -4.0, 4.0), wl.midpoint_grid(nv, -4.0, 4.0),
                                                wl.midpoint_grid(nv, U - 4.0, U + 4.0))
    p.wall_u = np.array(p.wall_u, dtype=float)
    p.wall_u[:, 2] += U
    W0 = wl.perturbed_state(p, seed=3, amp=0.02)
    W0[:, 3] += U
    g = gsis.Solver(p, precision="f64", mode="dvm", kinetic_presteps=0, init_W=W0, **({"n_sweeps": 2} if kind == "cylinder" else {}))
    g.step()
    f0, f1 = g.get_f(both=True)
    H = g.half_moments()
    g.close()
    rho, u, q, qr = _exact(p, f0, f1)
    assert float(np.abs(q).max()) > 1e-3 and float(np.abs(qr).max()) > 1e-4
    assert float((np.abs(H[:, 0] - rho) / rho).max()) < 1e-14
    for got, want, name in ((H[:, 12:15], q, "q"), (H[:, 15:18], qr, "q_r")):
        err = float((np.abs(got - want) / rho[:, None]).max())
        assert err < 2e-13, f"{kind} {nv}^3: {name} off by {err:.2e}"
