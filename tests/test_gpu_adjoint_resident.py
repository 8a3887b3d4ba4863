"""The resident reverse sweep (one cooperative launch per checkpoint segment) against the launched
stages on the same handle: curved walls, open columns with walls at their corners, periodic
wraps, lattices one tile wide, segments of one step."""
import dataclasses

import numpy as np
import pytest

from paper_1707_00198_gb300 import inputs as I

pytestmark = pytest.mark.gpu

FINGER = I.fingering_params(5.0, 0.1, 60.0)
CASES = [
    ("channel", I.displacement_channel(W=13, L=61, x_I=25.0, seed=1), FINGER),
    ("Poiseuille", I.displacement_channel(W=8, L=40, x_I=12.0, seed=2), dataclasses.replace(FINGER, inlet_profile=1)),
    ("cylinder", I.cylinder_droplet(40, 35, Rs=7.0, cx=20.0, cy=12.0, Rd=7.0, theta=1.2, noise=1e-2, seed=3,
                                    analytic_normal=False), I.Params(theta=1.2, sigma=0.02)),
    ("capillary", I.capillary_filling(L=20, d=8, reservoir=13, wall=5, red_into=6, noise=1e-2, seed=4), I.Params(theta=0.7)),
    ("narrow", I.flat_wall_droplet(6, 30, R=3.0, noise=1e-2, seed=5), I.Params(theta=1.0)),
]


@pytest.mark.parametrize("ckpt", [1, 7])
@pytest.mark.parametrize("name,g,p", CASES, ids=[c[0] for c in CASES])
def test_resident_reverse_equals_the_launched_stages(name, g, p, ckpt):
    # FP64: the sums of the two differ in order only; a changed poll limit keeps a handle on the
    # launched stages
    from paper_1707_00198_gb300.lbcg import Lattice
    rng = np.random.default_rng(7)
    w = rng.standard_normal((g.ny, g.nx)) * (g.solid == 0)
    out = []
    for launched in (False, True):
        L = Lattice(g, p, "fp64")
        L.set_tile(4)
        if launched:
            L.set_poll_limit(1 << 21)
        out.append(L.adjoint(21, ckpt, w))
        pops = L.populations()
        out[-1]["populations"] = pops
        L.close()
    a, b = out
    assert np.array_equal(a["populations"], b["populations"])
    scale = max(1e-12, float(np.abs(b["dtheta_node"]).max()))
    assert float(np.abs(a["dtheta_node"] - b["dtheta_node"]).max()) <= 1e-11 * scale
    for k in ("J", "dsigma", "dnu_R", "dnu_B", "dtheta"):
        assert abs(a[k] - b[k]) <= 1e-10 * max(abs(b[k]), scale), (k, a[k], b[k])
