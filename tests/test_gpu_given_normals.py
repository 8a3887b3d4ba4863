"""Given solid normals that are not of unit length enter Eq. 34-36 as they are, in FP64 as in the oracle:
the corrected gradient carries their length, n = g_c / |g_c| does not."""
import dataclasses
import math

import numpy as np
import pytest
import torch

from oracle import lbcg_oracle as O
from paper_1707_00198_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _scaled(g, how):
    rng = np.random.default_rng(5)
    if how == "unit":
        return g
    if how == "rounded":     # as read from a file with seven digits
        return dataclasses.replace(g, normal=np.round(g.normal, 7))
    f = {"short": 0.5, "long": 3.0}.get(how, None)
    return dataclasses.replace(g, normal=g.normal * (f if f else rng.uniform(0.2, 5.0, (g.ny, g.nx))))


@pytest.mark.parametrize("schedule", ["resident", "launched", "sweep"])
@pytest.mark.parametrize("how", ["unit", "rounded", "short", "long", "mixed"])
def test_fp64_steps_follow_the_oracle(how, schedule):
    from paper_1707_00198_gb300.lbcg import Lattice
    th = math.radians(70)
    g = _scaled(I.cylinder_droplet(60, 50, Rs=10.0, cx=30.0, cy=18.0, Rd=9.0, theta=th, noise=1e-3, seed=6), how)
    assert g.normal is not None
    p = I.Params(theta=th, sigma=0.02)
    lat = O.make_lattice(g, p.theta)
    s0 = O.init_state(lat, g.rhoN0, p.rho0, p)
    want = np.stack([f.numpy() for f in O.run(lat, p, *s0, 20)])
    L = Lattice(g, p, "fp64")
    L.set_sweep() if schedule == "sweep" else L.set_tile(8)
    if schedule == "resident":
        L.step(20)
    else:
        for _ in range(20):
            L.step(1)
    # (1e-10 after 100 steps is the framework's bound for FP64)
    assert float(np.abs(L.populations() - want).max()) <= 2e-11
    L.close()
