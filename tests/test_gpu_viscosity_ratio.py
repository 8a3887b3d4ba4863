"""FP64 tiles: the local viscosity (Eq. 18) of one fluid does not hang on the other's."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import lbcg_oracle as O
from paper_1707_00198_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("schedule", ["resident", "launched"])
@pytest.mark.parametrize("fluid", ["red", "blue"])
def test_pure_fluid_with_a_thin_other_one(fluid, schedule):
    # one fluid of viscosity 0.17 alone in a box, the absent one thinner by 10^11: 1/nu of the absent one
    # has an ulp of 10^-4.  After 10 steps from populations off equilibrium by 10^-2 the form of the equation is
    # within rounding (10 steps of about a hundred operations on values below 1: 10 * 100 * 1.1e-16)
    from paper_1707_00198_gb300.lbcg import Lattice
    g = I.periodic_box_droplet(21, 18, R=5.0)
    sign = 1.0 if fluid == "red" else -1.0
    g = dataclasses.replace(g, rhoN0=np.full((g.ny, g.nx), sign))
    thin = 0.17e-11
    p = I.Params(nu_R=0.17, nu_B=thin) if fluid == "red" else I.Params(nu_R=thin, nu_B=0.17)
    lat = O.make_lattice(g, p.theta)
    s0 = np.stack([f.numpy() for f in O.init_state(lat, g.rhoN0, p.rho0, p)])
    k = 0 if fluid == "red" else 1
    s0[k] += 1e-2 * np.random.default_rng(1).standard_normal(s0[k].shape) * s0[k]
    L = Lattice(g, p, "fp64")
    L.set_tile(4)
    L.set_populations(s0)
    if schedule == "launched":
        for _ in range(10):
            L.step(1)
    else:
        L.step(10)
    want = np.stack([f.numpy() for f in O.run(lat, p, torch.from_numpy(s0[0].copy()), torch.from_numpy(s0[1].copy()), 10)])
    assert float(np.abs(L.populations() - want).max()) <= 1.1e-13
    L.close()
