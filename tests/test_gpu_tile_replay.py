"""The step graph of the tile schedule (lattices that the cooperative kernel does not take, and handles
with a changed poll limit): replays give the bits of direct steps, and in 16-bit storage, whose rounding
keys count replays, those of the cooperative kernel."""
import math

import numpy as np
import pytest

from paper_1707_00198_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("ty", [4, 8, 16])
@pytest.mark.parametrize("batch", [False, True], ids=["one", "batch"])
def test_replays_of_the_tile_graph(prec, ty, batch):
    from paper_1707_00198_gb300.lbcg import Lattice
    g1 = I.displacement_channel(W=20, L=110, x_I=25.0, seed=6, noise=1e-3)
    p1 = I.fingering_params(M=5.0, Ca=0.1, theta_deg=60.0)
    g2 = I.cylinder_droplet(60, 50, Rs=10.0, cx=30.0, cy=18.0, Rd=9.0, theta=math.radians(110), noise=1e-3,
                            seed=13, analytic_normal=False)
    p2 = I.Params(theta=math.radians(110), sigma=0.02)
    gs, ps = ([g1, g2, g1, g2], [p1, p2, p1, p2]) if batch else ([g1], [p1])
    A, B = Lattice(gs, ps, prec), Lattice(gs, ps, prec)
    for L in (A, B):
        L.set_tile(ty)
    B.set_poll_limit(1 << 21)       # off the cooperative kernel
    B.step(100)
    # three replays of 32 steps (a batch's graph: three branches of two kernels a step; 16-bit
    # storage: one kernel a replay that counts it) and four direct steps
    sr = 3 if prec in ("fp16", "bf16") else 0
    assert B.step_launches == 96 * 2 * (3 if batch else 1) + 4 * 2 + sr
    if sr:
        A.step(100)
        assert A.step_launches == 2
    else:
        for _ in range(100):
            A.step(1)
    for i in range(len(gs)):
        b = B.populations(i)
        assert np.isfinite(b).all()
        assert np.array_equal(A.populations(i), b), i
    A.close()
    B.close()
