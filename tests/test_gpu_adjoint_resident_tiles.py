"""The resident reverse sweep against the launched stages where a tile's nodes fill several warps (its
halves synchronise by barriers of their own), in every pair of arithmetics, on both sides of the
largest tile it takes; and that it is the one that runs."""
import dataclasses

import numpy as np
import pytest

from paper_1707_00198_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LBCG_E_TIMEOUT = 6
FINGER = I.fingering_params(5.0, 0.1, 60.0)
POISEUILLE = dataclasses.replace(FINGER, inlet_profile=1)
# lattice, parameters, and the nodes of the largest tile in FP64 and in FP32 on 152 SMs; the kernel
# takes 128 at most
CASES = {
    "400x42": (*I.config_adjoint(), 112, 56),
    "Poiseuille 389x43": (I.displacement_channel(W=41, L=389, x_I=25.0, seed=1), POISEUILLE, 128, 64),
    "Poiseuille 397x45": (I.displacement_channel(W=43, L=397, x_I=25.0, seed=1), POISEUILLE, 132, 63),
    "curved wall": (I.cylinder_droplet(131, 111, Rs=20.0, cx=66.0, cy=41.0, Rd=19.0, theta=1.2, noise=1e-2, seed=3,
                                       analytic_normal=False), I.Params(theta=1.2, sigma=0.02), 98, 48),
    "620x62": (I.displacement_channel(W=60, L=620, x_I=25.0, seed=2), FINGER, 264, 135),
}
NSTEPS = 21


def _gradient(g, p, prec, fp32_reverse, ckpt, launched):
    from paper_1707_00198_gb300.lbcg import Lattice
    w = np.random.default_rng(7).standard_normal((g.ny, g.nx)) * (g.solid == 0)
    L = Lattice(g, p, prec)
    L.set_tile(4)
    if launched:
        L.set_poll_limit(1 << 21)      # keeps a handle on the launched stages
    out = L.adjoint(NSTEPS, ckpt, w, reverse_fp32=fp32_reverse)
    out["populations"] = L.populations()
    L.close()
    return out


def _runs_resident(g, p, prec, fp32_reverse, launched):
    # with a checkpoint at every step nothing but the reverse sweep waits for other tiles: with no
    # polls allowed it gives up
    from paper_1707_00198_gb300.lbcg import Lattice, LBCGError
    L = Lattice(g, p, prec)
    L.set_tile(4)
    L.set_tile_poll_limit(0)
    if launched:
        L.set_poll_limit(1 << 21)
    try:
        L.adjoint(2, 1, np.ones((g.ny, g.nx)), reverse_fp32=fp32_reverse)
        return False
    except LBCGError as e:
        assert e.status == LBCG_E_TIMEOUT
        return True
    finally:
        L.close()


@pytest.mark.parametrize("prec,fp32_reverse", [("fp64", False), ("fp32", False), ("fp32", True)])
@pytest.mark.parametrize("name", CASES)
def test_resident_reverse_equals_the_launched_stages(name, prec, fp32_reverse):
    g, p, nodes64, nodes32 = CASES[name]
    assert _runs_resident(g, p, prec, fp32_reverse, False) == ((nodes64 if prec == "fp64" else nodes32) <= 128)
    assert not _runs_resident(g, p, prec, fp32_reverse, True)
    a = _gradient(g, p, prec, fp32_reverse, 8, False)
    b = _gradient(g, p, prec, fp32_reverse, 8, True)
    assert np.array_equal(a["populations"], b["populations"])
    assert a["J"] == b["J"]
    scale = float(np.abs(b["dtheta_node"]).max())
    err = float(np.abs(a["dtheta_node"] - b["dtheta_node"]).max())
    keys = ("dsigma", "dnu_R", "dnu_B", "dtheta")
    if not fp32_reverse:
        # sums in another order: 64 rounded operations a step on a node's path, in FP32 states times
        # the 1 / |grad rho^N| <= 10^5 that n's reverse multiplies with
        tol = NSTEPS * 64 * 2.0 ** -53 * (1e5 if prec == "fp32" else 1e2)
        assert err <= tol * scale
        for k in keys:
            assert abs(a[k] - b[k]) <= 10 * tol * max(abs(b[k]), scale), k
    else:
        # as far from the FP64 reverse of the same states as the launched stages, but for the sums' order
        ref = _gradient(g, p, prec, False, 8, True)
        tol = NSTEPS * 64 * 2.0 ** -24
        off = float(np.abs(b["dtheta_node"] - ref["dtheta_node"]).max())
        assert float(np.abs(a["dtheta_node"] - ref["dtheta_node"]).max()) <= 2 * off + tol * scale
        for k in keys:
            assert abs(a[k] - ref[k]) <= 2 * abs(b[k] - ref[k]) + 10 * tol * max(abs(ref[k]), scale), k
