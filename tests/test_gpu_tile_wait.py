"""The bounded wait of the cooperative kernels (k_run, k_reverse) of a tile for the tiles around it,
without any GPU fault: with a bound of 0 every wait gives up at once, the blocks return, the next
synchronising call reports LBCG_E_TIMEOUT, and with the default bound back a state set afresh steps
to the same bits as on a new handle."""
import numpy as np
import pytest

from paper_1707_00198_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LBCG_E_TIMEOUT = 6
G = I.displacement_channel(W=20, L=110, x_I=25.0, seed=6, noise=1e-3)
P = I.fingering_params(M=5.0, Ca=0.1, theta_deg=60.0)


def _lattice(prec):
    from paper_1707_00198_gb300.lbcg import Lattice
    L = Lattice(G, P, prec)
    L.set_tile(4)
    return L


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16"])
def test_step_reports_a_wait_that_ran_out_and_recovers(prec):
    from paper_1707_00198_gb300.lbcg import LBCGError
    A, L = _lattice(prec), _lattice(prec)
    s0 = A.populations()
    for n in (8, 100, 8192 + 50):     # (the last: two launches)
        L.set_tile_poll_limit(0)
        L.step(n)
        with pytest.raises(LBCGError) as ei:
            L.populations()
        assert ei.value.status == LBCG_E_TIMEOUT, str(ei.value)
        L.populations()               # reported once: the word is cleared
        # the flags of the tiles that gave up lag behind: the next calls count on from the launches
        L.set_tile_poll_limit(-1)
        L.set_populations(s0)
        L.step(70)
        L.step(9)
        got = L.populations()
        assert np.isfinite(got).all()
        if prec != "fp16":            # (16-bit storage draws other rounding keys by now)
            A.set_populations(s0)
            A.step(70)
            A.step(9)
            assert np.array_equal(got, A.populations())
    A.close()
    L.close()


@pytest.mark.parametrize("fp32_reverse", [False, True])
@pytest.mark.parametrize("ckpt", [1, 7, 50])
def test_adjoint_reports_a_wait_that_ran_out_and_recovers(ckpt, fp32_reverse):
    # checkpoints every step: only the reverse sweep waits (one step is launched, and nothing is
    # recomputed); every 7: the recompute does too; every 50: and the forward steps
    from paper_1707_00198_gb300.lbcg import LBCGError
    prec = "fp32" if fp32_reverse else "fp64"
    A, L = _lattice(prec), _lattice(prec)
    s0 = A.populations()
    w = np.random.default_rng(7).standard_normal((G.ny, G.nx)) * (G.solid == 0)
    want = A.adjoint(60, ckpt, w, reverse_fp32=fp32_reverse)
    L.set_tile_poll_limit(0)
    with pytest.raises(LBCGError) as ei:
        L.adjoint(60, ckpt, w, reverse_fp32=fp32_reverse)
    assert ei.value.status == LBCG_E_TIMEOUT, str(ei.value)
    L.set_tile_poll_limit(-1)
    L.set_populations(s0)
    got = L.adjoint(60, ckpt, w, reverse_fp32=fp32_reverse)
    for k in want:                    # (no atomics in the resident sweep: the same bits)
        assert np.array_equal(got[k], want[k]), k
    A.close()
    L.close()


def test_autotune_leaves_out_a_kernel_that_steps_do_not_take():
    # a changed lbcg_set_poll_limit keeps steps off the cooperative kernel: it is no candidate then (its
    # waits, which would give up at once, are not reached)
    from paper_1707_00198_gb300.lbcg import LBCGError
    L = _lattice("fp32")
    L.set_tile_poll_limit(0)
    L.set_poll_limit(1 << 21)
    s0 = L.populations()
    L.autotune(4)
    assert np.array_equal(L.populations(), s0)
    L.set_poll_limit(-1)
    L.autotune(4)               # as a candidate it does
    with pytest.raises(LBCGError) as ei:
        L.populations()
    assert ei.value.status == LBCG_E_TIMEOUT
    L.close()
