"""lbcg_adjoint where device memory is refused."""
import numpy as np
import pytest

from paper_1707_00198_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_adjoint_with_one_block_refused():
    # every allocation of a call refused in turn: LBCG_E_NOMEM and nothing kept, or for the progress
    # words of the two cooperative kernels (an extra) the gradient by the launched stages, whose sums
    # differ in order only
    import torch
    from paper_1707_00198_gb300 import lbcg
    g = I.displacement_channel(W=13, L=61, x_I=25.0, seed=1)
    p = I.fingering_params(5.0, 0.1, 60.0)
    w = np.random.default_rng(7).standard_normal((g.ny, g.nx)) * (g.solid == 0)
    held, calls = {}, [0, -1]

    def alloc(nbytes, stream):
        calls[0] += 1
        if calls[0] - 1 == calls[1]:
            return 0
        t = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
        q = (t.data_ptr() + 255) & ~255
        held[q] = t
        return q

    def release(q, stream):
        torch.cuda.synchronize()
        held.pop(q)

    lbcg.lbcg_set_allocator(alloc, release)
    try:
        L = lbcg.Lattice(g, p, "fp64")
        L.set_tile(4)
        s0 = L.populations()
        L.fields()                      # (the fields' buffer is the handle's)
        kept = len(held)
        calls[0] = 0
        want = L.adjoint(21, 7, w)
        total = calls[0]
        refused = given = 0
        for k in range(total):
            L.set_populations(s0)
            calls[:] = [0, k]
            try:
                got = L.adjoint(21, 7, w)
            except lbcg.LBCGError as e:
                assert e.status == 8
                refused += 1
            else:
                given += 1
                scale = float(np.abs(want["dtheta_node"]).max())
                assert float(np.abs(got["dtheta_node"] - want["dtheta_node"]).max()) <= 1e-11 * scale
                for key in ("J", "dsigma", "dnu_R", "dnu_B", "dtheta"):
                    assert abs(got[key] - want[key]) <= 1e-10 * max(abs(want[key]), scale), key
            calls[1] = -1
            assert len(held) == kept
        assert given == 2 and refused == total - 2
        L.close()
    finally:
        lbcg.lbcg_set_allocator()
    assert not held


def test_refused_memory_is_not_the_next_launch_s_error():
    # 10^10 states of checkpoint segments: cudaMalloc refuses them, the call reports it, and the handle
    # and others step on
    from paper_1707_00198_gb300 import lbcg
    g, p = I.config_static_droplet()
    L, other = lbcg.Lattice(g, p, "fp32"), lbcg.Lattice(g, p, "fp32")
    w = np.ones((g.ny, g.nx))
    for schedule in (lambda: L.set_tile(8), lambda: L.set_sweep()):
        schedule()
        with pytest.raises(lbcg.LBCGError) as ei:
            L.adjoint(2, 10 ** 10, w)
        assert ei.value.status == 8
        L.step(1)
        L.step(8)
        with pytest.raises(lbcg.LBCGError):
            L.adjoint(2, 10 ** 10, w)
        other.step(1)
        assert np.isfinite(L.populations()).all() and np.isfinite(other.populations()).all()
    L.close()
    other.close()
