"""The resident kernel of the tile schedule (calls of more than 32 steps): the same bits as one
launch per kernel and step, in every storage form, on lattices where a tile's halo wraps, clamps
or covers the whole lattice, on walls of every kind, open columns and batches."""
import dataclasses
import math

import numpy as np
import pytest

from paper_1707_00198_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _porous(nx, ny, seed):
    """Periodic box with random solid nodes (about a tenth)."""
    rng = np.random.default_rng(seed)
    g = I.periodic_box_droplet(nx, ny, R=0.3 * ny, noise=1e-3, seed=seed)
    solid = (rng.random((ny, nx)) < 0.1).astype(np.uint8)
    return dataclasses.replace(g, solid=solid)


def _theta_node(g, seed):
    rng = np.random.default_rng(seed)
    return dataclasses.replace(g, theta_node=rng.uniform(0.6, 2.4, (g.ny, g.nx)))


def _cases():
    P = I.Params
    finger = I.fingering_params(5.0, 0.1, 60.0)
    yield "tiny periodic", [I.periodic_box_droplet(5, 5, R=1.6, noise=1e-2, seed=1)], [P(sigma=0.02)]
    yield "one tile wide", [I.flat_wall_droplet(7, 40, R=3.0, noise=1e-2, seed=2)], [P(theta=1.0)]
    yield "odd closed", [I.flat_wall_droplet(61, 33, R=14.0, seed=3, closed_x=True)], [P(theta=1.9, nu_B=0.05)]
    yield "odd periodic", [I.periodic_box_droplet(97, 45, R=15.0, noise=1e-3, seed=4)], [P(sigma=0.02)]
    yield "porous", [_porous(67, 50, 5)], [P(theta=0.8)]
    yield "cylinder", [I.cylinder_droplet(60, 50, Rs=10.0, cx=30.0, cy=18.0, Rd=9.0, theta=1.9, noise=1e-3, seed=6)], \
        [P(theta=1.9, sigma=0.02)]
    yield "angle per node", [_theta_node(I.flat_wall_droplet(64, 30, R=12.0, seed=7), 8)], [P()]
    yield "channel", [I.displacement_channel(W=21, L=115, x_I=25.0, seed=9, noise=1e-3)], [finger]
    yield "Poiseuille channel", [I.displacement_channel(W=20, L=110, x_I=25.0, seed=10)], \
        [dataclasses.replace(finger, inlet_profile=1)]
    for w in (1, 2):
        yield f"wetting {w}", [I.flat_wall_droplet(50, 30, R=12.0, seed=11)], [P(theta=1.2, wetting=w)]
    yield "capillary", [I.capillary_filling(L=60, d=20, reservoir=31, wall=7, red_into=20, noise=1e-3, seed=12)], [P(theta=0.6)]
    yield "batch", [I.displacement_channel(W=20, L=110, x_I=25.0, seed=13), I.periodic_box_droplet(33, 40, R=9.0, seed=14),
                    I.flat_wall_droplet(48, 20, R=8.0, seed=15)], [finger, P(nu_B=0.05), P(theta=1.2)]


CASES = list(_cases())


def _handles(gs, ps, prec, n=2):
    from paper_1707_00198_gb300.lbcg import Lattice
    out = [Lattice(gs, ps, prec) for _ in range(n)]
    for L in out:
        L.set_tile(8)
    return out


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name,gs,ps", CASES, ids=[c[0] for c in CASES])
def test_resident_steps_equal_single_steps(name, gs, ps, prec):
    A, B = _handles(gs, ps, prec)
    for _ in range(70):
        A.step(1)
    B.step(70)
    assert B.step_launches == 1 and A.step_launches == 70 * A.launches_per_step
    B.step(1)      # from the other pool, then again
    B.step(41)
    for _ in range(42):
        A.step(1)
    for i in range(len(gs)):
        b = B.populations(i)
        assert np.isfinite(b).all()
        assert np.array_equal(A.populations(i), b), (name, prec, i)
    A.close()
    B.close()


@pytest.mark.parametrize("prec", ["fp16", "bf16"])
@pytest.mark.parametrize("name,gs,ps", CASES, ids=[c[0] for c in CASES])
def test_resident_16bit_steps_draw_the_keys_of_graph_replays(name, gs, ps, prec):
    # calls of 32 steps are graph replays of one launch per kernel and step; a call of 65 steps
    # draws the keys of two replays and a direct step, also when it starts with a direct step
    A, B = _handles(gs, ps, prec)
    for n in (32, 32, 1, 1, 32, 2):
        A.step(n)
    B.step(65)
    B.step(35)     # starts from the other pool: one direct step, a replay, two direct steps
    for i in range(len(gs)):
        assert np.array_equal(A.populations(i), B.populations(i)), (name, prec, i)
    A.close()
    B.close()


def test_long_call_and_configuration_sizes():
    # several launches of one call, and the tiles of the configurations' lattices
    (A, B) = _handles([I.flat_wall_droplet(20, 12, R=5.0, seed=1)], [I.Params(theta=math.radians(70))], "fp32")
    A.step(9001)
    for _ in range(300):
        B.step(30)
    B.step(1)
    assert A.step_launches == 2
    assert np.array_equal(A.populations(), B.populations())
    for g, p in (I.config_capillary(), I.config_fingering(M=5.0)):
        A, B = _handles([g], [p], "fp32")
        A.step(64)
        B.step(32)
        B.step(32)
        assert A.step_launches == 1
        assert np.array_equal(A.populations(), B.populations()), g.name
        A.close()
        B.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16"])
def test_handles_of_several_sizes_step_in_turn(prec):
    # the kernel's shared-memory limit is the process's: a handle with larger tiles still steps after
    # handles with smaller ones were created, and the other way round
    from paper_1707_00198_gb300.lbcg import Lattice
    sizes = [(600, 100), (40, 20), (300, 60)]
    gs = [I.displacement_channel(W=w, L=l, x_I=15.0, seed=l) for l, w in sizes]
    p = I.fingering_params(5.0, 0.1, 60.0)
    hs = [Lattice(g, p, prec) for g in gs]
    for L in hs:
        L.set_tile(8)
    for _ in range(2):
        for L in hs:
            L.step(40)
    hs[0].autotune(4)
    for g, L in zip(gs, hs):
        one = Lattice(g, p, prec)
        one.set_tile(8)
        one.step(40)
        one.step(40)
        assert np.array_equal(L.populations(), one.populations()), (g.name, prec)
        one.close()
        L.close()


def test_handles_on_their_own_streams_run_at_once():
    # four handles, each with a stream of its own, stepped from four threads: cooperative launches of
    # one process beside each other give the bits of one after another
    import threading
    from paper_1707_00198_gb300.lbcg import Lattice
    cases = [("fp32", I.config_fingering(M=5.0)), ("fp32", I.config_static_droplet()),
             ("fp64", I.config_static_droplet()), ("fp16", I.config_capillary())]
    one = []
    for prec, (g, p) in cases:
        L = Lattice(g, p, prec)
        for _ in range(4):
            L.step(100)
        one.append(L.populations())
        L.close()
    hs = [Lattice(g, p, prec) for prec, (g, p) in cases]

    def work(L):
        for _ in range(4):
            L.step(100)

    ts = [threading.Thread(target=work, args=(L,)) for L in hs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for L, want, (prec, (g, _)) in zip(hs, one, cases):
        assert np.array_equal(L.populations(), want), (prec, g.name)
        L.close()


def test_allocator_that_refuses_one_block():
    # every allocation of a handle refused in turn: an error, and nothing kept, or for the two of the
    # resident kernel's plan (an extra) a handle that steps one launch per kernel and step
    import torch
    from paper_1707_00198_gb300 import lbcg
    g, p = I.config_static_droplet()
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
        L = lbcg.Lattice(g, p, "fp32")
        total = calls[0]
        L.step(40)
        assert L.step_launches == 1
        want = L.populations()
        L.close()
        launched = 0
        for k in range(total):
            calls[:] = [0, k]
            try:
                L = lbcg.Lattice(g, p, "fp32")
            except lbcg.LBCGError as e:
                assert e.status == 8 and not held
                continue
            launched += 1
            L.step(40)
            assert L.step_launches > 40
            assert np.array_equal(L.populations(), want)
            L.close()
        assert launched == 2
    finally:
        lbcg.lbcg_set_allocator()
    assert not held


@pytest.mark.parametrize("schedule", ["tiles", "sweep"])
def test_gradient_along_the_walls_normal_at_90_degrees(schedule):
    # Eq. 36 picks between two normals along the wall; a gradient along the wall's own normal (one
    # mixed node in pure fluid beside the wall) leaves them equally near but for rounding, so that every
    # operation of the chain before has to be the oracle's
    from oracle import lbcg_oracle as O
    from paper_1707_00198_gb300.lbcg import Lattice
    rng = np.random.default_rng(3)
    g = I.flat_wall_droplet(120, 90, R=20.0, closed_x=True)
    rho_n = np.full((90, 120), -1.0)
    for k in range(4, 86, 6):
        rho_n[k, 1] = rho_n[k, 118] = -1.0 + 1e-3 * rng.random()
    for k in range(6, 114, 6):
        rho_n[1, k] = rho_n[88, k] = -1.0 + 1e-3 * rng.random()
    g = dataclasses.replace(g, rhoN0=rho_n)
    p = I.Params(theta=math.pi / 2)
    L = Lattice(g, p, "fp64")
    L.set_tile(8) if schedule == "tiles" else L.set_sweep()
    L.step(1)
    lat = O.make_lattice(g, p.theta)
    fR, fB = O.run(lat, p, *O.init_state(lat, g.rhoN0, p.rho0, p), 1)
    # (a pick the other way round moves populations by 1e-5 and more; rounding by 1e-15)
    assert float(np.abs(L.populations() - np.stack([fR.numpy(), fB.numpy()])).max()) <= 1e-12
    L.close()
