"""The observable sums at sizes where their reduction changes path: warps and blocks without a
node, warps without an interface point, one to three nodes per thread, long rows of partials."""
import math

import numpy as np
import pytest
import torch

from paper_1707_00198_gb300 import inputs as I

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


def _terms(f, mask):
    """Per quantity the terms that it sums, and the size that bounds the error of one."""
    rR, rB, ux, uy = f
    ny, nx = rR.shape
    fluid, fit = (mask & 1) == 0, (mask & 9) == 0
    rn, rho = (rR - rB) / (rR + rB), rR + rB
    red, blue = fluid & (rn > 0.9), fluid & (rn < -0.9)
    xs, ys = [], []
    y, x = np.nonzero(fit[:, :-1] & fit[:, 1:] & ((rn[:, :-1] >= 0) != (rn[:, 1:] >= 0)))
    xs.append(x + rn[y, x] / (rn[y, x] - rn[y, x + 1]) - 0.5 * nx)
    ys.append(y - 0.5 * ny)
    y, x = np.nonzero(fit[:-1] & fit[1:] & ((rn[:-1] >= 0) != (rn[1:] >= 0)))
    xs.append(x - 0.5 * nx)
    ys.append(y + rn[y, x] / (rn[y, x] - rn[y + 1, x]) - 0.5 * ny)
    px, py = np.concatenate(xs), np.concatenate(ys)
    z, s = px * px + py * py, float(nx + ny)
    pts = [(np.ones_like(px), 0.0), (px, s), (py, s), (px * px, s**2), (py * py, s**2), (px * py, s**2),
           (z * px, s**3), (z * py, s**3), (z, s**2)]
    one = lambda m: np.ones(int(m.sum()))
    return [(rR[fluid], 0.0), (rB[fluid], 0.0), None, *pts, (rho[red] / 3, 0.0), (one(red), 0.0), (rho[blue] / 3, 0.0),
            (one(blue), 0.0)], math.sqrt((ux[fluid]**2 + uy[fluid]**2).max(initial=0.0))


@pytest.mark.parametrize("nx,ny", [(1, 1), (31, 1), (1, 33), (32, 8), (257, 3), (609, 130), (500, 401)])
@pytest.mark.parametrize("interface", ["none", "everywhere", "one line"])
def test_sums_match_a_node_by_node_evaluation(nx, ny, interface):
    from paper_1707_00198_gb300 import lbcg
    rng = np.random.default_rng(nx + 7 * ny)
    rn = {"none": 0.2 + 0.79 * rng.random((ny, nx)), "everywhere": rng.uniform(-1, 1, (ny, nx)),
          "one line": np.where(np.arange(nx)[None, :] < nx // 2, 0.95, -0.95) + 0.01 * rng.random((ny, nx))}[interface]
    rho = rng.uniform(0.9, 1.1, (ny, nx))
    f = np.stack([rho * (1 + rn) / 2, rho * (1 - rn) / 2, *rng.uniform(-0.1, 0.1, (2, ny, nx))])
    mask = np.where(rng.random((ny, nx)) < 0.05, 1, np.where(rng.random((ny, nx)) < 0.1, 8, 0)).astype(np.uint8)
    dev, dmask = torch.tensor(f, device="cuda").contiguous(), torch.tensor(mask, device="cuda").contiguous()
    out = torch.full((17,), -7.0, dtype=torch.float64, device="cuda")
    lbcg.lbcg_field_moments_noalloc(dev.data_ptr(), dmask.data_ptr(), nx, ny, torch.cuda.current_stream().cuda_stream,
                                    out.data_ptr())
    got = out.cpu().numpy()
    terms, umax = _terms(f, mask)
    assert abs(got[2] - umax) <= 2 * EPS * umax and got[16] == 0.0
    for k, t in enumerate(terms):
        if t is None:
            continue
        t, size = t
        # at most 32 additions in a chain, and 16 roundings in a term
        tol = 0.0 if k in (3, 13, 15) else 48 * EPS * (np.abs(t).sum() + size * len(t))
        assert abs(got[k] - math.fsum(t)) <= tol, (k, got[k], math.fsum(t))


def test_diagnostics_sums_match_the_fields():
    from paper_1707_00198_gb300.lbcg import Lattice
    g, p = I.flat_wall_droplet(400, 201, R=60.0, noise=1e-3, seed=4), I.Params(theta=1.2)
    L = Lattice(g, p, "fp64")
    L.step(20)
    u0 = L.fields()[2:]
    L.diagnostics((200.0, 40.0, 55.0))
    L.step(20)
    rho, rn, ux, uy = L.fields()
    d = L.diagnostics((200.0, 40.0, 55.0))
    y, x = np.mgrid[:g.ny, :g.nx]
    inside, fluid = (x - 200.0)**2 + (y - 40.0)**2 < 55.0**2, g.solid == 0
    for key, part, where in (("m_R_in", (1 + rn) / 2, inside), ("m_R_out", (1 + rn) / 2, ~inside),
                             ("m_B_in", (1 - rn) / 2, inside), ("m_B_out", (1 - rn) / 2, ~inside)):
        t = (rho * part)[where & fluid]
        # (the colours are recovered from rho and rho^N: two roundings of rho more per node)
        assert abs(d[key] - math.fsum(t)) <= 48 * EPS * rho[where & fluid].sum(), key
    assert d["e1"] == max(np.abs(ux - u0[0])[fluid].max(), np.abs(uy - u0[1])[fluid].max())
    L.close()
