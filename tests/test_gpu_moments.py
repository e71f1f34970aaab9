"""The moment kernels against FP64 sums over the exported populations: densities and
velocity, read with and without the totals, at sizes with remainders in every direction,
with walls and in both layouts of in-place streaming.

Densities: exact sums in FP32 pairs are good to 2^-46 of the largest value, FP64 sums of 38
values to 2^-48: 1e-13.  Velocity: momentum and force as good as the densities times O(10)
couplings, 2e-12 (walls, dense gas: divided by rho >= 0.03).  Multirange self forces are FP32
sums of at most 92 terms of total weight < 1 times |Psi G Psi| <= 12: 92 2^-24 12 / rho, 1e-4.
"""
import numpy as np
import pytest
import torch

from paper_2110_05197_gb300 import lbm

pytestmark = pytest.mark.gpu
BELT = {1: 4 / 135, 2: 1 / 63, 3: 2 / 315, 4: 5 / 1512, 5: 1 / 945, 6: 1 / 1890, 8: 1 / 15120}
P3 = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]
P2 = [(1, 0, 0), (0, 1, 0), (1, 1, 0), (1, -1, 0)]


def _gradient(a, solid, pairs):
    """sum over +-c of w a(x + c) c, a wall neighbour replaced by the centre; a is [z, y, x]."""
    def at(c):
        s = (-c[2], -c[1], -c[0])
        return np.where(np.roll(solid, s, (0, 1, 2)), a, np.roll(a, s, (0, 1, 2)))

    out = np.zeros((3,) + a.shape)
    for c, w in pairs:
        d = w * (at(c) - at(tuple(-s for s in c)))
        for t in range(3):
            out[t] += c[t] * d
    return out


@pytest.mark.parametrize("prec", [lbm.FP64, lbm.FP32, lbm.FP16])
@pytest.mark.parametrize("model,shape,walls,aa", [
    ("cg", (7, 5, 1), False, False), ("cg", (33, 9, 5), True, False), ("cg", (33, 9, 5), True, True),
    ("cg", (64, 16, 8), False, True), ("sc", (31, 3, 1), True, False), ("sc", (40, 11, 6), False, True),
    ("sc2c", (19, 8, 7), True, False), ("mr", (2, 3, 2), False, False), ("mr", (37, 13, 9), True, False)])
def test_moments(prec, model, shape, walls, aa):
    nx, ny, nz = shape
    kw = {"cg": dict(model=lbm.CG, rho_r0=1.0, rho_b0=0.5, A=4e-3, body_force=(1e-4, 0.0, 0.0) if walls else (0.0, 0.0, 0.0)),
          "sc": dict(model=lbm.SC_MP, G=-5.0, rho0_psi=1.0),
          "sc2c": dict(model=lbm.SC_2C, G=0.9, rho0_psi=0.577),
          "mr": dict(model=lbm.SC_MR, Ga=(-9.0, -8.0), Gr=(8.1, 7.1), G=1.215, rho0_psi=0.83)}[model]
    p = lbm.Params(lattice=lbm.D3Q19 if nz > 1 else lbm.D2Q9, precision=prec, nx=nx, ny=ny, nz=nz, tau_r=1.0, tau_b=0.9,
                   streaming=lbm.STREAM_AA if aa else lbm.STREAM_AB, **kw)
    g = np.random.default_rng(5)
    n, K = p.n, p.ncomp
    solid = np.zeros((nz, ny, nx), bool)
    if walls:
        solid[:, 0, :] = True
        solid[nz // 2, ny // 2, 1:3] = True
    rho = [np.where(solid, 0, 0.6 + 0.1 * g.random((nz, ny, nx))).ravel() for _ in range(K)]
    lat = lbm.Lattice(p)
    for steps in (0, 1, 2):  # both buffers, both in-place layouts
        lat.init(rho[0], rho[1] if K == 2 else None, solid=solid.astype(np.uint8).ravel() if walls else None)
        lat.step(steps)
        pops = lat.pops().cpu().numpy().reshape(K, -1, nz, ny, nx)
        pairs = P3 if nz > 1 else P2
        w = {1: 1 / 18, 2: 1 / 36} if nz > 1 else {1: 1 / 9, 2: 1 / 36}
        rs = [pops[k].sum(0) for k in range(K)]
        j = np.zeros((3, nz, ny, nx))
        for k in range(K):
            for q, c in enumerate(pairs):
                for t in range(3):
                    j[t] += c[t] * (pops[k, 2 * q + 1] - pops[k, 2 * q + 2])
        F = np.zeros_like(j) + np.array(p.body_force)[:, None, None, None]
        near = [(c, w[sum(s * s for s in c)]) for c in pairs]
        psi = [p.rho0_psi * (1 - np.exp(-r / p.rho0_psi)) for r in rs]
        if model == "sc":
            F += -p.G * psi[0] * _gradient(psi[0], solid, near)
        elif model in ("sc2c", "mr"):
            G = p.G / p.rho0_psi ** 2
            for s in range(2):
                F += -G * rs[s] * _gradient(rs[1 - s], solid, near)
                if model == "mr":
                    span = range(-2, 3)
                    belt = [(c, BELT[sum(t * t for t in c)]) for c in ((x, y, z) for x in span for y in span for z in span)
                            if c > (0, 0, 0) and sum(t * t for t in c) in BELT]
                    F += -p.Ga[s] * psi[s] * _gradient(psi[s], solid, near)
                    F += -p.Gr[s] * psi[s] * _gradient(psi[s], solid, belt)
        total = np.where(solid, 1.0, sum(rs))
        u = np.where(solid, 0.0, (j + 0.5 * F) / total)
        tol = 1e-4 if model == "mr" and prec != lbm.FP64 else 2e-12
        big = torch.full((2 * n + 3 * n + 3,), -7.0, dtype=torch.float64, device=lat.device)
        for off, totals in ((0, None), (1, np.zeros(10))):  # aligned and not, without and with the totals
            rr, uu = big[off:off + n], big[off + 2 * n:off + 5 * n]
            rb = big[off + n:off + 2 * n] if K == 2 else None
            lat.moments_into(rr, rb, uu, totals=totals)
            torch.cuda.synchronize()
            # in place, the slots of wall nodes hold bounced populations: fluid nodes only
            fluid = ~solid.ravel()
            assert np.abs(rr.cpu().numpy() - rs[0].ravel())[fluid].max() <= 1e-13
            if K == 2:
                assert np.abs(rb.cpu().numpy() - rs[1].ravel())[fluid].max() <= 1e-13
            assert np.abs(uu.cpu().numpy() - u.reshape(3, -1).ravel()).max() <= tol, (steps, off)
            if totals is not None:
                assert abs(totals[0] - rs[0].sum()) <= 1e-13 * n
                assert abs(totals[6] - np.sqrt((u ** 2).sum(0).max())) <= 2 * tol
                assert abs(totals[8] - rs[0][~solid].min()) <= 1e-13
