"""The repulsion force at sizes with remainders in every direction, with walls and in place:
the FP64 velocity (F/2) / rho at rest against the force computed here from its definition
(1e-12), and one step of the other precisions against the FP64 step.

From rest every storage precision starts from the same state (deviations 0).  FP32: about 50
operations on populations <= 0.5, 3e-6.  FP16: deviations up to 0.1 rounded to 2^-11, 1e-4.
The least gradient that counts as an interface lies between the noise (2e-3) and the
interfaces (0.1 and more): at a node whose gradient is near it, recolouring is ill-conditioned.
The force jumps where n.c passes 0, by at most Pi |n'.c| (1e-3 in a population): rounding
decides at a normal within 1e-6 of perpendicular, 1e-5 of the (node, direction) pairs, each
seen in 38 values of its node: 1e-3 of the values.
"""
import numpy as np
import pytest
import torch

from paper_2110_05197_gb300 import lbm

pytestmark = pytest.mark.gpu
P3 = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]
P2 = [(1, 0, 0), (0, 1, 0), (1, 1, 0), (1, -1, 0)]
PI, CHI, EPS = 0.012, 2.0, 1e-2


def _force(colour, solid, d2):
    pairs = P2 if d2 else P3
    w = {1: 1 / 9, 2: 1 / 36} if d2 else {1: 1 / 18, 2: 1 / 36}

    def roll(a, c):
        return np.roll(a, (-c[2], -c[1], -c[0]), (-3, -2, -1))

    g = np.zeros((3,) + colour.shape)
    for c in pairs:
        m = tuple(-s for s in c)
        vp, vm = np.where(roll(solid, c), colour, roll(colour, c)), np.where(roll(solid, m), colour, roll(colour, m))
        for t in range(3):
            g[t] += 3 * w[sum(s * s for s in c)] * c[t] * (vp - vm)
    a = np.sqrt((g ** 2).sum(0))
    n = np.where((a > EPS) & ~solid, g / np.where(a > 0, a, 1), 0.0)
    acc = np.zeros_like(n)
    for c in pairs + [tuple(-s for s in c) for c in pairs]:
        m = roll(n, c)
        nc, pc = sum(c[t] * n[t] for t in range(3)), sum(c[t] * m[t] for t in range(3))
        on = (nc * pc < 0) / np.sqrt(sum(s * s for s in c))
        acc += on * (nc * n + pc * m)
    return -PI * (1 - np.abs(colour)) ** CHI * acc


@pytest.mark.parametrize("shape,walls,aa", [((64, 16, 8), False, False), ((37, 11, 9), False, False),
                                            ((31, 3, 2), False, False), ((40, 13, 1), False, False),
                                            ((96, 88, 44), False, False), ((33, 10, 7), True, False),
                                            ((33, 10, 7), True, True)])
def test_repulsion(shape, walls, aa):
    nx, ny, nz = shape
    rng = np.random.default_rng(3)
    z, y, x = np.meshgrid(*(np.arange(v) for v in (nz, ny, nx)), indexing="ij")
    near = np.abs(x - nx // 3 - 0.5) < 1  # a film of two nodes: opposite normals side by side
    solid = np.zeros(near.shape, np.uint8)
    if walls:
        solid[:, 0, :] = 1
    rr = np.where(near, 1.2, 0.1) * (1 + 0.01 * rng.random(near.shape)) * (solid == 0)
    rb = np.where(near, 0.1, 1.2) * (1 + 0.01 * rng.random(near.shape)) * (solid == 0)
    out = {}
    for prec in (lbm.FP64, lbm.FP32, lbm.FP16):
        p = lbm.Params(lattice=lbm.D3Q19 if nz > 1 else lbm.D2Q9, model=lbm.CG, precision=prec, nx=nx, ny=ny, nz=nz,
                       rho_r0=1.36, rho_b0=1.36, tau_r=1.0, tau_b=1.0, A=0.0518, rep_pi=PI, rep_chi=CHI, grad_eps=EPS,
                       streaming=lbm.STREAM_AA if aa else lbm.STREAM_AB)
        lat = lbm.Lattice(p)
        lat.init(rr.ravel(), rb.ravel(), solid=solid.ravel() if walls else None)
        if prec == lbm.FP64:
            u = torch.empty(3 * p.n, dtype=torch.float64, device=lat.device)
            lat.moments_into(None, None, u)
            with np.errstate(invalid="ignore"):
                c = np.where(solid == 1, 0.0, (rr - rb) / (rr + rb))
            want = np.where(solid == 1, 0.0, 0.5 * _force(c, solid == 1, nz == 1) / np.where(solid == 1, 1, rr + rb))
            assert np.abs(want).max() > 1e-5
            assert np.abs(u.cpu().numpy().reshape(want.shape) - want).max() <= 1e-12
        lat.step(1)
        out[prec] = lat.pops().cpu().numpy()
    for prec, tol in ((lbm.FP32, 3e-6), (lbm.FP16, 1e-4)):
        err = np.abs(out[prec] - out[lbm.FP64])
        assert (err > tol).mean() <= 1e-3 and err.max() <= 1e-3, (prec, err.max(), (err > tol).mean())
