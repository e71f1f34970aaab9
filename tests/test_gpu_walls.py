"""Walls on the pair kernel, whose walled collision a plane of a tile row takes with walls in
sight: partial tiles, odd heights and every orientation of walls, planes with and without walls
in sight in one lattice and long enough runs for both collisions, against the batched kernel's
one-node-per-thread code at the bounds of test_gpu_pair; and what walls may cost.

Time: with a wall in sight of nearly every node the collision takes about half as long again
as without any (two more selections for each of 36 neighbours); a second pass over the nodes
beside walls takes five times as long.  Less than 2.5 times tells the two apart.
"""
import numpy as np
import pytest

from tests import cases as C
from tests.test_gpu_pair import _case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

# short runs; widths of 1 and 31 in the last tile, odd heights; runs of more than 16 planes with
# a clear middle (the planes beyond z = 3)
SHAPES = [(97, 41, 5), (63, 65, 4), (64, 48, 3), (96, 72, 330)]


def _solid(shape, kind, seed=3):
    nx, ny, nz = shape
    x, y, z = C.inputs.grid(nx, ny, nz)
    if kind == "y":
        s = (y == 0) | (y == ny - 1)
    elif kind == "x":
        s = (x == 0) | (x == 31) | ((x == nx - 1) & (y % 5 == 0))
    elif kind == "z":
        s = (z == 0) | ((z == nz - 1) & (x % 3 == 0))
    else:  # porous, in the first planes only where there are many
        s = (np.random.default_rng(seed).random(nx * ny * nz) < 0.15) & (z < max(4, nz // 2))
    return s.astype(np.uint8)


@pytest.mark.parametrize("kind", ["x", "y", "z", "porous"])
@pytest.mark.parametrize("model", [0, 1, 2])
@pytest.mark.parametrize("shape", SHAPES)
def test_walls_against_the_generic_code(lbm, shape, model, kind):
    case = _case(model, shape, False)
    case.solid = _solid(shape, kind)
    case.rho_r = np.where(case.solid, 0.0, case.rho_r)
    case.rho_b = None if case.rho_b is None else np.where(case.solid, 0.0, case.rho_b)
    case.kw["body_force"] = (1e-5, -2e-6, 2e-6)
    for precision, tol in ((lbm.FP32, 1e-6), (lbm.FP16, 2e-4), (lbm.BF16, 1e-2)):
        lat = C.gpu_lattice(lbm, case, precision).step(2)
        ref = C.gpu_lattice(lbm, case, precision)
        batch = lbm.Batch(precision, 1, lbm.Batch.units(ref), stream=ref.stream)
        batch.set([ref], [2])
        batch.step(2)
        a, b = lat.pops(), ref.pops()
        assert bool(torch.isfinite(b).all())
        assert float((a - b).abs().max()) <= tol * float(b.abs().max()), precision
        for l in (lat, ref):
            l.close()


@pytest.mark.parametrize("model", [0, 2])
def test_cost_of_a_porous_mask(lbm, model):
    shape = (128, 128, 64)
    case = _case(model, shape, False)
    solid = (np.random.default_rng(3).random(case.rho_r.size) < 0.15).astype(np.uint8)

    def step_ms(mask):
        case.solid = mask
        lat = C.gpu_lattice(lbm, case, lbm.FP32)
        lat.step(5)
        best = np.inf
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(lat.stream)
            lat.step(20)
            b.record(lat.stream)
            b.synchronize()
            best = min(best, a.elapsed_time(b) / 20)
        return best

    free, porous = step_ms(None), step_ms(solid)
    print(f"model {model}: {1e3 * free:.1f} us without walls, {1e3 * porous:.1f} porous")
    assert porous < 2.5 * free
