"""Every step kernel on lattices that it, and no other, runs (asserted), against other code.

* The pair kernel with partial tiles and odd heights, in every model and storage type (walls:
  test_gpu_walls), and on aligned lattices over 20 steps, against the batched kernel's
  one-node-per-thread code.  Bounds as in test_gpu_pair and test_gpu_parity: 1e-6 of the largest
  population in FP32, one rounding of the stored deviations in 16 bits (2e-4 FP16, 1e-2 BF16).
* Its repulsion force with partial tiles, as in test_gpu_repulsion.
* The TMA-staged kernel, which steps lattices of more than 512 columns, in every model, with walls,
  for chunked and persistent grids, against the same code.
* The generic kernel with 64-bit indices in FP32 (K Q N >= 2^31), against its 32-bit form: a lattice
  that repeats a smaller one 4 x 4 times keeps its period, and the same code gives the same bits."""
import numpy as np
import pytest

from tests import cases as C
from tests.test_gpu_pair import _case
from tests.test_gpu_repulsion import test_repulsion as _repulsion

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

TOL = {1: 1e-6, 2: 2e-4, 3: 1e-2}


def _against_batch(lbm, case, precision, steps, tiling=None, uses_tiling=False):
    lat = C.gpu_lattice(lbm, case, precision)
    if tiling:
        lat.set_tiling(*tiling)
    assert lat.tiling_used() is uses_tiling
    lat.step(steps)
    ref = C.gpu_lattice(lbm, case, precision)
    batch = lbm.Batch(precision, 1, lbm.Batch.units(ref), stream=ref.stream)
    batch.set([ref], [steps])
    batch.step(steps)
    a, b = lat.pops(), ref.pops()
    assert bool(torch.isfinite(b).all())
    assert float((a - b).abs().max()) <= TOL[precision] * float(b.abs().max())


@pytest.mark.parametrize("precision", [1, 2, 3])
@pytest.mark.parametrize("model", [0, 1, 2])
@pytest.mark.parametrize("shape", [(97, 41, 5), (63, 65, 4), (45, 47, 3), (481, 9, 2), (12, 170, 3)])
def test_pair_kernel_partial_tiles(lbm, shape, model, precision):
    _against_batch(lbm, _case(model, shape, False), precision, 2)


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("model", [0, 1, 2])
@pytest.mark.parametrize("shape", [(64, 24, 20), (96, 64, 48), (256, 16, 6)])
def test_pair_kernel_aligned(lbm, shape, model, precision):
    case = (C.cg_drop3d, C.sc_mp3d, C.sc_2c3d)[model](*shape)  # the inputs of the 20-step bounds
    _against_batch(lbm, case, precision, 20)


def test_pair_kernel_repulsion_partial_tiles(lbm):
    for precision in (lbm.FP32, lbm.FP16):
        kw = dict(nx=97, ny=41, nz=6, precision=precision, rep_pi=0.012)
        assert not lbm.Lattice(lbm.Params(**kw)).tiling_used()
    _repulsion((97, 41, 6), False, False)


@pytest.mark.parametrize("tiling", [(32, 8, 3), (32, 8, 0), (32, 16, 0)])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("model", [0, 1, 2])
def test_tma_kernel(lbm, model, walls, tiling):
    for shape in ((544, 8, 5), (576, 16, 7)):
        case = _case(model, shape, walls)
        for precision in (1, 2, 3):
            _against_batch(lbm, case, precision, 2, tiling, True)


def test_generic_kernel_64_bit_indices(lbm):
    free, _ = torch.cuda.mem_get_info()
    if free < 40 * 2 ** 30:
        pytest.skip("needs about 25 GB of free device memory")
    nx, ny, nz, reps = 516, 83, 83, 4
    assert 38 * nx * ny * nz * reps ** 2 >= 2 ** 31 > 38 * nx * ny * nz
    case = _case(0, (nx, ny, nz), False)
    small = C.gpu_lattice(lbm, case, lbm.FP32)

    def tile(a):
        return a.reshape(-1, nz, ny, nx).repeat(1, reps, reps, 1)

    big = lbm.Lattice(lbm.Params(precision=lbm.FP32, **dict(case.kw, ny=ny * reps, nz=nz * reps)))
    big.init(*[tile(torch.as_tensor(a, device=big.device)).reshape(-1) for a in (case.rho_r, case.rho_b)])
    assert big.tiling_used() and small.tiling_used()
    small.step(3)
    big.step(3)
    for a, b in zip(small.moments()[:3], big.moments()[:3]):
        assert torch.equal(tile(a).reshape(-1), b.reshape(-1))
