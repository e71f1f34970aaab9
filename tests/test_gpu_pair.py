"""The pair kernel (two nodes per thread) at the sizes where it can go wrong: widths around
its 32-column tiles and the largest cluster, heights around its 8- and 16-row tiles and odd
ones (half-filled pairs), one-node extents, planes fewer than a run, with walls in every
orientation, against the batched kernel's one-node-per-thread code (held to the oracle by
test_gpu_batch); and the raw-state copies of its padded rows.

Two steps apart by at most what the kernels of one storage type may differ by
(test_gpu_parity): 1e-6 of the largest population in FP32, one rounding of the stored
deviations (at most a tenth of it) in 16 bits: 2e-4 in FP16, 1e-2 in BF16."""
import numpy as np
import pytest

from tests import cases as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

SHAPES = [(1, 1, 1), (2, 3, 4), (5, 9, 3), (31, 8, 5), (33, 15, 4), (64, 17, 3), (97, 7, 6), (288, 16, 3), (511, 10, 2),
          (512, 8, 3)]


def _case(model, shape, walls, seed=11):
    nx, ny, nz = shape
    n = nx * ny * nz
    x, y, z = C.inputs.grid(nx, ny, nz)
    inside = ((x - nx / 2) ** 2 / max(nx / 3, 1) ** 2 + (y - ny / 2) ** 2 / max(ny / 3, 1) ** 2 +
              (z - nz / 2) ** 2 / max(nz / 3, 1) ** 2) <= 1
    noise = 0.01 * C.inputs.uniform_pm1(seed, n)
    if model == 0:
        rr, rb = C.inputs.two_fluid(inside, 1.0, 0.5, 0.01, seed)
        kw = dict(rho_r0=1.0, rho_b0=0.5, tau_r=0.9, tau_b=0.7, A=4e-3)
    elif model == 1:
        rr, rb = np.where(inside, C.SC_LIQ, C.SC_GAS) * (1 + noise), None
        kw = dict(G=-5.0, rho0_psi=1.0, tau_r=0.9)
    else:
        rr, rb = np.where(inside, 1.03, 0.03) * (1 + noise), np.where(inside, 0.03, 1.03) * (1 - noise)
        kw = dict(G=0.9, rho0_psi=0.577, tau_r=1.0, tau_b=0.8)
    solid = None
    if walls:  # planes, an edge, and single nodes
        solid = ((y == 0) | ((x == nx - 1) & (z == 0)) | ((x * 7 + y * 5 + z * 3) % 29 == 13)).astype(np.uint8)
        rr = np.where(solid, 0.0, rr)
        rb = None if rb is None else np.where(solid, 0.0, rb)
        kw["body_force"] = (1e-5, -2e-6, 2e-6)
    kw.update(lattice=1, model=model, nx=nx, ny=ny, nz=nz)
    return C.Case("pair", kw, rr, rb, None, solid)


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("model", [0, 1, 2])
@pytest.mark.parametrize("shape", SHAPES)
def test_pair_kernel_shapes(lbm, shape, model, walls):
    if walls and min(shape[0], shape[1]) < 3:
        pytest.skip("no fluid node left between the walls")
    case = _case(model, shape, walls)
    for precision, tol in ((lbm.FP32, 1e-6), (lbm.FP16, 2e-4), (lbm.BF16, 1e-2)):
        lat = C.gpu_lattice(lbm, case, precision).step(2)
        ref = C.gpu_lattice(lbm, case, precision)
        batch = lbm.Batch(precision, 1, 4096, stream=ref.stream)
        batch.set([ref], [2])
        batch.step(2)
        a, b = lat.pops().cpu().numpy(), ref.pops().cpu().numpy()
        assert np.all(np.isfinite(b))
        assert np.max(np.abs(a - b)) <= tol * np.max(np.abs(b)), precision


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("shape", [(13, 9, 7), (40, 8, 6)])
def test_padded_rows_state_copies(lbm, shape, precision):
    """Raw state out of and into padded rows, whole and by planes, is dense and bitwise."""
    case = _case(0, shape, True)
    a = C.gpu_lattice(lbm, case, precision).step(5)
    state = a.save_state()
    n, elt = np.prod(shape), 4 if precision == 1 else 2
    assert state.numel() == 38 * n * elt + 2 * n * 4
    solid = torch.as_tensor(case.solid, device=a.device)
    b = lbm.Lattice(lbm.Params(precision=precision, **case.kw)).load_state(state, solid)
    assert torch.equal(b.state_planes(0, shape[2]), state)
    c = lbm.Lattice(lbm.Params(precision=precision, **case.kw)).load_state(torch.zeros_like(state), solid)
    for z0, k in ((0, 2), (2, shape[2] - 2)):
        c.set_state_planes(z0, k, a.state_planes(z0, k))
    for lat in (a, b, c):
        lat.step(4)
    want = a.save_state()
    assert torch.equal(b.save_state(), want) and torch.equal(c.save_state(), want)
