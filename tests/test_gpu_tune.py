"""The tuner times what makes a difference: one candidate where the step kernel picks its own
shape, several where the tiling shapes it; the state is restored bit for bit."""
import pytest

from tests import cases as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.mark.parametrize("make,precision,own_shape", [
    (lambda: C.cg_drop3d(nx=64, ny=32, nz=20), 1, True), (lambda: C.sc_mp3d(nx=61, ny=57, nz=20), 2, True),
    (C.cg_walls3d, 1, False), (lambda: C.cg_walls3d(nx=32, ny=16, nz=9), 2, True), (C.sc_mp3d, 1, False),
    (lambda: C.cg_drop3d(nx=64, ny=32, nz=20), 0, False), (C.cg_drop2d, 1, False), (C.sc_mr3d, 1, True)])
def test_candidates(lbm, make, precision, own_shape):
    from paper_2110_05197_gb300 import tune
    case = make()
    lat = C.gpu_lattice(lbm, case, precision).step(2)
    state = lat.save_state()
    best, timings = tune.autotune(lat, use_cache=False, steps=2, trials=1)
    assert lat.tiling_used() is not own_shape
    assert (len(timings) == 1) is own_shape and best in timings
    assert torch.equal(lat.save_state(), state)
