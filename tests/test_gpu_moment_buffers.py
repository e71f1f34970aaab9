"""Where lbm_moments puts its results: device buffers at every alignment, a velocity buffer that
is not aligned to its elements included, pinned and pageable ones, and ones that overlap, against
the aligned device buffers, bit for bit."""
import ctypes

import numpy as np
import pytest

from tests import cases as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.mark.parametrize("kind", ["device", "pinned", "pageable"])
@pytest.mark.parametrize("model", ["cg_drop3d", "sc_mp3d", "sc_2c3d", "sc_mr3d"])
def test_moment_buffers(lbm, model, kind):
    case = C.SMALL_CASES[model]()
    lat = C.gpu_lattice(lbm, case, lbm.FP32).step(3)
    n = lat.params.n
    rr, rb, u, _, _ = lat.moments()
    want = [a.cpu().numpy().ravel() for a in (rr, rb, u)]
    for shift in (0, 4, 8, 12):  # bytes
        raw = torch.zeros(5 * n * 8 + 64, dtype=torch.uint8, device="cuda" if kind == "device" else "cpu")
        raw = raw.pin_memory() if kind == "pinned" else raw
        at = [raw.data_ptr() + shift + 8 * k for k in (0, n, 2 * n)]
        rc = lbm.lib().lbm_moments(lat._h, *[ctypes.c_void_p(a) for a in at], None, None)
        assert rc == lbm.OK
        torch.cuda.synchronize()
        got = raw.cpu().numpy()[shift:shift + 5 * n * 8].copy().view(np.float64)
        for k, (a, b) in enumerate(zip((0, n, 2 * n), (n, 2 * n, 5 * n))):
            assert np.array_equal(got[a:b], want[k]), (shift, k)
    # the densities in the velocity's buffer: they are copied last
    both = torch.zeros(3 * n, dtype=torch.float64, device="cuda")
    lat.moments_into(both[:n], both[n:2 * n], both)
    torch.cuda.synchronize()
    got = both.cpu().numpy()
    assert np.array_equal(got[:n], want[0]) and np.array_equal(got[n:2 * n], want[1])
    assert np.array_equal(got[2 * n:], want[2][2 * n:])
