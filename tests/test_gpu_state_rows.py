"""Raw state of lattices with padded rows, whole and by planes, to and from device, pinned and
pageable buffers at every alignment: dense, and the bytes of the populations in node order.

Time: loading from the host may take no more than 4 times what it takes for a lattice of the same
size whose rows need no padding (copied row by row it took 16 times as long)."""
import time

import numpy as np
import pytest

from tests import cases as C
from tests.test_gpu_pair import _case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


def _buffer(kind, n, shift):
    whole = torch.zeros(n + 8, dtype=torch.uint8, device="cuda" if kind == "device" else "cpu")
    if kind == "pinned":
        whole = whole.pin_memory()
    return whole[shift:shift + n]


@pytest.mark.parametrize("kind", ["device", "pinned", "pageable"])
@pytest.mark.parametrize("model", [0, 1])
@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("shape", [(97, 33, 3), (45, 47, 5), (33, 130, 17)])
def test_state_copies(lbm, shape, precision, model, kind):
    nx, ny, nz = shape
    case = _case(model, shape, False)
    a = C.gpu_lattice(lbm, case, precision).step(3)
    K, n, elt = (2, 1)[model], nx * ny * nz, (4, 2)[precision - 1]
    state = a.save_state()
    host = state.cpu().numpy()
    # what is stored, phi r + deviation, against the exported populations
    g = host[:K * 19 * n * elt].view((np.float32, np.float16)[precision - 1]).reshape(K, 19, n).astype(np.float64)
    r = host[K * 19 * n * elt:].view(np.float32).reshape(K, 1, n).astype(np.float64)
    f = a.pops().cpu().numpy()
    phi = np.stack([((f - g)[k, :, at] / r[k, 0, at]) for k, at in enumerate(r[:, 0].argmax(1))])
    assert np.abs(f - g - phi[:, :, None] * r).max() < 1e-12
    solid = None
    for shift in (0, 1, 2, 4):
        out = _buffer(kind, state.numel(), shift)
        a.save_state(out)
        assert torch.equal(out.cpu(), state.cpu())
        b = lbm.Lattice(lbm.Params(precision=precision, **case.kw)).load_state(out, solid)
        assert torch.equal(b.save_state(), state)
        c = lbm.Lattice(lbm.Params(precision=precision, **case.kw)).load_state(torch.zeros_like(state), solid)
        for z0, k in ((0, 1), (1, nz - 1)):
            nb = a.state_planes(z0, k).numel()
            part = _buffer(kind, nb, shift)
            a.state_planes(z0, k, part)
            a.stream.synchronize()
            c.set_state_planes(z0, k, part)
            c.stream.synchronize()
        assert torch.equal(c.save_state(), state)
        want = a.save_state()
        for lat in (b, c):  # both buffers hold it: two steps read the second
            x = lat.step(2).save_state()
            lat.close()
            y = lbm.Lattice(lbm.Params(precision=precision, **case.kw)).load_state(want, solid).step(2).save_state()
            assert torch.equal(x, y)


def test_loading_padded_rows_from_the_host_is_as_fast(lbm):
    def ms(nx):
        case = _case(0, (nx, 75, 67), False)
        lat = C.gpu_lattice(lbm, case, lbm.FP32)
        host = lat.save_state().cpu().pin_memory()
        best = np.inf
        for _ in range(5):
            t = time.perf_counter()
            lat.load_state(host)
            best = min(best, 1e3 * (time.perf_counter() - t))
        return best

    padded, dense = ms(101), ms(104)
    print(f"load from the host: {padded:.2f} ms padded, {dense:.2f} ms dense")
    assert padded < 4 * dense
