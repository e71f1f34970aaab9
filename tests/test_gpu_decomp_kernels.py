"""z-slabs against the single domain, bit for bit, where what steps a lattice could depend on its
number of planes: lattices with partial tiles of a few hundred thousand nodes, whose slabs are
much smaller; tiles of 16 rows on large SC lattices only; the walled collision for all nodes
where runs are short, for planes with walls in sight where they are long."""
import pytest

import tests.cases as C
from tests.test_gpu_pair import _case
from tests.test_gpu_walls import _solid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

CASES = {
    "cg_walls_fp32": ((101, 75, 67), 0, 1, "y", 4),
    "cg_walls_fp16": ((101, 75, 90), 0, 2, "porous", 2),
    "sc_fp16": ((97, 65, 64), 1, 2, None, 3),
    "sc_fp32": ((75, 77, 71), 1, 1, None, 3),
    "cg_fp16_narrow": ((33, 40, 260), 0, 2, None, 4),
    "sc_fp32_rows_of_16": ((64, 64, 48), 1, 1, None, 2),
    "cg_long_runs": ((96, 72, 330), 0, 1, "porous", 3),
    "sc2c_long_runs": ((96, 72, 330), 2, 1, "y", 3),
}


@pytest.mark.parametrize("name", list(CASES))
def test_slabs_run_what_the_whole_runs(lbm, name):
    from paper_2110_05197_gb300 import decomp
    shape, model, precision, walls, world = CASES[name]
    case = _case(model, shape, False)
    if walls:
        case.solid = _solid(shape, walls)
        case.rho_r = case.rho_r * (case.solid == 0)
        case.rho_b = None if case.rho_b is None else case.rho_b * (case.solid == 0)
        case.kw["body_force"] = (1e-5, -2e-6, 2e-6)
    full = C.gpu_lattice(lbm, case, precision)
    params = lbm.Params(precision=precision, **case.kw)
    doms = [decomp.lattice_slab(params, decomp.Slab(shape[2], world, r, 2), case.rho_r, case.rho_b, None, case.solid)
            for r in range(world)]
    decomp.local_exchange(doms)
    for _ in range(4):
        full.step(1)
        for d in doms:
            d.engine.step(1)
        decomp.local_exchange(doms)
    torch.cuda.synchronize()
    for d in doms:
        s = d.slab
        assert torch.equal(d.engine.lat.state_planes(s.halo, s.z1 - s.z0), full.state_planes(s.z0, s.z1 - s.z0)), s.rank
