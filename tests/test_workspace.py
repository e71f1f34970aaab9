"""Workspace of lattices that the pair kernel does not run: what they store, and a few per cent."""
import ctypes

import pytest

from paper_2110_05197_gb300 import build as lbm_build
from paper_2110_05197_gb300 import lbm


@pytest.mark.parametrize("kw", [
    dict(nx=1, ny=300, nz=200), dict(nx=3, ny=200, nz=200, precision=lbm.FP16), dict(nx=5, ny=100, nz=400, model=lbm.SC_MP),
    dict(lattice=lbm.D2Q9, nx=128, ny=128, nz=1, model=lbm.SC_MP, precision=lbm.FP16),
    dict(lattice=lbm.D2Q9, nx=64, ny=64, nz=1, precision=lbm.FP64), dict(nx=33, ny=40, nz=50, streaming=lbm.STREAM_AA)])
def test_workspace_is_what_a_lattice_stores(kw):
    lbm_build.build()
    p = lbm.Params(**kw)
    need = ctypes.c_size_t(0)
    assert lbm.lib().lbm_create(ctypes.byref(p.to_c()), None, ctypes.byref(need), None, None) == lbm.OK
    elt, ref = {lbm.FP64: (8, 8), lbm.FP32: (4, 4), lbm.FP16: (2, 4)}[p.precision]
    buffers = 1 if p.streaming == lbm.STREAM_AA else 2
    # populations, reference densities, wall mask, moments' staging; then block partials (80 bytes for
    # 64 nodes) and the tiles' wall words (8 bytes for up to 32 nodes, where the shape has them)
    stored = p.n * (buffers * p.ncomp * (p.q * elt + ref) + 1 + 48)
    assert stored <= need.value <= 1.03 * stored + 8192


def test_pair_lattices_have_room_for_the_tables_of_walls():
    """Also where only one component's arrays stay within 32-bit indices (rows padded for SC only)."""
    lbm_build.build()
    for model, ncomp in ((lbm.SC_MP, 1), (lbm.CG, 2)):
        p = lbm.Params(nx=33, ny=1300, nz=1300 if model == lbm.SC_MP else 1400, model=model)
        need = ctypes.c_size_t(0)
        assert lbm.lib().lbm_create(ctypes.byref(p.to_c()), None, ctypes.byref(need), None, None) == lbm.OK
        rows = p.ny * p.nz
        assert need.value >= 2 * ncomp * 20 * 4 * 40 * rows + 49 * p.n + 2 * 8 * rows + (p.ny + 7) // 8 * p.nz
