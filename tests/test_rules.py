"""The rules of csrc/lbm_rules.h, which decide what kernel a lattice runs and how it is stored,
compiled for the host: z-slabs run the kernel of the whole lattice; rows are padded only where the
pair kernel reads them, and never beyond what the batched launch takes."""
import ctypes
import itertools
import os
import subprocess

import pytest

from paper_2110_05197_gb300 import lbm

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include "lbm_rules.h"
extern "C" int pair_steps(const lbm_params* p, int walls) { return lbm::pair_steps(*p, walls != 0); }
extern "C" int row_pitch(const lbm_params* p) { return lbm::row_pitch(*p); }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cpp").write_text(SRC)
    so = d / "rules.so"
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2110_05197_gb300", "csrc"), str(d / "rules.cpp"), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


def _c(**kw):
    return ctypes.byref(lbm.Params(**kw).to_c())


def test_slabs_run_the_kernel_of_the_whole_lattice(rules):
    for (nx, ny), model, precision, walls in itertools.product(
            [(8, 200), (33, 33), (61, 57), (97, 75), (101, 75), (64, 64), (200, 203), (512, 40)], (0, 1, 2), (1, 2, 3),
            (False, True)):
        kinds = {rules.pair_steps(_c(nx=nx, ny=ny, nz=nz, model=model, precision=precision), walls)
                 for nz in (4, 17, 60, 67, 300, 1000)}
        assert len(kinds) == 1, (nx, ny, model, precision, walls)


def test_rows_are_padded_only_for_the_pair_kernel(rules):
    for nx, ny, model, precision, aa in itertools.product((1, 2, 3, 7, 11, 12, 33, 61, 97, 511, 513), (1, 9, 33, 75),
                                                          (0, 1, 2, 3), (0, 1, 2), (0, 1)):
        p = dict(nx=nx, ny=ny, nz=20, model=model, precision=precision, streaming=aa)
        runs = rules.pair_steps(_c(**p), 0) or rules.pair_steps(_c(**p), 1)
        assert rules.row_pitch(_c(**p)) == ((nx + 7) // 8 * 8 if runs else nx), p


def test_padding_does_not_leave_32_bit_indices(rules):
    """K Q N below 2^31 and 38 times the padded size above: dense, as the batched launch needs."""
    n = dict(nx=33, ny=1300, nz=1300)
    assert 38 * 33 * 1300 ** 2 < 2 ** 31 <= 38 * 40 * 1300 ** 2
    assert rules.row_pitch(_c(model=0, precision=1, **n)) == 33 and not rules.pair_steps(_c(model=0, precision=1, **n), 0)
    assert rules.row_pitch(_c(model=1, precision=1, **n)) == 40  # 19 arrays
    assert rules.row_pitch(_c(model=0, precision=1, nx=33, ny=1400, nz=1400)) == 40  # no batch in any case


def test_lattices_beyond_the_pair_kernels_indices(rules):
    """One array below 2^31 elements, below 2^30 with walls; 288 GB hold up to 2^31 nodes (SC in FP16)."""
    for nz, free, walled in ((1000, 1, 1), (1024, 1, 0), (2000, 1, 0), (2048, 0, 0), (2100, 0, 0)):
        p = dict(nx=512, ny=2048, nz=nz, model=1, precision=2)
        assert rules.pair_steps(_c(**p), 0) == free and rules.pair_steps(_c(**p), 1) == walled, nz
