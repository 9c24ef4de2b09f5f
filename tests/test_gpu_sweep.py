"""ILU(0) sweeps at the sizes where their schedule can go wrong: rows longer
than the edge rings (the rings wrap, progress reports come into play), rows
shorter than a chunk, 2D grids of one and of several tiles, a single tile, and
blocks of tiles that the grid does not fill.  The pipelined schedules (with
and without clusters) equal the level-scheduled sweeps bit for bit, in FP64
and in mixed precision."""
import os

import numpy as np
import pytest

from _cases import gpu_handle, make_case

pytestmark = pytest.mark.gpu

MODES = {"level": {"CAMS_ILU_LEVEL": "1"}, "tile": {"CAMS_ILU_LEVEL": "0", "CAMS_ILU_CTA": "0"},
         "cluster": {"CAMS_ILU_LEVEL": "0", "CAMS_ILU_CTA": "1"}}


@pytest.fixture(scope="module")
def cams():
    from paper_1705_05783_gb300 import cams
    return cams


def _iterate(cams, monkeypatch, case, mode):
    with monkeypatch.context() as m:
        for k, v in MODES[mode].items():
            m.setenv(k, v)
        h, bc, keep = gpu_handle(case)
    try:
        rng = np.random.default_rng(11)
        p_nu, p_n = rng.uniform(0, 1, case.N), rng.uniform(0, 1, case.N)
        cams.cams_assemble(h, p_nu, p_n, case.inp["dt"], bc)
        cams.cams_update_basis(h, True)
        res = cams.cams_iterate(h, 2)
        return res, cams.cams_get(h, cams.CAMS_Q_PRESSURE, np.zeros(case.N))
    finally:
        cams.cams_destroy(h)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape,coarse", [
    ((540, 9, 5), (9, 3, 5)),      # rows longer than either precision's ring, tiles of one row
    ((540, 72, 1), (9, 9, 1)),     # the same in 2D: three tiles
    ((3, 34, 21), (3, 2, 3)),      # a row shorter than a chunk
    ((6, 4, 1), (3, 2, 1)),        # one 2D tile, hardly filled
    ((9, 8, 4), (3, 4, 2)),        # one 3D tile, exactly
    ((21, 41, 17), (7, 41, 17)),   # six by five tiles: blocks that stick out of the grid
])
def test_sweeps_equal_level_schedule(cams, monkeypatch, shape, coarse, precision):
    case = make_case("3d-200x200x100", nx=shape[0], ny=shape[1], nz=shape[2], coarse=coarse,
                     n_post=2, precision=precision)
    r0, p0 = _iterate(cams, monkeypatch, case, "level")
    for mode in ("tile", "cluster"):
        r1, p1 = _iterate(cams, monkeypatch, case, mode)
        assert np.array_equal(p1, p0), mode
        assert np.array_equal(r1, r0), mode


@pytest.mark.parametrize("prec", [0, 1])
def test_a_row_of_more_than_two_million_cells(prec):
    """65,536 pieces of a row and more in the layout conversions (32 cells a
    piece in FP64).  On one row A is tridiagonal and ILU(0) is its LU
    factorisation, so one smoothing step solves the system: the residual falls
    to rounding (FP32 in the mixed preconditioner, whose residual is then below
    1e-3 of the first: u times the condition number of D^-1 A, diagonally
    dominant by dt here)."""
    from paper_1705_05783_gb300 import cams
    n = 65535 * 32 + 1000 + 64
    n -= n % 1000
    k = np.exp(np.random.default_rng(3).standard_normal(n))
    h = cams.cams_setup(cams.cams_grid(n, 1, 1, 1.0, 1.0, 1.0), cams.cams_fluid(0, 0.1, 1.0, 1.0, 1.0),
                        cams.make_options((1000, 1, 1), precision=prec, n_post=1), k)
    try:
        bc, keep = cams.make_bc(True, 1.0, 0.0)
        p0 = np.random.default_rng(4).uniform(0.0, 1.0, n)
        cams.cams_assemble(h, p0, p0, 1e-2, bc)
        cams.cams_update_basis(h, True)
        norms = cams.cams_iterate(h, 1)
        assert norms[1] <= (1e-3 if prec else 1e-9) * norms[0]
    finally:
        cams.cams_destroy(h)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape,coarse", [((5, 8, 90), (5, 4, 9)),     # one tile wide in y: clusters along z
                                          ((30, 150, 4), (5, 10, 2)),  # ... in z: clusters along y
                                          ((560, 3, 34), (8, 3, 17))]) # rows longer than the rings, one tile wide
def test_sweeps_of_one_row_of_tiles(cams, monkeypatch, shape, coarse, precision):
    test_sweeps_equal_level_schedule(cams, monkeypatch, shape, coarse, precision)
