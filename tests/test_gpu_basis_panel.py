"""The panel form of the local basis solves at the edges of its split: boxes of
one cell, flat and ragged ones, half-widths around multiples of the tile (8
rows) and of the panel (16 columns), boxes longer than the ring of columns,
and blocks whose interiors stay with the general solver.

Tolerance: P solves local SPD problems, backward stably, so two solvers differ
by the local condition number times the unit roundoff; the parity test's bound
for P (p_tolerance) holds here too, in FP32 with FP32's roundoff."""
import numpy as np
import pytest

import oracle
from oracle.basis import basis_operator, prolongation
from oracle.wirebasket import build_wirebasket

from _cases import gpu_handle, make_case, p_from_gpu
from test_gpu_parity import p_tolerance

pytestmark = pytest.mark.gpu

# mild fields, so that the bound says something in FP32 too
CASES = {
    "flat": dict(name="2d-40x40", nx=36, ny=27, coarse=(9, 9, 1)),
    "cells": dict(name="3d-200x200x100", nx=8, ny=6, nz=6, coarse=(2, 2, 2)),
    "m8": dict(name="3d-200x200x100", nx=15, ny=15, nz=15, coarse=(5, 3, 5)),
    "m16": dict(name="3d-200x200x100", nx=15, ny=15, nz=24, coarse=(5, 5, 8)),
    "m48": dict(name="3d-100x100x50-wells", nx=14, ny=18, nz=27, coarse=(7, 9, 9)),
    "m64": dict(name="3d-200x200x100", nx=27, ny=27, nz=27, coarse=(9, 9, 9)),
    "long": dict(name="3d-200x200x100", nx=96, ny=9, nz=9, coarse=(32, 3, 3)),
    "m121": dict(name="3d-200x200x100", nx=24, ny=24, nz=24, coarse=(12, 12, 12)),
    "lines": dict(name="3d-64x64x64-lines-a5", nx=16, ny=16, nz=16),
}


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("cname", list(CASES))
def test_panel_basis_against_the_oracle(cname, precision):
    from paper_1705_05783_gb300 import cams
    case = make_case(**CASES[cname], precision=precision, sigma=0.5)
    h, bc, keep = gpu_handle(case)
    try:
        rng = np.random.default_rng(5)
        p = rng.uniform(-0.2, 1.1, case.N)
        if len(case.inp["fix_cell"]):
            p[case.inp["fix_cell"]] = case.inp["fix_value"]
        cams.cams_assemble(h, p, p, case.inp["dt"], bc)
        cams.cams_update_basis(h, True)
        lin = oracle.assemble(case.pb, p, p, case.inp["dt"])
        wb = build_wirebasket(case.pb.grid, case.w.coarse)
        Ab = basis_operator(case.pb, case.w.basis, lin.rho, lin.c, p, case.inp["dt"])
        P = prolongation(Ab, wb).to_csr(wb.Nc)
        got, vals, cols = p_from_gpu(h, case.N, wb.Nc)
        assert np.all(vals[cols < 0] == 0.0)
        # FP32 rounds at 2^-24 instead of 2^-53
        tol = p_tolerance(Ab, wb) * (2.0 ** 29 if precision else 1.0)
        assert abs(got - P).max() <= tol
    finally:
        cams.cams_destroy(h)
