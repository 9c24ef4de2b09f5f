"""The two-ended coarse factorisation and its solve against the one-ended ones
(the schedule without the cluster solve), at the sizes where the split can go
wrong: the smallest coarse grid that is split, middles of m rows and of m + 63,
rows past the last block, a chain (m = 1), and a grid too small to be split.

Both solve the same SPD system backward stably, so iterates agree to the
coarse condition number times the unit roundoff; the schedules' test holds
them to 1e-12 relative on such grids, and so does this one."""
import numpy as np
import pytest

from _cases import gpu_handle, make_case

pytestmark = pytest.mark.gpu

# coarse nodes: 12x12 = 144, m 13 (H 64, middle 16); 5x5x9 = 225, m 31 (H 96,
# middle 33); 6x6x7 = 252, m 43 (H 96, middle 60); 190x1 chain, m 1 (H 64,
# middle 62); 3x4x20 = 240, m 16 (H 96, middle 48); 4x4x4 = 64 (not split)
GRIDS = [dict(name="2d-40x40", nx=60, ny=60, coarse=(5, 5, 1)),
         dict(name="3d-200x200x100", nx=15, ny=15, nz=27, coarse=(3, 3, 3)),
         dict(name="3d-200x200x100", nx=18, ny=18, nz=21, coarse=(3, 3, 3)),
         dict(name="2d-40x40", nx=570, ny=3, coarse=(3, 3, 1)),
         dict(name="3d-100x100x50-wells", nx=12, ny=16, nz=80, coarse=(4, 4, 4)),
         dict(name="3d-200x200x100", nx=12, ny=12, nz=12, coarse=(3, 3, 3))]


@pytest.mark.parametrize("kw", GRIDS, ids=[f"{g['nx']}x{g['ny']}x{g.get('nz', 1)}" for g in GRIDS])
def test_two_ended_coarse_solve(kw):
    from paper_1705_05783_gb300 import cams
    case = make_case(**kw, sigma=1.0, n_pre=0, n_post=1)
    h, bc, keep = gpu_handle(case)
    try:
        if cams.cams_get_schedule(h)[1] != 1:
            pytest.skip("no cluster coarse solve here")
        p0 = np.random.default_rng(2).uniform(0, 1, case.N)
        runs, factors = [], []
        for cl in (1, 0, 1):
            cams.cams_set_schedule(h, coarse_cluster=cl)
            cams.cams_assemble(h, p0, p0, case.inp["dt"], bc)
            if not runs:
                cams.cams_update_basis(h, True)
            norms = cams.cams_iterate(h, 2)
            runs.append((norms, cams.cams_get(h, cams.CAMS_Q_PRESSURE, np.zeros(case.N))))
            nc = int(cams.cams_get_int(h, cams.CAMS_Q_SIZES, np.zeros(8, np.int32))[1])
            m = int(cams.cams_get_int(h, cams.CAMS_Q_COARSE_ORDER, np.zeros(nc + 1, np.int32))[0])
            factors.append(cams.cams_get(h, cams.CAMS_Q_COARSE_FACTOR, np.zeros(nc * (m + 1))))
        for norms, p in runs[1:]:
            assert np.abs(p - runs[0][1]).max() <= 1e-12 * np.abs(runs[0][1]).max()
        assert np.array_equal(runs[0][1], runs[2][1])
        assert np.array_equal(factors[0], factors[1]) and np.array_equal(factors[0], factors[2])
        # both after a fresh factorisation in the schedule's own layout
        cams.cams_update_basis(h, True)
        cams.cams_assemble(h, p0, p0, case.inp["dt"], bc)
        cams.cams_iterate(h, 2)
        assert np.array_equal(cams.cams_get(h, cams.CAMS_Q_PRESSURE, np.zeros(case.N)), runs[0][1])
    finally:
        cams.cams_destroy(h)
