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
# middle 62); 3x4x20 = 240, m 16 (H 96, middle 48); 4x4x4 = 64 (not split);
# 13x13x13 = 2197, m 183 (the two bands' tiles are more than 152: two a CTA)
GRIDS = [dict(name="2d-40x40", nx=60, ny=60, coarse=(5, 5, 1)),
         dict(name="3d-200x200x100", nx=15, ny=15, nz=27, coarse=(3, 3, 3)),
         dict(name="3d-200x200x100", nx=18, ny=18, nz=21, coarse=(3, 3, 3)),
         dict(name="2d-40x40", nx=570, ny=3, coarse=(3, 3, 1)),
         dict(name="3d-100x100x50-wells", nx=12, ny=16, nz=80, coarse=(4, 4, 4)),
         dict(name="3d-200x200x100", nx=12, ny=12, nz=12, coarse=(3, 3, 3)),
         dict(name="3d-200x200x100", nx=39, ny=39, nz=39, coarse=(3, 3, 3))]


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


@pytest.mark.parametrize("kw", GRIDS, ids=[f"{g['nx']}x{g['ny']}x{g.get('nz', 1)}" for g in GRIDS])
def test_two_ended_inverse_factor(kw, monkeypatch):
    """The mixed preconditioner's coarse solve by the inverse factors of the
    two bands against its substitution with the same FP64 factor's FP32 copy:
    both are FP32 solves of one SPD system, so an iterate's correction agrees
    to FP32's unit roundoff times the coarse conditioning (mild field: below
    1e4), and iterating on brings both residuals down alike."""
    from paper_1705_05783_gb300 import cams
    case = make_case(**kw, sigma=0.5, n_pre=0, n_post=1, precision=1)
    p0 = np.random.default_rng(2).uniform(0, 1, case.N)
    runs = []
    for off in ("1", "0"):
        monkeypatch.setenv("CAMS_COARSE_INV", off)
        h, bc, keep = gpu_handle(case)
        try:
            cams.cams_assemble(h, p0, p0, case.inp["dt"], bc)
            cams.cams_update_basis(h, True)
            norms = cams.cams_iterate(h, 4)
            runs.append((np.asarray(norms), cams.cams_get(h, cams.CAMS_Q_PRESSURE, np.zeros(case.N))))
        finally:
            cams.cams_destroy(h)
    (na, pa), (nb, pb) = runs
    assert np.all(np.abs(na - nb) <= 1e-3 * nb[0])
    assert np.abs(pa - pb).max() <= 1e4 * 2.0 ** -24 * np.abs(pb - p0).max()


def test_one_band_with_two_tiles_a_cta():
    """A half-width of 273 (16x16x17 coarse nodes): too wide to be split, and
    more tiles than SMs.  R A P = L D L^T within the componentwise
    backward-error bound of the factorisation's own test."""
    from paper_1705_05783_gb300 import cams
    from test_gpu_coarse_factor import _factor
    case = make_case("3d-200x200x100", nx=48, ny=48, nz=51, coarse=(3, 3, 3), sigma=1.0)
    A, L, d, m = _factor(cams, case)
    assert m == 273 and np.all(d > 0)
    bound = (m + 2) * np.finfo(float).eps * (np.abs(L) * d) @ np.abs(L).T
    assert (np.abs((L * d) @ L.T - A) - 2.0 * bound).max() <= 0.0
