"""The backward error of the two-ended coarse factorisation as the solve uses it.

An iteration without smoothing adds P x, A_c x = R r, to the iterate, and P is one
at the coarse vertices, so from p = 0 the iterate holds x there.  A_c, P and r are
read from the engine; R r = P^T r is formed in extended precision.

Tolerance.  For an SPD A_c, elimination in any order and substitution give
(A_c + dA) x = b, |dA| <= 3 (m + 2) u |L| D |L|^T with at most m + 1 products a
sum (Higham, Accuracy and Stability, Thm 10.4 in L D L^T form), and |L| D |L|^T
<= sqrt(a_ii a_jj) entrywise.  The substitution multiplies by inverses of L's
32-row diagonal blocks, which adds 2 * 32 u |L_J||L_J^-1| times the same; kappa
below is the largest row sum of |L_J||L_J^-1| in the two-ended order, from a
factorisation here.  All of it stays inside the band, whichever end the
elimination starts from.  b carries the rounding of its sums, u P^T |r| times the
additions that a product goes through: a cell's turn of a thread (at most the
cells of a dual block over 32), the folds of a warp and over 8 warps, 8 blocks,
below 64 in all.  (u = 2^-52, twice the unit roundoff, for the terms of second order.)"""
import numpy as np
import pytest

from _cases import coarse_from_gpu, gpu_handle, make_case, p_from_gpu
from test_gpu_twist import GRIDS

pytestmark = pytest.mark.gpu

KCB = 32


def _kappa(A):
    """Largest row sum of |L_J||L_J^-1| over the diagonal blocks of 32 rows."""
    C = np.linalg.cholesky(A)
    L = C / np.diag(C)
    worst = 1.0
    for j in range(0, len(A), KCB):
        B = L[j:j + KCB, j:j + KCB]
        worst = max(worst, (np.abs(B) @ np.abs(np.linalg.inv(B))).sum(axis=1).max())
    return worst


@pytest.mark.parametrize("kw", GRIDS, ids=[f"{g['nx']}x{g['ny']}x{g.get('nz', 1)}" for g in GRIDS])
def test_backward_error_of_the_coarse_solve(kw):
    from paper_1705_05783_gb300 import cams
    case = make_case(**kw, sigma=1.5, n_pre=0, n_post=0)
    h, bc, keep = gpu_handle(case)
    try:
        if cams.cams_get_schedule(h)[1] != 1:
            pytest.skip("no cluster coarse solve here")
        N = case.N
        zero = np.zeros(N)
        cams.cams_assemble(h, zero, np.random.default_rng(1).uniform(0, 1, N), case.inp["dt"], bc)
        cams.cams_update_basis(h, True)
        sizes = cams.cams_get_int(h, cams.CAMS_Q_SIZES, np.zeros(8, np.int32))
        Nc, nc = int(sizes[1]), [int(v) for v in sizes[2:5]]
        order = cams.cams_get_int(h, cams.CAMS_Q_COARSE_ORDER, np.zeros(Nc + 1, np.int32))
        m, pos = int(order[0]), order[1:]
        A, _ = coarse_from_gpu(h, nc)
        P, _, _ = p_from_gpu(h, N, Nc)
        r = cams.cams_get(h, cams.CAMS_Q_RESIDUAL, np.zeros(N))
        cams.cams_iterate(h, 1)
        p = cams.cams_get(h, cams.CAMS_Q_PRESSURE, np.zeros(N))
    finally:
        cams.cams_destroy(h)
    b, bmag = np.zeros(Nc, np.longdouble), np.zeros(Nc)
    coo = P.tocoo()
    np.add.at(b, coo.col, coo.data.astype(np.longdouble) * r[coo.row].astype(np.longdouble))
    np.add.at(bmag, coo.col, np.abs(coo.data * r[coo.row]))
    # the vertex of coarse node J: the one cell whose row of P is J's unit vector
    x = np.full(Nc, np.nan)
    rows = P.tocsr()
    one = np.flatnonzero((np.diff(rows.indptr) >= 1) & (np.asarray((rows == 1.0).sum(axis=1)).ravel() == 1)
                         & (np.asarray((rows != 0.0).sum(axis=1)).ravel() == 1))
    off = [w // 2 for w in case.w.coarse]
    nx, ny = case.w.nx, case.w.ny
    for i in one:
        c = (i % nx, i // nx % ny, i // (nx * ny))
        if all((c[d] - off[d]) % case.w.coarse[d] == 0 for d in range(3)):
            J = int(rows[i].indices[np.argmax(rows[i].data)])
            x[J] = p[i]
    assert np.isfinite(x).all()
    # the two-ended order: H rows from either end, then the middle
    H = KCB * ((Nc - m) // (2 * KCB)) if Nc > m else 0
    place = np.empty(Nc, int)
    place[pos] = np.arange(Nc)                                    # natural node at a band position
    two = np.concatenate([place[:H], place[::-1][:H], place[H:Nc - H]])
    kappa = max(_kappa(A[np.ix_(two, two)]), _kappa(A[np.ix_(place, place)]))
    u = 2.0 ** -52
    res = np.abs(b - A.astype(np.longdouble) @ x.astype(np.longdouble)).astype(float)
    d = np.sqrt(np.diag(A))
    inside = np.abs(pos[:, None] - pos[None, :]) <= m
    assert max(case.w.coarse) ** 3 // 32 + 5 + 8 + 8 < 64
    bound = u * (3 * (m + 2) + 2 * KCB * kappa) * d * (inside @ (d * np.abs(x))) + 64 * u * bmag
    print(f"{Nc} nodes, m {m}, kappa {kappa:.1f}: largest residual / bound {np.max(res / bound):.2e}")
    assert np.all(res <= bound)
