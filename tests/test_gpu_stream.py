"""The streaming FP64 kernels at the edges of their split of the grid: pieces
of 256 (or 1024) columns, runs of planes that share a face, one cluster for
the smallest calls.

Tolerances: a residual is a sum of eight products in another order, a few
ulps of the terms' magnitudes; a matrix entry is a product of sums of two,
1e-13 relative to the largest entry as in the small-grid parity tests."""
import numpy as np
import pytest

import oracle

from _cases import gpu_handle, make_case, matrix_from_gpu
from test_gpu_parity import _rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cams():
    from paper_1705_05783_gb300 import cams
    return cams


# one cell; one piece; the last cluster size and the first grid beyond it;
# one column; flat, thin and ragged grids; two and more planes a run
@pytest.mark.parametrize("n", [(1, 1, 1), (40, 40, 1), (32, 32, 32), (32, 32, 33), (1025, 1, 3), (1, 1, 77),
                               (3, 257, 5), (181, 181, 1), (97, 101, 103), (128, 65, 130)])
def test_noalloc_residual_over_the_split(cams, n):
    import torch
    nx, ny, nz = n
    N = nx * ny * nz
    gen = torch.Generator(device="cuda").manual_seed(N)
    d, ax, ay, az, f, p = (torch.rand(nz, ny, nx, generator=gen, device="cuda", dtype=torch.float64) - 0.3
                           for _ in range(6))
    want, mag = f - d * p, f.abs() + (d * p).abs()
    for a, dim in ((ax, 2), (ay, 1), (az, 0)):
        m = a.shape[dim]
        c = a.narrow(dim, 1, m - 1) if m > 1 else a.narrow(dim, 0, 0)
        lo, up = p.narrow(dim, 0, max(m - 1, 0)), p.narrow(dim, 1, m - 1) if m > 1 else p.narrow(dim, 0, 0)
        want.narrow(dim, 1 if m > 1 else 0, m - 1).sub_(c * lo)
        mag.narrow(dim, 1 if m > 1 else 0, m - 1).add_((c * lo).abs())
        want.narrow(dim, 0, m - 1).sub_(c * up)
        mag.narrow(dim, 0, m - 1).add_((c * up).abs())
        a.narrow(dim, 0, 1).fill_(float("nan"))          # outside the grid: never used
    r = torch.full((N,), float("nan"), device="cuda", dtype=torch.float64)
    args = [v.reshape(-1).contiguous() for v in (d, ax, ay, az, f, p)]
    code, norm = cams.cams_residual_norm_noalloc(nx, ny, nz, *args, r, torch.cuda.current_stream().cuda_stream)
    assert code == cams.CAMS_OK
    assert bool(((r - want.reshape(-1)).abs() <= 32 * np.finfo(float).eps * mag.reshape(-1)).all())
    assert abs(norm - r.norm().item()) <= 1e-12 * norm
    again = cams.cams_residual_norm_noalloc(nx, ny, nz, *args, None, torch.cuda.current_stream().cuda_stream)
    assert again == (cams.CAMS_OK, norm)


@pytest.mark.parametrize("jacobian", [0, 1])
@pytest.mark.parametrize("case", [dict(name="3d-200x200x100", nx=140, ny=120, nz=65, coarse=(10, 10, 5)),
                                  dict(name="3d-100x100x50-wells", nx=140, ny=120, nz=65, coarse=(10, 10, 5)),
                                  dict(name="3d-64x64x64-lines-a5", nx=112, ny=104, nz=88)],
                         ids=["dirichlet", "wells", "lines"])
def test_assembly_on_runs_of_planes(cams, case, jacobian):
    case = make_case(**case)
    h, bc, keep = gpu_handle(case, jacobian=jacobian)
    try:
        N, nx, ny = case.N, case.w.nx, case.w.ny
        rng = np.random.default_rng(3)
        p_nu, p_n = rng.uniform(-0.2, 1.1, N), rng.uniform(-0.2, 1.1, N)
        if len(case.inp["fix_cell"]):
            p_nu[case.inp["fix_cell"]] = case.inp["fix_value"]
        eps = cams.cams_assemble(h, p_nu, p_n, case.inp["dt"], bc)
        lin = oracle.assemble(case.pb, p_nu, p_n, case.inp["dt"], **(dict(full_jacobian=True) if jacobian else {}))
        A = lin.A.tocsr()
        i = np.arange(N)
        got = matrix_from_gpu(h, N)
        assert _rel(got[0], A.diagonal()) < 1e-13
        up = cams.cams_get(h, cams.CAMS_Q_MATRIX_UPPER, np.zeros(3 * N)) if jacobian else None
        for k, (off, ok) in enumerate(((1, i % nx > 0), (nx, (i // nx) % ny > 0), (nx * ny, i // (nx * ny) > 0))):
            lo = np.zeros(N)
            lo[off:] = A.diagonal(-off)
            assert not lo[~ok].any()
            assert _rel(got[1 + k], lo) < 1e-13
            if jacobian:
                tr = np.zeros(N)
                tr[off:] = A.diagonal(off)
                assert _rel(up[k * N:(k + 1) * N], tr) < 1e-13
        assert _rel(cams.cams_get(h, cams.CAMS_Q_RHS, np.zeros(N)), lin.f) < 1e-12
        want = np.linalg.norm(lin.eps)
        assert abs(eps - want) <= 1e-11 * want
    finally:
        cams.cams_destroy(h)


@pytest.mark.parametrize("n", [(256, 256, 256), (40, 40, 1)])
def test_noalloc_residual_after_another_calls_error(cams, n):
    """An error left pending by an earlier call (a convolution that no CTA's
    shared memory holds: refused by the host, nothing launched) is not the
    residual's: the call succeeds, and its kernels are done when it returns."""
    import torch
    N = int(np.prod(n))
    gen = torch.Generator(device="cuda").manual_seed(1)
    args = [torch.rand(N, generator=gen, device="cuda", dtype=torch.float64) for _ in range(6)]
    s = torch.cuda.current_stream()
    want = cams.cams_residual_norm_noalloc(*n, *args, None, s.cuda_stream)
    assert want[0] == cams.CAMS_OK
    t = torch.zeros(16, device="cuda")
    with pytest.raises(cams.CamsError):
        cams.cams_net_conv_forward(1, 40, 5000, 1, t, t, t, 0, t)
    torch.cuda.synchronize()
    got = cams.cams_residual_norm_noalloc(*n, *args, None, s.cuda_stream)
    assert s.query()
    assert got == want


# planes of fewer columns than a CTA has threads: one column, fewer than a warp,
# a CTA and a bit more, with runs of one plane and of several
@pytest.mark.parametrize("n", [(1, 1, 1025), (1, 1, 1000003), (2, 3, 4001), (4, 4, 65537), (5, 7, 30011), (17, 17, 4099),
                               (33, 33, 67)])
def test_noalloc_residual_of_thin_grids(cams, n):
    import torch
    nx, ny, nz = n
    N, eps = nx * ny * nz, np.finfo(float).eps
    gen = torch.Generator(device="cuda").manual_seed(N)
    d, ax, ay, az, f, p = (torch.rand(N, generator=gen, device="cuda", dtype=torch.float64) - 0.3 for _ in range(6))
    i = torch.arange(N, device="cuda")
    want, mag = f - d * p, f.abs() + (d * p).abs()
    for a, st, c in ((ax, 1, i % nx), (ay, nx, i // nx % ny), (az, nx * ny, i // (nx * ny))):
        up = i[c > 0]                                  # the face between up - st and up
        t = a[up] * p[up - st]
        want[up] -= t
        mag[up] += t.abs()
        t = a[up] * p[up]
        want[up - st] -= t
        mag[up - st] += t.abs()
        a[c == 0] = float("nan")                       # outside the grid: never used
    r = torch.full((N,), float("nan"), device="cuda", dtype=torch.float64)
    code, norm = cams.cams_residual_norm_noalloc(nx, ny, nz, d, ax, ay, az, f, p, r,
                                                 torch.cuda.current_stream().cuda_stream)
    assert code == cams.CAMS_OK
    assert bool(((r - want).abs() <= 32 * eps * mag).all())
    assert abs(norm - r.norm().item()) <= 1e-12 * norm


def test_a_thin_grid_costs_as_much_as_a_long_one(cams):
    """A column of 10^6 cells along z takes no more than five times what the
    same cells along x do (30 times with a CTA for every plane of one cell)."""
    import torch
    N = 1000000
    args = [torch.ones(N, device="cuda", dtype=torch.float64) for _ in range(6)]
    s = torch.cuda.current_stream()

    def best(n):
        times = []
        for _ in range(8):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record(s)
            assert cams.cams_residual_norm_noalloc(*n, *args, None, s.cuda_stream)[0] == cams.CAMS_OK
            b.record(s)
            b.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)
    assert best((1, 1, N)) <= 5 * best((N, 1, 1))


@pytest.mark.parametrize("mu, dz", [(1e3, 0.5), (1.0, 0.5), (1e-3, 1e-170)])
def test_transmissibilities_over_the_exponent_range(cams, mu, dz):
    """The two-point formula as it stands, wherever it is finite, for
    permeabilities from the smallest normal number to 1.6e308: sums of two that
    overflow, ratios that underflow.  The formula and the library's form of it are
    each within five roundings of the exact value (16 eps covers both), as far as
    the formula's own quotients are normal numbers."""
    k = np.array([1e-13, 1.0, 3e5, 1e-290, 1e290, 1.6e308, 1.2e308, 1.6e308, 3e-308, 1e200, 1e-200, 1e-13, 1e140, 1e-140,
                  1e138, 1e308, 1e150, 7.0])
    nx, h = len(k), (1.0, 0.25, dz)
    g = cams.cams_grid(nx, 2, 2, *h)
    kf = np.tile(k, 4)
    o = cams.make_options((2, 2, 2))
    hd = cams.cams_setup(g, cams.cams_fluid(0, 0.1, 1.0, mu, 1.0), o, kf)
    try:
        T = cams.cams_get(hd, cams.CAMS_Q_TRANS, np.zeros(3 * 4 * nx)).reshape(3, 4 * nx)
    finally:
        cams.cams_destroy(hd)
    eps, tiny = np.finfo(float).eps, np.finfo(float).tiny
    with np.errstate(all="ignore"):
        def want(ka, kb, d):
            area = {0: np.float64(h[1]) * h[2], 1: np.float64(h[0]) * h[2], 2: np.float64(h[0]) * h[1]}[d]
            qa, qb = h[d] / (2.0 * (ka / mu)), h[d] / (2.0 * (kb / mu))
            t = area / (qa + qb)
            ok = np.isfinite(t) & (t >= tiny) & (qa + qb >= tiny)
            for q, v in ((qa, ka), (qb, kb)):
                ok &= np.isfinite(q) & (q >= tiny) & np.isfinite(2.0 * (v / mu)) & (v / mu >= tiny)
            return t, ok
        i = np.arange(4 * nx)
        used = 0
        for d, st, c in ((0, 1, i % nx), (1, nx, i // nx % 2), (2, 2 * nx, i // (2 * nx))):
            up = i[c > 0]
            t, ok = want(kf[up - st], kf[up], d)
            assert np.all(np.abs(T[d][up] - t)[ok] <= 16 * eps * t[ok])
            used += int(ok.sum())
    assert used >= 40


def test_transmissibilities_are_correctly_rounded(cams):
    """T = 2 A k_a k_b / (h mu (k_a + k_b)) to one rounding, u = 2^-53: numerator,
    denominator and the quotient's remainder carry their rounding errors, so what is
    left beside the last rounding is of the order of u^2 (a hundredth of u here)."""
    nx, ny, nz, h, mu = 45, 34, 23, (0.3, 1.7, 0.9), 0.77
    N = nx * ny * nz
    k = np.exp(3.0 * np.random.default_rng(8).standard_normal(N))
    k[::97] *= 1e40
    hd = cams.cams_setup(cams.cams_grid(nx, ny, nz, *h), cams.cams_fluid(0, 0.1, 1.0, mu, 1.0),
                         cams.make_options((5, 2, 23)), k)
    try:
        T = cams.cams_get(hd, cams.CAMS_Q_TRANS, np.zeros(3 * N)).reshape(3, N)
    finally:
        cams.cams_destroy(hd)
    Q = np.longdouble
    assert np.finfo(Q).eps <= 2.0 ** -60
    i = np.arange(N)
    for d, st, c in ((0, 1, i % nx), (1, nx, i // nx % ny), (2, nx * ny, i // (nx * ny))):
        up = i[c > 0]
        ka, kb = k[up - st].astype(Q), k[up].astype(Q)
        area = Q(h[0]) * Q(h[1]) * Q(h[2]) / Q(h[d])
        t = 2 * area * ka * kb / (Q(h[d]) * Q(mu) * (ka + kb))
        assert float((np.abs(T[d][up] - t) / t).max()) <= 1.01 * 2.0 ** -53
