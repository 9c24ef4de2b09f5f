"""The network's FP32 convolutions on both sides of the lines between the general
kernels (few warps, where latency is the time) and the tiled ones: which of them
the weight gradient takes, and the values of the tiled ones at batches that reach
them (tests/test_gpu_conv.py has the small ones, and the bounds' reasons)."""
import numpy as np
import pytest

from _cases import gpu_handle, make_case
from test_gpu_conv import U, _ref, env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,S,ci,co", [(300, 2, 3, 32), (130, 5, 12, 33), (20, 11, 32, 17), (70, 7, 9, 16), (16, 9, 33, 9),
                                       (64, 12, 17, 8)])
def test_tiled_convolutions_match_fp64(env, B, S, ci, co):  # noqa: F811
    torch, cams = env
    g = torch.Generator().manual_seed(B * 1000 + S)
    x = torch.randn(B, ci, S, S, S, generator=g)
    w = torch.randn(co, ci, 3, 3, 3, generator=g)
    b = torch.randn(co, generator=g)
    gy = torch.randn(B, co, S, S, S, generator=g) * (torch.rand(B, co, S, S, S, generator=g) > 0.3)
    dev = [t.cuda().contiguous() for t in (x, w, b, gy)]
    y, gx = torch.full_like(dev[3], float("nan")), torch.full_like(dev[0], float("nan"))
    gw, gb = torch.full_like(dev[1], float("nan")), torch.full_like(dev[2], float("nan"))
    cams.cams_net_conv_forward(B, S, ci, co, dev[0], dev[1], dev[2], 0, y)
    cams.cams_net_conv_backward(B, S, ci, co, dev[0], dev[1], dev[3], None, gx, gw, gb)
    torch.cuda.synchronize()
    ref = _ref(torch, x, w, b, gy)
    mag = _ref(torch, x.abs(), w.abs(), b.abs(), gy.abs())
    for got, r, m, n in zip((y, gx, gw, gb), ref, mag, (27 * ci + 1, 27 * co, B * S ** 3, B * S ** 3)):
        err = (got.double().cpu() - r).abs()
        assert bool((err <= (n + 2) * U * m + 1e-30).all()), float((err / (m + 1e-30)).max())


# kernels of a weight gradient: the general one, or the tiles and the sum of their
# chunks.  (One patch and three of 6^3 took 1.5 and 1.9 times as long in tiles.)
@pytest.mark.parametrize("B,S,ci,co,kernels", [(1, 11, 32, 8, 1), (3, 6, 11, 10, 1), (1, 11, 32, 32, 1), (4, 11, 32, 8, 2),
                                               (64, 3, 12, 32, 2), (1, 4, 256, 256, 2)])
def test_which_kernels_a_weight_gradient_takes(env, B, S, ci, co, kernels):  # noqa: F811
    torch, cams = env
    h, bc, keep = gpu_handle(make_case("2d-40x40", nx=20, ny=20, coarse=(5, 5, 1)))   # (it counts the launches)
    try:
        x, gy = torch.zeros(B, ci, S ** 3, device="cuda"), torch.zeros(B, co, S ** 3, device="cuda")
        w, gw, gb = torch.zeros(co, ci, 27, device="cuda"), torch.zeros(co, ci, 27, device="cuda"), torch.zeros(co, device="cuda")
        n0 = cams.cams_get(h, cams.CAMS_Q_LAUNCHES, np.zeros(1))[0]
        cams.cams_net_conv_backward(B, S, ci, co, x, w, gy, None, None, gw, gb)
        torch.cuda.synchronize()
        assert cams.cams_get(h, cams.CAMS_Q_LAUNCHES, np.zeros(1))[0] - n0 == kernels
    finally:
        cams.cams_destroy(h)


@pytest.mark.parametrize("what", ["an inf", "all nan", "nan weights"])
def test_non_finite_inputs_take_no_longer_than_without_tiles(env, what):  # noqa: F811
    """A sum that padding or a zero gradient may have made non-finite is formed again
    by a whole CTA: the call stays within three times its time on finite inputs
    plus the general kernel's 1.4 ms (ten times that with a thread a sum), and
    what is non-finite is what FP64 makes non-finite from the pairs of voxels
    inside the patch with a gradient."""
    torch, cams = env
    B, S, ci, co = 64, 11, 32, 32
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(B, ci, S, S, S, generator=g, device="cuda")
    w = torch.randn(co, ci, 27, generator=g, device="cuda")
    gy = torch.randn(B, co, S, S, S, generator=g, device="cuda")
    gy[:, :, 0, 0, :3] = 0.0
    gw, gb, gx = torch.zeros_like(w), torch.zeros(co, device="cuda"), torch.zeros_like(x)

    def best():
        ts = []
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            cams.cams_net_conv_backward(B, S, ci, co, x, w, gy, None, gx, gw, gb)
            b.record()
            b.synchronize()
            ts.append(a.elapsed_time(b))
        return min(ts)
    base = best()
    finite = gw.clone()
    if what == "an inf":
        x[5, 7, 0, 0, 0] = float("inf")
        # g is zero at the voxel itself and beside it along x: those two taps stay as they were
        # (dx = 0 and -1 of dy = dz = 0), other channels too; others see the infinity
        want = torch.zeros(co, ci, 27, dtype=torch.bool, device="cuda")
        for t in range(27):
            dx, dy, dz = t % 3 - 1, t // 3 % 3 - 1, t // 9 - 1
            if dx <= 0 and dy <= 0 and dz <= 0 and not (dy == 0 and dz == 0):
                want[:, 7, t] = True
    elif what == "all nan":
        x[:] = float("nan")
        want = torch.ones(co, ci, 27, dtype=torch.bool, device="cuda")
    else:
        w[:] = float("nan")
        want = torch.zeros(co, ci, 27, dtype=torch.bool, device="cuda")
    t = best()
    assert bool((torch.isfinite(gw) != want).all())
    if what == "an inf":
        rest = ~want
        rest[:, 7] = False
        assert torch.equal(gw[rest], finite[rest])
        assert bool(((gw - finite).abs() <= 2 * B * S ** 3 * U * 64.0)[~want].all())
    assert bool(torch.isnan(gx).all()) == (what == "nan weights")
    assert t <= 3 * base + 1.4
