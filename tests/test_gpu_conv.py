"""The network's FP32 convolution kernels at the sizes where their tiling can
go wrong: patches from one voxel to the first size past the tiles, rows that
are and are not whole strips, channel counts around the tiles of 8 and 32.
Reference: torch's convolution and its gradients in FP64.  Every result is a
sum of n products formed in some order in FP32, so its error is at most
(n + 2) u times the sum of the products' magnitudes, u = 2^-24."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    from paper_1705_05783_gb300 import cams
    return torch, cams


def _ref(torch, x, w, b, gy):
    """conv(x, w) + b, and the gradients of sum(conv * gy), on the CPU in FP64."""
    x, w, b = (t.double().cpu().requires_grad_(True) for t in (x, w, b))
    y = torch.nn.functional.conv3d(x, w, b, padding=1)
    y.backward(gy.double().cpu())
    return y.detach(), x.grad, w.grad, b.grad


@pytest.mark.parametrize("B,S,ci,co", [(1, 1, 1, 1), (2, 2, 3, 8), (3, 4, 9, 7), (2, 5, 8, 9), (5, 6, 12, 32),
                                       (3, 11, 32, 8), (2, 12, 33, 17), (1, 13, 40, 33), (120, 3, 5, 4),
                                       (1, 30, 3, 2)])
def test_convolutions_match_fp64(env, B, S, ci, co):
    torch, cams = env
    g = torch.Generator().manual_seed(B * 1000 + S)
    x = torch.randn(B, ci, S, S, S, generator=g)
    w = torch.randn(co, ci, 3, 3, 3, generator=g)
    b = torch.randn(co, generator=g)
    gy = torch.randn(B, co, S, S, S, generator=g) * (torch.rand(B, co, S, S, S, generator=g) > 0.3)
    act = torch.randn(B, ci, S, S, S, generator=g)
    dev = [t.cuda().contiguous() for t in (x, w, b, gy, act)]
    y, gx = torch.full_like(dev[3], float("nan")), torch.full_like(dev[0], float("nan"))
    gw, gb = torch.full_like(dev[1], float("nan")), torch.full_like(dev[2], float("nan"))
    cams.cams_net_conv_forward(B, S, ci, co, dev[0], dev[1], dev[2], 1, y)
    cams.cams_net_conv_backward(B, S, ci, co, dev[0], dev[1], dev[3], dev[4], gx, gw, gb)
    gw2, gb2 = torch.zeros_like(gw), torch.zeros_like(gb)
    cams.cams_net_conv_backward(B, S, ci, co, dev[0], dev[1], dev[3], None, None, gw2, gb2)
    torch.cuda.synchronize()
    assert torch.equal(gw, gw2) and torch.equal(gb, gb2)          # reproducible, with and without gx
    ref = _ref(torch, x, w, b, gy)
    mag = _ref(torch, x.abs(), w.abs(), b.abs(), gy.abs())
    keep = (act > 0).double()
    for got, r, m, n in ((y, ref[0].clamp_min(0), mag[0], 27 * ci + 1), (gx, ref[1] * keep, mag[1], 27 * co),
                         (gw, ref[2], mag[2], B * S ** 3), (gb, ref[3], mag[3], B * S ** 3)):
        err = (got.double().cpu() - r).abs()
        assert bool((err <= (n + 2) * U * m + 1e-30).all()), float((err / (m + 1e-30)).max())


def test_non_finite_inputs_stay_where_they_are(env):
    """Zero padding and zero gradients do not spread a non-finite input: the
    sums run over the voxel pairs inside the patch with a nonzero gradient."""
    torch, cams = env
    B, S, ci, co = 1, 6, 2, 3
    g = torch.Generator().manual_seed(5)
    x = torch.randn(B, ci, S, S, S, generator=g)
    w = torch.randn(co, ci, 3, 3, 3, generator=g)
    gy = torch.randn(B, co, S, S, S, generator=g)
    x[0, 1, 2, 3, S - 1] = float("inf")
    gy[0, :, 1:4, 2:5, S - 2:] = 0.0                              # every pair of that voxel
    w[1, 0, 0, 0, 0] = float("inf")
    dx, dw, dg = x.cuda(), w.cuda(), gy.cuda()
    gx, gw, gb = torch.zeros_like(dx), torch.zeros_like(dw), torch.zeros(co, device="cuda")
    cams.cams_net_conv_backward(B, S, ci, co, dx, dw, dg, None, gx, gw, gb)
    torch.cuda.synchronize()
    assert bool(torch.isfinite(gw).all())
    fin = torch.isfinite(gx.cpu())
    # the tap (-1, -1, -1) of input channel 0 reads gy at v + (1, 1, 1): voxels
    # of the last planes have no such pair and stay finite
    assert bool(fin[0, 1].all()) and bool(fin[0, 0, S - 1].all()) and bool(fin[0, 0, :, S - 1].all())
    assert bool(fin[0, 0, :, :, S - 1].all())


@pytest.mark.parametrize("S,ci,co", [(5, 12, 32), (6, 32, 32), (5, 32, 8)])
def test_tensor_core_conv_is_the_same_in_any_batch(env, S, ci, co):
    """More patches than CTAs (one or two an SM): every CTA runs several, and a
    patch's result is bit for bit the one it has alone."""
    torch, cams = env
    B = 700
    g = torch.Generator().manual_seed(S)
    x = torch.randn(B, ci, S, S, S, generator=g).cuda()
    w = (0.1 * torch.randn(co, ci, 27, generator=g)).cuda()
    b = torch.randn(co, generator=g).cuda()

    def run(xb):
        n = xb.shape[0]
        nb = cams.cams_net_tc_work_bytes(n, S)
        work = torch.full((nb,), 255, dtype=torch.uint8, device="cuda")   # not cleared by the caller
        y = torch.full((n, co, S, S, S), float("nan"), device="cuda")
        assert cams.cams_net_conv_forward_tc(n, S, ci, co, xb, w, b, 1, y, work, nb) == cams.CAMS_OK
        return y

    y = run(x)
    assert bool(torch.isfinite(y).all())
    for k in (0, 1, 151, 152, 303, 304, 456, B - 1):
        assert torch.equal(run(x[k:k + 1].contiguous())[0], y[k]), k
