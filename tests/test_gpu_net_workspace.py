"""The workspace of the weight gradient (cams_net_conv_backward): bounded for any
number of channels, given back with a handle, and of the context that uses it."""
import os
import subprocess
import sys

import pytest

from _cases import gpu_handle, make_case

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MB = 1 << 20


def _backward(cams, torch, B, S, ci, co, seed=0):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(B, ci, S, S, S, generator=gen, device="cuda")
    gy = torch.randn(B, co, S, S, S, generator=gen, device="cuda")
    w = torch.randn(co, ci, 27, generator=gen, device="cuda")
    gw, gb = torch.full_like(w, float("nan")), torch.full((co,), float("nan"), device="cuda")
    return x, gy, gw, gb, lambda: cams.cams_net_conv_backward(B, S, ci, co, x, w, gy, None, None, gw, gb)


@pytest.mark.parametrize("ci, co", [(32, 32), (128, 96), (512, 512), (700, 700)])
def test_workspace_is_bounded_and_given_back(ci, co):
    """At most 64 MB (and the pool's granularity) while the call is queued, nothing
    after a handle is destroyed; with 700 x 700 channels one chunk alone is more
    than that, and the kernel without a workspace runs."""
    import torch
    from paper_1705_05783_gb300 import cams
    B, S = 40, 3
    x, gy, gw, gb, call = _backward(cams, torch, B, S, ci, co)
    call()                                             # (the code is loaded, the pool exists)
    h, bc, keep = gpu_handle(make_case("2d-40x40", nx=20, ny=20, coarse=(5, 5, 1)))
    torch.cuda.synchronize()
    cams.cams_destroy(h)
    before = torch.cuda.mem_get_info()[0]
    call()
    during = torch.cuda.mem_get_info()[0]
    torch.cuda.synchronize()
    assert before - during <= 68 * MB
    h, bc, keep = gpu_handle(make_case("2d-40x40", nx=20, ny=20, coarse=(5, 5, 1)))
    cams.cams_destroy(h)
    assert before - torch.cuda.mem_get_info()[0] <= 4 * MB

    def sums(a, g):                                    # [co][ci][27], in FP64
        t = torch.nn.functional.conv3d(a.double().transpose(0, 1), g.double().transpose(0, 1), padding=1)
        return t.transpose(0, 1).reshape(co, ci, 27)
    # n products in FP32, in any order: n u sum |x| |gy|
    assert bool(((gw.double() - sums(x, gy)).abs() <= B * S ** 3 * 2.0 ** -24 * sums(x.abs(), gy.abs())).all())


RESET = """
import ctypes as C, sys
import numpy as np, torch
torch.zeros(1, device="cuda")
rt = C.CDLL([l.split()[-1] for l in open("/proc/self/maps") if "libcudart" in l][0])
from paper_1705_05783_gb300 import cams
B, S, ci, co = 40, 3, 5, 6
rng = np.random.default_rng(0)
host = [rng.standard_normal(n).astype(np.float32) for n in (B * ci * 27, co * ci * 27, B * co * 27)]
def run():
    dev = []
    for a in [*host, np.zeros(co * ci * 27, np.float32), np.zeros(co, np.float32)]:
        p = C.c_void_p()
        assert rt.cudaMalloc(C.byref(p), C.c_size_t(a.nbytes)) == 0
        assert rt.cudaMemcpy(p, a.ctypes.data_as(C.c_void_p), C.c_size_t(a.nbytes), 1) == 0
        dev.append(p.value)
    x, w, gy, gw, gb = dev
    cams.cams_net_conv_backward(B, S, ci, co, x, w, gy, None, None, gw, gb)
    out = np.zeros(co * ci * 27, np.float32)
    assert rt.cudaMemcpy(out.ctypes.data_as(C.c_void_p), C.c_void_p(gw), C.c_size_t(out.nbytes), 2) == 0
    return out
first = run()
assert first.any()
print("first", flush=True)
assert rt.cudaDeviceReset() == 0
second = run()
assert np.array_equal(first, second)
print("second", flush=True)
"""


def test_the_workspace_is_of_the_present_context():
    r = subprocess.run([sys.executable, "-c", RESET], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "second" in r.stdout, (r.returncode, r.stdout, r.stderr[-2000:])
