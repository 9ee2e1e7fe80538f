"""The device memory that finished csc2d_solve calls keep for later ones: how it is given
back, and what becomes of it when the device is reset between two calls."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests.test_gpu_csc2d import capi  # noqa: E402,F401

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RESET = r"""
import ctypes
import sys

import numpy as np

sys.path.insert(0, sys.argv[1])
from paper_1705_10087_gb300 import capi, synth

try:
    rt = ctypes.CDLL("/usr/local/cuda/lib64/libcudart.so")
except OSError:
    sys.exit(77)
pbs = [synth.make_problem2d(K=3, P=1, h=4, w=5, H=H, W=W, rho=0.01, sigma=0.05, seed=H)
       for H, W in ((40, 60), (300, 200))]


def solve():
    out = []
    for pb in pbs:
        Z = np.zeros((3, pb.X.shape[1] - 3, pb.X.shape[2] - 4), np.float32)
        status, E, _ = capi.csc2d_solve(pb.D, pb.X, 0.5, 1e-6, Z_out=Z)
        assert status == capi.CSC_OK
        out.append((E, Z))
    return out


def same(a, b):
    return all(x[0] == y[0] and np.array_equal(x[1], y[1]) for x, y in zip(a, b))


want = solve()
assert same(solve(), want)
for sizes in ([1 << 20] * 32 + [32 << 20] * 4, [8 << 20] * 8):
    assert rt.cudaDeviceReset() == 0
    # a new owner: its allocations get the addresses of what the reset took
    owned = []
    for n in sizes:
        p = ctypes.c_void_p()
        assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(n)) == 0
        assert rt.cudaMemset(p, 0x5A, ctypes.c_size_t(n)) == 0
        owned.append((p, n))
    assert same(solve(), want)
    assert same(solve(), want)
    for p, n in owned:
        got = np.empty(n, np.uint8)
        assert rt.cudaMemcpy(ctypes.c_void_p(got.ctypes.data), p, ctypes.c_size_t(n), 2) == 0
        assert (got == 0x5A).all()
"""


def test_a_device_reset_ends_the_kept_memory(capi):  # noqa: F811
    # (a process of its own: the reset ends its context)
    r = subprocess.run([sys.executable, "-c", RESET, ROOT], capture_output=True, text=True,
                       timeout=300)
    if r.returncode == 77:
        pytest.skip("no CUDA runtime library to reset the device with")
    assert r.returncode == 0, r.stdout + r.stderr


def test_trim_gives_the_kept_memory_back(capi):  # noqa: F811
    D = torch.randn((8, 1, 8, 8), device="cuda")
    X = torch.randn((1, 512, 512), device="cuda")
    need = 3 * 4 * 8 * 505 * 505  # beta0, r and Z alone

    def solve_and_free_bytes():
        capi.csc2d_solve(D, X, 1e6, 1e-6)  # (lambda above lambda_max: Z = 0)
        return torch.cuda.mem_get_info()[0]

    solve_and_free_bytes()  # (kernels loaded)
    capi.csc2d_trim()
    empty = torch.cuda.mem_get_info()[0]
    for _ in range(2):
        assert solve_and_free_bytes() <= empty - need
        capi.csc2d_trim()
        assert torch.cuda.mem_get_info()[0] == empty
    capi.csc2d_trim()  # (nothing left: no effect)
    assert torch.cuda.mem_get_info()[0] == empty
