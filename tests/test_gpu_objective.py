"""E(Z) of a given Z at the edges of its kernel's loops (csrc/kernels_fp64.cu, obj_pass)
against the FP64 oracle: channel counts around the packed pairs and the passes of 8,
buckets with no, one, an odd number of and more than 64 nonzeros, kernels around the
32-column buckets.  A sample sums at most K L products in double-float, each within
2^-47 of the largest partial sum: 240 x 2^-47 = 2e-12 of the residual and twice that of
its square for the dense case; the bar is 1e-11."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests.test_gpu_parity import capi, cuda  # noqa: E402,F401

CASES = [
    # K, P, L, T, density of Z
    (1, 1, 1, 37, 0.5),
    (3, 1, 5, 300, 0.02),
    (5, 2, 33, 700, 0.01),
    (4, 3, 32, 513, 0.1),
    (6, 4, 40, 600, 1.0),     # every bucket holds more than 64 nonzeros
    (25, 5, 64, 1000, 0.005),
    (20, 7, 64, 3000, 0.1),   # around 64 nonzeros in a bucket: both walks
    (12, 8, 17, 900, 0.02),
    (7, 9, 64, 800, 0.01),
    (3, 11, 129, 1024, 0.05),
    (17, 7, 31, 400, 0.0),
]


@pytest.mark.parametrize("K,P,L,T,density", CASES)
def test_objective_of_any_z_matches_oracle(capi, K, P, L, T, density):  # noqa: F811
    rng = np.random.default_rng(K * 1000 + P * 100 + L)
    D = rng.standard_normal((K, P, L)).astype(np.float32)
    X = rng.standard_normal((P, T)).astype(np.float32)
    Z = rng.standard_normal((K, T - L + 1)).astype(np.float32)
    Z *= rng.random(Z.shape) < density
    E = capi.csc_objective_noalloc(cuda(D), cuda(X), cuda(Z), 0.3)
    Er = oracle.objective(D, X, Z.astype(np.float64), 0.3)
    assert abs(E - Er) <= 1e-11 * abs(Er)
