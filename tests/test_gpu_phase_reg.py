"""The block form of the phase kernel with thread-private r (csrc/phase_reg_impl.cuh)
at the edges of its layout, against the FP64 oracle: atom counts around its
float4 groups and around one and several groups of threads, windows of just
under, exactly and just over a multiple of 32 columns, segments of one, two and
more columns per thread, one update per visit, and more nonzeros in a segment
than its active list holds.  Bars of tests/test_gpu_parity.py."""
import pytest

import oracle
from paper_1705_10087_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests.test_gpu_parity import assert_parity, capi, gpu_solve  # noqa: E402,F401

CASES = [
    # K, P, L, T, M, u, lambda / lambda_max
    (1, 1, 1, 300, 3, 0, 0.1),       # no halo, one quad, Tz = T
    (3, 2, 5, 5, 1, 0, 0.1),         # a single column
    (4, 2, 16, 1200, 20, 0, 0.1),    # 31 window columns in 32 threads
    (5, 3, 17, 1200, 20, 24, 0.1),   # 33 window columns in 64 threads
    (12, 4, 33, 3000, 40, 3, 0.1),   # three quads, 65 window columns
    (25, 7, 64, 2500, 19, 1, 0.1),   # one column per thread, one update per visit
    (25, 7, 64, 2500, 10, 24, 0.1),  # two columns per thread
    (25, 7, 64, 2500, 3, 0, 0.1),    # seven columns per thread
    (28, 7, 40, 2500, 25, 0, 0.1),   # seven whole quads
    (32, 7, 48, 2500, 25, 24, 0.1),  # eight quads, one group
    (33, 8, 20, 1500, 30, 0, 0.1),   # two groups, the last with one quad
    (64, 8, 64, 2000, 15, 24, 0.1),  # two whole groups
    (100, 16, 12, 800, 25, 0, 0.1),  # four groups
    (8, 4, 70, 4000, 20, 24, 0.1),   # 139 window columns in 160 threads
    (4, 8, 8, 1500, 2, 0, 0.05),     # more nonzeros in a segment than the active list
]


@pytest.mark.parametrize("K,P,L,T,M,u,frac", CASES)
def test_phase_layout_edges_match_oracle(capi, K, P, L, T, M, u, frac):  # noqa: F811
    dense = frac < 0.1
    pb = synth.make_problem(K=K, P=P, L=L, T=T, rho=0.2 if dense else 0.01, sigma=0.1, seed=K + L)
    lam = frac * oracle.lambda_max(pb.D, pb.X)
    ref = oracle.locally_greedy_cd(pb.D, pb.X, lam, 1e-10, M=M, mode="phase")
    assert ref["converged"]
    if dense:
        assert (ref["Z"] != 0).sum() > 2 * 128 * M
    r = gpu_solve(capi, pb, lam, 1e-6, M=M, u=u)
    assert r["status"] == 0 and r["stats"]["segments"] == M, r["stats"]
    assert_parity(r["Z"], r["E"], ref["Z"], oracle.objective(pb.D, pb.X, ref["Z"], lam))


@pytest.mark.parametrize("K,P,L,T,M", [
    (4, 4, 70, 20_000, 100),   # 192-thread blocks, all resident in the form with more registers
    (4, 4, 70, 88_000, 632),   # and more than that
    (4, 2, 150, 30_000, 90),   # 352-thread blocks
    (4, 2, 150, 93_000, 306),
])
def test_few_and_many_segments_match_oracle(capi, K, P, L, T, M):  # noqa: F811
    pb = synth.make_problem(K=K, P=P, L=L, T=T, rho=0.001, sigma=0.1, seed=K + L)
    lam = 0.1 * oracle.lambda_max(pb.D, pb.X)
    ref = oracle.locally_greedy_cd(pb.D, pb.X, lam, 1e-10, M=M, mode="phase")
    assert ref["converged"]
    r = gpu_solve(capi, pb, lam, 1e-6, M=M, u=24)
    assert r["status"] == 0 and r["stats"]["segments"] == M, r["stats"]
    assert_parity(r["Z"], r["E"], ref["Z"], oracle.objective(pb.D, pb.X, ref["Z"], lam))
