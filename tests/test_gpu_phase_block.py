"""The block form of the phase kernel in csrc/kernel_phase.cu at sizes that the
thread-private form (csrc/phase_reg_impl.cuh) does not hold, just past its bounds,
against the FP64 oracle: windows of more than 512 columns, several groups of atoms
times a window of more than 512 threads, segments too wide for shared memory; per
segment and drained from a queue.  Bars of tests/test_gpu_parity.py."""
import pytest

import oracle
from paper_1705_10087_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests.test_gpu_parity import assert_parity, capi, cuda, gpu_solve  # noqa: E402,F401

CASES = [
    # K, P, L, T, M, u: staged (r and Z in shared memory) unless the segments are too wide
    (3, 2, 257, 4000, 0, 0),     # 513 window columns: blocks of 1024 threads
    (25, 2, 257, 3000, 5, 24),
    (25, 2, 300, 3000, 1, 0),    # the same in place
    (5, 1, 512, 6000, 0, 3),     # the longest atoms
    (40, 4, 130, 1500, 0, 24),   # two groups of 288 threads: blocks of 512 threads
    (40, 4, 130, 1500, 1, 0),    # in place
    (64, 4, 130, 1500, 0, 0),    # K = 64 fixed at compile time, staged
    (64, 4, 130, 1500, 2, 24),   # in place
    (100, 8, 70, 800, 0, 0),     # four groups of 160 threads
    (33, 6, 20, 789, 1, 64),     # a segment between the two forms' shared memory: 128 threads
    (33, 6, 20, 1200, 1, 0),     # in place
    (5, 2, 16, 4000, 1, 100),    # few atoms, a segment of 3985 columns, in place
    (25, 4, 40, 2500, 1, 0),     # K = 25 in place, 128 threads
    (25, 2, 70, 2500, 1, 24),    # and 512
    (64, 5, 20, 1200, 1, 24),    # K = 64 in place, 128 threads
]


@pytest.mark.parametrize("K,P,L,T,M,u", CASES)
def test_block_form_matches_oracle(capi, K, P, L, T, M, u):  # noqa: F811
    pb = synth.make_problem(K=K, P=P, L=L, T=T, rho=0.002, sigma=0.1, seed=K + L)
    lam = 0.1 * oracle.lambda_max(pb.D, pb.X)
    Mr = M if M else max(1, pb.Tz // (2 * L - 2))
    ref = oracle.locally_greedy_cd(pb.D, pb.X, lam, 1e-10, M=Mr, mode="phase")
    assert ref["converged"]
    r = gpu_solve(capi, pb, lam, 1e-6, M=M, u=u)
    assert r["status"] == 0 and r["stats"]["segments"] == Mr, r["stats"]
    assert_parity(r["Z"], r["E"], ref["Z"], oracle.objective(pb.D, pb.X, ref["Z"], lam))


@pytest.mark.parametrize("K,L,T", [
    (2, 257, 650_000),   # more than 608 segments in a phase, one block of 1024 threads per SM
    (33, 130, 320_000),  # of 512
])
def test_drained_block_form_matches_oracle(capi, K, L, T):  # noqa: F811
    pb = synth.make_problem(K=K, P=1, L=L, T=T, rho=1e-4, sigma=0.05, seed=K + L)
    lam = 0.3 * oracle.lambda_max(pb.D, pb.X)
    M = pb.Tz // (2 * L - 2)
    assert M > 2 * 608
    ref = oracle.locally_greedy_cd(pb.D, pb.X, lam, 1e-10, M=M, mode="phase")
    assert ref["converged"]
    r = gpu_solve(capi, pb, lam, 1e-6, u=24)
    assert r["status"] == 0 and r["stats"]["segments"] == M, r["stats"]
    assert_parity(r["Z"], r["E"], ref["Z"], oracle.objective(pb.D, pb.X, ref["Z"], lam))


@pytest.mark.parametrize("L,T,M,u", [(64, 20_000, 64, 0), (64, 20_000, 313, 24),
                                     (40, 9_000, 90, 3), (1, 500, 20, 0), (17, 5_000, 9, 7)])
def test_forms_agree_bit_for_bit(capi, L, T, M, u):  # noqa: F811
    """One warp per segment (the arithmetic of the block form) and the thread-private
    form make the same updates in the same order with the same roundings."""
    pb = synth.make_problem(K=25, P=3, L=L, T=T, rho=0.005, sigma=0.1, seed=L)
    lam = 0.1 * oracle.lambda_max(pb.D, pb.X)
    got = []
    for tps in (32, 0):
        h = capi.csc_setup(cuda(pb.D), capi.make_opts(segments=M, updates_per_visit=u,
                                                      threads_per_segment=tps))
        try:
            capi.csc_init(h, cuda(pb.X), lam)
            Z = torch.zeros((pb.K, pb.Tz), dtype=torch.float32, device="cuda")
            status, E, st = capi.csc_solve(h, 1e-6, 1 << 40, Z)
        finally:
            capi.csc_destroy(h)
        got.append((status, E, st["updates"], Z))
    assert got[0][:3] == got[1][:3] and torch.equal(got[0][3], got[1][3])
