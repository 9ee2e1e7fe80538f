"""One-row atoms up to the documented limit of (2h-1)(2w-1) <= 4096 positions, against
the 2-D FP64 oracle: the atoms that csc2d_solve stages for beta0 take up to 64 KB of
shared memory there.  Bars of tests/test_gpu_csc2d.py."""
import pytest

from oracle import csc2d
from paper_1705_10087_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests.test_gpu_csc2d import assert_parity, capi  # noqa: E402,F401


@pytest.mark.parametrize("K,P,w,H,W", [
    (2, 1, 1536, 3, 4000),  # 48 KB: the most without a raised limit
    (2, 1, 1537, 3, 4000),
    (9, 2, 1600, 2, 3500),  # two groups of staged atoms, two channels
    (1, 1, 2048, 2, 4500),  # 64 KB: the widest
])
def test_wide_one_row_atoms_match_oracle(capi, K, P, w, H, W):  # noqa: F811
    pb = synth.make_problem2d(K=K, P=P, h=1, w=w, H=H, W=W, rho=0.001, sigma=0.05, seed=K + w)
    lam = 0.1 * csc2d.lambda_max(pb.D, pb.X)
    ref = csc2d.locally_greedy_cd(pb.D, pb.X, lam, 1e-10, M=H, mode="phase")
    assert ref["converged"]
    Z = torch.zeros((K, H, W - w + 1), dtype=torch.float32, device="cuda")
    status, E, st = capi.csc2d_solve(torch.from_numpy(pb.D).cuda(), torch.from_numpy(pb.X).cuda(),
                                     lam, 1e-6, Z_out=Z)
    assert status == capi.CSC_OK and st["converged"] == 1, st
    assert_parity(Z.cpu().numpy(), E, ref["Z"], csc2d.objective(pb.D, pb.X, ref["Z"], lam))
