"""The 2-D tile visit with thread-private positions (csrc/csc2d_tile.cuh) at the
edges of its layout, against the 2-D FP64 oracle: atom counts around its float4
groups, windows of just under and just over a multiple of 32 positions, one-row
and one-column windows, tiles wider than the window (several positions per
thread), tiles as large as the image, one update per visit, and more nonzeros in
a tile than its active list holds.  Bars of tests/test_gpu_csc2d.py."""
import pytest

from oracle import csc2d
from paper_1705_10087_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests.test_gpu_csc2d import assert_parity, capi  # noqa: E402,F401

CASES = [
    # K, P, h, w, H, W, M, N, u, lambda / lambda_max, rho
    (1, 1, 1, 1, 20, 33, 0, 0, 0, 0.1, 0.05),    # no halo, one position per window
    (4, 2, 1, 7, 12, 60, 0, 0, 0, 0.1, 0.02),    # one-row windows
    (5, 2, 8, 1, 50, 14, 0, 0, 3, 0.1, 0.02),    # one-column windows
    (8, 2, 3, 4, 40, 41, 0, 0, 1, 0.1, 0.01),    # 35 window positions, one update a visit
    (9, 3, 3, 3, 33, 47, 2, 3, 0, 0.1, 0.01),    # tiles several windows wide
    (20, 6, 5, 5, 40, 40, 0, 0, 0, 0.1, 0.005),  # five quads
    (32, 8, 4, 4, 30, 34, 0, 0, 8, 0.1, 0.005),  # eight quads, the most
    (33, 8, 4, 4, 30, 34, 0, 0, 8, 0.1, 0.005),  # one more atom: the shared form
    (3, 2, 4, 4, 16, 17, 1, 1, 0, 0.1, 0.02),    # one tile
    (2, 4, 3, 3, 24, 26, 1, 1, 0, 0.03, 0.3),    # more nonzeros than the active list
]


@pytest.mark.parametrize("K,P,h,w,H,W,M,N,u,frac,rho", CASES)
def test_tile_layout_edges_match_oracle(capi, K, P, h, w, H, W, M, N, u, frac, rho):  # noqa: F811
    pb = synth.make_problem2d(K=K, P=P, h=h, w=w, H=H, W=W, rho=rho, sigma=0.05, seed=K + h)
    lam = frac * csc2d.lambda_max(pb.D, pb.X)
    Hz, Wz = H - h + 1, W - w + 1
    Mr = M if M else max(1, Hz // max(1, 2 * h - 2))
    ref = csc2d.locally_greedy_cd(pb.D, pb.X, lam, 1e-10, M=Mr, mode="phase")
    assert ref["converged"]
    if frac < 0.1:
        assert (ref["Z"] != 0).sum() > 2 * 128
    Z = torch.zeros((K, Hz, Wz), dtype=torch.float32, device="cuda")
    status, E, st = capi.csc2d_solve(torch.from_numpy(pb.D).cuda(), torch.from_numpy(pb.X).cuda(),
                                     lam, 1e-6, M=M, N=N, updates_per_visit=u, Z_out=Z)
    assert status == capi.CSC_OK and st["converged"] == 1, st
    assert_parity(Z.cpu().numpy(), E, ref["Z"], csc2d.objective(pb.D, pb.X, ref["Z"], lam))


def test_calls_of_two_threads_share_no_workspace(capi):  # noqa: F811
    # finished calls leave their device memory for later ones: calls that run at
    # the same time on two streams must not meet in it, whatever their sizes
    import threading

    pbs = [synth.make_problem2d(K=3, P=1, h=4, w=5, H=40 + 30 * i, W=60 - 9 * i, rho=0.01,
                                sigma=0.05, seed=20 + i) for i in range(2)]
    lams = [0.1 * csc2d.lambda_max(pb.D, pb.X) for pb in pbs]

    def solve(i, stream=None):
        pb = pbs[i]
        Z = torch.zeros((3, pb.X.shape[1] - 3, pb.X.shape[2] - 4), dtype=torch.float32,
                        device="cuda")
        torch.cuda.synchronize()
        _, E, _ = capi.csc2d_solve(torch.from_numpy(pb.D).cuda(), torch.from_numpy(pb.X).cuda(),
                                   lams[i], 1e-6, Z_out=Z, stream=stream)
        return Z.cpu(), E

    want = [solve(i) for i in range(2)]
    bad = []

    def run(i):
        stream = torch.cuda.Stream()
        for _ in range(6):
            Z, E = solve(i, stream)
            if not torch.equal(Z, want[i][0]) or E != want[i][1]:
                bad.append(i)

    threads = [threading.Thread(target=run, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
