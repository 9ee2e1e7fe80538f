"""Calls of several threads at once, each on its own stream and, in 1-D, its own
handle: they share kernels, whose dynamic shared-memory limit is state of the
device, and 2-D calls share the list of kept workspaces.  Every thread must finish
all its calls, with the bits that the same calls gave alone."""
import threading

import pytest

from paper_1705_10087_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests.test_gpu_csc2d import capi  # noqa: E402,F401

ROUNDS = 12


def run_together(jobs):
    """Every job (a function of its stream) ROUNDS times, all jobs at once; the
    results of each, after the one that it gave alone."""
    torch.cuda.synchronize()
    got = [[job(None)] for job in jobs]
    errors = []
    start = threading.Barrier(len(jobs))

    def run(i):
        try:
            stream = torch.cuda.Stream()
            start.wait(60)
            for _ in range(ROUNDS):
                got[i].append(jobs[i](stream))
        except BaseException as e:  # an exception ends only its thread
            errors.append((i, e))

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join(300)
    assert not errors, errors
    for g in got:
        assert len(g) == 1 + ROUNDS
        for status, E, Z in g:
            assert status == 0 and E == g[0][1] and torch.equal(Z, g[0][2])


def image_job(capi, K, P, h, w, H, W, seed, **opts):  # noqa: F811
    pb = synth.make_problem2d(K=K, P=P, h=h, w=w, H=H, W=W, rho=0.01, sigma=0.05, seed=seed)
    D, X = torch.from_numpy(pb.D).cuda(), torch.from_numpy(pb.X).cuda()

    def job(stream):
        Z = torch.empty((K, H - h + 1, W - w + 1), device="cuda")
        torch.cuda.synchronize()
        status, E, _ = capi.csc2d_solve(D, X, 0.5, 1e-6, Z_out=Z, stream=stream, **opts)
        return status, E, Z.cpu()
    return job


@pytest.mark.parametrize("atoms,sizes", [
    # (K, P, h, w): one kernel; ((H, W), options) per thread: its tiles
    ((3, 1, 4, 5), [((40, 60), {}), ((70, 51), {})]),
    ((12, 2, 9, 9), [((120, 120), {}), ((60, 70), {"M": 20, "N": 20})]),    # one above 48 KB
    ((33, 8, 4, 4), [((50, 90), {"M": 2, "N": 4}), ((40, 40), {}), ((41, 40), {})]),  # tile_kernel
])
def test_images(capi, atoms, sizes):  # noqa: F811
    run_together([image_job(capi, *atoms, H, W, seed=30 + i, **opts)
                  for i, ((H, W), opts) in enumerate(sizes)])


def signal_job(capi, K, P, L, T, M, tps, seed):  # noqa: F811
    pb = synth.make_problem(K=K, P=P, L=L, T=T, rho=0.01, sigma=0.05, seed=seed)
    D, X = torch.from_numpy(pb.D).cuda(), torch.from_numpy(pb.X).cuda()

    def job(stream):
        # (a new handle and plan: its phases are launched one by one)
        Z = torch.empty((K, T - L + 1), device="cuda")
        torch.cuda.synchronize()
        h = capi.csc_setup(D, capi.make_opts(segments=M, threads_per_segment=tps), stream=stream)
        try:
            capi.csc_init(h, X, 0.5)
            status, E, _ = capi.csc_solve(h, 1e-6, 1 << 40, Z)
        finally:
            capi.csc_destroy(h)
        return status, E, Z.cpu()
    return job


@pytest.mark.parametrize("K,P,L,tps,plans", [
    (5, 2, 16, 0, [(900, 2), (9_000, 300), (3_000, 30)]),    # thread-private form
    (25, 4, 40, 32, [(2_000, 6), (8_000, 90)]),              # one warp per segment
    (3, 2, 260, 0, [(4_000, 1), (9_000, 17), (9_001, 3)]),   # the block form of wide windows
])
def test_signals(capi, K, P, L, tps, plans):  # noqa: F811
    run_together([signal_job(capi, K, P, L, T, M, tps, seed=40 + i)
                  for i, (T, M) in enumerate(plans)])
