"""csc_get_trace's objective decrease of a launch: summed in the order of the updates
in more than float32, so that a solve gives the same bits every time, although the
lanes that hold the nonzero coordinates of a segment differ from run to run."""
import numpy as np
import pytest

import oracle
from paper_1705_10087_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests.test_gpu_parity import capi  # noqa: E402,F401


@pytest.mark.parametrize("K,P,L,T,u", [
    (5, 2, 16, 1500, 31),    # one short of what is added up at a time
    (5, 2, 16, 1500, 32),
    (5, 2, 16, 1500, 33),
    (25, 4, 40, 1400, 200),  # several times that
    (40, 6, 20, 700, 64),    # two groups of atoms
])
def test_decrease_is_the_same_on_every_run(capi, K, P, L, T, u):  # noqa: F811
    # one segment: a launch is one visit (the sums of several blocks are added up
    # in FP64, in the order of their ends)
    pb = synth.make_problem(K=K, P=P, L=L, T=T, rho=0.05, sigma=0.1, seed=K + u)
    D, X = torch.from_numpy(pb.D).cuda(), torch.from_numpy(pb.X).cuda()
    Z, beta0 = (torch.empty((K, T - L + 1), device="cuda") for _ in range(2))
    h = capi.csc_setup(D, capi.make_opts(segments=1, updates_per_visit=u))
    try:
        runs = []
        for _ in range(8):
            capi.csc_init(h, X, 0.2)
            capi.csc_get_beta(h, beta0)
            status, E, st = capi.csc_solve(h, 1e-4, 1 << 40, Z)
            assert status == capi.CSC_OK and st["updates"] > 10 * u, st
            runs.append((capi.csc_get_trace(h), E))
    finally:
        capi.csc_destroy(h)
    first, E = runs[0]
    assert first["n"] == len(first["decrease"]) and first["updates"].max() == u
    for tr, _ in runs[1:]:
        assert np.array_equal(tr["updates"], first["updates"])
        assert np.array_equal(tr["decrease"], first["decrease"])
    # and it accounts for the whole descent, on the problem of the computed beta0 (bar and
    # offset of the trace in tests/test_gpu_parity.py)
    offset = float((Z.double().cpu().numpy() *
                    (beta0.double().cpu().numpy() - oracle.dtx(pb.D, pb.X))).sum())
    assert first["E_start"] - first["decrease"].sum() == pytest.approx(E - offset, rel=1e-6)
