"""Runs whose device workspace is limited: at the smallest limit that is not
refused a sweep takes the forms with the smallest buffers (per-gate dataflow
steps, the FP64 target product), and still gives the oracle's sweep."""
import numpy as np
import pytest

from oracle import qfs_oracle as o
from paper_2405_12866_gb300 import workloads as w

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qfs():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2405_12866_gb300 import build, qfs as q
    build.build()
    return q


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("n, layers, M, S", [(4, 3, 6, 2), (7, 4, 24, 5), (9, 3, 33, 3)])
def test_smallest_accepted_workspace(qfs, n, layers, M, S, mixed):
    pairs = w.brick_pairs(n, layers)
    U = w.target_unitary(w.haar_gates(41, w.STREAM_TARGET_GATES, len(pairs)), pairs, n)
    Psi, G = w.sample_states(42, n, M), w.initial_gates(43, S, len(pairs))
    prec = qfs.QFS_MIXED if mixed else qfs.QFS_FP64

    def sweep(cap):
        with qfs.Context(0) as c:
            c.set_option(qfs.QFS_OPT_WORKSPACE_CAP, cap)
            try:
                return c.sweep_once(n, pairs, U, Psi, G, prec)
            except qfs.QfsError as e:
                assert e.code == qfs.QFS_ENOMEM
                return None

    lo, hi = 1 << 10, 1 << 28  # refused, accepted
    while hi - lo > 256:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if sweep(mid) is not None else (mid, hi)
    g, e, cost = sweep(hi)
    UPsi, tol = U @ Psi, 1e-4 if mixed else 1e-10
    for s in range(S):
        r = o.sweep(UPsi, Psi, G[s], pairs, n)
        assert np.max(np.abs(g[s] - r.gates)) < tol
        assert np.max(np.abs(e[s] - r.envs)) < tol * max(1.0, np.max(np.abs(r.envs)))
        assert abs(cost[s] - r.cost) < (1e-4 if mixed else 1e-12)
