"""FP64 runs from initial gates that are not unitary: the first sweep is plain FP64
(by the cluster sweep or, from 2048 entries a CTA on, by the dataflow sweep), the
next ones in fixed point.  Against the oracle, to the FP64 sweep tolerances (1e-10
on gates a sweep, 1e-12 on the cost, four sweeps)."""
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
    from paper_2405_12866_gb300 import build, qfs
    build.build()
    return qfs


def _problem(n, layers, M, S, seed):
    pairs = w.brick_pairs(n, layers)
    U = w.target_unitary(w.haar_gates(seed, w.STREAM_TARGET_GATES, len(pairs)), pairs, n)
    G = w.initial_gates(seed + 2, S, len(pairs)) * np.linspace(0.9, 1.2, S)[:, None, None, None]
    G[:, 0, 1, 2] += 0.1
    return pairs, U, w.sample_states(seed + 1, n, M), G


@pytest.mark.parametrize("n, layers, M, S", [(4, 3, 4, 1), (7, 3, 12, 3), (10, 2, 32, 2), (10, 2, 48, 1), (11, 2, 20, 2)])
@pytest.mark.parametrize("sweeps", [1, 4])
def test_runs_match_the_oracle(qfs, n, layers, M, S, sweeps):
    pairs, U, Psi, G = _problem(n, layers, M, S, 40 + n)
    want, costs = [], []
    for s in range(S):
        g = G[s]
        for _ in range(sweeps):
            r = o.sweep(U @ Psi, Psi, g, pairs, n)
            g = r.gates
        want.append(g)
        costs.append(r.cost)
    prm = qfs.default_params(M=M, multistarts=S, max_sweeps=sweeps, dist_tol=1e-30)
    with qfs.Context(0) as c:
        for _ in range(2):  # (a run leaves nothing for the next)
            r = c.instantiate(n, pairs, U, prm, samples=Psi, init_gates=G)
            assert np.max(np.abs(r.start_costs - costs)) < 1e-12 * sweeps
            best = int(np.argmin(costs))
            assert np.max(np.abs(r.gates.reshape(want[best].shape) - want[best])) < 1e-10 * sweeps
        if sweeps == 1:
            g, e, cost = c.sweep_once(n, pairs, U, Psi, G, qfs.QFS_FP64)
            assert np.max(np.abs(g - np.array(want))) < 1e-10


def test_slots_with_and_without_unitary_gates(qfs):
    """Targets of one call, some with unitary initial gates and some without, more targets than
    slots: each gets the run it gets alone, to rounding."""
    n, M, S = 10, 32, 2
    pairs, U, Psi, G = _problem(n, 2, M, S, 60)
    Gu = w.initial_gates(62, S, len(pairs))
    T = 5
    gates = np.stack([G if t % 2 else Gu for t in range(T)])
    prm = qfs.default_params(M=M, multistarts=S, max_sweeps=4, dist_tol=1e-30, concurrent_targets=2)
    with qfs.Context(0) as c:
        got = c.instantiate_many(n, pairs, np.stack([U] * T), prm, np.stack([Psi] * T), gates)
        alone = [c.instantiate(n, pairs, U, prm, samples=Psi, init_gates=g) for g in (Gu, G)]
    for t in range(T):
        assert abs(got[t].cost - alone[t % 2].cost) < 1e-12 * 4
        assert np.max(np.abs(got[t].gates.reshape(-1) - alone[t % 2].gates.reshape(-1))) < 1e-10 * 4
