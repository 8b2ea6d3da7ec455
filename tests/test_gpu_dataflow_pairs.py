"""The dataflow sweep's steps for two gates at once (both environments from
one pass over B and Phi, Phi carried past both) against the CPU oracle: pairs
and single gates in every neighbourhood, at the start, in the middle and at the
end of the circuit, so that a step follows a pair, a single gate or nothing, and
the residual follows a pair or a single gate.

Small starts take the cluster sweep; a dataflow trace keeps them here."""
import numpy as np
import pytest

from oracle import qfs_oracle as o
from paper_2405_12866_gb300 import workloads as w

pytestmark = pytest.mark.gpu

CASES = {
    # all pairs (the residual follows a pair)
    "even_pairs": (6, [(0, 1), (2, 3), (4, 5), (1, 0), (2, 4), (3, 5)], 8, 3),
    # one gate left over: it is gate 1 (the residual follows a single gate)
    "odd_pairs": (6, [(4, 5), (0, 1), (2, 3), (5, 4), (1, 3)], 8, 3),
    # a single gate between pairs, and after them
    "single_inside": (6, [(0, 1), (2, 3), (2, 1), (1, 5), (0, 4), (2, 3)], 6, 2),
    "single_last": (6, [(0, 1), (2, 3), (4, 5), (3, 4), (3, 5)], 10, 2),
    # no pair at all
    "chain": (5, [(0, 1), (1, 2), (2, 3), (3, 4), (3, 2)], 8, 2),
    "one_gate": (4, [(1, 3)], 4, 2),
    "two_gates": (4, [(3, 1), (0, 2)], 8, 2),
    # several chunks a start, ragged rounds
    "brick_n9": (9, w.brick_pairs(9, 4), 26, 2),
    "brick_n11": (11, w.brick_pairs(11, 3), 34, 2),
}


@pytest.fixture(scope="module")
def qfs():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2405_12866_gb300 import build, qfs as q
    build.build()
    return q


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("beta", [0.0, 0.2])
def test_pair_steps_match_oracle(qfs, name, beta):
    n, pairs, M, S = CASES[name]
    U = w.target_unitary(w.haar_gates(31, w.STREAM_TARGET_GATES, len(pairs)), pairs, n)
    Psi, G = w.sample_states(32, n, M), w.initial_gates(33, S, len(pairs))
    with qfs.Context(0) as c:
        c.dataflow_trace(1 << 20)
        g, e, cost = c.sweep_once(n, pairs, U, Psi, G, qfs.QFS_MIXED, beta=beta)
        steps, _ = c.dataflow_trace_read()
    assert steps.shape[0] > 0  # (the dataflow sweep ran)
    UPsi = U @ Psi
    for s in range(S):
        r = o.sweep(UPsi, Psi, G[s], pairs, n, beta)
        assert np.max(np.abs(g[s] - r.gates)) < 1e-4
        assert np.max(np.abs(e[s] - r.envs)) < 1e-4 * max(1.0, np.max(np.abs(r.envs)))
        assert abs(cost[s] - r.cost) < 1e-4


def test_pair_steps_of_several_targets_give_each_what_it_gets_alone(qfs):
    n, pairs, M, S, T = 6, w.brick_pairs(6, 3), 8, 3, 3
    U = np.stack([w.target_unitary(w.haar_gates(40 + t, w.STREAM_TARGET_GATES, len(pairs)), pairs, n) for t in range(T)])
    Psi = np.stack([w.sample_states(50 + t, n, M) for t in range(T)])
    G = np.stack([w.initial_gates(60 + t, S, len(pairs)) for t in range(T)])
    prm = qfs.default_params(M=M, multistarts=S, max_sweeps=5, dist_tol=1e-30, precision=qfs.QFS_MIXED, concurrent_targets=2)
    with qfs.Context(0) as c:
        c.dataflow_trace(1 << 20)
        many = c.instantiate_many(n, pairs, U, prm, Psi, G)
        for t in range(T):
            one = c.instantiate(n, pairs, U[t], prm, Psi[t], G[t])
            assert np.array_equal(one.gates, many[t].gates) and np.array_equal(one.start_costs, many[t].start_costs)
