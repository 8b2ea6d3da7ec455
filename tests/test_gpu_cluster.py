"""The cluster sweep (a start's columns split over a thread-block cluster,
FP64 in fixed point) and the one-launch FP64 check against the CPU oracle, at
the sizes where a split, a slice or a bound of the fixed point changes."""
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


@pytest.fixture(scope="module")
def ctx(qfs):
    with qfs.Context(0) as c:
        yield c


def _problem(n, pairs, M, S, seed=71):
    U = w.target_unitary(w.haar_gates(seed, w.STREAM_TARGET_GATES, len(pairs)), pairs, n)
    return U, w.sample_states(seed + 1, n, M), w.initial_gates(seed + 2, S, len(pairs))


def _kappa(E):
    s = np.linalg.svd(E, compute_uv=False)
    return s[..., 0] / np.maximum(s[..., 3], 1e-300)


# (n, pairs, M, S): one gate; two qubits; uneven column splits (M not a
# multiple of the CTAs); pairs with qubits apart and in both orders; more
# columns per CTA than 4 and 8 (smaller fixed-point scales); many starts
# (several rounds of clusters); one column more or less than a split; slices
# that are no multiple of 16 entries.
CASES = {
    "one_gate": (3, [(0, 2)], 4, 3),
    "two_qubits": (2, [(0, 1), (1, 0), (0, 1)], 4, 2),
    "two_qubits_odd": (2, [(0, 1)], 3, 200),  # (E has rank 3: the gate is not unique)
    "three_qubits_odd": (3, w.chain_pairs(3, 6), 7, 17),
    "three_qubits_five": (3, w.chain_pairs(3, 4), 5, 160),
    "apart_both_orders": (5, [(0, 4), (3, 1), (2, 0), (4, 2), (1, 3), (0, 1)], 7, 4),
    "uneven_columns": (7, w.brick_pairs(7, 4), 13, 5),
    "one_more_column": (6, w.brick_pairs(6, 4), 17, 3),
    "full_unitary_n6": (6, w.brick_pairs(6, 3), 64, 2),
    "full_unitary_n7": (7, w.brick_pairs(7, 3), 128, 2),
    "full_unitary_n8": (8, w.brick_pairs(8, 2), 256, 1),
    "many_starts": (4, w.brick_pairs(4, 4), 6, 170),
    "largest_slice": (10, w.brick_pairs(10, 2), 33, 2),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("beta", [0.0, 0.25])
def test_fp64_sweep_matches_oracle(qfs, ctx, name, beta):
    n, pairs, M, S = CASES[name]
    U, Psi, G = _problem(n, pairs, M, S)
    g, e, c = ctx.sweep_once(n, pairs, U, Psi, G, qfs.QFS_FP64, beta=beta)
    UPsi = U @ Psi
    for s in range(0, S, max(1, S // 6)):
        r = o.sweep(UPsi, Psi, G[s], pairs, n, beta)
        scale = max(1.0, np.max(np.abs(r.envs)))
        # 1e-14 kappa, the growth of the polar factor's rounding with its condition.
        tol = 1e-11 + 1e-14 * np.max(_kappa(r.envs))
        assert np.max(np.abs(g[s] - r.gates)) < tol
        assert np.max(np.abs(e[s] - r.envs)) < tol * scale
        assert abs(c[s] - r.cost) < 1e-12
        assert np.max(np.abs(np.einsum("kij,klj->kil", g[s], g[s].conj()) - np.eye(4))) < 1e-14


@pytest.mark.parametrize("name", sorted(CASES))
def test_complex64_sweep_matches_oracle(qfs, ctx, name):
    n, pairs, M, S = CASES[name]
    U, Psi, G = _problem(n, pairs, M, S)
    g, e, c = ctx.sweep_once(n, pairs, U, Psi, G, qfs.QFS_MIXED)
    UPsi = U @ Psi
    for s in range(0, S, max(1, S // 6)):
        r = o.sweep(UPsi, Psi, G[s], pairs, n)
        if np.max(_kappa(r.envs)) < 1e4:
            assert np.max(np.abs(g[s] - r.gates)) < 1e-4
        else:
            got = np.real(np.einsum("kij,kji->k", g[s], e[s]))
            assert np.max(np.abs(got - np.sum(np.linalg.svd(e[s], compute_uv=False), axis=-1))) < 1e-4
        assert np.max(np.abs(e[s] - r.envs)) < 1e-4 * max(1.0, np.max(np.abs(r.envs)))
        assert abs(c[s] - r.cost) < 1e-4
        assert np.max(np.abs(np.einsum("kij,klj->kil", g[s], g[s].conj()) - np.eye(4))) < 1e-14


@pytest.mark.parametrize("what", ["gates_not_unitary", "target_times_3", "target_times_1e-6", "states_times_1e5"])
def test_fp64_sweep_of_inputs_without_unit_norms(qfs, ctx, what):
    """Columns of any norm (their own fixed-point scale) and initial gates
    that are not unitary (the plain FP64 form)."""
    n, pairs, M, S = 6, w.brick_pairs(6, 3), 8, 3
    U, Psi, G = _problem(n, pairs, M, S)
    if what == "gates_not_unitary":
        G = G * np.linspace(0.5, 4.0, S)[:, None, None, None]
    elif what == "states_times_1e5":
        Psi = Psi * 1e5
    else:
        U = U * float(what.rsplit("_", 1)[1])
    g, e, _ = ctx.sweep_once(n, pairs, U, Psi, G, qfs.QFS_FP64)
    for s in range(S):
        r = o.sweep(U @ Psi, Psi, G[s], pairs, n)
        assert np.max(np.abs(g[s] - r.gates)) < 1e-11 + 1e-14 * np.max(_kappa(r.envs))
        assert np.max(np.abs(e[s] - r.envs)) < 1e-11 * np.max(np.abs(r.envs))


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("M", [1, 2])
def test_rank_deficient_environments_get_an_optimal_unitary(qfs, ctx, prec, M):
    """n = 3 with one or two states: E has rank 2 M at most, any completion is
    optimal: Re tr(g E) is the sum of the singular values."""
    n, pairs, S = 3, [(0, 1)], 4
    U, Psi, G = _problem(n, pairs + [(1, 2)], M, S)
    g, e, _ = ctx.sweep_once(n, pairs, U, Psi, G[:, :1], qfs.QFS_FP64 if prec == "fp64" else qfs.QFS_MIXED)
    tol = 1e-12 if prec == "fp64" else 1e-5
    for s in range(S):
        best = np.sum(np.linalg.svd(e[s, 0], compute_uv=False))
        assert abs(np.real(np.trace(g[s, 0] @ e[s, 0])) - best) < tol
        assert np.max(np.abs(g[s, 0] @ g[s, 0].conj().T - np.eye(4))) < 1e-13


@pytest.mark.parametrize("n,M,S,sweeps", [(3, 4, 1, 70), (5, 9, 3, 20), (8, 12, 4, 18)])
def test_runs_match_the_per_step_sweeps(qfs, ctx, n, M, S, sweeps):
    """Several sweeps per launch (one CTA per start) and several launches per
    round trip end where one per-step sweep at a time does, also when the
    tolerance is met on the way."""
    pairs = w.brick_pairs(n, 4)
    U, Psi, G = _problem(n, pairs, M, S)
    with qfs.Context(0) as steps:
        steps.set_option(qfs.QFS_OPT_DATAFLOW, 0)
        prm = qfs.default_params(M=M, multistarts=S, max_sweeps=sweeps, dist_tol=1e-30)
        a, b = (c.instantiate(n, pairs, U, prm, Psi, G) for c in (ctx, steps))
        assert a.sweeps == b.sweeps == sweeps and a.best_start == b.best_start
        assert np.max(np.abs(a.start_costs - b.start_costs)) < 1e-9
        # A tolerance between two sweeps' costs: both stop at the same sweep.
        prm = qfs.default_params(M=M, multistarts=S, max_sweeps=max(1, sweeps // 2), dist_tol=1e-30)
        mid = steps.instantiate(n, pairs, U, prm, Psi, G).cost
        prm = qfs.default_params(M=M, multistarts=S, max_sweeps=sweeps, dist_tol=mid * (1 + 1e-6))
        a, b = (c.instantiate(n, pairs, U, prm, Psi, G) for c in (ctx, steps))
        assert a.converged and b.converged and a.sweeps == b.sweeps and a.best_start == b.best_start
        assert np.max(np.abs(a.gates - b.gates)) < 1e-7


@pytest.mark.parametrize("n,M", [(3, 4), (6, 7), (9, 3), (11, 2), (13, 1)])
def test_one_launch_check_gives_the_cost_of_the_returned_gates(qfs, ctx, n, M):
    pairs = w.brick_pairs(n, 3)
    U, Psi, G = _problem(n, pairs, M, 2)
    prm = qfs.default_params(M=M, multistarts=2, max_sweeps=2, dist_tol=0.0, precision=qfs.QFS_MIXED)
    r = ctx.instantiate(n, pairs, U, prm, Psi, G)
    assert abs(r.cost - o.sample_cost(U @ Psi, Psi, r.gates, pairs, n)) < 1e-13
