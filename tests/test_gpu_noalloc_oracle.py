"""The allocation-free sweep against the CPU oracle on each of its routes, and
what it leaves where a wait runs out.

Routes: the cluster sweep (behind the fixed-point product, and behind the digits
at 9 qubits and, in fewer splits for want of room, at 10) and the per-step launches (more gates than the cluster sweep takes,
with either product).  Tolerances as for every FP64 sweep: 1e-10 on gates and
environments, 1e-12 on the cost."""
import ctypes as C

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


def _run(qfs, n, pairs, M, S, seed, wait_limit=None, beta=0.0):
    import torch
    L = len(pairs)
    U = w.target_unitary(w.haar_gates(seed, w.STREAM_TARGET_GATES, L), pairs, n)
    Psi, G = w.sample_states(seed + 1, n, M), w.initial_gates(seed + 2, S, L)
    tU, tP, tG = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (U, Psi, G))
    out = [torch.zeros((S, L, 4, 4), dtype=torch.complex128, device="cuda") for _ in range(2)]
    cost = torch.zeros(S, dtype=torch.float64, device="cuda")
    cir = qfs._CircuitArg(n, pairs)
    args = [torch.cuda.current_stream().cuda_stream, C.byref(cir.c), tU.data_ptr(), tP.data_ptr(), M, S, beta, tG.data_ptr(),
            out[0].data_ptr(), cost.data_ptr(), out[1].data_ptr()]
    lib = qfs.lib()
    code = lib.qfs_sweep_once_noalloc(*args) if wait_limit is None else lib.qfs_sweep_once_noalloc_limit(*args, wait_limit)
    torch.cuda.synchronize()
    return code, out[0].cpu().numpy(), out[1].cpu().numpy(), cost.cpu().numpy(), (U, Psi, G)


@pytest.mark.parametrize("n, layers, chain, M, S", [(6, 3, 0, 16, 3), (3, 0, 4, 4, 1), (9, 2, 0, 4, 1), (10, 2, 0, 32, 1), (4, 0, 130, 8, 3),
                                                    (9, 0, 130, 1, 1)])
def test_routes_match_the_oracle(qfs, n, layers, chain, M, S):
    pairs = w.brick_pairs(n, layers) if layers else w.chain_pairs(n, chain)
    code, g, e, c, (U, Psi, G) = _run(qfs, n, pairs, M, S, 601)
    assert code == qfs.QFS_OK
    for s in range(S):
        r = o.sweep(U @ Psi, Psi, G[s], pairs, n)
        assert np.max(np.abs(g[s] - r.gates)) < 1e-10
        assert np.max(np.abs(e[s] - r.envs)) < 1e-10
        assert abs(c[s] - r.cost) < 1e-12


def test_a_wait_that_runs_out_leaves_nan(qfs):
    """One poll for the exchange of a gate's environment (some hundred ns): starts that
    give up get NaN everywhere, the others their sweep; the next call is as ever."""
    case = (8, w.brick_pairs(8, 4), 16, 8, 602)
    code, g0, e0, c0, _ = _run(qfs, *case)
    assert code == qfs.QFS_OK and np.isfinite(c0).all()
    code, g, e, c, _ = _run(qfs, *case, wait_limit=1)
    assert code == qfs.QFS_OK
    bad = np.isnan(c)
    assert bad.any()
    assert np.isnan(g[bad]).all() and np.isnan(e[bad]).all()
    assert np.array_equal(g[~bad], g0[~bad]) and np.array_equal(c[~bad], c0[~bad])
    code, g, e, c, _ = _run(qfs, *case)
    assert code == qfs.QFS_OK and np.array_equal(g, g0) and np.array_equal(e, e0) and np.array_equal(c, c0)


def test_wait_limit_below_one_is_refused(qfs):
    code, *_ = _run(qfs, 3, [(0, 1), (1, 2)], 4, 1, 603, wait_limit=0)
    assert code == qfs.QFS_EINVAL


@pytest.mark.parametrize("n, S", [(8, 8), (12, 32)])
def test_both_whole_sweep_forms_time_out(qfs, n, S):
    """QFS_OPT_WAIT_LIMIT = 1: the cluster sweep (8 qubits) and the dataflow sweep (12
    qubits, 32 starts) return QFS_ETIMEOUT and leave the context usable."""
    p = w.brick_n12(target_seed=7) if n == 12 else w.brick_n8(target_seed=7)
    prm = qfs.default_params(M=p.M, multistarts=S, max_sweeps=2, dist_tol=1e-30, precision=qfs.QFS_MIXED)
    Psi, G = p.samples(), p.init_gates()[:S]
    with qfs.Context(0) as c:
        want = c.instantiate(p.n, p.pairs, p.U, prm, Psi, G)
        c.set_option(qfs.QFS_OPT_WAIT_LIMIT, 1)
        with pytest.raises(qfs.QfsError) as e:
            c.instantiate(p.n, p.pairs, p.U, prm, Psi, G)
        assert e.value.code == qfs.QFS_ETIMEOUT
        c.set_option(qfs.QFS_OPT_WAIT_LIMIT, 1 << 25)
        got = c.instantiate(p.n, p.pairs, p.U, prm, Psi, G)
    assert np.array_equal(got.gates, want.gates) and np.array_equal(got.start_costs, want.start_costs)
