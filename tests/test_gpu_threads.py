"""Contexts of several host threads at once: each thread keeps its own, and a
call's launches must not depend on what another thread's calls set up.  What a
kernel may take of shared memory is a property of the function on the device,
shared by all threads; sizes that need different amounts run side by side here.

Answers are compared with those of the same arrays in a call that ran alone: the
same bits for a product and for an FP64 sweep.  A batch's cost is the cost of
the gates it came with, to 1e-9 (of costs near 1, formed in FP64)."""
import threading

import numpy as np
import pytest

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


def _together(work):
    """work: a list of functions; each runs in a thread of its own.  Their errors."""
    errors, start = [], threading.Barrier(len(work))

    def run(f):
        start.wait()
        try:
            f()
        except Exception as e:  # (reported by the test, not by the thread)
            errors.append(repr(e))
    threads = [threading.Thread(target=run, args=(f,)) for f in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors


def _target(n, seed, layers=2):
    pairs = w.brick_pairs(n, layers)
    return pairs, w.target_unitary(w.haar_gates(seed, w.STREAM_TARGET_GATES, len(pairs)), pairs, n)


def test_products_of_two_sizes_side_by_side(qfs):
    import torch
    lib, ctxs, work = qfs.lib(), [], []
    for n in (7, 8) * 4:
        U = torch.from_numpy(_target(n, 5)[1]).cuda()
        Psi = torch.from_numpy(w.sample_states(6, n, 8)).cuda()
        c = qfs.Context(0)
        ctxs.append(c)
        first = c.target_product(n, U, Psi, 0).clone()
        got = torch.empty_like(first)
        torch.cuda.synchronize()

        def loop(c=c, n=n, U=U, Psi=Psi, first=first, got=got):
            for i in range(3000):
                code = lib.qfs_target_product_dev(c._h, n, 8, U.data_ptr(), Psi.data_ptr(), 0, got.data_ptr())
                assert code == qfs.QFS_OK, f"n = {n}, call {i}: {lib.qfs_last_error().decode()}"
            assert torch.equal(got, first)
        work.append(loop)
    errors = _together(work)
    for c in ctxs:
        c.close()
    assert not errors, errors[0]


def test_sweeps_of_two_sizes_side_by_side(qfs):
    ctxs, work = [], []
    for n in (7, 8) * 3:
        pairs, U = _target(n, 5)
        both = [U, _target(n, 8)[1]]  # (in turn, so that a product left out leaves the other target's)
        Psi, G = w.sample_states(6, n, 8), w.initial_gates(7, 1, len(pairs))
        c = qfs.Context(0)
        ctxs.append(c)
        first = [c.sweep_once(n, pairs, u, Psi, G, qfs.QFS_FP64)[0] for u in both]

        def loop(c=c, n=n, pairs=pairs, both=both, Psi=Psi, G=G, first=first):
            for i in range(400):
                got = c.sweep_once(n, pairs, both[i % 2], Psi, G, qfs.QFS_FP64)[0]
                assert np.array_equal(got, first[i % 2]), f"n = {n}, call {i}: other gates"
        work.append(loop)
    errors = _together(work)
    for c in ctxs:
        c.close()
    assert not errors, errors[0]


def _cost(n, pairs, U, Psi, gates):
    return np.linalg.norm(U @ Psi - w.target_unitary(gates, pairs, n) @ Psi) ** 2 / Psi.shape[1]


def test_batches_of_two_sizes_side_by_side(qfs):
    ctxs, work = [], []
    for n, M in ((3, 4), (6, 16)) * 3:
        pairs, U = _target(n, 5)
        both = [U, _target(n, 8)[1]]
        Psi, G = w.sample_states(6, n, M), w.initial_gates(7, 2, len(pairs))
        c = qfs.Context(0)
        ctxs.append(c)
        prm = qfs.default_params(M=M, multistarts=2, max_sweeps=2, dist_tol=1e-30, refine_sweeps_max=0, precision=qfs.QFS_MIXED)

        def call(i, c=c, n=n, pairs=pairs, both=both, Psi=Psi, G=G, prm=prm):
            P, U = 1 + i % 7, both[i % 2]  # (seven shapes, so every call captures its launches anew)
            gates, info = c.instantiate_batch([(n, pairs, U)] * P, prm, [Psi] * P, [G] * P)
            for g, r in zip(gates, info):
                want = _cost(n, pairs, U, Psi, g)
                assert abs(r["cost"] - want) < 1e-9, f"n = {n}, call {i}: cost {r['cost']} of gates with {want}"
        for i in range(7):
            call(i)

        def loop(call=call):
            for i in range(100):
                call(i)
        work.append(loop)
    errors = _together(work)
    for c in ctxs:
        c.close()
    assert not errors, errors[0]
