"""Messages and codes of calls: a call that succeeds by a smaller plan leaves no
message behind."""
import pytest

from paper_2405_12866_gb300 import workloads as w

pytestmark = pytest.mark.gpu


def test_no_message_after_a_run_that_fell_back_to_smaller_buffers():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2405_12866_gb300 import build, qfs
    build.build()
    n, pairs = 9, w.brick_pairs(9, 3)
    U = w.target_unitary(w.haar_gates(41, w.STREAM_TARGET_GATES, len(pairs)), pairs, n)
    Psi, G = w.sample_states(42, n, 33), w.initial_gates(43, 3, len(pairs))
    lo, hi = 1 << 10, 1 << 28
    with qfs.Context(0) as c:
        while hi - lo > 256:  # to the smallest limit, where only the smallest plan fits
            mid = (lo + hi) // 2
            c.set_option(qfs.QFS_OPT_WORKSPACE_CAP, mid)
            try:
                c.sweep_once(n, pairs, U, Psi, G, qfs.QFS_MIXED)
                hi = mid
                assert qfs.lib().qfs_last_error() == b""
            except qfs.QfsError as e:
                assert e.code == qfs.QFS_ENOMEM
                lo = mid
